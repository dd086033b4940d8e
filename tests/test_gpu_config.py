"""Launch configurations: what a grid or batch reports can be set again and is
what runs."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_09713_gb300 import build

    build.build()
    from paper_1709_09713_gb300 import sbli

    sbli.lib()
    return sbli


# 128^3 lies above the planes a CTA slot from which fused grids take the TMEM queue
@pytest.mark.parametrize("n", [24, 128])
@pytest.mark.parametrize("variant,precision", [("SBLI_FUSED", 0), ("SBLI_FUSED", 1), ("SBLI_FUSED", 2), ("SBLI_FUSED", 3),
                                               ("SBLI_STORE_ALL", 0), ("SBLI_STORE_ALL", 1), ("SBLI_RS", 0),
                                               ("SBLI_SS", 0), ("SBLI_RA", 0), ("SBLI_SN", 0), ("SBLI_SN2", 0)])
def test_reported_config_can_be_set(S, variant, precision, n):
    g = S.Grid(n, precision, getattr(S, variant))
    cfg = g.config()
    g.set_config(*cfg)
    assert g.config() == cfg
    g.close()


def test_configured_planes_are_launched(S):
    """The kinetic energy shows which planes a CTA sums: 2 at x2 = 0 and 2^-53 at
    x2 = 4, 5, 6 of one column.  CTAs of four planes form 3 x 2^-53 first, which moves
    the total by a unit in the last place; singly each would be lost."""
    n = (32, 32, 32)
    q = torch.zeros((5, n[2], n[1], n[0]), dtype=torch.float64)
    q[0], q[4] = 1.0, 200.0
    q[1, 0, 0, 0] = 2.0
    q[1, 4:7, 0, 0] = 2.0**-26
    for precision in (S.SBLI_FP32, S.SBLI_FP32_DF):
        g = S.Grid(n, precision)
        start = g.config()
        for cfg in ((8, 4, 0, 1), (8, 4, 1, 1)):  # one of them the grid's own default, of fewer planes
            g.set_config(*cfg)
            g.set_state(q)
            assert g.step_n_history(1, 1e-6)[0, 0].item() == (2.0 + 2.0**-51) / 32**3, (start, cfg)
        g.close()


@pytest.mark.parametrize("precision", [1, 2])
def test_batch_keeps_its_own_planes(S, precision):
    """A batch too small for 32 planes an item: setting the z-queue mode alone, and
    a tuned batch set back to what it reported, launch what they did."""
    sizes = [(64, 64, 64), (48, 40, 64)]
    b = S.Batch(sizes, precision)
    own = b.work_items()
    assert own > sum(-(-n[0] // 32) * -(-n[1] // 8) * 2 for n in sizes)  # more than items of 32 planes
    zq, planes = b.schedule()
    b.set_schedule(zq)
    assert b.work_items() == own and b.schedule() == (zq, planes)
    b.set_schedule(1 - zq)
    b.set_schedule(zq)
    assert b.work_items() == own
    b.set_schedule(zq, [32, 32])  # set: 32 planes are 32 planes
    items = b.work_items()
    assert items < own
    b.set_schedule(zq)
    assert b.work_items() == items
    b.close()


@pytest.mark.parametrize("precision", [0, 3])
def test_even_batch_reports_what_it_launches(S, precision):
    """Binary64-register members: work items are planes of 16 x 8 tiles, and the
    planes per item, which nothing launches, stay as they are through a tuning."""
    sizes = [(40, 17, 61), (33, 9, 7), (64, 64, 64)]
    b = S.Batch(sizes, precision)
    assert b.work_items() == sum(-(-n[0] // 16) * -(-n[1] // 8) * n[2] for n in sizes)
    planes = b.schedule()[1]
    b.init_tgv()
    zq, ms = b.autotune(1)
    assert b.schedule() == (zq, planes) and ms > 0
    b.close()
