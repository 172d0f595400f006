"""The finest level's sweep: the marching sweep's rule stands before a saved
choice (files of an earlier version hold choices timed against other kernels),
and the choice that a handle reports can be run on its level."""
import pytest

from paper_1410_8568_gb300 import gbmg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def solver(shape, bc):
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    rho = torch.exp(torch.rand(shape[::-1], dtype=torch.float64, device="cuda", generator=g))
    return gbmg.Solver(shape, bc, rho=rho)


@pytest.mark.parametrize("saved", [0, 1, 7])
def test_a_saved_choice_does_not_replace_the_rule(tmp_path, saved):
    shape, bc = (128, 128, 128), (1, 1, 0)
    gbmg.tune_cache_clear()
    with solver(shape, bc) as S:
        rule = S.tile_choice(gbmg.TILE_SWEEP, 0)
    assert gbmg.sweep_shape(rule)[2] > 0  # it marches
    src = tmp_path / "tune.txt"
    src.write_text("3 1 3 128 128 128 %d\n" % saved)
    gbmg.tune_cache_clear()
    assert gbmg.tune_cache_load(str(src)) == 1
    with solver(shape, bc) as S:
        assert S.tile_choice(gbmg.TILE_SWEEP, 0) == rule
        # below the march's sizes the saved choice is taken
    src.write_text("3 1 3 64 64 64 3\n")
    assert gbmg.tune_cache_load(str(src)) == 1
    with solver((64, 64, 64), bc) as S:
        assert S.tile_choice(gbmg.TILE_SWEEP, 0) == 3
    gbmg.tune_cache_clear()


@pytest.mark.parametrize("shape,bc", [((192, 160, 128), (1, 1, 0)), ((320, 128, 96), (0, 1, 0))])
def test_the_reported_choice_runs_on_its_level(shape, bc):
    gbmg.tune_cache_clear()
    with solver(shape, bc) as S:
        choice = S.tile_choice(gbmg.TILE_SWEEP, 0)
        assert gbmg.sweep_shape(choice)[2] > 0
        g = torch.Generator(device="cuda").manual_seed(7)
        x = torch.randn(shape[::-1], dtype=torch.float32, device="cuda", generator=g)
        b = torch.randn(shape[::-1], dtype=torch.float32, device="cuda", generator=g)
        want, work = x.clone(), torch.zeros_like(x)
        S.smooth(0, b, want, 2, prec=gbmg.MIXED)
        S.smooth_onepass(0, b, x, work, 2, prec=gbmg.MIXED, variant=choice)
        assert torch.equal(x, want)


def test_a_right_hand_side_at_an_odd_element():
    """The marching sweep copies quads of b: an unaligned one is refused by number, and
    the handle's choice runs a whole-row shape on it."""
    shape, bc = (192, 160, 128), (1, 1, 0)
    with solver(shape, bc) as S:
        g = torch.Generator(device="cuda").manual_seed(8)
        x = torch.randn(shape[::-1], dtype=torch.float32, device="cuda", generator=g)
        b = torch.empty(x.numel() + 1, dtype=torch.float32, device="cuda")[1:].view(x.shape)
        b.copy_(torch.randn(shape[::-1], dtype=torch.float32, device="cuda", generator=g))
        assert b.data_ptr() % 16 == 4
        want, work = x.clone(), torch.zeros_like(x)
        S.smooth(0, b, want, 2, prec=gbmg.MIXED)
        S.smooth_onepass(0, b, x, work, 2, prec=gbmg.MIXED, variant=0)
        assert torch.equal(x, want)
    shape = (256, 32, 16)
    with solver(shape, bc) as S:
        x = torch.zeros(shape[::-1], dtype=torch.float32, device="cuda")
        b = torch.zeros(x.numel() + 1, dtype=torch.float32, device="cuda")[1:].view(x.shape)
        for v in (7, 10):
            with pytest.raises(gbmg.MGError) as e:
                S.smooth_onepass(0, b, x, x.clone(), 1, prec=gbmg.MIXED, variant=v)
            assert e.value.code == gbmg.EINVAL
