"""lbm_steps_per_launch says which launches a call takes, and what lbm_profile
and lbm_step_variant therefore describe."""
import pytest

from tests.test_gpu_multi_steps import lbm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,storage,want", [(96, 80, 0, 64), (96, 80, 3, 64), (2048, 2048, 1, 2),
                                                (2048, 2048, 2, 1), (1024, 1024, 0, 1)])
def test_steps_per_launch(lbm, monkeypatch, nx, ny, storage, want):  # noqa: F811
    L = lbm.Lattice(nx, ny, c=6.0, omega=1.9, storage=storage)
    lbm.lbm_set_material(L.ctx, 1, [1.5, 0.75])
    assert lbm.lbm_steps_per_launch(L.ctx, 1000) == want
    assert lbm.lbm_steps_per_launch(L.ctx, 3) == min(want, 3)
    assert lbm.lbm_steps_per_launch(L.ctx, 1) == 1
    lbm.lbm_profile(L.ctx, True)
    assert lbm.lbm_steps_per_launch(L.ctx, 1000) == 1
    lbm.lbm_profile(L.ctx, False)
    monkeypatch.setenv("LBM_DYN", "0")
    lbm.lbm_set_material(L.ctx, 1, [1.5, 0.75])
    assert lbm.lbm_steps_per_launch(L.ctx, 1000) == 1
    with pytest.raises(lbm.LbmError):
        lbm.lbm_steps_per_launch(L.ctx, 0)
    L.close()


@pytest.mark.parametrize("storage,periodic,want", [(2, True, 1), (3, True, 1), (2, False, 2), (1, True, 2)])
def test_two_steps_of_a_16_bit_lattice(lbm, storage, periodic, want):  # noqa: F811
    L = lbm.Lattice(300, 300, c=6.0, omega=1.9, storage=storage)
    lbm.lbm_set_material(L.ctx, 1, [1.5, 0.75])
    if not periodic:
        for e in (0, 1):
            lbm.lbm_set_boundary(L.ctx, e, lbm.LBM_BC_VELOCITY)
    assert lbm.lbm_steps_per_launch(L.ctx, 2) == want
    assert lbm.lbm_steps_per_launch(L.ctx, 3) == 3
    L.close()
