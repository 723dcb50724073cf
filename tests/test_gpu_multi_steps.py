"""Many steps of a small lattice in one launch: bit for bit the state that the
same number of lbm_step calls of one step each gives (those are launches of
the step kernel). Sizes: one node, one warp and a ragged second one, a row
longer than a block, more tasks than resident warps; step counts around the
64 steps of a launch; edges with profiles and time functions."""
import numpy as np
import pytest

from tests.cases import smooth_field

pytestmark = pytest.mark.gpu

PARAMS = {0: [1.5, 0.75], 1: [1.5, 0.75], 2: [1.5, 0.75], 3: [1.5, 0.25, 0.125], 4: [1.5, 0.375, 0.05, 0.01],
          5: [1.5, 0.75, 20.0]}


@pytest.fixture(scope="module")
def lbm():
    from paper_2605_26677_gb300 import build

    build.build()
    from paper_2605_26677_gb300 import lbm as m

    return m


def bits(lbm, L):
    U, P, t = lbm.lbm_read_state(L.ctx)
    return [x.view(np.uint64) for x in (U, P, lbm.lbm_read_displacement(L.ctx))] + [np.array([t])]


def compare(lbm, nx, ny, storage, law, edges, steps, b=(0.0, 0.0)):
    U0 = smooth_field(nx, ny, seed=nx + ny, amp=0.03, periodic=edges == "pppp")
    res = []
    for chunks in (steps, [1] * sum(steps)):
        L = lbm.Lattice(nx, ny, c=6.0, omega=1.9, storage=storage)
        lbm.lbm_set_material(L.ctx, law, PARAMS[law])
        lbm.lbm_set_body_force(L.ctx, *b)
        for e, k in enumerate(edges):
            n = ny if e < 2 else nx
            if k == "v":
                lbm.lbm_set_boundary(L.ctx, e, lbm.LBM_BC_VELOCITY, (0.003, -0.002), lbm.LBM_T_SIN_PULSE, (9.0,))
            if k == "t":
                lbm.lbm_set_boundary(L.ctx, e, lbm.LBM_BC_TRACTION, (0.02, 0.01), lbm.LBM_T_SIN2_RAMP, (15.0,),
                                     np.linspace(0.5, 1.5, n) if e & 1 else None)
        lbm.lbm_init(L.ctx, U0)
        for n in chunks:
            lbm.lbm_step(L.ctx, n)
        res.append(bits(lbm, L))
        L.close()
    for x, y in zip(*res):
        assert np.all(np.isfinite(x.view(np.float64)))
        assert np.array_equal(x, y)


@pytest.mark.parametrize("storage", [0, 1, 2, 3])
@pytest.mark.parametrize("nx,ny,edges", [(1, 1, "pppp"), (3, 3, "vttt"), (33, 5, "ppvt"), (64, 64, "pppp"),
                                         (257, 130, "tvtv")])
def test_many_steps_equal_single_steps(lbm, storage, nx, ny, edges):
    compare(lbm, nx, ny, storage, 1, edges, [67, 2, 64, 1], b=(1e-5, -2e-5))


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("law", [0, 2, 3, 4, 5])
def test_every_closure(lbm, storage, law):
    compare(lbm, 150, 70, storage, law, "vttt", [30])


@pytest.mark.parametrize("nx,ny", [(1030, 700), (64, 9000)])
def test_more_tasks_than_resident_warps(lbm, nx, ny):
    compare(lbm, nx, ny, 1, 1, "vttt", [9])


def test_status_is_latched(lbm):
    """A step of a many-steps launch that reaches J <= 0 reports it."""
    U0 = smooth_field(40, 30, seed=2, amp=0.01)
    U0[0] += 4.0 * np.sin(2 * np.pi * np.arange(40) / 40)[None, :]
    L = lbm.Lattice(40, 30, c=6.0, omega=1.9, storage=1)
    lbm.lbm_set_material(L.ctx, 1, PARAMS[1])
    lbm.lbm_init(L.ctx, U0)
    with pytest.raises(lbm.LbmError) as e:
        lbm.lbm_step(L.ctx, 60)
    assert e.value.status in (lbm.LBM_ERR_NONPOSITIVE_J, lbm.LBM_ERR_NONFINITE)
    L.close()
