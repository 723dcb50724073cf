"""Which lattices the two-step kernel takes, and that every route gives the
bits of single steps: forced wherever it can run (LBM_PAIR=1), chosen by the
comparison inside the first long call, and after a change of the edges."""
import numpy as np
import pytest

from tests.cases import smooth_field
from tests.test_gpu_multi_steps import PARAMS, bits, compare, lbm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,edges,law", [(8, 140000, "vttt", 1), (45000, 24, "vttt", 1), (140000, 8, "vvpp", 1),
                                             (60, 20000, "pppp", 1), (101, 11001, "ppvt", 1), (121, 9001, "tvpp", 1),
                                             (1100, 1003, "vttt", 0), (1100, 1003, "vttt", 2), (1100, 1003, "vttt", 3),
                                             (1100, 1003, "vttt", 4), (1100, 1003, "vttt", 5), (2049, 1025, "vttt", 5),
                                             (613, 4894, "vttt", 1), (725, 5794, "vttt", 4), (6929, 217, "vvvv", 1)])
def test_forced_pairs_equal_single_steps(lbm, monkeypatch, nx, ny, edges, law):  # noqa: F811
    monkeypatch.setenv("LBM_PAIR", "1")
    compare(lbm, nx, ny, 1, law, edges, [2, 5], b=(1e-5, -2e-5))


def lattice(lbm, nx, ny, law, edges, edges_first=False):  # noqa: F811
    L = lbm.Lattice(nx, ny, c=6.0, omega=1.9, storage=1)
    if not edges_first:
        lbm.lbm_set_material(L.ctx, law, PARAMS[law])
    for e, k in enumerate(edges):
        if k != "p":
            lbm.lbm_set_boundary(L.ctx, e, lbm.LBM_BC_VELOCITY if k == "v" else lbm.LBM_BC_TRACTION, (0.002, -0.001))
    if edges_first:
        lbm.lbm_set_material(L.ctx, law, PARAMS[law])
    return L


@pytest.mark.parametrize("nx,ny,law,edges,want", [(1100, 1003, 1, "vvpp", 2), (1100, 1003, 1, "ppvt", 1),
                                                  (1100, 1003, 2, "vttt", 1), (9000, 130, 3, "vttt", 1),
                                                  (53, 46980, 2, "pppp", 1), (4096, 2048, 1, "vttt", 2)])
def test_choice_in_either_order_of_the_calls(lbm, nx, ny, law, edges, want):  # noqa: F811
    for first in (False, True):
        L = lattice(lbm, nx, ny, law, edges, first)
        assert lbm.lbm_steps_per_launch(L.ctx, 40) == want, first
        L.close()


@pytest.mark.parametrize("nx,ny,law,edges", [(1100, 1003, 5, "vttt"), (130, 9000, 1, "vvpp"), (300, 4000, 3, "ppvt")])
@pytest.mark.parametrize("steps", [[3, 11, 4], [45, 2]])
def test_comparison_and_changed_edges(lbm, monkeypatch, nx, ny, law, edges, steps):  # noqa: F811
    """The first call of 10 steps or more compares the kernels on its own
    steps; then another kind of edge, another comparison."""
    U0 = smooth_field(nx, ny, seed=7, amp=0.02, periodic=edges == "pppp")
    res = []
    for env in (None, "0"):
        if env:
            monkeypatch.setenv("LBM_PAIR", env)
        L = lattice(lbm, nx, ny, law, edges)
        lbm.lbm_init(L.ctx, U0)
        for n in steps:
            lbm.lbm_step(L.ctx, n)
        if edges[2] != "p":
            lbm.lbm_set_boundary(L.ctx, 3, lbm.LBM_BC_VELOCITY, (0.001, 0.0))
        for n in steps:
            lbm.lbm_step(L.ctx, n)
        assert lbm.lbm_info(L.ctx)[0] == 2 * sum(steps)
        res.append(bits(lbm, L))
        L.close()
    for x, y in zip(*res):
        assert np.all(np.isfinite(x.view(np.float64)))
        assert np.array_equal(x, y)
