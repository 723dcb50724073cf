"""Two steps of a large FP32 lattice in one pass: bit for bit the state that the
same number of lbm_step calls of one step each gives (those are launches of
the step kernel). Widths around the 120 columns of a strip and below the 8
lanes' worth of a warp, the narrowest and lowest lattices it takes, every
kind of edge, odd step counts, profiles and time functions on the edges."""
import numpy as np
import pytest

from tests.test_gpu_multi_steps import compare, lbm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,edges", [(8, 140000, "vttt"), (45000, 24, "vttt"), (140000, 8, "vvpp"),
                                         (101, 11001, "pppp"),
                                         (119, 9001, "ppvt"), (120, 9001, "tvpp"), (121, 9001, "vttt"),
                                         (122, 9001, "pppp"), (1199, 1001, "pppp"), (1200, 999, "vtpp"),
                                         (1201, 1001, "tttv"), (1322, 1000, "ppvt")])
def test_pairs_equal_single_steps(lbm, nx, ny, edges):  # noqa: F811
    compare(lbm, nx, ny, 1, 1, edges, [2, 5], b=(1e-5, -2e-5))


@pytest.mark.parametrize("law", [0, 2, 3, 4, 5])
def test_every_closure(lbm, law):  # noqa: F811
    compare(lbm, 1100, 1003, 1, law, "vttt", [6])


def test_asynchronous_steps_and_checkpoint(lbm):  # noqa: F811
    """lbm_step_async takes the same path; a checkpoint between pairs resumes."""
    nx, ny = 1030, 1021
    U0 = np.zeros((6, ny, nx))
    U0[2] = U0[5] = 1.0
    U0[0] = 0.02 * np.sin(2 * np.pi * np.arange(nx) / nx)[None, :]
    res = []
    for cut in (False, True):
        L = lbm.Lattice(nx, ny, c=6.0, omega=1.9, storage=1)
        lbm.lbm_set_material(L.ctx, 1, [1.5, 0.75])
        lbm.lbm_init(L.ctx, U0)
        lbm.lbm_step_async(L.ctx, 4)
        if cut:
            buf = lbm.lbm_save(L.ctx)
            lbm.lbm_step(L.ctx, 3)
            lbm.lbm_load(L.ctx, buf)
        lbm.lbm_step(L.ctx, 4)
        res.append(lbm.lbm_read_state(L.ctx)[0].view(np.uint64))
        L.close()
    assert np.array_equal(*res)


@pytest.mark.parametrize("nx,ny,storage", [(96, 80, 0), (1300, 900, 1)])
def test_captured_steps_can_be_replayed(lbm, nx, ny, storage):  # noqa: F811
    """A graph of two steps replayed three times makes six steps."""
    import torch

    U0 = np.zeros((6, ny, nx))
    U0[2] = U0[5] = 1.0
    U0[0] = 0.02 * np.sin(2 * np.pi * np.arange(nx) / nx)[None, :]
    res = []
    for graph in (False, True):
        s = torch.cuda.Stream()
        L = lbm.Lattice(nx, ny, c=6.0, omega=1.9, storage=storage, stream=s)
        lbm.lbm_set_material(L.ctx, 1, [1.5, 0.75])
        lbm.lbm_init(L.ctx, U0)
        lbm.lbm_step_async(L.ctx, 1)
        lbm.lbm_sync(L.ctx)
        if graph:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                lbm.lbm_step_async(L.ctx, 2)
            with torch.cuda.stream(s):
                for _ in range(3):
                    g.replay()
        else:
            lbm.lbm_step(L.ctx, 6)
        lbm.lbm_sync(L.ctx)
        res.append(lbm.lbm_read_state(L.ctx)[0].view(np.uint64))
        L.close()
    assert np.array_equal(*res)
