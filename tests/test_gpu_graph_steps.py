"""Captured work replayed between direct calls. A graph holds the address of
the buffer that the state lay in when it was captured, so every call of an
even number of steps has to leave the state in the buffer it took it from,
and the counters of a dynamic task order as it found them."""
import numpy as np
import pytest

from tests.test_gpu_multi_steps import lbm  # noqa: F401

pytestmark = pytest.mark.gpu


def start(lbm, L):  # noqa: F811
    nx, ny = L.nx, L.ny
    U0 = np.zeros((6, ny, nx))
    U0[2] = U0[5] = 1.0
    U0[0] = 0.02 * np.sin(2 * np.pi * np.arange(nx) / nx)[None, :] * np.cos(2 * np.pi * np.arange(ny) / ny)[:, None]
    lbm.lbm_set_material(L.ctx, 1, [1.5, 0.75])
    lbm.lbm_init(L.ctx, U0)


@pytest.mark.parametrize("nx,ny,storage,dynamic", [(96, 80, 0, "0"), (1300, 900, 1, "0"), (1300, 900, 1, "1")])
def test_direct_steps_between_replays(lbm, monkeypatch, nx, ny, storage, dynamic):  # noqa: F811
    """A graph of two steps, replayed before and after direct calls of 2, 6
    and 4 steps (1 + 2 + 2 + 2 + 6 + 2 + 4 + 2 steps)."""
    import torch

    res = []
    for graph in (False, True):
        s = torch.cuda.Stream()
        # the variable at lbm_create sets the task order; without it at
        # lbm_set_material the steps may go several to a launch
        monkeypatch.setenv("LBM_DYN", dynamic)
        L = lbm.Lattice(nx, ny, c=6.0, omega=1.9, storage=storage, stream=s)
        monkeypatch.delenv("LBM_DYN")
        start(lbm, L)
        lbm.lbm_step_async(L.ctx, 1)
        lbm.lbm_sync(L.ctx)
        if graph:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                lbm.lbm_step_async(L.ctx, 2)

        def two():
            if graph:
                with torch.cuda.stream(s):
                    g.replay()
            else:
                lbm.lbm_step(L.ctx, 2)

        two()
        two()
        for n in (2, 6, 4):
            lbm.lbm_step(L.ctx, n)
            two()
        lbm.lbm_sync(L.ctx)
        res.append(lbm.lbm_read_state(L.ctx)[0].view(np.uint64))
        L.close()
    assert np.array_equal(*res)


def test_captured_read_out_after_direct_steps(lbm):  # noqa: F811
    """A captured read-out, replayed after calls of an even number of steps,
    gives the present state."""
    import torch

    nx, ny = 1100, 1000
    s = torch.cuda.Stream()
    L = lbm.Lattice(nx, ny, c=6.0, omega=1.9, storage=1, stream=s)
    start(lbm, L)
    U = torch.zeros((6, ny, nx), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        lbm.lbm_read_state_device(L.ctx, U)
    for n in (2, 4, 6):
        lbm.lbm_step(L.ctx, n)
        with torch.cuda.stream(s):
            g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(U.cpu().numpy().view(np.uint64), lbm.lbm_read_state(L.ctx)[0].view(np.uint64))
    L.close()
