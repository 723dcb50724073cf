"""What a many-steps launch does when it cannot run: runs in child processes,
because the switches in the environment are read once per process."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def child(out_path, stall=0):
    """200 steps of a 96 x 80 FP32 lattice with edges; saves the final state.
    stall: before them, a call that has to report LBM_ERR_CUDA."""
    import time

    from paper_2605_26677_gb300 import lbm
    from tests.cases import smooth_field

    nx, ny = 96, 80
    L = lbm.Lattice(nx, ny, c=5.0, omega=1.9, storage=lbm.LBM_STORE_F32)
    lbm.lbm_set_material(L.ctx, lbm.LBM_LAW_NH, [1.5, 0.75])
    for e in range(4):
        lbm.lbm_set_boundary(L.ctx, e, lbm.LBM_BC_VELOCITY if e == 0 else lbm.LBM_BC_TRACTION)
    status, secs = 0, 0.0
    if stall:
        lbm.lbm_init(L.ctx, smooth_field(nx, ny, seed=5, amp=0.02))
        t0 = time.time()
        try:
            lbm.lbm_step(L.ctx, 70)
        except lbm.LbmError as e:
            status = e.status
        secs = time.time() - t0
    lbm.lbm_init(L.ctx, smooth_field(nx, ny, seed=5, amp=0.02))
    lbm.lbm_step(L.ctx, 200)
    U, _, t = lbm.lbm_read_state(L.ctx)
    np.savez(out_path, U=U, t=t, step=lbm.lbm_info(L.ctx)[0], status=status, secs=secs)
    L.close()


def run(tmp_path, stall=0, **env):
    out = str(tmp_path / ("out%d.npz" % len(list(tmp_path.iterdir()))))
    code = "import sys; sys.path.insert(0, %r); import tests.test_gpu_multi_failures as m; m.child(%r, %d)" % (
        ROOT, out, stall)
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, **env), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    return dict(np.load(out))


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_26677_gb300 import build

    build.build()


@pytest.mark.parametrize("launch", ["1", "3"])
def test_refused_launch_falls_back_to_single_steps(tmp_path, launch):
    """CUDA refuses a grid that does not fit (here the first or the third of
    the four launches): the remaining steps are single launches."""
    ref, got = run(tmp_path), run(tmp_path, LBM_MULTI_REFUSE_TEST=launch)
    assert int(got["step"]) == 200 and float(got["t"]) == float(ref["t"])
    assert np.array_equal(got["U"].view(np.uint64), ref["U"].view(np.uint64))


@pytest.mark.parametrize("launch", ["1", "2"])
def test_wait_between_steps_runs_out(tmp_path, launch):
    """A barrier whose count starts one too low is never passed: each block
    gives up after a second, the launch ends, the call reports LBM_ERR_CUDA,
    and the context runs normally after the next initialization."""
    from paper_2605_26677_gb300 import lbm

    ref, got = run(tmp_path), run(tmp_path, stall=1, LBM_MULTI_STALL_TEST=launch)
    assert int(got["status"]) == lbm.LBM_ERR_CUDA
    assert 0.5 < float(got["secs"]) < 30.0
    assert np.array_equal(got["U"].view(np.uint64), ref["U"].view(np.uint64))
