"""What the compiler reports of the FP64 kernels of the laws with a logarithm:
no stack frame. A call inside them (a Newton solve of its own, say) brings one,
and the registers around it follow the calling convention: MR, Yeoh and Gent
steps took 8 to 15% longer, on every lattice."""
import concurrent.futures as cf
import os
import re
import subprocess

import pytest

from paper_2605_26677_gb300 import build

KERNELS = {"lbm_step_kernels.cuh": "template __global__ void k_step<double, %s, 2, true>(const StepArgs<double>);",
           "lbm_multi_kernels.cuh": "template __global__ void k_multi<double, %s>(const __grid_constant__ StepArgs<double>, "
                                    "const __grid_constant__ StepTimes<double>, int, unsigned *);"}
LAWS = ["LAW_LOGNH", "LAW_MR", "LAW_YEOH", "LAW_GENT"]


@pytest.mark.parametrize("header", sorted(KERNELS))
def test_fp64_kernels_have_no_stack_frame(tmp_path, header):
    if not os.path.exists(build._nvcc()):
        pytest.skip("nvcc not found")

    def frame(law):
        src = str(tmp_path / (law + ".cu"))
        with open(src, "w") as fh:
            fh.write('#include "%s"\nnamespace tlv {\n%s\n}\n' % (header, KERNELS[header] % law))
        r = subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-Xptxas", "-v", "-c", src, "-o", src + ".o"],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-3000:]
        return [int(n) for n in re.findall(r"(\d+) bytes stack frame", r.stderr)]

    with cf.ThreadPoolExecutor() as ex:
        for law, got in zip(LAWS, ex.map(frame, LAWS)):
            assert got and not any(got), (law, got)
