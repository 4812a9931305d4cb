"""The fixed-point exponential of the LavaMD pair loop (csrc/exp_fixed.cuh): a
checker compiled from tests/cuda/exp_fixed_check.cu compares it with the host's
long-double expl, and the forces are compared with the oracle for scales that
take its range test to the library's exponential."""
import os
import subprocess
import tempfile

import numpy as np
import pytest

from paper_2308_16877_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2308_16877_gb300", "csrc")


def test_fixed_point_exp_accuracy():
    from paper_2308_16877_gb300 import build
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "exp_fixed_check")
        subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-I", CSRC, "-o", exe,
                        os.path.join(HERE, "cuda", "exp_fixed_check.cu")], check=True)
        r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("a2", [0.0, 1e-12, 0.5, 37.5, 600.0, 9000.0])
@pytest.mark.parametrize("B,NP", [(2, 37), (3, 300)])
def test_forces_over_scales(orc, a2, B, NP):
    """Each exponential is within |u| 2^-53 (the oracle rounds u = -a2 r2) of
    the other side's, |u| <= 745 where it is not 0: 1e-13 of a term, below
    1e-12 of the particle's potential in all."""
    from paper_2308_16877_gb300 import hpac as H
    rq = W.lavamd_inputs(B, NP, seed=int(a2) + NP)
    rq[:3, ::7] *= 40.0      # some pairs far apart
    fv = H.lavamd(torch.from_numpy(rq).cuda(), B, NP, a2).cpu().numpy()
    ofv = orc.lavamd(B, NP, a2, rq)[0]
    err = np.abs(fv - ofv)
    # a force sums q v d with |d| up to 62 here, against a potential of q v
    assert np.all(err[0] <= 1e-12 * np.abs(ofv[0]))
    assert np.all(err[1:] <= 1e-12 * 2 * 62 * np.abs(ofv[0]))
