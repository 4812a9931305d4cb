"""The fixed-point exponential of the LavaMD pair loop (csrc/exp_fixed.cuh): a
program compiled from tests/cuda/exp_fixed_check.cu compares it with the host's
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


@pytest.mark.parametrize("a2", [3e291, 1e300, 1e305, 1.7e308])
def test_own_term_at_the_largest_scales(a2):
    """At scales this large every pair but a particle's own (r2 = 0) underflows:
    the potential is the particle's charge and the force is zero, exactly."""
    from paper_2308_16877_gb300 import hpac as H
    rq = W.lavamd_inputs(2, 37, seed=9)
    fv = H.lavamd(torch.from_numpy(rq).cuda(), 2, 37, a2).cpu().numpy()
    assert np.array_equal(fv[0], rq[3]) and not fv[1:].any()


@pytest.mark.parametrize("kind", ["tied", "signs", "tiny", "large", "outlier", "nan"])
@pytest.mark.parametrize("tech", [0, 1])
def test_forces_on_and_off_the_grid(orc, kind, tech):
    """The pair loop's fixed-point grid: positions tied to their boxes, mixed
    signs with zeros and binade edges, very small and large coordinates (with
    a2 to match), one particle far outside (its box and its neighbours' steps
    take FP64) and one NaN. TAF at an infinite threshold predicts by window
    counts alone, so steps without computing threads lie between the others.
    The bound is that of test_forces_over_scales."""
    from paper_2308_16877_gb300 import hpac as H
    B, NP, a2 = 3, 45, 0.5
    P = B ** 3 * NP
    rq = W.lavamd_inputs(B, NP, seed=77)
    g = np.random.default_rng(5)
    if kind == "tied":
        box = np.arange(P) // NP
        rq[0] += box % B
        rq[1] += box // B % B
        rq[2] += box // (B * B)
    elif kind == "signs":
        rq[:3] = g.uniform(-1.0, 1.0, (3, P))
        edge = np.array([0.0, -0.0, 0.5, -0.5, 1.0, -1.0, 2.0 ** -30, 5e-324, np.nextafter(1.0, 0.0)])
        rq[:3, ::5] = g.choice(edge, (3, rq[:, ::5].shape[1]))
    elif kind == "tiny":
        rq[:3] *= 2.0 ** -300
        a2 = 0.5 * 2.0 ** 600
    elif kind == "large":
        rq[:3] *= 2.0 ** 200
        a2 = 0.5 * 2.0 ** -400
    elif kind == "outlier":
        rq[1, 13 * NP + 7] = 1e3
        rq[0, 2 * NP + 3] = -6.0
    else:
        rq[2, 26 * NP + 1] = np.nan
    kw = dict(technique=1, level=2, hsize=2, psize=3, thresh=float("inf")) if tech else {}
    fv = H.lavamd(torch.from_numpy(rq).cuda(), B, NP, a2, **kw).cpu().numpy()
    okw = dict(technique=1, level=2, hsize=2, psize=3, thresh=float("inf")) if tech else {}
    ofv = orc.lavamd(B, NP, a2, rq, **okw)[0]
    bad = np.isnan(ofv)
    assert np.array_equal(np.isnan(fv), bad) and (bad.any() == (kind == "nan"))
    reach = 2.0 * np.nanmax(np.abs(rq[:3]))
    err = np.where(bad, 0.0, np.abs(fv - ofv))
    pot = np.where(bad[0], 1.0, np.abs(ofv[0]))
    assert np.all(err[0] <= 1e-12 * pot)
    assert np.all(err[1:] <= 1e-12 * 2 * reach * pot)
