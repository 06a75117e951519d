"""The CUDA-core joint backward where one spin is far weaker than the other: gZ = g Z / |Z| weighs
a weak Z like any other, so Z has to be summed with rounding errors of its own size and not of the
strong spin's.  The scalogram handed to the backward holds one modulation, whose phase along
lambda matches one wavelet's spin, and 2^-10 of its mirror image; the cotangent lies on the weak
spin alone.  Y has rounding errors of its own: the error that FP32 rounding of Y makes in the gradient is
computed in 64 bits, and twice that is allowed (an FFT leaves about four roundings in a sample, and
independent ones add in squares), plus 16 units of FP32 rounding (1e-6) for the stages after gZ."""
import numpy as np
import pytest

from oracle import jtfs_oracle as O
from parity_checks import relative_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CFG = dict(N=2 ** 15, J=12, Q=16, J_fr=5, Q_fr=1, T=2 ** 14, F=1, average_fr=False)
WEAK = 2.0 ** -10


@pytest.mark.parametrize("beta", [2, 3, 4])
def test_weak_spin_gradient(beta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_08269_gb300 import JTFSPlan, build
    build.build()
    op = O.Plan(O.Config(**CFG))
    sc = O.Schedule(op, 0)
    ops = O.Operators(op, sc)
    rng = np.random.default_rng(beta)
    x = rng.standard_normal(op.N).astype(np.float32)
    a = op.n2 - 2
    lm, sa = int(sc.lam_min[a]), int(sc.s2[a])
    u1 = []
    for lam in range(op.n1):
        L = int(sc.L1[lam])
        t = 2 * np.pi * round(op.xi2[a] * op.N) / L * np.arange(L)
        phi = 2 * np.pi * op.xi_fr[beta] * lam
        u1.append((2 + np.cos(t + phi) + WEAK * np.cos(t - phi)).astype(np.float32))
    Y = np.zeros((op.n1, int(sc.L2[a])), dtype=np.complex128)
    for lam in range(lm, op.n1):
        Y[lam] = ops.psi2(u1[lam].astype(np.float64), lam, a)
    c = min((beta, beta + op.n_fr), key=lambda q: np.abs(ops.wfr(Y, q, lm)).mean())
    g = np.zeros((op.n2, op.C, op.n_lam_out, op.n_t), dtype=np.float32)
    g[a, c] = 1 + rng.random((op.n_lam_out, op.n_t))
    g_abs = ops.pool_T_T(ops.pool_F_T(g[a, c].astype(np.float64)), sa)
    phase = O._safe_phase(ops.wfr(Y, c, lm))
    rounded = O._safe_phase(ops.wfr(Y.astype(np.complex64).astype(np.complex128), c, lm))
    tol = 2 * np.linalg.norm(g_abs * (rounded - phase)) / np.linalg.norm(g_abs) + 1e-6
    gY = ops.wfr_T(g_abs * phase, c, lm)
    xh = ops.x_hat(x.astype(np.float64))
    g_xh = sum(ops.psi1_T(ops.psi2_T(gY[lam - lm], lam, a) * O._safe_phase(ops.psi1(xh, lam)), lam)
               for lam in range(lm, op.n1))
    plan = JTFSPlan(**CFG, precision="fp32_simt")
    gx = plan.backward(torch.from_numpy(x).cuda()[None],
                       torch.from_numpy(np.concatenate(u1)).cuda()[None].contiguous(), None, None,
                       torch.from_numpy(g).cuda()[None].contiguous())
    plan.sync()
    assert relative_l2(gx[0].cpu().numpy(), ops.x_hat_T(g_xh)) <= tol
