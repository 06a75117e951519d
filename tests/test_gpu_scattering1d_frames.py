"""Time scattering over the frame counts and row lengths where its pooling kernels change form:
one, two, four and eight or more frames, rows with fewer and more than 32 samples per frame,
rows shared by several warps, and more frames than the shared-row form takes.  Outputs and
gradient against the FP64 oracle, at the tolerances of the other time-scattering tests."""
import numpy as np
import pytest

import synth_signals as SS
from oracle import jtfs_oracle as O
from parity_checks import relative_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL, GTOL = 1e-4, 1e-3


@pytest.mark.parametrize("N,J,T", [
    (1024, 5, 1024), (1024, 5, 512), (1024, 5, 256), (1024, 5, 128), (1024, 5, 8),
    (2 ** 14, 9, 2 ** 11), (2 ** 14, 9, 2 ** 9), (2 ** 15, 9, 2 ** 9)])
def test_time_scattering_frames(N, J, T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_08269_gb300 import JTFSPlan, build
    build.build()
    cfg = dict(N=N, J=J, Q=4, J_fr=2, Q_fr=1, T=T, F=4)
    plan = JTFSPlan(**cfg, precision="fp32_simt")
    op = O.Plan(O.Config(**cfg))
    sc = O.Schedule(op, 0)
    xs = SS.white_noise_batch(2, N, 700)
    x = torch.from_numpy(xs).cuda()
    s0, s1, s2t, u1 = plan.scattering1d(x)
    rng = np.random.default_rng(T)
    g = [rng.standard_normal(tuple(t.shape)).astype(np.float32) for t in (s0, s1, s2t)]
    gx = plan.scattering1d_backward(x, u1, *[torch.from_numpy(v).cuda() for v in g]).cpu().numpy()
    ref = O.scattering1d_one(xs[1].astype(np.float64), op, sc)
    for got, name in ((s0, "S0"), (s1, "S1"), (s2t, "S2t")):
        assert relative_l2(got[1].cpu().numpy(), ref[name]) <= TOL, name
    gref = O.scattering1d_backward_one(xs[1].astype(np.float64), *[v[1] for v in g], op, sc)
    assert relative_l2(gx[1], gref) <= GTOL
