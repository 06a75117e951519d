"""The CUDA-core joint backward where its thread tiles and column tiles change: row counts that
are and are not multiples of 8, rates whose first row is not 0, one to 64 frames, Eq. 4 outputs,
columns short of a tile, and a row and frame count that needs the 16-column form.  Gradient
against the FP64 oracle at the repository's gradient tolerance."""
import numpy as np
import pytest

import synth_signals as SS
from oracle import jtfs_oracle as O
from parity_checks import relative_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GTOL = 1e-3


@pytest.mark.parametrize("cfg", [
    dict(N=256, J=4, Q=3, J_fr=2, Q_fr=2, T=16, F=3),
    dict(N=512, J=5, Q=4, J_fr=3, Q_fr=1, T=8, F=4),                         # 64 frames
    dict(N=1024, J=6, Q=2, J_fr=2, Q_fr=1, T=1024, F=1),                     # one frame
    dict(N=1024, J=6, Q=16, J_fr=3, Q_fr=2, T=64, F=16, average_fr=False),
    dict(N=2048, J=8, Q=40, J_fr=2, Q_fr=1, T=64, F=8)])                     # 16 columns
def test_simt_gradient(cfg):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_08269_gb300 import JTFSPlan, build
    build.build()
    plan = JTFSPlan(**cfg, precision="fp32_simt")
    op = O.Plan(O.Config(**cfg))
    sc = O.Schedule(op, 0)
    xs = SS.white_noise_batch(2, cfg["N"], 800)
    sh = plan.shapes
    rng = np.random.default_rng(cfg["N"])
    g = [rng.standard_normal(f(2)).astype(np.float32) for f in (sh.s0, sh.s1, sh.s2)]
    out = plan.forward_backward(torch.from_numpy(xs).cuda(),
                                *[torch.from_numpy(v).cuda() for v in g])
    gref = O.backward_one(xs[1].astype(np.float64), *[v[1] for v in g], op, sc)
    assert relative_l2(out[3][1].cpu().numpy(), gref) <= GTOL
