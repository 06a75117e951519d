"""The CUDA-core joint backward at the ends of its block shapes: a few rows, where most of a block's
threads only stage; the most rows that take 32 columns, and more rows, which take 16.  Gradient
against the FP64 oracle at the repository's gradient tolerance."""
import numpy as np
import pytest

import synth_signals as SS
from oracle import jtfs_oracle as O
from parity_checks import relative_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GTOL = 1e-3


@pytest.mark.parametrize("cfg,B", [
    (dict(N=512, J=4, Q=2, J_fr=2, Q_fr=1, T=16, F=1), 1),             # 9 rows
    (dict(N=512, J=4, Q=2, J_fr=2, Q_fr=1, T=16, F=1), 33),            # without the surplus threads
    (dict(N=2048, J=9, Q=42, J_fr=2, Q_fr=1, T=2048, F=8), 2),
    (dict(N=2048, J=9, Q=44, J_fr=2, Q_fr=1, T=2048, F=8), 2)])
def test_simt_gradient_rows(cfg, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_08269_gb300 import JTFSPlan, build
    build.build()
    plan = JTFSPlan(**cfg, precision="fp32_simt")
    op = O.Plan(O.Config(**cfg))
    sc = O.Schedule(op, 0)
    xs = SS.white_noise_batch(B, cfg["N"], 900)
    sh = plan.shapes
    rng = np.random.default_rng(sh.n1)
    g = [rng.standard_normal(f(B)).astype(np.float32) for f in (sh.s0, sh.s1, sh.s2)]
    out = plan.forward_backward(torch.from_numpy(xs).cuda(),
                                *[torch.from_numpy(v).cuda() for v in g])
    gref = O.backward_one(xs[B - 1].astype(np.float64), *[v[B - 1] for v in g], op, sc)
    assert relative_l2(out[3][B - 1].cpu().numpy(), gref) <= GTOL
