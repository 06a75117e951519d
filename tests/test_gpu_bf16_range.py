"""BF16 forward of quiet signals: BF16 has the exponent range of FP32, so a signal scaled by 2^-60
has its coefficients scaled by 2^-60, although most |Z|^2 are then below the smallest normal FP32
number (their own rounding, 2^-150, is within a thousandth of them down to |Z| = 1e-21).  Against
the FP64 oracle of the unscaled signal at the repository's BF16 tolerance; the loud signal of each
batch and the silent one keep theirs."""
import numpy as np
import pytest

import synth_signals as SS
from oracle import jtfs_oracle as O
from parity_checks import check_orders

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 2e-2
SCALE = 2.0 ** -60


@pytest.mark.parametrize("cfg", [
    dict(N=2 ** 12, J=6, Q=8, J_fr=3, Q_fr=1, T=2 ** 8, F=8),       # 16 frames
    dict(N=2 ** 12, J=6, Q=8, J_fr=3, Q_fr=1, T=2 ** 7, F=8)])      # 32 frames
def test_bf16_quiet_signals(cfg):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_08269_gb300 import JTFSPlan, build
    build.build()
    plan = JTFSPlan(**cfg, precision="bf16")
    op = O.Plan(O.Config(**cfg))
    sc = O.Schedule(op, 0)
    x = SS.white_noise_batch(1, cfg["N"], 901)[0]
    scales = [1.0, SCALE, 0.0]
    batch = np.stack([x * np.float32(s) for s in scales])
    out = plan.forward(torch.from_numpy(batch).cuda())
    plan.sync()
    s0, s1, s2 = (t.cpu().numpy().astype(np.float64) for t in out[:3])
    ref = O.forward_one(x.astype(np.float64), op, sc)
    for b, s in enumerate(scales[:2]):
        check_orders({"S0": s0[b] / s, "S1": s1[b] / s, "S2": s2[b].reshape(ref["S2"].shape) / s},
                     ref, TOL, s)
    assert not s2[2].any()
