"""The 64-frame (channel-row) contraction forward with its rates in parts: batches of up to 48
signals walk this configuration's rates in two parts on 152 SMs, 64 signals whole.  The split walk
against the FP64 oracle and against the whole one, whose sums differ in order alone."""
import numpy as np
import pytest

import synth_signals as SS
from oracle import jtfs_oracle as O
from parity_checks import check_orders

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CFG = dict(N=2 ** 12, J=6, Q=8, J_fr=3, Q_fr=1, T=2 ** 6, F=8)
TOL = {"fp32": 1e-4, "bf16": 2e-2}
WHOLE = 64


@pytest.mark.parametrize("precision", list(TOL))
def test_split_rates_64_frames(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_08269_gb300 import JTFSPlan, build
    build.build()
    plan = JTFSPlan(precision=precision, **CFG)
    xs = SS.white_noise_batch(WHOLE, CFG["N"], 902)
    x = torch.from_numpy(xs).cuda()
    whole = [t.clone() for t in plan.forward(x)[:3]]
    plan.sync()
    op = O.Plan(O.Config(**CFG))
    ref = O.forward_one(xs[0].astype(np.float64), op, O.Schedule(op, 0))
    # S2 sums non-negative terms: re-ordering moves an element by at most its additions times 2^-23,
    # 4 per 16 samples of at most 2^12
    tol = 2 ** 12 / 16 * 4 * 2 ** -23
    for B in (1, 5, 40):
        s0, s1, s2 = plan.forward(x[:B].contiguous())[:3]
        plan.sync()
        got = {"S0": s0[0].cpu().numpy(), "S1": s1[0].cpu().numpy(),
               "S2": s2[0].cpu().numpy().reshape(ref["S2"].shape)}
        check_orders(got, ref, TOL[precision], B)
        assert ((s2 - whole[2][:B]).abs() <= tol * whole[2][:B].abs()).all()
        # another order of sums, so not the same bits throughout: the parts were taken
        assert not torch.equal(s2, whole[2][:B])
