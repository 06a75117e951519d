"""Small batches split the contraction's longest rates (and the three-atom items of its backward)
over several CTAs; a batch that fills the GPU walks them whole.  Both must give the same signals'
outputs up to the order of FP32 sums."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# 16 and 32 frames (spin-pair forms; n1 = 151 and 87 rows), 64 frames (channel-row form), and rates
# past the tensor-core backward's rows (n1 = 167)
CONFIGS = {
    "16 frames": dict(N=2 ** 16, J=12, Q=16, J_fr=4, Q_fr=2, T=2 ** 12, F=16),
    "8 frames": dict(N=2 ** 15, J=12, Q=16, J_fr=4, Q_fr=2, T=2 ** 12, F=16),
    "32 frames": dict(N=2 ** 13, J=8, Q=16, J_fr=3, Q_fr=2, T=2 ** 8, F=16),
    "64 frames": dict(N=2 ** 12, J=6, Q=8, J_fr=3, Q_fr=1, T=2 ** 6, F=8),
    "n1 = 167": dict(N=2 ** 17, J=13, Q=16, J_fr=4, Q_fr=2, T=2 ** 13, F=16),
}


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("config", list(CONFIGS))
def test_small_batches_match_a_full_one(config, precision):
    from paper_2204_08269_gb300 import JTFSPlan
    plan = JTFSPlan(precision=precision, **CONFIGS[config])
    sh, many = plan.shapes, 40
    gen = torch.Generator(device="cuda").manual_seed(11)
    x = torch.randn(many, CONFIGS[config]["N"], device="cuda", generator=gen)
    g = [torch.randn(s, device="cuda", generator=gen) for s in (sh.s0(many), sh.s1(many), sh.s2(many))]
    full = [t.clone() for t in plan.forward_backward(x, *g)]
    # S2 sums non-negative terms: re-ordering moves an element by at most its additions times 2^-23,
    # 4 per 16 samples of at most 2^13; g_x likewise in norm, with 8 additions per 16 rows of W and
    # at most 2^11 rows
    tol_s, tol_g = 2 ** 13 / 16 * 4 * 2 ** -23, 2 ** 11 / 16 * 8 * 2 ** -23
    for B in (1, 2, 3, 5, 11):
        out = plan.forward_backward(x[:B].contiguous(), *[t[:B].contiguous() for t in g])
        plan.sync()
        for a, f in zip(out[:2], full[:2]):
            assert torch.equal(a, f[:B])
        assert ((out[2] - full[2][:B]).abs() <= tol_s * full[2][:B].abs()).all()
        assert (out[3] - full[3][:B]).norm() <= tol_g * full[3][:B].norm()
