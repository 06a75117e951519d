"""Buffers rewritten in place between calls on one stream.  Kernels of a call start before the ones
ahead of them end, and some read their inputs without waiting for the kernel just before them (S0,
and the later forms of the contraction stages), so each call must still see what was written last:
the input by a kernel directly ahead of the call, and the workspace by the call's own stages.
Every call gives the same bits as the same call with the device idle before it."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CONFIGS = {
    "16 frames": dict(N=2 ** 15, J=12, Q=16, J_fr=4, Q_fr=2, T=2 ** 11, F=16),   # every backward form
    "64 frames": dict(N=2 ** 12, J=6, Q=8, J_fr=3, Q_fr=1, T=2 ** 6, F=8),
}


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("config", list(CONFIGS))
@pytest.mark.parametrize("B", [1, 24])
def test_inputs_rewritten_in_place(config, precision, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_08269_gb300 import JTFSPlan, build
    build.build()
    plan = JTFSPlan(precision=precision, **CONFIGS[config])
    sh = plan.shapes
    gen = torch.Generator(device="cuda").manual_seed(B)
    base = torch.randn(B, CONFIGS[config]["N"], device="cuda", generator=gen)
    cot = [torch.randn(f(B), device="cuda", generator=gen) for f in (sh.s0, sh.s1, sh.s2)]
    x, g = torch.empty_like(base), [torch.empty_like(c) for c in cot]

    def call(k, idle):
        torch.mul(base, float(2 ** k), out=x)
        for c, v in zip(cot, g):
            torch.mul(c, float(2 ** -k), out=v)
        if idle:
            torch.cuda.synchronize()
        return plan.forward_backward(x, *g)

    want = []
    for k in range(4):
        want.append(call(k, True))
        torch.cuda.synchronize()
    got = [call(k % 4, False) for k in range(24)]
    plan.sync()
    for k, out in enumerate(got):
        for a, b in zip(out, want[k % 4]):
            assert torch.equal(a, b), k
    # (the calls do differ)
    assert not torch.equal(want[0][0], want[1][0]) and not torch.equal(want[0][3], want[3][3])
