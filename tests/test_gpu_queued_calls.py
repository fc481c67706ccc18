"""Sequences of calls queued without synchronisation against the same sequences synchronised after every call, bit for bit: a state carried
from call to call, feature-level steps, half passes, and weights that kernels of the caller rewrite between the calls."""
import pytest
import torch

from paper_2602_12128_b200 import binding

pytestmark = pytest.mark.gpu


class Case:
    def __init__(self, B, H, N, d, phi="mlp", F=3, **kw):
        g = torch.Generator(device="cuda")
        g.manual_seed(7)
        r = lambda *s: torch.randn(s, generator=g, device="cuda")
        self.bf = torch.float32 if kw.get("dtype") == "f32" else torch.bfloat16
        dphi = 6 if F == 3 else 12
        self.op = binding.Hla(B, H, N, d, phi=phi, F=F, d_phi=dphi, **kw)
        self.x = []
        for _ in range(3):
            V, dO = (r(B, H, N, d).to(self.bf) for _ in range(2))
            Q, K = [r(B, H, N, d).to(self.bf) for _ in range(2)] if phi == "mlp" else (r(B, H, N, dphi).abs_(), r(B, H, F, N, dphi).abs_())
            self.x.append((Q, K, V, dO))
        if phi == "mlp":
            self.sets = [[tuple(t.to(self.bf) for t in (r(d, d) / d ** 0.5, 0.1 * r(d), 0.3 * r(d, dphi) / d ** 0.5, 0.5 + 0.1 * r(dphi).abs())) for _ in range(1 + F)]
                         for _ in range(2)]
            self.w = [tuple(t.clone() for t in m) for m in self.sets[0]]
            self.op.set_phi(self.w[0], self.w[1:])

    def rewrite(self, which):
        for m, s in zip(self.w, self.sets[which]):
            for t, u in zip(m, s):
                t.copy_(u)


def compare(c, calls):
    def play(sync):
        out = []
        for f in calls:
            out += [t.clone() for t in f(c)]
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert c.op.device_status() == 0
        return out
    want = play(True)
    for _ in range(3):
        for i, (a, b) in enumerate(zip(want, play(False))):
            assert torch.equal(a, b), i


def chunk(i, carry):
    def f(c):
        c.op.set_carry(carry)
        return (c.op.forward(*c.x[i][:3]),)
    return f


def step(i, weights=False):
    def f(c):
        Q, K, V, dO = c.x[i]
        O = c.op.forward(Q, K, V)
        out = [O, *c.op.backward(Q, K, V, O, dO)]
        if weights:
            gq, gk = c.op.backward_weights(Q, K)
            out += [*gq, *(t for m in gk for t in m)]
        return out
    return f


def rewrite(which):
    def f(c):
        c.rewrite(which)
        return ()
    return f


@pytest.mark.parametrize("phi,B,H,N,d", [("mlp", 1, 3, 500, 128), ("mlp", 8, 40, 130, 64), ("mlp", 1, 1, 2300, 64), ("none", 1, 5, 1100, 128)])
def test_carried_chunks(phi, B, H, N, d):
    state = lambda c: (c.op.state_region(),)
    compare(Case(B, H, N, d, phi=phi, causal=True), [chunk(0, False), chunk(1, True), chunk(2, True), chunk(0, True), state, chunk(1, False), chunk(2, True), state])


@pytest.mark.parametrize("B,H,N,d,F,kw", [(1, 12, 1500, 128, 3, {"causal": True}), (1, 3, 5000, 64, 3, {"causal": True}), (1, 12, 1500, 64, 3, {}),
                                          (2, 40, 300, 128, 2, {}), (1, 3, 300, 64, 3, {"dtype": "f32"})])
def test_feature_level_steps(B, H, N, d, F, kw):
    compare(Case(B, H, N, d, phi="none", F=F, **kw), [step(i % 3) for i in range(8)])


@pytest.mark.parametrize("B,H,N,d,F,kw", [(1, 4, 1000, 128, 3, {}), (1, 4, 1000, 64, 2, {}), (1, 4, 1000, 128, 3, {"causal": True}), (1, 2, 300, 32, 3, {"dtype": "f32"})])
def test_weights_rewritten_between_calls(B, H, N, d, F, kw):
    compare(Case(B, H, N, d, F=F, **kw), [s for i in range(6) for s in (rewrite(i % 2), step(i % 3, weights="dtype" not in kw))])


def test_weights_rewritten_between_forward_and_backward():
    def fwd(c):
        c.O = c.op.forward(*c.x[0][:3])
        return (c.O,)

    def bwd(c):
        Q, K, V, dO = c.x[0]
        return c.op.backward(Q, K, V, c.O, dO)
    compare(Case(1, 4, 3000, 128), [rewrite(0), fwd, rewrite(1), bwd, rewrite(0), fwd, bwd])


@pytest.mark.parametrize("phi,B,H,N,d", [("mlp", 2, 12, 2000, 128), ("none", 1, 5, 1500, 64)])
def test_half_passes(phi, B, H, N, d):
    def halves(i):
        def f(c):
            Q, K, V, dO = c.x[i]
            O, dQ, dK, dV = torch.empty_like(V), torch.empty_like(Q), torch.empty_like(K), torch.empty_like(V)
            ws = c.op.workspace
            binding.hla_forward_keys(c.op.ctx, K, V, ws)
            binding.hla_forward_queries(c.op.ctx, Q, O, ws)
            binding.hla_backward_queries(c.op.ctx, Q, K, V, O, dO, dQ, dK, dV, ws)
            binding.hla_backward_keys(c.op.ctx, Q, K, V, O, dO, dQ, dK, dV, ws)
            return O, dQ, dK, dV
        return f
    c = Case(B, H, N, d, phi=phi)
    compare(c, [halves(i % 3) for i in range(6)])
    for a, b in zip(halves(1)(c), step(1)(c)):
        assert torch.equal(a, b)
