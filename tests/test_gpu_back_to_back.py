"""Calls that follow one another on a stream without synchronisation, on the same context and workspace: kernels that start beside
their predecessor must see what the kernels before it wrote, and must not touch what it still reads.  Steps on inputs A and B
alternate; every result of A must be bit for bit that of a step on A alone."""
import pytest
import torch

from paper_2602_12128_b200 import binding

pytestmark = pytest.mark.gpu


def _inputs(seed, dims, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return tuple(torch.randn(dims, generator=g, device="cuda").to(dtype) for _ in range(4))


def _weights(seed, d, dphi, n, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    mk = lambda *s: (torch.randn(s, generator=g, device="cuda") / d ** 0.5).to(dtype)
    return [(mk(d, d), mk(d), mk(d, dphi), mk(dphi)) for _ in range(n)]


@pytest.mark.parametrize("kind,B,H,N,d,dtype,F", [("step", 1, 3, 200, 64, "f32", 3), ("step", 1, 40, 300, 64, "f32", 2), ("weights", 1, 2, 300, 128, "bf16", 3),
                                                  ("weights", 1, 8, 2500, 64, "bf16", 2), ("causal", 1, 3, 500, 128, "bf16", 3), ("vmod", 1, 4, 700, 128, "bf16", 3)])
def test_alternating_steps(kind, B, H, N, d, dtype, F):
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    dphi = 6 if F == 3 else 12
    op = binding.Hla(B, H, N, d, dtype=dtype, F=F, d_phi=dphi, causal=kind == "causal", value_mod=kind == "vmod")
    w = _weights(1, d, dphi, 1 + F, dt)
    op.set_phi(w[0], w[1:])
    if kind == "vmod":
        g = torch.Generator(device="cuda")
        g.manual_seed(9)
        mk = lambda *s: (0.1 * torch.randn(s, generator=g, device="cuda") + (1.0 if len(s) == 1 else 0.0)).to(dt)
        op.set_phi_v(*[(mk(d), mk(d), mk(d, d), mk(d), mk(d, d), mk(d)) for _ in range(2)])

    def step(x):
        Q, K, V, dO = x
        O = op.forward(Q, K, V)
        out = [O]
        if kind == "vmod":
            out.append(op.value_mod_forward(O, V))
            dO, dV = op.value_mod_backward(O, V, dO)
            out += [dO, dV]
        out += list(op.backward(Q, K, V, O, dO))
        if kind == "weights":
            gq, gk = op.backward_weights(Q, K)
            out += list(gq) + [t for m in gk for t in m]
        return out

    a, b = (_inputs(s, (B, H, N, d), dt) for s in (3, 4))
    ref = step(a)
    torch.cuda.synchronize()
    got = []
    for _ in range(6):
        step(b)
        got.append(step(a))
    torch.cuda.synchronize()
    assert op.device_status() == 0
    for out in got:
        for x, y in zip(ref, out):
            assert torch.equal(x, y)
