"""A state carried through many short calls against the sum, in 64 bits, of the states of the calls on their own."""
import pytest
import torch

from paper_2602_12128_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("phi,B,H,N,d", [("mlp", 1, 2, 128, 64), ("mlp", 1, 3, 300, 128), ("mlp", 8, 40, 130, 64), ("none", 1, 2, 256, 64)])
def test_state_of_many_calls(phi, B, H, N, d):
    calls = 400
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")
    carried, fresh = (binding.Hla(B, H, N, d, phi=phi, causal=True) for _ in range(2))
    if phi == "mlp":
        w = [tuple(t.to(torch.bfloat16) for t in (r(d, d) / d ** 0.5, 0.1 * r(d), 0.2 * r(d, 6) / d ** 0.5, 0.8 + 0.1 * r(6).abs())) for _ in range(4)]
        for op in (carried, fresh):
            op.set_phi(w[0], w[1:])
    total = 0.0
    rows = lambda op: op.state_region().view(B * H, op.layout.state_rows, op.layout.state_ld)[:, :, : d + 1].double()
    for c in range(calls):
        if c < 8 or c % 50 == 0:      # (positive: the partial sums grow, so that a relative bound holds for every entry)
            if phi == "mlp":
                Q, K = (r(B, H, N, d).to(torch.bfloat16) for _ in range(2))
            else:
                Q, K = r(B, H, N, 6).abs_(), r(B, H, 3, N, 6).abs_()
            V = r(B, H, N, d).abs_().to(torch.bfloat16)
        carried.set_carry(c > 0)
        carried.forward(Q, K, V)
        fresh.forward(Q, K, V)
        total = total + rows(fresh)
    assert carried.device_status() == 0
    got = rows(carried)
    # every call adds its own state to the carried one in one or two fp32 additions per piece of the sequence, rounded to nearest
    # (2^-24 of a partial sum each; the partial sums grow about linearly, so half of that in all), and the state of a call is that of a
    # call on its own up to its own sum over the pieces
    pieces = 2 if N > 128 else 1
    err = ((got - total).abs() / total.abs().clamp_min(1e-30))[total.abs() > 0].max()
    print("relative error of the carried state", float(err), "bound", calls * pieces * 2.0 ** -24)
    assert err < calls * pieces * 2.0 ** -24
