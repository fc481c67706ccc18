"""Gradients written over inputs (the combinations that hla.h allows): bit for bit the results of separate buffers."""
import pytest
import torch

from paper_2602_12128_b200 import binding

pytestmark = pytest.mark.gpu


def _rand(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return lambda *s: torch.randn(s, generator=g, device="cuda")


@pytest.mark.parametrize("phi,dtype,causal,F,d,over", [
    ("mlp", "bf16", False, 3, 128, {"dQ": "V"}), ("mlp", "bf16", False, 2, 64, {"dQ": "V"}), ("mlp", "bf16", False, 3, 64, {"dQ": "dO", "dK": "K"}),
    ("mlp", "bf16", False, 3, 128, {"dQ": "Q"}), ("mlp", "bf16", True, 3, 128, {"dQ": "dO"}), ("mlp", "bf16", True, 3, 64, {"dQ": "V", "dK": "K"}),
    ("mlp", "bf16", True, 3, 128, {"dQ": "O"}), ("none", "bf16", True, 3, 128, {"dK": "K"}), ("none", "bf16", False, 3, 128, {"dQ": "Q", "dK": "K"}),
    ("mlp", "f32", False, 3, 64, {"dQ": "V"}), ("mlp", "f32", False, 2, 32, {"dQ": "dO", "dK": "K"}), ("none", "f32", False, 3, 64, {"dQ": "Q"}),
    ("none", "f32", False, 2, 128, {"dK": "K"}), ("none", "f32", False, 2, 12, {"dQ": "dO"})])
def test_backward(phi, dtype, causal, F, d, over):
    B, H, N, dphi = 1, 12, 3000, 6 if F == 3 else 12
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    r = _rand(1)
    op = binding.Hla(B, H, N, d, dtype=dtype, phi=phi, F=F, d_phi=dphi, causal=causal)
    x = {"V": r(B, H, N, d).to(dt), "dO": r(B, H, N, d).to(dt)}
    if phi == "mlp":
        w = [tuple(t.to(dt) for t in (r(d, d) / d ** 0.5, 0.1 * r(d), r(d, dphi) / d ** 0.5, 0.5 + 0.1 * r(dphi).abs())) for _ in range(1 + F)]
        op.set_phi(w[0], w[1:])
        x["Q"], x["K"] = r(B, H, N, d).to(dt), r(B, H, N, d).to(dt)
    else:
        x["Q"], x["K"] = r(B, H, N, dphi).abs_(), r(B, H, F, N, dphi).abs_()
    x["O"] = op.forward(x["Q"], x["K"], x["V"])
    want = op.backward(x["Q"], x["K"], x["V"], x["O"], x["dO"])
    want = [t.clone() for t in want]
    for _ in range(3):
        y = {k: v.clone() for k, v in x.items()}
        got = op.backward(y["Q"], y["K"], y["V"], y["O"], y["dO"], **{k: y[v] for k, v in over.items()})
        for a, b in zip(want, got):
            assert torch.equal(a, b)
    assert op.device_status() == 0


@pytest.mark.parametrize("over", [{"dV": "dOut"}, {"dV": "T"}, {"dV": "V", "dT": "T"}])
def test_value_modulation(over):
    B, H, N, d = 1, 12, 3000, 128
    r = _rand(2)
    op = binding.Hla(B, H, N, d, value_mod=True)
    op.set_phi_v(*[tuple(t.to(torch.bfloat16) for t in (1 + 0.1 * r(d), 0.1 * r(d), r(d, d) / d ** 0.5, 0.1 * r(d), r(d, d) / d ** 0.5, 0.1 * r(d))) for _ in range(2)])
    x = {k: r(B, H, N, d).to(torch.bfloat16) for k in ("T", "V", "dOut")}
    want = [t.clone() for t in op.value_mod_backward(x["T"], x["V"], x["dOut"])]
    for _ in range(3):
        y = {k: v.clone() for k, v in x.items()}
        got = op.value_mod_backward(y["T"], y["V"], y["dOut"], **{k: y[v] for k, v in over.items()})
        for a, b in zip(want, got):
            assert torch.equal(a, b)
