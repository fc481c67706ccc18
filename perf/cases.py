"""What the performance of the operator is measured on: calls that a user of this library makes, from a few hundred
tokens in fp32 to the long video sequences, through the public classes and functions of the package.

A case is a plain dict.  `call` says what one pass does:

    forward   O = HLA(Q, K, V)                                                   (inference)
    step      forward, then dQ, dK, dV from dO                                   (training with the feature maps fixed)
    weights   step, then the gradients of the feature networks                   (training, Section 5)
    vmod      T = forward; Out = T + phi_v1(T) * phi_v2(V); the backward of both (training with Section 4.5)
    chunks    causal forward of a sequence that arrives in `chunks` pieces of N tokens each, the state carried
              from call to call (Section 4.4, sequential updates: prefill in chunks and decode in blocks)

The other keys are the arguments of `binding.Hla`.  Inputs have the distribution of the video-DiT workloads: Q and K
RMS-normalised per head, V and the upstream gradient N(0,1).  The feature networks stand for trained ones, which keep
the normaliser away from zero: a few directions of the input matter, one feature of each map is dead and the others
stay above the kink of the ReLU.  Results are then well conditioned in every output; with random networks a query all
of whose features are about zero has an output that jumps, and two correct programs differ there by O(1)."""
from __future__ import annotations

import math

import torch

from paper_2602_12128_b200 import binding, flops

DEVICE = "cuda"


def _case(name, call, B, H, N, d, dtype="bf16", phi="mlp", F=3, d_phi=6, causal=False, chunks=1):
    c = {"call": call, "B": B, "H": H, "N": N, "d": d, "dtype": dtype, "phi": phi, "F": F, "d_phi": d_phi, "causal": causal, "chunks": chunks}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: the fp32 configuration of the parity checks, where launches and latency count
        _case("tiny_f32_forward", "forward", 1, 2, 256, 16, dtype="f32"),
        # fp32 training step at a ragged length: what a user runs to validate a model before going to bf16
        _case("f32_step", "step", 1, 12, 3000, 64, dtype="f32"),
        # a short sequence at the narrow head width: three launches of a few microseconds each
        _case("small_forward", "forward", 2, 12, 4096, 64),
        # one attention call of a video DiT, 21x39x40 latent grid
        _case("dit_forward", "forward", 1, 24, 32760, 128),
        # the long sequence, 21x60x60 latent grid
        _case("long_forward", "forward", 1, 40, 75600, 128),
        # training step of the headline configuration
        _case("train_step", "step", 2, 24, 32760, 128),
        # the lower resolution of the paper (12 heads, 12600 tokens) trained with the feature networks
        _case("r2_step_weights", "weights", 1, 12, 12600, 128),
        # the 2-factor variant at the paper's higher resolution
        _case("two_factor_step", "step", 1, 12, 32760, 128, F=2, d_phi=12),
        # causal training step
        _case("causal_step", "step", 1, 24, 32760, 128, causal=True),
        # a causal sequence handed over in blocks, state carried
        _case("causal_chunks", "chunks", 1, 12, 500, 128, causal=True, chunks=8),
        # value modulation in a training step
        _case("value_mod_step", "vmod", 1, 12, 32760, 128),
        # the core on given features (the listings' signature), ragged, forward and backward
        _case("features_step", "step", 2, 6, 4999, 64, phi="none"),
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same kinds with other sizes: B, H, N over the whole range, N mostly not a multiple of a tile."""
    kind = rng.choice(["f32", "forward", "forward", "step", "step", "weights", "two_factor", "causal", "chunks", "vmod", "features"])
    if kind == "f32":
        F, d_phi = rng.choice([(3, 6), (2, 12)])
        H, N, d = rng.randint(1, 12), _log_between(rng, 64, 4096), rng.choice([16, 32, 64, 128])
        return _case(None, rng.choice(["forward", "step"]), 1, H, N, d, dtype="f32", F=F, d_phi=d_phi)
    d = rng.choice([64, 128, 128])
    B, H = rng.choice([1, 1, 2]), rng.randint(2, 40)
    most = {"forward": 120_000_000, "step": 60_000_000}.get(kind, 30_000_000) * 3 // d     # token-heads, inside the largest listed case
    N = min(_log_between(rng, 128, 75600), most // (B * H))
    if kind == "two_factor":
        return _case(None, rng.choice(["forward", "step"]), B, H, N, d, F=2, d_phi=12)
    if kind == "causal":
        return _case(None, rng.choice(["forward", "step"]), B, H, N, d, causal=True)
    if kind == "chunks":
        return _case(None, "chunks", 1, H, _log_between(rng, 64, 4096), d, causal=True, chunks=rng.randint(2, 8))
    if kind == "features":
        F, d_phi = rng.choice([(3, 6), (2, 12)])
        return _case(None, rng.choice(["forward", "step"]), B, H, N, d, phi="none", F=F, d_phi=d_phi)
    return _case(None, kind, B, H, N, d)


# ---- inputs --------------------------------------------------------------------------------------------------------
class _Draw:
    def __init__(self, seed, dtype):
        self.g = torch.Generator(device=DEVICE)
        self.g.manual_seed(seed)
        self.dtype = dtype

    def normal(self, *dims):
        return torch.randn(dims, generator=self.g, device=DEVICE, dtype=torch.float32)

    def tokens(self, *dims):
        return self.normal(*dims).to(self.dtype)

    def rms_tokens(self, *dims):
        x = self.normal(*dims)
        return x.mul_(torch.rsqrt(x.square().mean(-1, keepdim=True))).to(self.dtype)

    def feature_map(self, d, d_phi):
        """(W1, b1, W2, b2) of one feature network.  Hidden unit j follows one of d_phi directions of the input, feature m
        averages the units of its own direction; noise on everything; one feature is dead."""
        own = torch.arange(d, device=DEVICE) % d_phi
        directions = self.normal(d, d_phi)
        directions /= directions.norm(dim=0)
        W1 = directions[:, own] + 0.3 * self.normal(d, d) / math.sqrt(d)
        W2 = torch.nn.functional.one_hot(own, d_phi).float()
        W2 = W2 / W2.sum(0) + 0.1 * self.normal(d, d_phi) / d
        b2 = 0.5 + 0.05 * self.normal(d_phi)
        b2[int(torch.randint(d_phi, (1,), generator=self.g, device=DEVICE))] = -8.0
        return tuple(w.to(self.dtype) for w in (W1, 0.1 * self.normal(d), W2, b2))

    def value_map(self, d):
        """(ln_g, ln_b, W1, b1, W2, b2) of one value-modulation network."""
        ws = (1.0 + 0.2 * self.normal(d), 0.1 * self.normal(d), self.normal(d, d) / math.sqrt(d), 0.1 * self.normal(d),
              self.normal(d, d) / math.sqrt(d), 0.1 * self.normal(d))
        return tuple(w.to(self.dtype) for w in ws)


def prepare(case, seed):
    c = case
    r = _Draw(seed, torch.bfloat16 if c["dtype"] == "bf16" else torch.float32)
    op = binding.Hla(c["B"], c["H"], c["N"], c["d"], dtype=c["dtype"], phi=c["phi"], F=c["F"], d_phi=c["d_phi"], causal=c["causal"],
                     value_mod=c["call"] == "vmod", device=DEVICE)
    dims = (c["B"], c["H"], c["N"], c["d"])
    s = {"op": op, "call": c["call"]}
    if c["phi"] == "mlp":
        op.set_phi(r.feature_map(c["d"], c["d_phi"]), [r.feature_map(c["d"], c["d_phi"]) for _ in range(c["F"])])
        s["parts"] = [(r.rms_tokens(*dims), r.rms_tokens(*dims), r.tokens(*dims)) for _ in range(c["chunks"])]
    else:
        scale = 1.0 / math.sqrt(c["d_phi"])
        qf = r.normal(c["B"], c["H"], c["N"], c["d_phi"]).abs_().mul_(scale)
        kf = r.normal(c["B"], c["H"], c["F"], c["N"], c["d_phi"]).abs_().mul_(scale)
        s["parts"] = [(qf, kf, r.tokens(*dims))]
    if c["call"] in ("step", "weights", "vmod"):
        s["dO"] = r.tokens(*dims)
    if c["call"] == "vmod":
        op.set_phi_v(r.value_map(c["d"]), r.value_map(c["d"]))
    return s


def run(state):
    op, call = state["op"], state["call"]
    if call == "chunks":
        outs = []
        for i, (Q, K, V) in enumerate(state["parts"]):
            op.set_carry(i > 0)
            outs.append(op.forward(Q, K, V))
        L, cfg = op.layout, op.cfg
        carried = op.state_region().view(cfg.B * cfg.H, L.state_rows, L.state_ld)[:, :, : cfg.d + 1]     # (C, z); the rest of a row is padding
        return {"O": outs, "state": carried}
    Q, K, V = state["parts"][0]
    O = op.forward(Q, K, V)
    if call == "forward":
        return O
    dO = state["dO"]
    if call == "vmod":
        Out = op.value_mod_forward(O, V)
        dT, dV = op.value_mod_backward(O, V, dO)
        dQ, dK, dVa = op.backward(Q, K, V, O, dT)
        dV += dVa
        return {"Out": Out, "dQ": dQ, "dK": dK, "dV": dV}
    dQ, dK, dV = op.backward(Q, K, V, O, dO)
    out = {"O": O, "dQ": dQ, "dK": dK, "dV": dV}
    if call == "weights":
        gq, gk = op.backward_weights(Q, K)
        out["phi_q"], out["phi_k"] = list(gq), [list(g) for g in gk]
    return out


def work(case):
    """Inputs read once, results written once; the FLOPs of the symmetry-folded scheme (what any program has to execute)."""
    c = case
    th = c["B"] * c["H"] * c["N"] * c["chunks"]
    elt, mlp = (2 if c["dtype"] == "bf16" else 4), c["phi"] == "mlp"
    d, F, d_phi = c["d"], c["F"], c["d_phi"]
    backward = c["call"] in ("step", "weights", "vmod")
    by = 2 * d * elt + (2 * d * elt if mlp else (1 + F) * d_phi * 4)                    # V, O, and Q, K or the features
    if backward:
        by += 2 * d * elt + (2 * d * elt if mlp else (1 + F) * d_phi * 4)               # dO, dV, and dQ, dK or the features' gradients
    fl = flops.folded_flops_per_token(d, F, d_phi, backward, mlp)
    if c["call"] == "weights":
        fl += (1 + F) * (2 * d * d + 2 * d * d_phi)                                     # dW1, dW2; the hidden layer is counted in the backward
    if c["call"] == "vmod":
        fl += flops.value_mod_flops_per_token(d, True)
    weights = (1 + F) * (d * d + d + d * d_phi + d_phi) if mlp else 0
    extra = weights * elt + (weights * 4 if c["call"] == "weights" else 0) + (2 * (2 * d * d + 4 * d) * elt if c["call"] == "vmod" else 0)
    if c["call"] == "chunks":
        extra += c["B"] * c["H"] * flops.n_monomials(F, d_phi) * (d + 1) * 4
    return {"bytes": th * by + extra, "flops": th * fl}


def tolerance(case):
    """About four times what each kind of call shows against the same operator in 64 bits on these inputs: fp32 results
    7e-7 (dQ) and below, bf16 outputs 2e-3 (one rounding of the operands and one of the result), gradients 2e-3 to 6e-3;
    1e-2 for the causal dQ (the first tokens attend to a few keys only, their gradients are small differences of large
    terms) and for the second-layer biases of the key maps (sums over all tokens that nearly cancel)."""
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 5e-4}
    if case["call"] in ("forward", "chunks"):
        return {"rel": 8e-3, "max": 0.3}
    if case["causal"] or case["call"] == "weights":
        return {"rel": 3e-2, "max": 0.9}
    return {"rel": 2e-2, "max": 0.5}
