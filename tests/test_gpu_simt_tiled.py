"""The register-tiled fp32 kernels (F = 3 with d_phi = 6, F = 2 with d_phi = 12) at the sizes where a tile can go wrong:
head widths at and beside the column groups (32, 64, 128), token counts at and beside the tiles of 32 and 64, one token,
more splits than tokens.  Against the fp64 oracle; the bound is the fp32 one of the other tests (1e-4 of the largest
value): sums of at most a few thousand fp32 terms, each rounded to 2^-24, stay two orders below it."""
import numpy as np
import pytest
import torch

from oracle import hla_oracle as orc
from paper_2602_12128_b200 import binding, synth
from hla_testlib import DeviceRun, TOL, oracle_state, relerr

pytestmark = pytest.mark.gpu
EPS = 1e-6
f64 = lambda a: np.asarray(a, np.float64)


# (the last three: enough heads for the tiles of 64 tokens, the others run on tiles of 16)
@pytest.mark.parametrize("F,dphi", [(3, 6), (2, 12)])
@pytest.mark.parametrize("H,d,N,splits", [(3, 4, 1, 0), (3, 28, 63, 0), (3, 32, 64, 5), (3, 36, 65, 0), (3, 64, 31, 0), (3, 64, 129, 3), (3, 68, 33, 0), (3, 128, 200, 0),
                                          (150, 32, 63, 0), (75, 64, 65, 0), (50, 128, 130, 2)])
def test_core_forward_backward(F, dphi, H, d, N, splits):
    s = synth.HlaShape("t", 1, H, N, d, "f32", "inv_sqrt_d", F=F, d_phi=dphi)
    _, _, V = synth.make_qkv(s)
    V = V * np.float32(np.sqrt(d))
    qf, kf = synth.make_features(s)
    dO = synth.make_dO(s)
    run = DeviceRun(s, "none", EPS, splits)
    O = run.forward(qf, kf, V)
    dq, dk, dv = run.backward(dO)
    Oq, eta = orc.hla_core_forward(f64(qf), f64(kf), f64(V), EPS, "quadratic")
    C, z = run.state()
    Co, zo = oracle_state(f64(kf), f64(V))
    assert relerr(O, Oq) < TOL["f32"] and relerr(run.eta(), eta) < TOL["f32"]
    assert relerr(C, Co) < TOL["f32"] and relerr(z, zo) < TOL["f32"]
    rq, rk, rv = orc.hla_core_backward(f64(qf), f64(kf), f64(V), f64(dO), EPS, "quadratic")
    assert relerr(dv, rv) < TOL["f32"]
    # dq and dk are differences of terms of size |dO_i . o_i| (with a single key they cancel completely)
    term = np.abs((f64(dO) * Oq).sum(-1)).max()
    assert np.abs(dq - rq).max() < TOL["f32"] * max(np.abs(rq).max(), term)
    assert np.abs(dk - rk).max() < TOL["f32"] * max(np.abs(rk).max(), term)


@pytest.mark.parametrize("F,dphi,H,d,N,dtype", [(3, 6, 2, 16, 70, "f32"), (2, 12, 2, 20, 64, "f32"), (3, 6, 2, 64, 65, "f32"), (2, 12, 2, 128, 33, "f32"),
                                                (3, 6, 2, 100, 130, "f32"), (3, 6, 2, 32, 65, "bf16"), (2, 12, 2, 72, 40, "bf16"), (3, 6, 75, 20, 63, "f32"),
                                                (2, 12, 38, 64, 129, "f32"), (3, 6, 38, 128, 129, "f32"), (3, 6, 75, 32, 63, "bf16")])
def test_with_phi_stage_by_stage(F, dphi, H, d, N, dtype):
    """Feature networks forward and backward, each stage on the features and feature gradients the library kept."""
    s = synth.HlaShape("t", 2, H, N, d, dtype, "rms_qk", F=F, d_phi=dphi)
    Q, K, V = synth.make_qkv(s)
    dO = synth.make_dO(s)
    pq, pk = synth.make_phi_weights(d, dphi, F, dtype)
    run = DeviceRun(s, "mlp", EPS)
    assert run.op.layout.tensor_core == 0
    run.set_weights(pq, pk)
    O = run.forward(Q, K, V)
    dQ, dK, dV = run.backward(dO)
    gq, gk = run.features()
    rows = lambda x: f64(x).reshape(-1, d)
    fq = orc.phi_mlp(rows(Q), *pq).reshape(gq.shape)
    fk = np.stack([orc.phi_mlp(rows(K), *w).reshape(gq.shape) for w in pk], axis=2)
    assert relerr(gq, fq) < TOL["f32"] and relerr(gk, fk) < TOL["f32"]
    Oc, _ = orc.hla_core_forward(gq, gk, f64(V), EPS, "factored")
    assert relerr(O, Oc) < TOL[dtype]
    n = gq.size
    dqf, dkf = run.region("dqf", n, gq.shape), run.region("dkf", n * F, gk.shape)
    # weights fixed, ReLU mask from the features the library kept: dx = W1 (GELU'(h) (W2 (df [feat > 0])))
    def back(x, w, df, feat):
        W1, b1, W2, _ = (f64(a) for a in w)
        h = rows(x) @ W1 + b1
        from math import pi
        from scipy.special import erf
        gp = 0.5 * (1 + erf(h / np.sqrt(2))) + h * np.exp(-0.5 * h * h) / np.sqrt(2 * pi)
        dp = (df * (feat > 0)).reshape(-1, dphi)
        return ((dp @ W2.T) * gp) @ W1.T
    rQ = back(Q, pq, dqf, gq).reshape(dQ.shape)
    rK = sum(back(K, pk[f], dkf[:, :, f], gk[:, :, f]) for f in range(F)).reshape(dK.shape)
    tol = max(TOL["f32"], 2.0 ** -8 if dtype == "bf16" else 0.0)      # bf16 results are rounded once
    assert relerr(dQ, rQ) < tol and relerr(dK, rK) < tol
