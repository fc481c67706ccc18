"""Causal forward with the phi maps whose sweep adds the pieces before its own: CTAs that begin several heads, with and without a carried
state; a head with more pieces than that is done for (the scan runs first); the state left for the next call, and a backward after it."""
import numpy as np
import pytest

from oracle import hla_oracle as orc
from paper_2602_12128_b200 import synth
from hla_testlib import DeviceRun, TOL, fold_symmetric, oracle_state, relerr

pytestmark = pytest.mark.gpu
EPS = 1e-6
f64 = lambda a: np.asarray(a, np.float64)


@pytest.mark.parametrize("d,N,H,chunks", [(128, 300, 61, 2), (64, 129, 100, 3), (128, 100, 1, 2), (64, 2177, 1, 2), (128, 16 * 128, 1, 2), (128, 16 * 128 + 1, 1, 2)])
def test_chunks_with_phi_maps(d, N, H, chunks):
    s = synth.HlaShape("t", 1, H, N * chunks, d, "bf16", "rms_qk")
    Q, K, V = synth.make_qkv(s)
    pq, pk = synth.make_phi_weights(d, 6, 3, s.dtype)
    lift = lambda w: (w[0], w[1], synth.bf16_round(w[2] * np.float32(0.25)), synth.bf16_round(np.abs(w[3]) + np.float32(0.5)))      # features away from zero
    run = DeviceRun(synth.HlaShape("t", 1, H, N, d, "bf16", "rms_qk"), "mlp", EPS, causal=True)
    run.set_weights(lift(pq), [lift(w) for w in pk])
    parts = [[np.ascontiguousarray(x[:, :, c * N:(c + 1) * N]) for x in (Q, K, V)] for c in range(chunks)]
    outs, gqs, gks = [], [], []
    for c in range(chunks):
        run.op.set_carry(c > 0)
        outs.append(run.forward(*parts[c]))
        gq, gk = run.features()
        gqs.append(gq)
        gks.append(gk)
    O, gq, gk = np.concatenate(outs, axis=2), np.concatenate(gqs, axis=2), np.concatenate(gks, axis=3)
    Oc, _ = orc.hla_core_forward(gq, gk, f64(V), EPS, "causal_streaming" if N * chunks > 1000 else "causal_quadratic")
    C, z = run.state()
    Co, zo = oracle_state(gk, f64(V))
    Co, zo = fold_symmetric(Co), fold_symmetric(zo[..., None])[..., 0]
    for h in range(H):      # per head: a piece or a carried state of another head would be wrong in one head only
        assert relerr(O[:, h], Oc[:, h]) < TOL["bf16"], h
        # the operands of the state product are rounded to bf16 once (2^-9 each), its sums are fp32
        assert relerr(C[:, h], Co[:, h]) < TOL["bf16"] / 4 and relerr(z[:, h], zo[:, h]) < TOL["bf16"] / 4, h
    # a fresh sequence in the same workspace forgets what was carried, and its backward finds its own pieces
    run.op.set_carry(False)
    assert np.array_equal(run.forward(*parts[0]), outs[0])
    dO = synth.make_dO(run.shape)
    _, _, dV = run.backward(dO)
    rq, _, rv = orc.hla_core_backward(gqs[0], gks[0], f64(parts[0][2]), f64(dO), EPS, "causal_quadratic")
    assert relerr(dV, rv) < TOL["bf16"]
    dq = run.region("dqf", gqs[0].size, gqs[0].shape)
    for h in range(H):      # differences of terms of size |dO_i . o_i|, each rounded to bf16
        term = np.abs((f64(dO[0, h]) * outs[0][0, h]).sum(-1)).max()
        assert np.abs(dq[0, h] - rq[0, h]).max() < TOL["bf16"] * max(np.abs(rq[0, h]).max(), term), h
