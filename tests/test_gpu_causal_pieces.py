"""Causal backward on the pieces the forward left: CTAs whose work crosses heads (more tiles than SMs, few tiles per head), a
piece that is one ragged tile, one head; the backward twice after one forward."""
import numpy as np
import pytest
import torch

from oracle import hla_oracle as orc
from paper_2602_12128_b200 import synth
from hla_testlib import DeviceRun, TOL, relerr

pytestmark = pytest.mark.gpu
f64 = lambda a: np.asarray(a, np.float64)


@pytest.mark.parametrize("d,N,H", [(128, 300, 61), (64, 700, 37), (128, 129, 100), (64, 100, 1), (128, 1000, 1)])
def test_backward_with_phi_maps(d, N, H):
    s = synth.HlaShape("t", 1, H, N, d, "bf16", "rms_qk")
    Q, K, V = synth.make_qkv(s)
    dO = synth.make_dO(s)
    pq, pk = synth.make_phi_weights(d, 6, 3, s.dtype)
    lift = lambda w: (w[0], w[1], synth.bf16_round(w[2] * np.float32(0.25)), synth.bf16_round(np.abs(w[3]) + np.float32(0.5)))      # features away from zero
    run = DeviceRun(s, "mlp", 1e-6, causal=True)
    run.set_weights(lift(pq), [lift(w) for w in pk])
    O = run.forward(Q, K, V)
    a = run.backward(dO)
    gq, gk = run.features()
    dqf, dkf = run.region("dqf", gq.size, gq.shape), run.region("dkf", gk.size, gk.shape)
    Oc, _ = orc.hla_core_forward(gq, gk, f64(V), 1e-6, "causal_quadratic")
    rq, rk, rv = orc.hla_core_backward(gq, gk, f64(V), f64(dO), 1e-6, "causal_quadratic")
    assert relerr(O, Oc) < TOL["bf16"] and relerr(a[2], rv) < TOL["bf16"]
    # per head: a piece taken from another head's state would be wrong in one head only.  dq and dk are differences of terms of size
    # |dO_i . o_i| (every weight of a row is shifted by it), each of which is rounded to bf16, so the error is measured against that
    # size where the result is smaller: the features here are nearly constant along a row, which makes the gradients small.
    for h in range(H):
        term = np.abs((f64(dO[0, h]) * Oc[0, h]).sum(-1)).max()
        assert np.abs(dqf[0, h] - rq[0, h]).max() < TOL["bf16"] * max(np.abs(rq[0, h]).max(), term), h
        assert np.abs(dkf[0, h] - rk[0, h]).max() < TOL["bf16"] * max(np.abs(rk[0, h]).max(), term), h
    b = run.backward(dO)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
