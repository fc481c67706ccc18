"""Fused query side with uneven shares (its last CTAs start late and get fewer tiles): one and two tiles per CTA, shares that do not divide,
the longest calls and the most heads that do it and the first that does not.  Every row of O and eta is written, and right in the first, a middle and the last head."""
import numpy as np
import pytest
import torch

from oracle import hla_oracle as orc
from paper_2602_12128_b200 import binding, synth
from hla_testlib import TOL, dev_weights, relerr, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,H,N", [(128, 37, 512), (64, 37, 1025), (128, 5, 128 * 59 + 1), (64, 16, 128 * 148), (64, 16, 128 * 148 + 1),
                                     (128, 44, 300), (128, 45, 300), (64, 55, 300), (64, 56, 300),
                                     (64, 148, 100), (64, 149, 100)])
@pytest.mark.parametrize("F,dphi", [(3, 6), (2, 12)])
def test_every_tile_has_an_owner(d, H, N, F, dphi):
    s = synth.HlaShape("t", 1, H, N, d, "bf16", "rms_qk", F=F, d_phi=dphi)
    Q, K, V = synth.make_qkv(s)
    pq, pk = synth.make_phi_weights(d, dphi, F, s.dtype)
    lift = lambda w: (w[0], w[1], synth.bf16_round(w[2] * np.float32(0.25)), synth.bf16_round(np.abs(w[3]) + np.float32(0.5)))      # features away from zero
    op = binding.Hla(1, H, N, d, phi="mlp", F=F, d_phi=dphi, eps=1e-6)
    wq, wk = dev_weights(lift(pq), [lift(w) for w in pk], "bf16")
    op.set_phi(wq, wk)
    O = torch.full((1, H, N, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    op.region("eta")[: H * N] = float("nan")
    op.forward(to_dev(Q, "bf16"), to_dev(K, "bf16"), to_dev(V, "bf16"), O)
    assert op.device_status() == binding.HLA_OK
    assert bool(torch.isfinite(O.float()).all()) and bool(torch.isfinite(op.region("eta")[: H * N]).all())
    gq = to_np(op.region("qf")[: H * N * dphi]).reshape(1, H, N, dphi)
    gk = to_np(op.region("kf")[: H * F * N * dphi]).reshape(1, H, F, N, dphi)
    h = [0, H // 2, H - 1]
    Oc, _ = orc.hla_core_forward(gq[:, h], gk[:, h], V[:, h].astype(np.float64), 1e-6, "factored")
    got = to_np(O[:, h])
    for i in range(3):
        assert relerr(got[:, i], Oc[:, i]) < TOL["bf16"], h[i]
