"""Weight gradients where the split of a side's CTAs over its maps can go wrong: one tile (a CTA per map), fewer tiles than
CTAs (an uneven run of tiles per map), a ragged last tile, both geometries, one side alone."""
import numpy as np
import pytest
import torch

from paper_2602_12128_b200 import synth
from hla_testlib import DeviceRun, TOL, relerr, to_np
from test_gpu_wgrad import oracle_stagewise

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F,dphi,d,N,H", [(3, 6, 128, 1, 1), (3, 6, 64, 129, 1), (2, 12, 128, 128, 1), (2, 12, 64, 300, 1), (3, 6, 128, 1000, 7), (2, 12, 128, 640, 31)])
def test_stagewise(F, dphi, d, N, H):
    s = synth.HlaShape("t", 1, H, N, d, "bf16", "rms_qk", backward=True, F=F, d_phi=dphi)
    Q, K, V = synth.make_qkv(s)
    pq, pk = synth.make_phi_weights(d, dphi, F, s.dtype)
    run = DeviceRun(s, "mlp", 1e-6)
    run.set_weights(pq, pk)
    run.forward(Q, K, V)
    run.backward(synth.make_dO(s))
    gq, gk = run.op.backward_weights(run.Q, run.K)
    torch.cuda.synchronize()
    assert run.op.device_status() == 0
    qf, kf = run.features()
    dqf, dkf = run.region("dqf", qf.size, qf.shape), run.region("dkf", kf.size, kf.shape)
    for got, X, w, feat, dfeat in [(gq, Q, pq, qf, dqf)] + [(gk[f], K, pk[f], kf[:, :, f], dkf[:, :, f]) for f in range(F)]:
        for name, y, ref in zip(("dW1", "db1", "dW2", "db2"), got, oracle_stagewise(X, w, feat, dfeat)):
            # bf16 operands of the products, fp32 sums: the bound of the other weight-gradient tests, against the largest value
            # (a single token whose features are all clipped has gradients of exactly zero)
            assert relerr(to_np(y), ref) < TOL["bf16"], name
