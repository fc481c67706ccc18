"""An infinite value in V makes its channel of the output infinite, not NaN, and leaves the other channels alone (fp32, features given and
positive: every product of the state and of the readout that meets it is inf or a positive number)."""
import pytest
import torch

from paper_2602_12128_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F,d_phi,d,N", [(3, 6, 32, 100), (2, 12, 64, 2100), (3, 6, 128, 70)])
def test_one_infinite_value(F, d_phi, d, N):
    B, H = 1, 3
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    qf = torch.rand((B, H, N, d_phi), generator=g, device="cuda") + 0.1
    kf = torch.rand((B, H, F, N, d_phi), generator=g, device="cuda") + 0.1
    V = torch.randn((B, H, N, d), generator=g, device="cuda")
    op = binding.Hla(B, H, N, d, dtype="f32", phi="none", F=F, d_phi=d_phi)
    ref = op.forward(qf, kf, V)
    V2 = V.clone()
    V2[0, 1, N // 2, 5] = float("inf")
    out = op.forward(qf, kf, V2)
    want = ref.clone()
    want[0, 1, :, 5] = float("inf")
    assert torch.equal(out, want)
