"""The angle MSE is that of the angle images: on maps that differ by a radian, by a
thousandth and by a few units in the last place, with normals of every direction,
beside the z axis, at the cuts of the angles and masked ones, it equals the mean of
the squared differences of the images that nrm_spherical writes. (Their differences are the same floats,
squared and summed in FP32 over at most 32 pixels and then in FP64: 32 x 2^-24
= 1.9e-6 relative; allowed 4e-6.) Against the FP64 oracle where the difference is
far above the angles' own error of 3e-7."""
import pytest
import torch

import paper_2209_08241_gb300 as nrm
from oracle import evaluation

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def directions(H, W, spread, gen):
    """Unit vectors around +-z, `spread` wide (large: every direction)."""
    n = torch.zeros((H, W, 4), device=DEV, dtype=torch.float64)
    n[..., 2] = torch.where(torch.rand((H, W), generator=gen, device=DEV) < 0.5, -1.0, 1.0)
    n[..., :3] += spread * torch.randn((H, W, 3), generator=gen, device=DEV, dtype=torch.float64)
    return n / n.norm(dim=-1, keepdim=True)


@pytest.mark.parametrize("spread", [3.0, 0.1, 1e-4, 1e-12])
@pytest.mark.parametrize("apart", [1.0, 1e-3, 3e-7])
@pytest.mark.parametrize("length", [1.0, 1.37])
def test_equals_the_mse_of_the_angle_images(spread, apart, length):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(1e6 * apart))
    H, W = 411, 517
    a = directions(H, W, spread, gen)
    b = a.clone()
    b[..., :3] += apart * spread * torch.randn((H, W, 3), generator=gen, device=DEV, dtype=torch.float64)
    # (The angles do not depend on a vector's length, the roundings on the way do.)
    b = length * b / b.norm(dim=-1, keepdim=True)
    a, b = a.float(), b.float()
    a[0, :7, :2] = torch.tensor([[0.0, 0.0], [-0.0, 0.0], [0.0, -0.0], [-1e-14, 0.0], [1e-14, 1e-15], [-0.5, -0.0],
                                 [-0.5, 0.0]], device=DEV)
    va = (torch.rand((H, W), generator=gen, device=DEV) < 0.9).to(torch.uint8)
    vb = (torch.rand((H, W), generator=gen, device=DEV) < 0.9).to(torch.uint8)
    a, b = a * va[..., None], b * vb[..., None]
    est = nrm.BatchedEstimator()
    got = nrm.angle_mse(est, a, va, b, vb).cpu()
    est.sync_status()
    (pa, ta), (pb, tb) = nrm.spherical_images(a, va), nrm.spherical_images(b, vb)
    both = (va != 0) & (vb != 0)
    assert float(got[2]) == float(both.sum())
    for mse, x, y in ((got[0], ta, tb), (got[1], pa, pb)):
        d = (x - y)[both].double()  # (the difference of two floats, rounded to FP32 as the kernel's is)
        want = float((d * d).mean())
        assert float(mse) == pytest.approx(want, rel=4e-6, abs=0.0), (spread, apart)
    if spread >= 0.1 and apart >= 1e-3:
        mt, mp, _ = evaluation.angle_mse(a.double().cpu().numpy(), va.cpu().numpy(), b.double().cpu().numpy(),
                                         vb.cpu().numpy())
        assert float(got[0]) == pytest.approx(mt, rel=1e-2 if apart < 1 else 1e-4, abs=0.0)
