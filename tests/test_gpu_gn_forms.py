"""The GroupNorm forward's forms (channel slices, one block per image with six and with four
blocks an SM, a statistics and a normalise launch) against float64, at channel counts that do
and do not divide 256 and batches on both sides of the lines between the forms: four and six
images an SM. Inputs are O(1) with group means up to a few units: a sum of at most 100 values
and four roundings of an output below 8 leave 1e-5 (8 x 2^-24 x 4 = 2e-6 and the statistics'
relative 1e-6)."""
import pytest
import torch

from paper_1911_00357_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [6, 20, 32, 48, 72, 96, 112, 512])
@pytest.mark.parametrize("per_sm,over", [(4, -1), (4, 1), (6, 0), (6, 1)])
def test_forward_forms(C, per_sm, over):
    N, HW = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + over, 50
    g = torch.Generator(device="cuda").manual_seed(C + N)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)
    z, resid = r(N, HW, C) + r(1, 1, C), r(N, HW, C)
    gamma, beta = 1 + 0.1 * r(C), 0.1 * r(C)
    for res, relu in ((None, False), (resid, True)):
        out, mean, rstd = torch.zeros_like(z), r(N, C // 2), r(N, C // 2)
        B.ddppo_group_norm(z, gamma, beta, out, mean, rstd, resid=res, relu=relu)
        y = z.double().view(N, HW, C // 2, 2)
        m = y.mean((1, 3))
        rs = 1 / torch.sqrt(((y - m[:, None, :, None]) ** 2).mean((1, 3)) + 1e-5)
        ref = ((y - m[:, None, :, None]) * rs[:, None, :, None]).reshape(z.shape) * gamma.double() + beta.double()
        if res is not None:
            ref = torch.relu(ref + res.double())
        assert (mean.double() - m).abs().max() <= 1e-5 and (rstd.double() / rs - 1).abs().max() <= 1e-5
        assert (out.double() - ref).abs().max() <= 1e-5
