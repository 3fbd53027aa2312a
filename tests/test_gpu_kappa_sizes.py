"""counts_to_kappa on both sides of its size rules (division up to nside 64,
four pixels per thread above nside 512), at 16-byte aligned and other maps."""
import pytest
import torch

from oracle import binning
from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside", [1, 64, 128, 512, 1024])
@pytest.mark.parametrize("shift", [0, 1])
def test_kappa_is_bit_exact(nside, shift):
    c = ctx()
    npx = 12 * nside * nside
    counts = torch.randint(0, 6000, (npx + 1,), dtype=torch.int32, generator=torch.Generator().manual_seed(nside))
    out = torch.zeros(npx + 1, dtype=torch.float64, device="cuda")[shift:shift + npx]
    c.counts_to_kappa(counts.cuda()[shift:shift + npx], nside, 3.7, 1.3, kappa=out)
    c.sync()
    assert torch.equal(out.cpu(), binning.kappa_from_counts(counts[shift:shift + npx].long(), 3.7, 1.3))
