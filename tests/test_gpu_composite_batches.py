"""GPU: the composite latent at the edges of its batches of vectors (fewer
vectors than a batch, one more than a whole grid of them, rows of one and of
many vectors, periods of one and beyond the canvas): a bit copy."""
import numpy as np
import pytest
import torch

from gpu_util import bits, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("T,C,period", [(1, 8, 1), (3, 8, 2), (129, 64, 128), (1025, 72, 7), (152 * 8 * 256 * 4 + 5, 8, 1000),
                                        (40000, 512, 50000)])
def test_composite_batches(T, C, period):
    from paper_2609_23169_gb300 import ultratex as u
    g = np.random.Generator(np.random.PCG64([81, T]))
    mask = torch.from_numpy((g.random(T) < 0.4).astype(np.uint8)).cuda()
    z = torch.randint(-30000, 30000, (T, C), dtype=torch.int16, device="cuda").view(torch.bfloat16)
    tile = torch.randint(-30000, 30000, (period, C), dtype=torch.int16, device="cuda").view(torch.bfloat16)
    want = torch.where(mask[:, None].bool(), z.view(torch.int16),
                       tile.view(torch.int16)[torch.arange(T, device="cuda") % period])
    u.ut_fg_composite(mask, z, tile)
    assert np.array_equal(bits(z), want.cpu().numpy())
