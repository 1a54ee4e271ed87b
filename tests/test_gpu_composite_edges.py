"""GPU: the composite latent at the edges of the range that takes four vectors a
thread (one vector more than the threads of the largest grid, and four times as
many): a bit copy."""
import numpy as np
import pytest
import torch

from gpu_util import bits, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("batches,more,C,period", [(1, 0, 8, 77), (1, 1, 8, 1), (2, 300, 24, 1000), (4, 0, 8, 123456), (4, 1, 8, 5)])
def test_edges_of_the_batch_of_four(batches, more, C, period):
    from paper_2609_23169_gb300 import ultratex as u
    threads = torch.cuda.get_device_properties(0).multi_processor_count * 8 * 256
    T = batches * threads * 8 // C + more
    g = torch.Generator(device="cuda").manual_seed(T)
    mask = (torch.rand(T, generator=g, device="cuda") < 0.4).to(torch.uint8)
    z, tile = (torch.randint(-30000, 30000, (n, C), dtype=torch.int16, generator=g, device="cuda") for n in (T, period))
    want = torch.where(mask[:, None].bool(), z, tile[torch.arange(T, device="cuda") % period])
    u.ut_fg_composite(mask, z.view(torch.bfloat16), tile.view(torch.bfloat16))
    assert np.array_equal(bits(z), want.cpu().numpy())
