"""The autotuner starts from the launch that the library makes by itself."""

import pytest

from paper_2511_08498_gb300 import api, autotune


def item(nx, nz, n_lambda, capacity):
    it = api.BatchItem()
    it.nx, it.nz, it.n_lambda, it.capacity = nx, nz, n_lambda, capacity
    return it


@pytest.mark.parametrize("items,W,walk,packet,staging", [
    ([(128, 128, 32, 64)], 8, "per_batch", 128, 1),
    ([(512, 512, 32, 227), (64, 64, 4, 3)], 8, "per_batch", 128, 1),  # 908 and 3 packets
    ([(512, 512, 32, 227), (64, 64, 4, 3)], 8, "paired", 128, 1),
    ([(512, 512, 32, 228)], 8, "per_batch", 256, 1),                  # 912
    ([(1024, 1024, 20, 456)], 8, "paired", 256, 1),                   # a pair and a lone batch
    ([(2048, 1024, 32, 4000)], 8, "per_batch", 256, 1),
    ([(2048, 1040, 32, 4000)], 8, "per_batch", 256, 0),               # 8320 blocks
    ([(512, 512, 32, 227)], 4, "per_batch", 256, 1),
])
def test_default(items, W, walk, packet, staging):
    cfg = autotune.default_config([item(*i) for i in items], W, 152, walk)
    assert cfg == dict(ctas=152 * (6 if packet == 128 else 3), packet=packet, chunk=1, staging=staging, occupancy=0,
                       walk=walk)
