"""The tiled global transform (large aligned lists) against the oracle's
transform, bit for bit: list lengths around whole tiles, bins of one record,
empty bins, and bins that span many tiles."""
import numpy as np
import pytest

from oracle import oracle as O
from test_gpu_unatt_encode import dec  # noqa: F401
from test_gpu_xyz import _same_bits

pytestmark = pytest.mark.gpu

FROM = 1 << 22  # records from which the tiles are used


@pytest.mark.parametrize("n", [FROM - 1, FROM, FROM + 1, FROM + 1023, FROM + 7 * 1024 + 5])
@pytest.mark.parametrize("shape", ["uniform", "hot"])
def test_tiles(dec, n, shape):  # noqa: F811
    import torch
    rng = np.random.default_rng(n % 1000)
    w = np.ones(5472)
    if shape == "hot":  # most bins empty or of a few records, two of a million
        w = rng.random(5472) ** 12
        w[rng.permutation(5472)[:3000]] = 0
        w[[7, 4001]] = w.sum()
    cnt = np.floor(w / w.sum() * n).astype(np.int64)
    cnt[7] += n - cnt.sum()
    rs = np.concatenate([[0], np.cumsum(cnt)]).astype(np.uint32)
    native = rng.integers(0, 256, (n, 12), dtype=np.uint8)
    out = dec.global_xyz(torch.from_numpy(native).cuda(), torch.from_numpy(rs.view(np.int32)).cuda())
    torch.cuda.synchronize()
    _same_bits(out, O.global_xyz(native, rs), f"{n} {shape}")
