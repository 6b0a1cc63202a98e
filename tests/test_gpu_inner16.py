"""Key inner product fused with the last pass of the transform (N = 2^16): relinearised products at levels with one, full and partial
digits, batches that fill a block's four warps and that do not, several sources summed (deferred giant steps)."""
import numpy as np
import pytest

from gpu_util import add_key, ctx_pair, random_ct, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level,batch", [(1, 5), (4, 4), (6, 3), (9, 1)])
def test_relinearised_product(level, batch):
    import torch

    ctx, orc, _ = ctx_pair("full")
    a, b = random_ct(orc, 31, level, level, batch), random_ct(orc, 32, level, level, batch)
    out = torch.empty_like(to_dev(a))
    ctx.ct_ct_mul(to_dev(a), to_dev(b), out, batch, level)
    got = to_host(out)
    for i in range(batch):
        assert np.array_equal(got[i], orc.ct_ct_mul(a[i], b[i]))


@pytest.mark.parametrize("level,n_keys", [(3, 2), (10, 5)])
def test_hoisted_rotations_share_a_pass(level, n_keys):
    """Hoisted rotations by several keys: converted digits in shared memory, one division launch for all keys."""
    import torch

    pair = ctx_pair("full")
    ctx, orc, _ = pair
    ids = [600 + k for k in range(n_keys)]
    for k, i in enumerate(ids):
        add_key(pair, (3, -5, 128, 8192, -1)[k], i)
    ct = random_ct(orc, 33, level, level, 2)
    out = torch.empty((n_keys, 2, 2, level, orc.N), dtype=torch.int64, device="cuda")
    ctx.rotate_hoisted(to_dev(ct), out, 2, level, ids)
    got = to_host(out)
    for b in range(2):
        want = orc.rotate_hoisted(ct[b], ids)
        for k in range(n_keys):
            assert np.array_equal(got[k, b], want[k]), (k, b)
