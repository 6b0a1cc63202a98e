"""ModUp fused with the first pass of the N = 2^16 forward transform: every digit shape of the ring (full and partial last
digits, one to four source limbs), with random residues and with the largest ones, through a rotation."""
import numpy as np
import pytest

from gpu_util import add_key, ctx_pair, random_ct, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level,batch,largest", [(1, 1, False), (2, 3, True), (3, 1, True), (4, 2, False), (5, 1, True), (11, 1, False), (24, 1, True)])
def test_rotation_at_every_digit_shape(level, batch, largest):
    import torch

    pair = ctx_pair("full")
    ctx, orc, _ = pair
    add_key(pair, 8, 41)
    ct = random_ct(orc, 17, level, level, batch)
    if largest:
        ct[:, 1] = np.array(orc.q[:level], dtype=np.uint64)[None, :, None] - 1
    d = to_dev(ct)
    out = torch.empty_like(d)
    ctx.rotate(d, out, batch, level, 41)
    got = to_host(out)
    for b in range(batch):
        assert np.array_equal(got[b], orc.rotate(ct[b], 41))
