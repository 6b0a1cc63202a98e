"""The N = 2^16 transform kernels: both kinds of rows (primes below 2^50 in FP64, larger ones in integers) alone and in one
buffer, one row and several, with random residues and with residues at the ends of the range (the largest lazy values)."""
import numpy as np
import pytest

import fesc_synth as S
from gpu_util import ctx_pair, to_dev, to_host

pytestmark = pytest.mark.gpu


def _rows(orc, idx, kind, batch):
    if kind == "random":
        return np.stack([S.uniform_residues_np(9, b, [orc.q[i] for i in idx], orc.N) for b in range(batch)])
    out = np.empty((batch, len(idx), orc.N), dtype=np.uint64)
    for k, i in enumerate(idx):
        out[:, k] = orc.q[i] - 1
        if kind == "ends":              # 0 and q - 1 in a pattern that no transform stage is aligned with
            out[:, k, (np.arange(orc.N) * 2654435761 >> 7) % 3 == 0] = 0
    return out


@pytest.mark.parametrize("kind", ["random", "largest", "ends"])
@pytest.mark.parametrize("first,limbs,batch", [(0, 1, 1), (23, 2, 3), (24, 4, 1), (22, 6, 2)])
def test_rows_of_both_kinds(first, limbs, batch, kind):
    ctx, orc, _ = ctx_pair("full")
    idx = list(range(first, first + limbs))
    a = _rows(orc, idx, kind, batch)
    d = to_dev(a)
    ctx.ntt(d, batch, first, limbs)
    got = to_host(d)
    for b in range(batch):
        assert np.array_equal(got[b], orc.ntt(a[b], idx))
    d = to_dev(a)
    ctx.intt(d, batch, first, limbs)
    got = to_host(d)
    for b in range(batch):
        assert np.array_equal(got[b], orc.intt(a[b], idx))
