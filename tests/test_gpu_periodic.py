"""Accumulate for periodic diagonals on tcgen05: first and last rows of an output tile, one and several tiles of token blocks, first and
last k-step, shortest run, both kinds of primes, largest sums."""
import numpy as np
import pytest

from gpu_util import ctx_pair, to_dev, to_host
import fesc_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,tbs,gin,nout,shift", [("small", 1, 1, 64, 4), ("small", 5, 33, 130, 5), ("small", 4, 192, 128, 7),
                                                    ("wide", 3, 160, 65, 4)])
def test_periodic_accumulate(name, tbs, gin, nout, shift):
    import torch
    import paper_2608_17442_b200 as fesc

    ctx, orc, p = ctx_pair(name)
    level, N, n = 2, orc.N, orc.N >> shift
    q = np.array(orc.q[:level], dtype=np.uint64)[:, None]
    cts = np.stack([S.uniform_residues_np(p["seed"], 70000 + i, orc.q[:level], N) for i in range(tbs * gin * 2)])
    cts = cts.reshape(tbs, gin, 2, level, N)
    w = np.stack([S.uniform_residues_np(p["seed"], 90000 + i, orc.q[:level], n) for i in range(nout * gin)]).reshape(nout, 1, gin, 1, level, n)
    cts[0], w[nout - 1, 0] = q - 1, q - 1                # the largest sums
    desc = fesc.BsgsDesc(1, 1, gin, nout, tbs, level, 0, 0, 0, 0, 1, shift)
    image = torch.empty((ctx.linear_packed_bytes(desc),), dtype=torch.uint8, device="cuda")
    ctx.linear_pack_diags(to_dev(w.reshape(nout, gin, 1, level, n)), desc, 0, nout, image)
    out = torch.empty((tbs, nout, 2, level - 1, N), dtype=torch.int64, device="cuda")
    ctx.linear(to_dev(cts), image, desc, out)
    ctx.sync()
    got = to_host(out)
    for b in sorted({0, 1, 8, 63, nout // 2, nout - 2, nout - 1}):       # every output is a sum of its own
        full = np.repeat(w[b:b + 1], 1 << shift, axis=-1)
        assert np.array_equal(got[:, b:b + 1], orc.linear(cts, full, dict(n1=1, n2=1), {}, {})), (name, b)
