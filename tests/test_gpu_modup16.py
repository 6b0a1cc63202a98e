"""ModUp fused with the first pass of the N = 2^16 forward transform: every digit shape of the ring (full and partial last
digits, one to four source limbs), with random residues and with the largest conversion sums, through a rotation; and the same on
the prime sets next to 2^50, where the range of the converted sums is tightest."""
import numpy as np
import pytest

from gpu_util import add_key, ctx_pair, random_ct, to_dev, to_host
import fesc_synth as S
from test_modup_bound import SETS

pytestmark = pytest.mark.gpu


def extreme_c1(orc, level, seed):
    """EVAL rows whose digits have y_a = d_a (Q_j / q_a)^-1 next to 0 or next to q_a, independently per limb and coefficient: the sums
    against every sign pattern of the centred constants.  (The signs a rotation brings exchange the two ends.)"""
    g, rows = np.random.default_rng(seed), np.empty((level, orc.N), dtype=np.uint64)
    for first in range(0, level, orc.alpha):
        digit = range(first, min(first + orc.alpha, level))
        for a in digit:
            q, y = orc.q[a], g.integers(0, 4, orc.N)
            m = int(np.prod([orc.q[b] % q for b in digit if b != a], dtype=object)) % q
            ends = np.array([v * m % q for v in range(4)] + [(q - 1 - v) * m % q for v in range(4)], dtype=np.uint64)
            rows[a] = ends[y + 4 * g.integers(0, 2, orc.N)]
    return orc.ntt(rows, list(range(level)))


def check_rotation(pair, key, level, batch, largest):
    import torch

    ctx, orc, _ = pair
    ct = random_ct(orc, 17, level, level, batch)
    if largest:
        ct[0, 1] = extreme_c1(orc, level, level)
    d = to_dev(ct)
    out = torch.empty_like(d)
    ctx.rotate(d, out, batch, level, key)
    got = to_host(out)
    for b in range(batch):
        assert np.array_equal(got[b], orc.rotate(ct[b], key)), b


@pytest.mark.parametrize("level,batch,largest", [(1, 1, False), (2, 3, True), (3, 1, True), (4, 2, False), (5, 1, True), (11, 1, False), (24, 1, True)])
def test_rotation_at_every_digit_shape(level, batch, largest):
    pair = ctx_pair("full")
    add_key(pair, 8, 41)
    check_rotation(pair, 41, level, batch, largest)


@pytest.mark.parametrize("name,n_q,n_p,dnum", [("largest", 24, 4, 6), ("next", 24, 4, 6), ("found", 8, 4, 2), ("spread", 8, 3, 2),
                                               ("largest", 3, 1, 3), ("largest", 4, 2, 2)])
def test_rotation_on_primes_next_to_the_limit(name, n_q, n_p, dnum):
    import paper_2608_17442_b200 as fesc
    from oracle.ckks import Oracle

    data = (SETS[name] + S.ntt_primes(50, 16, 27, 0)[24:])[:n_q]
    args = (16, data + S.ntt_primes(60, 16, n_p, 0), n_q, n_p, dnum, 77)
    pair = (fesc.Context(*args), Oracle(*args), None)
    add_key(pair, 8, 41)
    check_rotation(pair, 41, n_q, 2, True)
