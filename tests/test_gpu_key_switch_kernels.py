"""Key switches over the sizes of special primes (N = 2^16) and sums over many products."""
import numpy as np
import pytest

import fesc_synth as S
from gpu_util import add_key, random_ct, to_dev, to_host

pytestmark = pytest.mark.gpu


def _pair(bits, n_p):
    import paper_2608_17442_b200 as fesc
    from oracle.ckks import Oracle

    args = (16, S.ntt_primes(50, 16, 5, 0) + S.ntt_primes(bits, 16, n_p, 0), 5, n_p, 2, 61)
    return fesc.Context(*args), Oracle(*args), None


@pytest.mark.parametrize("bits,n_p", [(60, 4), (55, 2), (51, 1), (61, 2), (49, 4), (40, 2)])
def test_key_switches_by_size_of_the_special_primes(bits, n_p):
    """Special primes next to 2^60 and next to 2^51 from below, 61 bits, which the fused division does not take, and 49 and 40 bits, whose rows
    (and key words) are FP64 rows like the data primes': their keys, their transforms at the ends of the range, a relinearisation, a
    rotation, hoisted rotations and their sum."""
    import torch

    pair = _pair(bits, n_p)
    ctx, orc, _ = pair
    for k, rot in enumerate((3, -8, 4096)):
        add_key(pair, rot, 70 + k)
    assert np.array_equal(to_host(ctx.export_key(71)), orc.keys[71][1])      # kept in another form, handed out as residues
    idx = list(range(5, 5 + n_p))
    rows = np.empty((2, n_p, orc.N), dtype=np.uint64)
    for k, i in enumerate(idx):
        rows[0, k] = orc.q[i] - 1
        rows[1, k] = np.where((np.arange(orc.N) * 2654435761 >> 7) % 3 == 0, 0, orc.q[i] // 2 + 1)
    for gpu, ref in ((ctx.ntt, orc.ntt), (ctx.intt, orc.intt)):
        d = to_dev(rows)
        gpu(d, 2, 5, n_p)
        got = to_host(d)
        for b in range(2):
            assert np.array_equal(got[b], ref(rows[b], idx))
    ct, ids = random_ct(orc, 5, 5, 5, 3), [70, 71, 72]
    d, out = to_dev(ct), torch.empty((3, 3, 2, 5, orc.N), dtype=torch.int64, device="cuda")
    ctx.rotate(d, out[0], 3, 5, 71)
    ctx.rotate_sum_hoisted(d, out[1], 3, 5, ids)
    ctx.ct_ct_mul(d, d, out[2], 3, 5)
    got = to_host(out)
    for b in range(3):
        assert np.array_equal(got[0, b], orc.rotate(ct[b], 71))
        assert np.array_equal(got[1, b], orc.rotate_sum_hoisted(ct[b], ids))
        assert np.array_equal(got[2, b], orc.ct_ct_mul(ct[b], ct[b]))
    ctx.rotate_hoisted(d, out, 3, 5, ids)
    got = to_host(out)
    for b in range(3):
        assert np.array_equal(got[:, b], np.stack(orc.rotate_hoisted(ct[b], ids)))


@pytest.mark.parametrize("batch,n_keys", [(2, 8), (4, 3), (1, 7)])
def test_sums_that_are_reduced_in_between(batch, n_keys):
    """Six digits of one limb: up to 48 products per sum, and batches of one, two and four ciphertexts per thread."""
    import torch
    import paper_2608_17442_b200 as fesc
    from oracle.ckks import Oracle

    args = (16, S.ntt_primes(50, 16, 6, 0) + S.ntt_primes(60, 16, 1, 0), 6, 1, 6, 62)
    pair = (fesc.Context(*args), Oracle(*args), None)
    ctx, orc, _ = pair
    ids = [700 + k for k in range(n_keys)]
    for k, i in enumerate(ids):
        add_key(pair, 16 * k + 1, i)
    ct = random_ct(orc, 41, 6, 6, batch)
    ct[0] = (np.array(orc.q[:6], dtype=np.uint64) - np.uint64(1))[None, :, None]
    out = torch.empty_like(to_dev(ct))
    ctx.rotate_sum_hoisted(to_dev(ct), out, batch, 6, ids)
    got = to_host(out)
    for b in sorted({0, batch - 1}):
        assert np.array_equal(got[b], orc.rotate_sum_hoisted(ct[b], ids))


def _launches(ctx, call):
    before = ctx.counters()[4]
    call()
    return ctx.counters()[4] - before


def _boundaries(ctx, orc, lv, key_id, most):
    """Batches on both sides of every change of the number of launches of a rotation, the first and the last; launches by batch."""
    import torch

    d = torch.zeros((most, 2, lv, orc.N), dtype=torch.int64, device="cuda")
    out = torch.empty_like(d)
    n = [_launches(ctx, lambda: ctx.rotate(d, out, b, lv, key_id)) for b in range(1, most + 1)]
    return sorted({1, most} | {b + k for b in range(1, most) if n[b - 1] != n[b] for k in (0, 1)}), n


def _small_pair(name):
    """Contexts of the test's own: their scratch goes with them (a later test of the suite fills the device)."""
    import paper_2608_17442_b200 as fesc
    from oracle.ckks import Oracle

    if name == "2048":
        args = (11, S.ntt_primes(50, 11, 6, 0) + S.ntt_primes(60, 11, 2, 0), 6, 2, 3, 65)
    else:
        p = S.params(name)
        args = (p["log_n"], p["primes"], p["n_q"], p["n_p"], p["dnum"], p["seed"])
    return fesc.Context(*args), Oracle(*args), None


@pytest.mark.parametrize("name,levels", [("tiny", {3: (1, 4), 2: (1, 4), 1: (1, 4)}), ("2048", {6: (4, 4), 4: (1, 4), 1: (1, 4)}),
                                         ("small", {24: (4, 4), 8: (1, 4), 5: (1, 4), 1: (1, 1)})])
def test_small_rings_in_one_launch_and_in_four(name, levels):
    """Key switches of small rings run as one launch while their clusters fit the device and convert few rows each, as four beyond that: the
    launches of 1 and of 64 ciphertexts by level, and the oracle's words on either side of every change."""
    import torch

    pair = _small_pair(name)
    ctx, orc, _ = pair
    add_key(pair, 5, 91)
    for lv, ends in levels.items():
        batches, launches = _boundaries(ctx, orc, lv, 91, 64)
        assert (launches[0], launches[-1]) == ends and set(launches) <= {1, 4}, (lv, launches)
        for batch in batches:
            ct = random_ct(orc, 51, lv, lv, batch)
            d, out = to_dev(ct), torch.empty((2, batch, 2, lv, orc.N), dtype=torch.int64, device="cuda")
            assert _launches(ctx, lambda: ctx.rotate(d, out[0], batch, lv, 91)) == launches[batch - 1]
            assert _launches(ctx, lambda: ctx.ct_ct_mul(d, d, out[1], batch, lv)) == 1 + launches[batch - 1]
            got = to_host(out)
            for b in sorted({0, batch // 2, batch - 1}):
                assert np.array_equal(got[0, b], orc.rotate(ct[b], 91)), (lv, batch, b)
                assert np.array_equal(got[1, b], orc.ct_ct_mul(ct[b], ct[b])), (lv, batch, b)


@pytest.mark.parametrize("log_n", [10, 11, 12])
def test_one_digit_of_more_limbs_than_the_level_and_the_special_primes(log_n):
    """Levels below the digit's size: every converted row belongs to the one digit there is."""
    import torch
    import paper_2608_17442_b200 as fesc
    from oracle.ckks import Oracle

    args = (log_n, S.ntt_primes(45, log_n, 4, 0) + S.ntt_primes(60, log_n, 1, 0), 4, 1, 1, 66)
    pair = (fesc.Context(*args), Oracle(*args), None)
    ctx, orc, _ = pair
    add_key(pair, 3, 92)
    for lv in (1, 2, 3, 4):
        ct = random_ct(orc, 52, lv, lv, 2)
        d, out = to_dev(ct), torch.empty((2, 2, lv, orc.N), dtype=torch.int64, device="cuda")
        assert _launches(ctx, lambda: ctx.rotate(d, out, 2, lv, 92)) == 1
        got = to_host(out)
        for b in range(2):
            assert np.array_equal(got[b], orc.rotate(ct[b], 92)), (lv, b)


@pytest.mark.parametrize("bits", [50, 55])
@pytest.mark.parametrize("log_n", [10, 11, 12])
def test_small_ring_transforms_and_rescale_at_the_ends_of_the_range(log_n, bits):
    """Rings with one, two and three stages after the rounds of three: transforms of the largest words and of words 0, (q +- 1)/2 and q - 1, and
    rescales of one CTA per SM and of several."""
    import torch
    import paper_2608_17442_b200 as fesc
    from oracle.ckks import Oracle

    args = (log_n, S.ntt_primes(bits, log_n, 3, 0) + S.ntt_primes(60, log_n, 1, 0), 3, 1, 3, 67)
    ctx, orc = fesc.Context(*args), Oracle(*args)
    at = np.arange(orc.N)
    rows = np.empty((3, 4, orc.N), dtype=np.uint64)
    for i, q in enumerate(orc.q):
        words = np.array([0, (q - 1) // 2, (q + 1) // 2, q - 1], dtype=np.uint64)
        rows[0, i] = q - 1
        rows[1, i] = words[(at * 2654435761 >> 7) % 4]
        rows[2, i] = np.where(at % 2 == 0, (q - 1) // 2, (q + 1) // 2)
    for gpu, ref in ((ctx.ntt, orc.ntt), (ctx.intt, orc.intt)):
        d = to_dev(rows)
        gpu(d, 3, 0, 4)
        got = to_host(d)
        for b in range(3):
            assert np.array_equal(got[b], ref(rows[b], list(range(4)))), b
    for batch in (1, 37, 150):      # 4, 148 and 600 CTAs
        ct = np.ascontiguousarray(np.broadcast_to(rows[:2, :3], (batch, 2, 3, orc.N)))
        ct[-1] = rows[1:, :3]
        out = torch.empty((batch, 2, 2, orc.N), dtype=torch.int64, device="cuda")
        ctx.rescale(to_dev(ct), out, batch, 3)
        got = to_host(out)
        for b in sorted({0, batch // 2, batch - 1}):
            assert np.array_equal(got[b], orc.rescale(ct[b])), (batch, b)


def test_steps_of_a_small_key_switch_are_timed_apart():
    """While the families of a key switch are timed, it runs as its four steps, one record each."""
    import torch

    pair = _small_pair("tiny")
    ctx, orc, _ = pair
    add_key(pair, 5, 91)
    ct = random_ct(orc, 53, 3, 3, 1)
    d, out = to_dev(ct), torch.empty((1, 2, 3, orc.N), dtype=torch.int64, device="cuda")
    families = ("ntt", "modup", "inner", "moddown")
    ctx.profile_enable(families, 64)
    try:
        ctx.rotate(d, out, 1, 3, 91)
        read = ctx.profile_read()
    finally:
        ctx.profile_enable(())
    assert [read[f][1] for f in families] == [1, 1, 1, 1]
    assert np.array_equal(to_host(out)[0], orc.rotate(ct[0], 91))
    assert _launches(ctx, lambda: ctx.rotate(d, out, 1, 3, 91)) == 1


@pytest.mark.parametrize("bits", [36, 50, 51, 55])
def test_products_of_the_largest_words(bits):
    """Products with relinearisation on both sides of 2^50, where FP64 products end: words 0, 1, (q +- 1)/2, q - 2 and q - 1 against each other."""
    import torch
    import paper_2608_17442_b200 as fesc
    from oracle.ckks import Oracle

    args = (12, S.ntt_primes(bits, 12, 3, 0) + S.ntt_primes(60, 12, 1, 0), 3, 1, 3, 63)
    ctx, orc = fesc.Context(*args), Oracle(*args)
    ct = np.empty((2, 2, 3, orc.N), dtype=np.uint64)
    at = np.arange(orc.N)
    for l in range(3):
        q = orc.q[l]
        words = np.array([0, 1, (q - 1) // 2, (q + 1) // 2, q - 2, q - 1], dtype=np.uint64)
        for k in range(4):
            ct[k // 2, k % 2, l] = words[at // 6**k % 6]
    out = torch.empty((2, 2, 3, orc.N), dtype=torch.int64, device="cuda")
    a, b = to_dev(ct), to_dev(ct[::-1].copy())
    ctx.ct_ct_mul(a, b, out[:1], 1, 3)
    ctx.ct_ct_mul(a, a, out[1:], 1, 3)
    got = to_host(out)
    assert np.array_equal(got[0], orc.ct_ct_mul(ct[0], ct[1]))
    assert np.array_equal(got[1], orc.ct_ct_mul(ct[0], ct[0]))


def test_threads_with_contexts_of_their_own():
    """Hoisted rotations of 1 and of 16 ciphertexts from two threads at a time: kernels whose shared memory depends on the call."""
    import threading

    import torch
    import paper_2608_17442_b200 as fesc

    args = (16, S.ntt_primes(50, 16, 8, 0) + S.ntt_primes(60, 16, 4, 0), 8, 4, 2, 64)
    errors, results = [], {}
    go = threading.Barrier(2)

    def work(batch):
        try:
            torch.cuda.set_device(0)
            with torch.cuda.stream(torch.cuda.Stream()):
                ctx = fesc.Context(*args)
                for k in (1, 2):
                    ctx.add_galois_key(k, k)
                ct = torch.arange(batch * 2 * 8 << 16, dtype=torch.int64, device="cuda").view(batch, 2, 8, 1 << 16)
                out = torch.empty((2, batch, 2, 8, 1 << 16), dtype=torch.int64, device="cuda")
                go.wait(60)
                for _ in range(300 if batch == 16 else 3000):
                    ctx.rotate_hoisted(ct, out, batch, 8, [1, 2])
                ctx.sync()
                results[batch] = out[:, 0].cpu()
        except Exception as e:      # reported by the test, not by the thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(b,)) for b in (1, 16)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.empty_cache()
    assert not errors, errors
    assert torch.equal(results[1], results[16])       # the first ciphertext of both batches is the same
