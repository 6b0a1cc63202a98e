"""Performance cases of the RNS-CKKS library: the work an encrypted Mamba-2 layer has it do, through its public calls.

Every case names a `kind` (below) and its sizes.  Inputs are residues drawn from a counter hash: ciphertext words, switching
keys and encoded plaintexts are all uniform below their primes in real use, so the values and the distributions are those
the kernels meet in earnest.  Contexts, switching keys and packed weights are what a program keeps; they are made in
`prepare`.  Outputs are whole residues and have to be equal to the last bit.

  tiny      plaintext product, then rotations by +1 and +5, on the ring N = 2^12 (3 primes of 36 bits)
  ntt       forward transform of one batch of polynomials and inverse transform of another
  rotate    plain rotations of a batch, one call per key
  hoisted   rotations that share one decomposition, each result returned (sum = False) or added up (sum = True)
  square    ciphertext product, relinearisation, rescale
  linear    plaintext-weight projection by baby and giant steps
  conv      causal depthwise convolution
  scale     per-token normalisation factor times per-channel weight
  scan      factorized scan-contract
"""
import math
import weakref

import torch

import fesc_synth as S
import paper_2608_17442_b200 as fesc

# "full" is the N = 2^16 ring of the layer: 24 primes of 50 bits, 4 special primes of 60 bits, digits of 4 limbs;
# "tiny" has N = 2^12, 3 primes and 1 special prime of 36 bits, digits of one limb
T_SEG = 128          # tokens per segment: a ciphertext of 32768 slots holds 128 tokens of 256 features
CHANNELS = 256


def listed():
    return [
        # smallest calls: four ciphertexts of the tiny ring, a product and two rotations (latency, launches)
        dict(name="tiny_product_rotations", kind="tiny", batch=4),
        # the transform sweep: 64 polynomials of 24 limbs in each direction
        dict(name="ntt_64x24", kind="ntt", batch=64, limbs=24),
        # one ciphertext, one rotation: what an interactive caller waits for
        dict(name="rotate_one", kind="rotate", batch=1, limbs=24, keys=1),
        # a batch of 32 ciphertexts by several amounts (baby and giant steps of a projection)
        dict(name="rotate_32x4", kind="rotate", batch=32, limbs=24, keys=4),
        # a rotate-and-add step of a broadcast chain in the middle of the modulus chain, odd batch
        dict(name="rotate_sum_5x3", kind="hoisted", batch=5, limbs=15, keys=3, sum=True),
        # squares before the normalisation: two token blocks of six channel blocks, part of the limbs used up
        dict(name="square_12", kind="square", batch=12, limbs=17),
        # projection 768 -> 512 of 2048 tokens with weights packed offline
        dict(name="linear_packed", kind="linear", token_blocks=16, in_blocks=3, out_blocks=2, n1=32, n2=8, limbs=24,
             hoist=1, defer=1, packed=1, period=0),
        # in_proj, 768 -> 3352 for 1024 tokens, in the token-major packing (periodic diagonals)
        dict(name="linear_token_major", kind="linear", token_blocks=8, in_blocks=3, out_blocks=14, n1=63, n2=15, limbs=24,
             hoist=1, defer=1, packed=1, period=7),
        # a short request low in the modulus chain: one token block, weights as residues, plain rotations
        dict(name="linear_residues", kind="linear", token_blocks=1, in_blocks=2, out_blocks=3, n1=16, n2=16, limbs=9,
             hoist=0, defer=0, packed=0, period=0),
        # the convolution of a layer: 1792 channels, 2048 tokens, four taps
        dict(name="conv_layer", kind="conv", token_blocks=16, blocks=7, taps=4, limbs=24),
        # the scaling after the normalisation: 1536 channels, 1024 tokens
        dict(name="scale_8x6", kind="scale", token_blocks=8, blocks=6, limbs=21),
        # one state chunk (2 heads) over one block of 256 tokens, the setting a layer runs
        dict(name="scan_chunk", kind="scan", tokens=256, heads=2, block=256, limbs=24, group=4, plain=0),
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], spread evenly over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["tiny", "ntt", "rotate", "hoisted", "square", "linear", "linear", "conv", "scale", "scan"])
    if kind == "tiny":
        return dict(kind=kind, batch=_log_int(rng, 1, 200))
    if kind == "ntt":
        return dict(kind=kind, batch=_log_int(rng, 1, 96), limbs=rng.randint(1, 24))
    if kind == "rotate":
        return dict(kind=kind, batch=_log_int(rng, 1, 40), limbs=rng.randint(2, 24), keys=rng.randint(1, 4))
    if kind == "hoisted":
        return dict(kind=kind, batch=_log_int(rng, 1, 24), limbs=rng.randint(2, 24), keys=rng.randint(1, 8),
                    sum=rng.random() < 0.5)
    if kind == "square":
        return dict(kind=kind, batch=_log_int(rng, 1, 48), limbs=rng.randint(2, 24))
    if kind == "linear":
        packed, split = rng.random() < 0.7, rng.choice([(32, 8), (16, 16), (63, 15), (31, 31)])
        period = 7 if packed and split[0] % 2 else 0
        if not period:
            split = rng.choice([(32, 8), (16, 16)])
        blocks, limbs = rng.randint(1, 3), rng.randint(4, 24)
        small = dict(in_blocks=blocks, out_blocks=rng.randint(1, 4 if period else 3), n1=split[0], n2=split[1])
        # plain rotations and separate divisions cost several times more per token block
        plain = rng.random() < 0.3
        return dict(kind=kind, token_blocks=_log_int(rng, 1, 16 if packed and not plain else 3),
                    limbs=limbs if packed else min(limbs, 12), hoist=int(not plain), defer=int(not plain), packed=int(packed),
                    period=period, **small)
    if kind == "conv":
        return dict(kind=kind, token_blocks=_log_int(rng, 1, 16), blocks=rng.randint(1, 7), taps=rng.randint(2, 4),
                    limbs=rng.randint(3, 24))
    if kind == "scale":
        return dict(kind=kind, token_blocks=_log_int(rng, 1, 16), blocks=rng.randint(1, 6), limbs=rng.randint(3, 24))
    block = rng.choice([32, 64, 128, 256])
    # a chunk holds 2 heads at the stride of 256 slots, 4 heads at 128
    heads = 2 if block == 256 else 4 * rng.randint(1, 2)
    lowest = 6 + 2 * int(math.log2(block))          # the levels the schedule uses, one left for the result
    return dict(kind=kind, tokens=block - rng.randrange(block // 4), heads=heads, block=block, limbs=rng.randint(lowest, 24),
                group=rng.choice([2, 4, 8]), plain=int(rng.random() < 0.4))


# ---------------------------------------------------------------------------------------------
# contexts and inputs
# ---------------------------------------------------------------------------------------------
_contexts = weakref.WeakValueDictionary()     # a context lives as long as a state uses it


def _context(params, amounts):
    """A context with Galois keys for `amounts`, (slot rotation, key id) pairs; shared by the states that need the same."""
    key = (params, tuple(amounts))
    ctx = _contexts.get(key)
    if ctx is None:
        p = S.params(params)
        ctx = fesc.Context(p["log_n"], p["primes"], p["n_q"], p["n_p"], p["dnum"], p["seed"])
        for rot, key_id in amounts:
            ctx.add_galois_key(rot, key_id)
        _contexts[key] = ctx
    return ctx


def _residues(ctx, seed, stream, limbs, *shape):
    """[*shape, limbs, words] residues: row i below prime i.  The last entry of `shape` is the words per limb."""
    *lead, words = shape
    r = S.hashed_residues(seed, stream, ctx.primes[:limbs], math.prod(lead) * words, device="cuda")
    return r.view(limbs, *lead, words).movedim(0, -2).contiguous()


def _empty(*shape):
    return torch.empty(shape, dtype=torch.int64, device="cuda")


def _scan_amounts(n, P, d_s, block, stride, group):
    """Left slot rotations of a scan with hoisted rotate-and-add chains and leaves built in groups (see include/fesc.h)."""
    log2 = lambda v: int(math.log2(v))
    seg = block // max(1, block // stride)               # tokens per segment
    dg, dgs = min(16, block), min(16, seg)
    c_state, R, am = n // stride, P * stride, set()
    chain = lambda unit, steps: ({unit * (1 << b) for b in range(steps)} |
                                 {3 * unit * (1 << b) for b in range(0, steps - 1, 2)})
    digits = lambda unit, count: ({unit * t for t in range(1, min(16, count))} |
                                  {unit * min(16, count) * t for t in range(1, count // min(16, count))})
    for unit in (1, P):                                  # offsets of x and a inside a segment
        am |= digits(unit, seg) | digits(group * unit, seg // group)
    am |= digits(d_s, block) | digits(group * d_s, block // group)
    am |= {-t for t in range(1, dgs)} | {-dgs * t for t in range(1, seg // dgs)}
    am |= chain(-1, log2(max(d_s, P))) | chain(-1, log2(P)) | chain(-1, log2(d_s)) | chain(1, log2(d_s))
    am |= chain(-P, log2(R // P)) | chain(-stride, log2(c_state))
    am |= chain(-group, log2(d_s // group)) | chain(-group * P, log2(R // (group * P)))
    am |= chain(-group * d_s, log2(n // (group * d_s)))
    for unit in (1, P, d_s):                             # class shifts inside a group
        am |= {k * unit for k in range(1, group)} | {-k * unit for k in range(1, group)}
    return sorted({a % n for a in am} - {0})


def _scan_shape(case):
    n, block = 1 << 15, case["block"]
    stride = max(128, block)
    l1 = case["limbs"] - 3
    linj = l1 - 2 * int(math.log2(block)) + 1
    return n, stride, case["heads"] * 64 // (n // stride), linj


def _prepare_scan(case, seed):
    n, stride, chunks, linj = _scan_shape(case)
    block, l0, G, base, P, d_s = case["block"], case["limbs"], case["group"], 100000, 64, 128
    amounts = [(r, base + r) for r in _scan_amounts(n, P, d_s, block, stride, G)] + [(fesc.CONJ, base + n)]
    ctx = _context("full", amounts)
    N, log_b = ctx.N, int(math.log2(block))
    one = lambda stream, limbs, *lead: _residues(ctx, seed, stream, limbs, *lead, N)
    s = dict(ctx=ctx, x=one(1, l0, 1, chunks, 1, 2), mask_x=one(5, l0), mask_out=one(8, linj - 2),
             adj=[(1 << 49) + 12345 * i for i in range((l0 + 1) ** 2)], out=_empty(1, chunks, 1, 2, linj - 3, N))
    s["groups"] = [one(9, l0), one(10, l0), one(11, l0 - 1, G), one(12, l0 - 1, G), one(13, l0), one(14, l0 - 1, G)]
    if case["plain"]:        # plaintext decay, input and output factors, one level per row at a pitch of l0 limbs
        s["plain"] = [one(15, l0 - 2), one(16, linj - 1), one(17, l0, log_b), one(18, l0, max(1, log_b - 1)), one(19, l0, 1),
                      one(20, linj, block)]
        s.update(a=None, B=None, C=None, mask_b=None, mask_a=None)
    else:
        s.update(plain=None, a=one(2, l0, 1, chunks, 1, 2), B=one(3, l0, 1, 2), C=one(4, l0, 1, 2), mask_b=one(6, l0),
                 mask_a=one(7, l0))
    s["desc"] = fesc.ScanDesc(case["tokens"], case["heads"], P, d_s, block, stride, l0, base, 1, fesc.NET_BRENT_KUNG, G,
                              case["plain"])
    return s


def _prepare_linear(case, seed):
    tbs, gin, nout, n1, n2, limbs, s = (case[k] for k in ("token_blocks", "in_blocks", "out_blocks", "n1", "n2", "limbs", "period"))
    # amounts in units of tokens (segment packing) or of features with their wrap twins (token-major packing)
    if s:
        h1 = (n1 + 1) // 2
        baby = list(range(1, h1)) + [q - CHANNELS for q in range(1, h1)]
        giant = [p * h1 for p in range(1, (n2 + 1) // 2)]
        giant += [g - CHANNELS for g in giant]
    else:
        baby, giant = [q * T_SEG for q in range(1, n1)], [p * n1 * T_SEG for p in range(1, n2)]
    ctx = _context("full", [(r, 1001 + i) for i, r in enumerate(baby)] + [(r, 2001 + i) for i, r in enumerate(giant)])
    N, pairs = ctx.N, nout * n2
    desc = fesc.BsgsDesc(n1, n2, gin, nout, tbs, limbs, 1000, 2000, case["hoist"], case["defer"], case["packed"], s)
    if case["packed"]:       # the one-off preparation of the weights, eight (output, giant step) pairs at a time
        diags = torch.empty((ctx.linear_packed_bytes(desc),), dtype=torch.uint8, device="cuda")
        for first in range(0, pairs, 8):
            count = min(8, pairs - first)
            part = _residues(ctx, seed, 100 + first, limbs, count, gin, n1, N >> s)
            ctx.linear_pack_diags(part, desc, first, count, diags)
    else:
        diags = _empty(pairs, gin, n1, limbs, N)
        for i in range(pairs):
            diags[i] = _residues(ctx, seed, 100 + i, limbs, gin, n1, N)
    return dict(ctx=ctx, x=_residues(ctx, seed, 1, limbs, tbs, gin, 2, N), diags=diags, desc=desc,
                out=_empty(tbs, nout, 2, limbs - 1, N))


def prepare(case, seed):
    s = _prepare(case, seed)
    s["kind"], s["case"] = case["kind"], case
    return s


def _prepare(case, seed):
    kind = case["kind"]
    if kind == "scan":
        return _prepare_scan(case, seed)
    if kind == "linear":
        return _prepare_linear(case, seed)
    if kind == "tiny":
        ctx, b = _context("tiny", ((1, 1), (5, 2))), case["batch"]
        return dict(ctx=ctx, ct=_residues(ctx, seed, 1, 3, b, 2, ctx.N), pt=_residues(ctx, seed, 2, 3, b, ctx.N),
                    prod=_empty(b, 2, 3, ctx.N), r1=_empty(b, 2, 3, ctx.N), r5=_empty(b, 2, 3, ctx.N))
    if kind == "ntt":
        ctx = _context("full", ())
        return dict(ctx=ctx, coef=_residues(ctx, seed, 1, case["limbs"], case["batch"], ctx.N),
                    evals=_residues(ctx, seed, 2, case["limbs"], case["batch"], ctx.N))
    if kind in ("rotate", "hoisted"):
        b, l, k = case["batch"], case["limbs"], case["keys"]
        ctx = _context("full", tuple((r, r) for r in range(1, 9)))
        shape = (b, 2, l, ctx.N) if case.get("sum") else (k, b, 2, l, ctx.N)
        return dict(ctx=ctx, ct=_residues(ctx, seed, 1, l, b, 2, ctx.N), out=_empty(*shape), ids=list(range(1, k + 1)))
    if kind == "square":
        ctx, b, l = _context("full", ()), case["batch"], case["limbs"]
        return dict(ctx=ctx, ct=_residues(ctx, seed, 1, l, b, 2, ctx.N), out=_empty(b, 2, l - 1, ctx.N))
    tbs, blocks, l = case["token_blocks"], case["blocks"], case["limbs"]
    if kind == "conv":
        d = case["taps"]
        ctx = _context("full", tuple((-r, 3000 + r) for r in range(1, d)) + tuple((T_SEG - r, 3000 + d + r) for r in range(1, d)))
        return dict(ctx=ctx, ct=_residues(ctx, seed, 1, l, tbs, blocks, 2, ctx.N), bias=_residues(ctx, seed, 3, l, blocks, ctx.N),
                    masks=_residues(ctx, seed, 2, l, blocks, 2 * d - 1, ctx.N), out=_empty(tbs, blocks, 2, l - 1, ctx.N),
                    desc=fesc.ConvDesc(d, T_SEG, blocks, tbs, l, 3000))
    ctx = _context("full", tuple((-(T_SEG << b), 3500 + b) for b in range(8)))
    return dict(ctx=ctx, ct=_residues(ctx, seed, 1, l, tbs, blocks, 2, ctx.N), s=_residues(ctx, seed, 2, l, tbs, 2, ctx.N),
                gamma=_residues(ctx, seed, 3, l - 1, blocks, ctx.N), out=_empty(tbs, blocks, 2, l - 2, ctx.N),
                desc=fesc.NormDesc(T_SEG, blocks, tbs, l, 3500))


def run(s):
    ctx, kind, case = s["ctx"], s["kind"], s["case"]
    if kind == "tiny":
        s["prod"].zero_()
        ctx.ct_pt_mac(s["ct"], s["pt"], s["prod"], case["batch"], 3)
        ctx.rotate(s["prod"], s["r1"], case["batch"], 3, 1)
        ctx.rotate(s["prod"], s["r5"], case["batch"], 3, 2)
        return s["prod"], s["r1"], s["r5"]
    if kind == "ntt":
        ctx.ntt(s["coef"], case["batch"], 0, case["limbs"])
        ctx.intt(s["evals"], case["batch"], 0, case["limbs"])
        return s["coef"], s["evals"]
    if kind == "rotate":
        for k, key_id in enumerate(s["ids"]):
            ctx.rotate(s["ct"], s["out"][k], case["batch"], case["limbs"], key_id)
    elif kind == "hoisted":
        rotate = ctx.rotate_sum_hoisted if case["sum"] else ctx.rotate_hoisted
        rotate(s["ct"], s["out"], case["batch"], case["limbs"], s["ids"])
    elif kind == "square":
        ctx.norm_square(s["ct"], s["out"], case["batch"], case["limbs"])
    elif kind == "linear":
        ctx.linear(s["x"], s["diags"], s["desc"], s["out"])
    elif kind == "conv":
        ctx.conv(s["ct"], s["masks"], s["bias"], s["desc"], s["out"])
    elif kind == "scale":
        ctx.norm_scale(s["ct"], s["s"], s["gamma"], s["desc"], s["out"])
    else:
        ctx.scan_contract(s["x"], s["a"], s["B"], s["C"], s["desc"], s["mask_x"], s["mask_b"], s["mask_a"], s["mask_out"],
                          s["adj"], s["adj"], s["out"], s["groups"], s["plain"])
    return s["out"]


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without: every input, key and weight read once, every output written once; 2 operations per
# modular product of the transforms (N/2 log2 N), the basis conversions, the inner products and the plaintext products
# ---------------------------------------------------------------------------------------------
def _keys(level, N=1 << 16, K=4, alpha=4):
    """Words of one switching key at `level`."""
    return -(-level // alpha) * 2 * (level + K) * N


def _decompose(level, N=1 << 16, K=4, alpha=4):
    """Products of one decomposition: inverse transform, conversion of every digit, forward transforms."""
    digits, t = -(-level // alpha), N // 2 * (N.bit_length() - 1)
    other = digits * (level + K) - level
    return level * t + other * (t + alpha * N)


def _inner(level, N=1 << 16, K=4, alpha=4):
    return _keys(level, N, K, alpha)


def _divide(level, N=1 << 16, K=4):
    """Products of the division by the special modulus, both polynomials."""
    t = N // 2 * (N.bit_length() - 1)
    return 2 * (K * t + level * (t + K * N))


def _switch(level, *ring):
    return _decompose(level, *ring) + _inner(level, *ring) + _divide(level, *ring[:2])


def _rescale(level, N=1 << 16):
    return 2 * level * (N // 2 * (N.bit_length() - 1) + N)


def _words_and_products(case):
    """64-bit words that have to move and modular products of a pass."""
    kind, N = case["kind"], 1 << 16
    if kind == "tiny":
        b, n = case["batch"], 1 << 12
        return b * 3 * n * (2 + 1 + 3 * 2) + 2 * _keys(3, n, 1, 1), b * (6 * n + 2 * _switch(3, n, 1, 1))
    if kind == "ntt":
        rows = case["batch"] * case["limbs"]
        return 4 * rows * N, 2 * rows * N // 2 * 16
    if kind in ("rotate", "hoisted"):
        b, l, k = case["batch"], case["limbs"], case["keys"]
        shared = kind == "hoisted"
        outs = 1 if case.get("sum") else k
        products = b * (_decompose(l) * (1 if shared else k) + k * _inner(l) + outs * _divide(l))
        return (1 + outs) * b * 2 * l * N + k * _keys(l), products
    if kind == "square":
        b, l = case["batch"], case["limbs"]
        return b * 2 * (2 * l - 1) * N + _keys(l), b * (4 * l * N + _switch(l) + _rescale(l))
    if kind == "linear":
        tbs, gin, nout, n1, n2, l = (case[k] for k in ("token_blocks", "in_blocks", "out_blocks", "n1", "n2", "limbs"))
        weights = nout * n2 * gin * n1 * l * (N >> case["period"])
        words = tbs * gin * 2 * l * N + tbs * nout * 2 * (l - 1) * N + (n1 + n2 - 2) * _keys(l)
        baby = tbs * gin * ((_decompose(l) if case["hoist"] else (n1 - 1) * _decompose(l)) + (n1 - 1) * (_inner(l) + _divide(l)))
        giant = tbs * nout * ((n2 - 1) * (_decompose(l) + _inner(l)) + (1 if case["defer"] else n2 - 1) * _divide(l) + _rescale(l))
        return words + weights * (7 / 8 if case["packed"] else 1), baby + giant + tbs * nout * n2 * gin * n1 * 2 * l * N
    if kind == "conv":
        tbs, blocks, d, l = case["token_blocks"], case["blocks"], case["taps"], case["limbs"]
        words = tbs * blocks * 2 * (2 * l - 1) * N + 2 * d * blocks * l * N + (d - 1) * (2 if tbs > 1 else 1) * _keys(l)
        rotations, macs = (2 * tbs - 1) * (d - 1) * blocks, ((2 * tbs - 1) * (d - 1) + tbs) * blocks
        return words, tbs * blocks * (_decompose(l) + _rescale(l)) + rotations * (_inner(l) + _divide(l)) + macs * 2 * l * N
    if kind == "scale":
        tbs, blocks, l = case["token_blocks"], case["blocks"], case["limbs"]
        words = tbs * (blocks * 2 * (2 * l - 2) + 2 * l) * N + blocks * (l - 1) * N + 9 * _keys(l)
        return words, tbs * (8 * _switch(l) + blocks * (4 * l * N + _switch(l) + _rescale(l) + 2 * (l - 1) * N + _rescale(l - 1)))
    return _scan_work(case)


def _scan_work(case):
    """Inputs, outputs, masks and keys once; products of the rotations, compositions and contractions at their levels."""
    N = 1 << 16
    n, stride, chunks, linj = _scan_shape(case)
    l0, block, G = case["limbs"], case["block"], case["group"]
    log_b, amounts = int(math.log2(block)), len(_scan_amounts(n, 64, 128, block, stride, G)) + 1
    enc = 1 if case["plain"] else 2
    words = (chunks * enc + 2 * (enc - 1)) * 2 * l0 * N + chunks * 2 * (linj - 3) * N + (1 + 3 * G) * l0 * N + amounts * _keys(l0)
    groups = block // G
    fill = lambda steps, level: _decompose(level) * -(-steps // 2) + steps * _inner(level) + _divide(level) * -(-steps // 2)
    log2 = lambda v: int(math.log2(v))
    per_x = 3 * _switch(l0) + fill(log2(128 // G), l0 - 1) + 2 * (G - 1) * (_inner(l0 - 1) + _divide(l0 - 1))
    per_token = _rescale(l0 - 1)
    shared, chunk = 0, groups * per_x + block * per_token
    for s in range(1, log_b + 1):                # up-sweep stages
        level = l0 - 3 - (s - 1)
        chunk += (block >> s) * (_rescale(level) + (0 if case["plain"] else 2 * _switch(level) + _rescale(level)))
    for s in range(log_b - 1, 0, -1):            # down-sweep stages; the first block forms no prefix decays
        level = l0 - 3 - log_b - (log_b - 1 - s)
        chunk += ((block >> s) - 1) * (_rescale(level) + (0 if case["plain"] else _switch(level)))
    low = linj - 1
    chunk += block * (_rescale(low) + (0 if case["plain"] else _switch(low)) + fill(7, linj - 2) // 2 + _rescale(linj - 2))
    if not case["plain"]:
        chunk += groups * (2 * per_x) + block * per_token              # br(a)
        shared = groups * per_x + block * (per_token + fill(log2(n // 128), linj - 1))      # br(B), br(C)
    return words, shared + chunks * chunk


def work(case):
    words, products = _words_and_products(case)
    return {"bytes": 8.0 * words, "flops": 2.0 * products}


def tolerance(case):
    return "exact"          # residues below their primes: one right answer
