"""Buffers need the alignment of their words only: the pair-wise loads and stores must take inputs and results that start on an odd word."""
import pytest

from gpu_util import add_key, ctx_pair, random_ct, to_dev

pytestmark = pytest.mark.gpu


def _odd(t):
    import torch

    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    buf[1:].copy_(t.reshape(-1))
    assert buf[1:].data_ptr() % 16 == 8
    return buf[1:]


@pytest.mark.parametrize("name", ["full", "small"])
def test_inputs_on_an_odd_word(name):
    import torch
    import paper_2608_17442_b200 as fesc

    pair = ctx_pair(name)
    ctx, orc, _ = pair
    level, N = 4, orc.N
    add_key(pair, 3, 640)
    add_key(pair, -5, 641)
    ct, pt = to_dev(random_ct(orc, 41, 0, level, 1)), to_dev(random_ct(orc, 42, 0, level, 1)[0])
    factor = to_dev(random_ct(orc, 43, 0, level, 1))
    conv, norm = fesc.ConvDesc(1, N // 2, 1, 1, level, 7800000), fesc.NormDesc(N // 2, 1, 1, level, 7800000)
    calls = [
        (2 * level, lambda out, *a: ctx.rotate(a[0], out, 1, level, 640)),
        (4 * level, lambda out, *a: ctx.rotate_hoisted(a[0], out, 1, level, [640, 641])),
        (2 * level, lambda out, *a: ctx.rotate_sum_hoisted(a[0], out, 1, level, [640, 641])),
        (2 * level, lambda out, *a: ctx.ct_ct_mul(a[0], a[2], out, 1, level)),
        (2 * (level - 1), lambda out, *a: ctx.conv(a[0], a[1][: level * N], a[1][level * N :], conv, out)),
        (2 * (level - 2), lambda out, *a: ctx.norm_scale(a[0], a[2], a[1][: (level - 1) * N], norm, out)),
    ]
    args = [t.reshape(-1) for t in (ct, pt, factor)]
    for i, (rows, call) in enumerate(calls):
        want, got = (torch.zeros(rows * N, dtype=torch.int64, device="cuda") for _ in range(2))
        call(want, *args)
        call(got, *(_odd(t) for t in args))
        ctx.sync()
        assert torch.equal(got, want) and bool(got.any()), (name, i)


@pytest.mark.parametrize("name,level", [("full", 3), ("full52", 2), ("small", 3)])
def test_rescale_transforms_and_results_on_an_odd_word(name, level):
    import torch
    import paper_2608_17442_b200 as fesc

    pair = ctx_pair(name)
    ctx, orc, _ = pair
    N = orc.N
    add_key(pair, 3, 640)
    add_key(pair, -5, 641)
    ct = to_dev(random_ct(orc, 44, 0, level, 1)).reshape(-1)
    pt = to_dev(random_ct(orc, 45, 0, level, 1)).reshape(-1)[: level * N]
    lin = fesc.BsgsDesc(1, 1, 1, 1, 1, level, 0, 0)
    calls = [
        (2 * (level - 1), lambda out, c, p: ctx.rescale(c, out, 1, level)),
        (2 * (level - 1), lambda out, c, p: ctx.rescale_static(c, out, 1, level)),
        (2 * level, lambda out, c, p: ctx.rotate(c, out, 1, level, 640)),
        (4 * level, lambda out, c, p: ctx.rotate_hoisted(c, out, 1, level, [640, 641])),
        (2 * level, lambda out, c, p: ctx.rotate_sum_hoisted(c, out, 1, level, [640, 641])),
        (2 * level, lambda out, c, p: ctx.ct_ct_mul(c, c, out, 1, level)),
        (2 * (level - 1), lambda out, c, p: ctx.norm_square(c, out, 1, level)),
        (2 * (level - 1), lambda out, c, p: ctx.linear(c, p, lin, out)),
        (2 * level, lambda out, c, p: (out.copy_(c), ctx.ntt(out, 2, 0, level))),
        (2 * level, lambda out, c, p: (out.copy_(c), ctx.intt(out, 2, 0, level))),
    ]
    for i, (rows, call) in enumerate(calls):
        want, got = torch.zeros(rows * N, dtype=torch.int64, device="cuda"), torch.zeros(rows * N + 2, dtype=torch.int64, device="cuda")
        call(want, ct, pt)
        call(got[1:-1], _odd(ct), _odd(pt))
        ctx.sync()
        assert torch.equal(got[1:-1], want) and bool(want.any()) and not got[0] and not got[-1], (name, i)


def test_a_packed_image_off_its_boundary_is_refused():
    import torch
    import paper_2608_17442_b200 as fesc

    ctx, orc, _ = ctx_pair("small")
    level, N = 2, orc.N
    ct = to_dev(random_ct(orc, 46, 0, level, 1))
    desc = fesc.BsgsDesc(1, 1, 1, 1, 1, level, 0, 0, 0, 0, 1, 0)
    image = torch.zeros((ctx.linear_packed_bytes(desc) + 16,), dtype=torch.uint8, device="cuda")
    out = torch.empty((2 * (level - 1) * N,), dtype=torch.int64, device="cuda")
    with pytest.raises(fesc.FescError):
        ctx.linear_pack_diags(ct.reshape(-1)[: level * N], desc, 0, 1, image[8:])
    with pytest.raises(fesc.FescError):
        ctx.linear(ct, image[8:], desc, out)
