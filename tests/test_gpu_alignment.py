"""Inputs need the alignment of their words only: the pair-wise loads must take buffers that start on an odd word."""
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
