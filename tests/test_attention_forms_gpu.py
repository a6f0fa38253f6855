"""GPU parity of the two bf16 tensor-core attention forms at the edges of their tiles.

Prefill form (many rows over all heads): 128-row tiles, chunks of 96 keys (64 at hd 128) through a
ring, an output rescale when a row's max grows.  Decode form (up to 16 rows per head, or few row tiles
in all): 16-row tiles, keys split over warps and clusters.  Tolerance 1e-2 as in test_attention_gpu.py (bf16
probabilities and outputs, 2^-9 each, fp32 sums).
"""
import pytest
import torch

import oracle as O
import paper_2608_17616_gb300 as mone
import workloads as wk
from harness import DeviceRun, rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2608_17616_gb300 import build
    build.build()
    assert torch.cuda.is_available()
    mone.lib()


def run_case(group, Lq, n_mem, hd, n_layers=2, n_kv=2, late_scale=1.0):
    """late_scale: factor on the keys of the last third of the cache, so later chunks raise the row max."""
    d_out = max(256, 2 * n_kv * hd)
    wl = wk.Workload("attn_forms", 41, 1, n_layers, 256, 256, d_out, d_out // (2 * hd), hd, 128, 128, 8, "bf16", wk.PLAIN)
    run = DeviceRun(wl)
    n_kv, S = wl.n_kv_heads, n_mem + Lq
    g = torch.Generator(device="cuda").manual_seed(group * 1000 + Lq * 10 + n_mem + hd)
    K = torch.randn(1, n_layers, n_kv, S, hd, generator=g, device="cuda")
    K[..., 2 * S // 3:, :] *= late_scale
    K, V = K.bfloat16(), torch.randn(K.shape, generator=g, device="cuda").bfloat16()
    Q = torch.randn(1, n_layers, group * n_kv, Lq, hd, generator=g, device="cuda").bfloat16()
    out = torch.full_like(Q, 7.0)
    mone.mone_attention(run.h, Q, group * n_kv, Lq, K, V, K.stride()[:4], n_mem, out)
    mone.mone_mem_sync(run.h)
    run.close()
    for layer in sorted({0, n_layers // 2, n_layers - 1}):
        ref = O.attention(Q[0, layer].cpu(), K[0, layer].cpu(), V[0, layer].cpu(), n_mem)
        assert rel_fro(out[0, layer].float().cpu(), ref) <= 1e-2, layer


@pytest.mark.parametrize("group,Lq,n_mem,hd,late_scale", [
    (4, 200, 70, 64, 1.0),    # 32-token tiles, the last ragged
    (1, 300, 513, 64, 1.0),   # 128-token tiles; nine chunks, a ring wrap
    (2, 33, 1000, 64, 1.0),   # one tile of 66 rows over eleven chunks
    (64, 2, 94, 64, 1.0),     # the largest group: 2 tokens a tile; exactly one chunk of keys
    (64, 2, 95, 64, 1.0),     # one key past it
    (3, 150, 0, 128, 1.0),    # padded rows (126 of 128), no memory, hd 128
    (4, 129, 383, 128, 1.0),  # hd 128: 64-key chunks, eight of them exactly, one token past the tiles
    (4, 100, 300, 64, 9.0),   # the row max grows in later chunks: O is rescaled
    (2, 140, 200, 128, 9.0),
])
def test_prefill_form(group, Lq, n_mem, hd, late_scale):
    run_case(group, Lq, n_mem, hd, n_layers=20, late_scale=late_scale)


def strided(kind, n_ctx, L, n_kv, S, hd, g):
    """A [n_ctx, L, n_kv, S, hd] cache with the strides of `kind`."""
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()  # noqa: E731
    if kind == "dense":
        return rn(n_ctx, L, n_kv, S, hd)
    if kind == "padded":  # rows of a wider buffer, spare positions after the last key
        return rn(n_ctx, L, n_kv, S + 37, hd + 24)[..., :S, :hd]
    if kind == "heads inner":  # [position][head]
        return rn(n_ctx, L, S, n_kv, hd).transpose(2, 3)
    if kind == "layers inner":  # [head][position][layer]
        return rn(n_ctx, n_kv, S, L, hd).permute(0, 3, 1, 2, 4)
    one = dict(zip(("context", "layer", "head"), range(3)))
    shape = [n_ctx, L, n_kv, S, hd]
    for name in kind.split("+"):  # shared by every context, layer or head
        shape[one[name]] = 1
    return rn(*shape).expand(n_ctx, L, n_kv, S, hd)


@pytest.mark.parametrize("kind", ["dense", "padded", "heads inner", "layers inner", "context", "layer", "head",
                                  "context+layer", "layer+head", "context+layer+head"])
@pytest.mark.parametrize("n_ctx,group,Lq,n_mem,hd", [(2, 2, 150, 200, 64), (3, 4, 70, 130, 128), (2, 1, 3, 300, 64)])
def test_cache_strides(kind, n_ctx, group, Lq, n_mem, hd):
    """Several contexts over several chunks of keys, through the tensor maps of the prefill form and the plain loads
    of the decode form; a shared dimension has stride 0."""
    n_kv, L = 2, 12
    run = DeviceRun(wk.Workload("attn_forms", 45, n_ctx, L, 256, 256, 2 * n_kv * hd, n_kv, hd, 128, 128, 8, "bf16", wk.PLAIN))
    g = torch.Generator(device="cuda").manual_seed(Lq + hd)
    K, V = (strided(kind, n_ctx, L, n_kv, n_mem + Lq, hd, g) for _ in range(2))
    assert K.stride() == V.stride() and K.stride(4) == 1
    Q = torch.randn(n_ctx, L, group * n_kv, Lq, hd, generator=g, device="cuda").bfloat16()
    out = torch.full_like(Q, 7.0)
    mone.mone_attention(run.h, Q, group * n_kv, Lq, K, V, K.stride()[:4], n_mem, out)
    mone.mone_mem_sync(run.h)
    run.close()
    for c in {0, n_ctx - 1}:
        for layer in {0, L - 1}:
            ref = O.attention(Q[c, layer].cpu(), K[c, layer].cpu(), V[c, layer].cpu(), n_mem)
            assert rel_fro(out[c, layer].float().cpu(), ref) <= 1e-2, (c, layer)


@pytest.mark.parametrize("hd,group,Lq,n_mem", [(64, 4, 200, 200), (128, 2, 150, 130), (64, 1, 3, 300)])
def test_keys_at_minus_infinity_count_for_nothing(hd, group, Lq, n_mem):
    """The memory keys, whole chunks of them, overflow to scores of -inf; the tokens' own keys are ordinary."""
    n_kv, L = 2, 20
    run = DeviceRun(wk.Workload("attn_forms", 43, 1, L, 256, 256, 2 * n_kv * hd, n_kv, hd, 128, 128, 8, "bf16", wk.PLAIN))
    g = torch.Generator(device="cuda").manual_seed(hd + Lq)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()  # noqa: E731
    K, V, Q = rn(1, L, n_kv, n_mem + Lq, hd), rn(1, L, n_kv, n_mem + Lq, hd), rn(1, L, group * n_kv, Lq, hd)
    K[..., 0] = 0
    K[..., :n_mem, 0] = -1e25
    Q[..., 0] = 1e25
    out = torch.full_like(Q, 7.0)
    mone.mone_attention(run.h, Q, group * n_kv, Lq, K, V, K.stride()[:4], n_mem, out)
    mone.mone_mem_sync(run.h)
    run.close()
    for layer in (0, L - 1):
        ref = O.attention(Q[0, layer].cpu(), K[0, layer].cpu(), V[0, layer].cpu(), n_mem)
        assert rel_fro(out[0, layer].float().cpu(), ref) <= 1e-2, layer


@pytest.mark.parametrize("group,Lq,n_mem,hd,n_layers", [
    (4, 200, 70, 64, 20),    # prefill: 32-token tiles; the tiles' last chunks hold later tokens' rows
    (3, 150, 0, 128, 20),    # 42-token tiles
    (1, 300, 77, 64, 20),    # 128-token tiles
    (1, 300, 31, 64, 1),     # decode: 16-row tiles of one head
    (7, 40, 500, 128, 1),    # rows of the group's heads, 18-token blocks
    (20, 40, 60, 64, 1),     # 6-token blocks
])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_value_rows_stay_with_their_tile(group, Lq, n_mem, hd, n_layers, bad):
    """A token's non-finite value and key rows reach no token of an earlier tile of 128 / group tokens."""
    n_kv = 2
    run = DeviceRun(wk.Workload("attn_forms", 44, 1, n_layers, 256, 256, 2 * n_kv * hd, n_kv, hd, 128, 128, 8, "bf16", wk.PLAIN))
    g = torch.Generator(device="cuda").manual_seed(group + Lq)
    rn = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()  # noqa: E731
    K, V, Q = (rn(1, n_layers, h, t, hd) for h, t in ((n_kv, n_mem + Lq), (n_kv, n_mem + Lq), (group * n_kv, Lq)))
    outs = []
    tile = 128 // group
    first = tile * ((Lq - 1) // tile)  # first token of the last tile
    for t in range(first, Lq, 3):
        V[..., n_mem + t, :] = bad
        K[..., n_mem + t, ::2] = bad
        outs.append(torch.full_like(Q, 7.0))
        mone.mone_attention(run.h, Q, group * n_kv, Lq, K, V, K.stride()[:4], n_mem, outs[-1])
    mone.mone_mem_sync(run.h)
    run.close()
    for layer in (0, n_layers - 1):
        sl = slice(0, n_mem + first)
        ref = O.attention(Q[0, layer, :, :first].cpu(), K[0, layer, :, sl].cpu(), V[0, layer, :, sl].cpu(), n_mem)
        for out in outs:
            assert rel_fro(out[0, layer, :, :first].float().cpu(), ref) <= 1e-2, layer


def test_prefill_form_many_tiles_repeat():
    """More CTAs than the SMs hold at once, repeated: every wait is met and the output repeats bit for bit."""
    n_kv, group, hd, Lq, n_mem, L = 8, 4, 128, 400, 64, 16
    wl = wk.Workload("attn_forms", 42, 1, L, 256, 256, 2 * n_kv * hd, n_kv, hd, 128, 128, 8, "bf16", wk.PLAIN)
    run = DeviceRun(wl)
    g = torch.Generator(device="cuda").manual_seed(3)
    K = torch.randn(1, L, n_kv, n_mem + Lq, hd, generator=g, device="cuda").bfloat16()
    V = torch.randn(K.shape, generator=g, device="cuda").bfloat16()
    Q = torch.randn(1, L, group * n_kv, Lq, hd, generator=g, device="cuda").bfloat16()
    outs = [torch.full_like(Q, 7.0) for _ in range(2)]
    for i in range(40):
        mone.mone_attention(run.h, Q, group * n_kv, Lq, K, V, K.stride()[:4], n_mem, outs[i % 2])
    mone.mone_mem_sync(run.h)
    run.close()
    assert torch.equal(*outs)


@pytest.mark.parametrize("group,Lq,n_mem,hd,n_layers", [
    (1, 1, 0, 64, 2),        # one row, one key
    (4, 1, 31, 64, 2),       # one whole 32-key block
    (4, 1, 32, 64, 2),       # one key past it
    (7, 2, 5000, 64, 1),     # a cluster of eight, 14 rows
    (8, 3, 700, 64, 3),      # 24 rows: two row tiles, causal rows
    (16, 32, 100, 64, 1),    # 512 rows: 32 row tiles of two heads
    (4, 1, 15, 128, 2),      # hd 128: one whole 16-key block
    (4, 1, 16, 128, 2),      # one key past it
    (5, 5, 3000, 128, 1),    # 25 rows over a cluster
])
def test_decode_form(group, Lq, n_mem, hd, n_layers):
    run_case(group, Lq, n_mem, hd, n_layers=n_layers, late_scale=3.0)
