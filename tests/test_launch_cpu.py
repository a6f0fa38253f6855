"""Host code of the launches, on a CUDA runtime without a GPU: two devices in one process."""
import shutil

import pytest

import paper_2608_17616_gb300 as mone
from fakert import Fake, build_fake

P = 1 << 30  # a made-up, aligned device address


@pytest.fixture()
def fake(tmp_path, monkeypatch, built):
    # a copy of its own for each test: the library's per-process state starts empty
    path = shutil.copy(built, tmp_path / "libmone_fakert.so")
    f = Fake(str(path))
    monkeypatch.setattr(mone, "_lib", mone.lib(str(path)))
    return f


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    return build_fake(tmp_path_factory.mktemp("fakert"))


def init(n_layers, d_in, d_hid, d_out, T, dtype, mode=mone.MONE_PLAIN, n_ctx=1, hd=64, **kw):
    meta = {k: P for k in ("alpha", "gamma", "w_eta", "b_eta", "w_beta", "b_beta", "gate")} if mode == mone.MONE_PAPER else None
    cfg = mone.make_config(n_ctx, n_layers, d_in, d_hid, d_out, d_out // (2 * hd), hd, T, dtype, mode, 1e-2, **kw)
    return mone.mone_mem_init(cfg, P, P, meta, 0)


F32_SHAPES = [
    (1, 256, 512, 256, 128),     # resident chain, four rows a CTA
    (8, 256, 512, 256, 128),     # resident chain, eight rows
    (4, 1024, 1024, 1024, 256),  # 64 x 64 tiles of phase A (55,296 bytes), 128 x 128 of phase B
]


@pytest.mark.parametrize("shape", F32_SHAPES)
def test_fp32_learning_on_either_device(fake, shape):
    for dev in (0, 1, 0):
        fake.device(dev)
        h = init(*shape, mone.MONE_FP32)
        mone.mone_ttl_context(h, P, P, P, 1000, 0)
        launches, _ = fake.drain()
        assert launches and {x["dev"] for x in launches} == {dev}
        mone.mone_mem_free(h)


@pytest.mark.parametrize("shape", F32_SHAPES)
def test_a_failed_opt_in_is_reported_and_tried_again(fake, shape):
    h = init(*shape, mone.MONE_FP32)
    fake.fail_opt_ins(1)
    with pytest.raises(mone.MoneError):
        mone.mone_ttl_context(h, P, P, P, 1000, 0)
    mone.mone_ttl_context(h, P, P, P, 1000, 0)
    mone.mone_mem_free(h)


BF16_SHAPES = [  # d_in, d_hid, d_out, T, layers, options
    (512, 512, 512, 256, 4, {}),                               # phase A on CTA pairs
    (512, 512, 512, 128, 4, {}),                               # one-CTA phase A
    (512, 512, 512, 1024, 4, {}),                              # phase B on CTA pairs
    (512, 512, 512, 128, 1, {}),                               # one chain: phase A over clusters
    (512, 512, 512, 256, 4, dict(loss=mone.MONE_LOSS_MSE)),
    (896, 224, 896, 512, 2, dict(memory=mone.MONE_MEM_SWIGLU, mem_heads=4)),
]


@pytest.mark.parametrize("d_in,d_hid,d_out,T,layers,kw", BF16_SHAPES)
def test_bf16_calls_on_either_device(fake, d_in, d_hid, d_out, T, layers, kw):
    for dev, sms in ((0, 152), (1, 100), (0, 152)):
        fake.device(dev)
        h = init(layers, d_in, d_hid, d_out, T, mone.MONE_BF16, mone.MONE_PAPER, **kw)
        fake.drain()
        mone.mone_ttl_context_host(h, P, P, P, 3 * T + 1, T, 0)
        launches, _ = fake.drain()
        assert {x["dev"] for x in launches} == {dev}
        for x in launches:  # the persistent learning kernels stay within the device's SMs
            if "phase_" in x["name"] or "swiglu_a" in x["name"] or "swiglu_b" in x["name"]:
                assert x["grid"][0] <= sms, x
        mone.mone_ttl_context(h, P, P, P, 3 * T + 1, 0)
        for Q in (3, 300, 4000):
            mone.mone_mem_generate_kv(h, P, Q, P, P, (0, 0, 0, 64), 0)
        for Lq in (1, 2000):
            mone.mone_attention(h, P, d_out // 128, Lq, P, P, mone.kv_strides(layers, d_out // 128, Lq + 8, 64), 8, P, 0)
        assert {x["dev"] for x in fake.drain()[0]} == {dev}
        mone.mone_mem_free(h)


def test_tile_rules_follow_the_devices_sm_count(fake):
    """Each rule at a size where 152 and 100 SMs decide differently."""
    want = {0: {}, 1: {}}
    for dev in (0, 1):
        fake.device(dev)
        h = init(3, 1024, 1024, 1024, 256, mone.MONE_FP32)  # 192 tiles of 64 x 64 in phase A
        mone.mone_ttl_context(h, P, P, P, 256, 0)
        want[dev]["phase_a"] = [x["grid"] for x in fake.drain()[0] if "phase_a_f32" in x["name"]]
        h = init(1, 1024, 1024, 512, 64, mone.MONE_FP32)    # 96 tiles of 128 x 128 in phase B
        mone.mone_ttl_context(h, P, P, P, 64, 0)
        want[dev]["phase_b"] = [x["grid"] for x in fake.drain()[0] if "phase_b_f32" in x["name"]]
        h = init(1, 512, 512, 512, 128, mone.MONE_BF16, mone.MONE_PAPER)
        mone.mone_ttl_context(h, P, P, P, 3000, 0)          # 384 CTAs of 8 rows in the input transform
        want[dev]["transform"] = [x["grid"] for x in fake.drain()[0] if "prepass" in x["name"]]
        h = init(16, 512, 512, 512, 128, mone.MONE_BF16)    # decode over 64 heads in all
        mone.mone_attention(h, P, 4, 1, P, P, mone.kv_strides(16, 4, 2048, 64), 2047, P, 0)
        want[dev]["decode"] = [x["cluster"] for x in fake.drain()[0] if "decode" in x["name"]]
    assert want[0]["phase_a"] == [(8, 16, 3)] and want[1]["phase_a"] == [(4, 16, 3)]
    assert want[0]["phase_b"] == [(24, 16, 1)] and want[1]["phase_b"] == [(12, 8, 1)]
    assert want[0]["transform"] == [(384, 1, 1)] and want[1]["transform"] == [(192, 1, 1)]
    assert want[0]["decode"] == [8] and want[1]["decode"] == [6]


@pytest.mark.parametrize("memory", [mone.MONE_MEM_MLP, mone.MONE_MEM_SWIGLU])
def test_a_failed_bf16_opt_in_fails_the_init_and_is_tried_again(fake, memory):
    args = (2, 512, 256, 512, 128, mone.MONE_BF16)
    fake.fail_opt_ins(1)
    with pytest.raises(mone.MoneError):
        init(*args, memory=memory, mem_heads=2)
    h = init(*args, memory=memory, mem_heads=2)
    mone.mone_ttl_context(h, P, P, P, 1000, 0)
    mone.mone_mem_free(h)


@pytest.mark.parametrize("strides", [(1, 1, 1), (0, 1, 1), (1, 0, 1), (1, 1, 0), (0, 0, 1), (0, 1, 0), (1, 0, 0), (0, 0, 0)])
def test_attention_over_shared_caches_stays_on_the_tensor_cores(fake, strides):
    """A cache that contexts, layers or heads share (stride 0) takes the prefill form, with one element of that dimension
    in its maps."""
    n_ctx, L, n_kv, hd, Lq, n_mem = 3, 8, 4, 64, 1000, 64
    h = init(L, 512, 256, 2 * n_kv * hd, 128, mone.MONE_BF16, n_ctx=n_ctx)
    dense = mone.kv_strides(L, n_kv, n_mem + Lq, hd)
    fake.drain()
    mone.mone_attention(h, P, n_kv, Lq, P, P + 4096, [s * k for s, k in zip(dense, strides)] + [hd], n_mem, P, 0)
    launches, maps = fake.drain()
    assert [x["name"] for x in launches if "prefill" in x["name"]] and len(launches) == 1
    assert [m[0] for m in maps[-3:]] == [P, P, P + 4096]
    for base, dims in maps[-2:]:  # K and V: (dimension, stride in bytes, box)
        assert [d for d, _, _ in dims] == [hd, n_mem + Lq, n_kv if strides[2] else 1, L if strides[1] else 1, n_ctx if strides[0] else 1]
        assert [s for (d, s, _), keep in zip(dims[2:], strides[::-1]) if keep] == [2 * s for s, keep in zip(dense[2::-1], strides[::-1]) if keep]
    mone.mone_mem_free(h)


def test_attention_maps_follow_the_calls_addresses_and_shape(fake):
    h = init(8, 512, 256, 512, 128, mone.MONE_BF16)

    def call(q, k, v, Lq=1000, n_mem=64, pad=0):
        fake.drain()
        mone.mone_attention(h, q, 4, Lq, k, v, mone.kv_strides(8, 4, n_mem + Lq + pad, 64), n_mem, P, 0)
        _, maps = fake.drain()
        assert [m[0] for m in maps[-3:]] == [q, k, v]
        assert maps[-3][1][1][0] == Lq and maps[-2][1] == maps[-1][1] and maps[-1][1][1][0] == n_mem + Lq
        assert maps[-1][1][2][1] == 2 * 64 * (n_mem + Lq + pad)
        return fake.encoded

    assert call(P, P + 256, P + 512) == 2
    assert call(P + 1024, P + 2048, P + 4096) == 0  # the same shape elsewhere
    assert call(P, P + 256, P + 512, n_mem=65) == 2
    assert call(P, P + 256, P + 512, n_mem=65, pad=8) == 2
    assert call(P, P + 256, P + 512) == 2
    mone.mone_mem_free(h)


@pytest.mark.parametrize("layers,mode,kw", [(2, mone.MONE_PAPER, {}), (1, mone.MONE_PAPER, {}), (2, mone.MONE_PLAIN, {}),
                                            (2, mone.MONE_PAPER, dict(memory=mone.MONE_MEM_SWIGLU, mem_heads=2))])
def test_a_host_context_in_the_librarys_chunks_renormalises_once(fake, layers, mode, kw):
    """The learning kernels of one mone_ttl_context, and its one pass over the weights at the end."""
    T, N = 128, 2 * (32 << 20) // (layers * 2048) + 3  # 2 KB a token and layer: chunks of 32 MB
    h = init(layers, 512, 256, 512, T, mone.MONE_BF16, mode, **kw)
    fake.drain()
    mone.mone_ttl_context(h, P, P, P, N, 0)
    one = [x["name"] for x in fake.drain()[0]]
    mone.mone_ttl_context_host(h, P, P, P, N, 0, 0)
    chunks = [x["name"] for x in fake.drain()[0]]
    for part in ("phase", "swiglu_a", "swiglu_b", "finalize", "swiglu_rows"):
        assert sum(part in n for n in chunks) == sum(part in n for n in one), part
    assert sum("stage" in n for n in chunks) == 3
    assert sum("finalize" in n or "swiglu_rows" in n for n in chunks) == (mode == mone.MONE_PAPER)
    mone.mone_mem_free(h)
