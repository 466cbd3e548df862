"""GPU parity of lla_encode (Eq. encode, Sec. 3) against the CPU float64 oracle.

The latents the GPU stored are read back from the paged pool through the documented layout and
compared with oracle.encode on the same inputs (bf16 storage: max abs <= 2e-2 and relative
L2 <= 5e-3; fp32 storage and fp32 x: relative L2 <= 1e-5).  The cases reach the kernel's
separate code paths: a reduction axis T*d longer than one shared-memory chunk of W_down (fp32
and bf16), ranks whose rows are not a multiple of 16 bytes (4-byte copies), token counts that
leave a ragged last tile, x in bf16 and fp32, with and without mu, a decode-step batch, and
prompts of more than 64 tokens (or 256, at small ranks) in bf16, which take the tcgen05 kernel.
"""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_parity, bf16_half_ulp, ensure_library, f64, unpack_head

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.fixture(scope="module")
def lla():
    ensure_library()
    from paper_2607_15456_gb300 import lla as m
    m.lla_clear_device_error()
    return m


def _dt(name):
    return torch.bfloat16 if name == "bf16" else torch.float32


def _encode_and_compare(lla, T, H, d, r_k, r_v, storage, x_dtype, lens, with_mu, seed):
    from paper_2607_15456_gb300 import workloads as W
    geom = lla.Geometry(T, H, d, r_k, r_v, storage)
    cod = W.codec_tensors(T, H, d, r_k, r_v, seed, 0, dtype=_dt(storage), device=DEV,
                          with_mu=with_mu)
    codec = lla.Codec(**cod)
    pt = W.page_table(lens, seed, extra_tokens=0)
    bb = lla.lla_cache_block_bytes(geom)
    pool = torch.full((pt.num_blocks * bb,), 0xFF, dtype=torch.uint8, device=DEV)
    cache = lla.Cache(pool, pt.num_blocks, pt.block_table.to(DEV), pt.max_blocks)
    N = sum(lens)
    x_k = W.normal((T, N, H, d), seed, 40, dtype=_dt(x_dtype), device=DEV)
    x_v = W.normal((T, N, H, d), seed, 41, dtype=_dt(x_dtype), device=DEV)
    slots = torch.cat([pt.slots(b, range(L)) for b, L in enumerate(lens)]).to(DEV)
    lla.lla_encode(geom, codec, cache, x_k, x_v, slots)
    torch.cuda.synchronize()
    assert lla.lla_get_device_error() == 0
    w = {k: (None if v is None else f64(v)) for k, v in cod.items()}
    xk, xv = f64(x_k), f64(x_v)
    pool_cpu = pool.cpu()
    off = 0
    for b, L in enumerate(lens):
        for h in range(H):
            gk, gv = unpack_head(pool_cpu, H, r_k, r_v, storage, pt.block_table[b], L, h)
            ck = oracle.encode(xk[:, off:off + L, h, :], None if w["mu_k"] is None else w["mu_k"][h],
                               w["w_down_k"][h])
            cv = oracle.encode(xv[:, off:off + L, h, :], None if w["mu_v"] is None else w["mu_v"][h],
                               w["w_down_v"][h])
            io = "bf16" if x_dtype == "bf16" else "fp32"
            assert_parity(gk, ck, storage, f"c_k b{b} h{h}", io=io)
            assert_parity(gv, cv, storage, f"c_v b{b} h{h}", io=io)
        off += L


@pytest.mark.parametrize("storage,x_dtype", [("bf16", "bf16"), ("bf16", "fp32"), ("fp32", "fp32")])
def test_encode_reduction_axis_longer_than_one_chunk(lla, storage, x_dtype):
    # T*d = 16 * 256 = 4096: 8 chunks of W_down in bf16, 16 in fp32; token tiles of 6
    _encode_and_compare(lla, 16, 2, 256, 96, 160, storage, x_dtype, [13, 1, 7], True, 3)


@pytest.mark.parametrize("r_k,r_v", [(18, 30), (72, 120), (192, 320)])
def test_encode_rank_shapes_and_ragged_tiles(lla, r_k, r_v):
    # 37 tokens: two full tiles of 16 and a ragged tile of 5; r = 18, 30 use 4-byte copies
    _encode_and_compare(lla, 4, 3, 128, r_k, r_v, "bf16", "bf16", [20, 17], False, 4)


def test_encode_fp32_small_ranks(lla):
    _encode_and_compare(lla, 4, 2, 128, 18, 30, "fp32", "fp32", [33], True, 5)


def test_encode_decode_step_batch(lla):
    # the decode-step shape: one completed token for each of 16 sequences, all 16 heads
    _encode_and_compare(lla, 4, 16, 128, 96, 160, "bf16", "bf16", [1] * 16, False, 6)


@pytest.mark.parametrize("r_k,r_v,with_mu", [(96, 160, True), (192, 320, False), (128, 128, True)])
def test_encode_prompt_on_tensor_cores(lla, r_k, r_v, with_mu):
    # 300 tokens in three sequences: three tiles of 128 tokens, the last one ragged (44 tokens)
    _encode_and_compare(lla, 4, 3, 128, r_k, r_v, "bf16", "bf16", [130, 101, 69], with_mu, 7)


@pytest.mark.parametrize("r_k,r_v", [(192, 320), (96, 160)])
def test_encode_prompt_many_units_per_cta(lla, r_k, r_v):
    # 4200 tokens (33 tiles, the last ragged) of 8 heads with mu: every CTA of the persistent
    # kernel takes several (head, tile, column group) units, alternates its two accumulator
    # slots and crosses a head boundary (the bias mu W_down is recomputed there); at (192, 320)
    # the two column groups of the V axis read the same x tile one after the other
    _encode_and_compare(lla, 4, 8, 128, r_k, r_v, "bf16", "bf16", [2000, 1500, 700], True, 10)


def test_encode_prompt_long_reduction_on_tensor_cores(lla):
    # T*d = 16 * 256 = 4096: 64 slabs of the reduction axis through the stage ring
    _encode_and_compare(lla, 16, 2, 256, 96, 160, "bf16", "bf16", [150], True, 8)


@pytest.mark.parametrize("N,storage", [(16, "bf16"), (16, "fp32"), (200, "bf16")])
def test_encode_layers_equals_per_layer_calls(lla, N, storage):
    """lla_encode_layers writes exactly what one lla_encode call per layer writes (one launch
    for a decode batch; prompts go layer by layer through the tensor-core kernel)."""
    from paper_2607_15456_gb300 import workloads as W
    T, H, d, r_k, r_v, L = 4, 16, 128, 96, 160, 3
    geom = lla.Geometry(T, H, d, r_k, r_v, storage)
    pt = W.page_table([N], 9, extra_tokens=0)
    bb = lla.lla_cache_block_bytes(geom)
    slots = pt.slots(0, range(N)).to(DEV)
    table = pt.block_table.to(DEV)
    codecs, caches_a, caches_b, xs_k, xs_v, pools = [], [], [], [], [], []
    for l in range(L):
        cod = W.codec_tensors(T, H, d, r_k, r_v, 9, l, dtype=_dt(storage), device=DEV, with_mu=(l == 1))
        codecs.append(lla.Codec(**cod))
        for lst in (caches_a, caches_b):
            pool = torch.full((pt.num_blocks * bb,), 0xFF, dtype=torch.uint8, device=DEV)
            pools.append(pool)
            lst.append(lla.Cache(pool, pt.num_blocks, table, pt.max_blocks))
        xs_k.append(W.normal((T, N, H, d), 9, 50, l, device=DEV))
        xs_v.append(W.normal((T, N, H, d), 9, 51, l, device=DEV))
    lla.lla_clear_device_error()
    lla.lla_encode_layers(geom, codecs, caches_a, xs_k, xs_v, slots)
    for l in range(L):
        lla.lla_encode(geom, codecs[l], caches_b[l], xs_k[l], xs_v[l], slots)
    torch.cuda.synchronize()
    assert lla.lla_get_device_error() == 0
    for l in range(L):
        assert torch.equal(caches_a[l].pool, caches_b[l].pool), l


@pytest.mark.parametrize("r_k,r_v,with_mu", [(72, 120, True), (8, 200, True), (104, 136, False),
                                             (18, 30, True), (18, 30, False), (24, 62, True), (2, 64, True)])
def test_encode_prompt_any_rank_on_tensor_cores(lla, r_k, r_v, with_mu):
    # ranks that are not multiples of 32 (the last columns of a group are padding), an axis in two
    # uneven groups (200 = 112 + 88), and rows of W_down that are not whole 16-byte words (resident
    # W_down, 4-byte granules of the K-plane or 16-byte ones); 3 heads, a ragged third tile
    _encode_and_compare(lla, 4, 3, 128, r_k, r_v, "bf16", "bf16", [128, 129, 33], with_mu, 11)


@pytest.mark.parametrize("r_k,r_v", [(72, 120), (18, 30)])
def test_encode_prompt_any_rank_many_units_per_cta(lla, r_k, r_v):
    # 33 tiles of 8 heads with mu: several units per CTA and a head boundary inside a CTA's range
    _encode_and_compare(lla, 4, 8, 128, r_k, r_v, "bf16", "bf16", [2000, 1500, 700], True, 12)


@pytest.mark.parametrize("N", [1, 7, 16, 17, 33, 127, 256])
@pytest.mark.parametrize("r_k,r_v,with_mu", [(96, 160, True), (72, 120, False), (8, 136, True), (128, 192, False),
                                             (18, 30, True), (24, 70, False)])
def test_encode_step_tokens_and_rank_edges(lla, N, r_k, r_v, with_mu):
    # token tiles of 16 and 32 with every kind of remainder; column groups of 1 to 8 chunks of 8
    # columns, or of up to 16 pairs when a row of W_down is not whole 16-byte words
    _encode_and_compare(lla, 4, 2, 128, r_k, r_v, "bf16", "bf16", [N], with_mu, 13)


@pytest.mark.parametrize("T,d", [(1, 32), (3, 96), (16, 128), (4, 64)])
def test_encode_step_reduction_lengths(lla, T, d):
    # fewer blocks of 32 rows than warps, blocks that do not divide by the warps, a long reduction
    _encode_and_compare(lla, T, 2, d, 40, 72, "bf16", "bf16", [21], True, 14)


def _mu_far_above_the_spread(lla, H, d, r_k, r_v, N, two_d=False, T=4):
    """Half of the stacked coordinates are channels whose mean is thousands of times the spread of the others,
    and which tokens do not vary in: x - mu is zero there, so those channels may not cost precision.
    Every latent is within its bf16 rounding of the 64-bit value, but for what a sum in 32 bits of the
    products (x - mu) w rounds off: less than 2^-23 of the sum of their magnitudes per step of 16 and part."""
    g = torch.Generator(device=DEV).manual_seed(15)
    rand = lambda *s: torch.randn(s, generator=g, device=DEV)
    Hh, Td = (1, T * H * d) if two_d else (H, T * d)
    geom = lla.Geometry(T, H, d, r_k, r_v)
    pages = -(-N // 64)
    bb = (lla.lla_cache_2d_block_bytes if two_d else lla.lla_cache_block_bytes)(geom)
    pool = torch.zeros(pages * bb, dtype=torch.uint8, device=DEV)
    x, mu, w = {}, {}, {}
    for ax, r in (("k", r_k), ("v", r_v)):
        big = rand(Hh, Td) > 0
        mu[ax] = torch.where(big, rand(Hh, Td).to(torch.bfloat16).float() * 65536, 0.5 * rand(Hh, Td))
        s = torch.where(big, mu[ax], 0.5 * rand(N, Hh, Td) + mu[ax]).to(torch.bfloat16)  # stacked x
        x[ax] = (s.view(N, T, H, d).permute(1, 0, 2, 3) if two_d else s.view(N, H, T, d).permute(2, 0, 1, 3)).contiguous()
        w[ax] = (rand(Hh, Td, r) * Td ** -0.5).to(torch.bfloat16)
        y = s.double() - mu[ax].double()
        x[ax + "64"] = torch.einsum("nhk,hkr->nhr", y, w[ax].double())
        x[ax + "abs"] = torch.einsum("nhk,hkr->nhr", y.abs(), w[ax].double().abs())
    sq = (lambda t: t[0].contiguous()) if two_d else (lambda t: t)
    codec = lla.Codec(sq(w["k"]), sq(w["v"]), None, None, sq(mu["k"]), sq(mu["v"]))
    (lla.lla_encode_2d if two_d else lla.lla_encode)(geom, codec, lla.Cache(pool, pages, None, 1), x["k"], x["v"],
                                                      torch.arange(N, device=DEV))
    torch.cuda.synchronize()
    assert lla.lla_get_device_error() == 0
    pool_cpu, table = pool.cpu(), list(range(pages))
    for h in range(Hh):
        for ax, got in zip("kv", unpack_head(pool_cpu, Hh, r_k, r_v, "bf16", table, N, h)):
            ref, mag = f64(x[ax + "64"][:, h]), f64(x[ax + "abs"][:, h])
            dev = np.abs(got - ref) - bf16_half_ulp(ref)
            assert (dev <= (Td / 8 + 8) * 2.0 ** -23 * mag).all(), (ax, h, (dev / mag).max() * 2 ** 23)


@pytest.mark.parametrize("N,r_k,r_v", [(1, 96, 160), (16, 18, 30), (33, 72, 120), (64, 24, 70)])
def test_encode_step_mu_far_above_the_spread(lla, N, r_k, r_v):
    _mu_far_above_the_spread(lla, 2, 128, r_k, r_v, N)


@pytest.mark.parametrize("N,r_k,r_v", [(100, 192, 320), (300, 96, 160), (300, 72, 120), (300, 18, 30), (300, 24, 62)])
def test_encode_prompt_mu_far_above_the_spread(lla, N, r_k, r_v):
    _mu_far_above_the_spread(lla, 2, 128, r_k, r_v, N)


@pytest.mark.parametrize("N,r_k,r_v", [(1, 288, 480), (130, 288, 480), (16, 1152, 1920)])
def test_encode_2d_mu_far_above_the_spread(lla, N, r_k, r_v):
    # the reduction split over clusters, each CTA with its part of (mu - m) W_down
    _mu_far_above_the_spread(lla, 16, 128, r_k, r_v, N, two_d=True)


@pytest.mark.parametrize("N,r_k,r_v", [(16, 96, 160), (33, 18, 30), (200, 96, 160), (200, 18, 30)])
def test_encode_infinite_input(lla, N, r_k, r_v):
    """An infinite coordinate of one token makes its latents infinite with the sign of w, and no other token's."""
    H, d, T = 2, 128, 2
    g = torch.Generator(device=DEV).manual_seed(16)
    rand = lambda *s: torch.randn(s, generator=g, device=DEV)
    geom = lla.Geometry(T, H, d, r_k, r_v)
    pages = -(-N // 64)
    pool = torch.zeros(pages * lla.lla_cache_block_bytes(geom), dtype=torch.uint8, device=DEV)
    w = [rand(H, T * d, r).to(torch.bfloat16) for r in (r_k, r_v)]
    x = rand(T, N, H, d).to(torch.bfloat16)
    x[1, 5, :, 7] = float("inf")
    codec = lla.Codec(w[0], w[1], None, None, rand(H, T * d), rand(H, T * d))
    lla.lla_encode(geom, codec, lla.Cache(pool, pages, None, 1), x, x, torch.arange(N, device=DEV))
    pool_cpu = pool.cpu()
    for h in range(H):
        for wa, got in zip(w, unpack_head(pool_cpu, H, r_k, r_v, "bf16", list(range(pages)), N, h)):
            assert np.isfinite(np.delete(got, 5, 0)).all()
            assert (got[5] == np.sign(f64(wa[h, d + 7])) * np.inf).all()


@pytest.mark.parametrize("with_mu", [False, True])
def test_encode_2d_long_sums_are_as_exact_as_fp32(lla, with_mu):
    """8192 products of one sign: sums in the tensor core are cut off, not rounded, so that a long one falls
    short by half a unit of 2^-23 per step on average.  In chains of 16 steps, added up by fp32 adds, a latent
    is short by 16 / 4 such units (the partial sums are half as large on average), 4.8e-7 of itself: one in
    11000 is then rounded to another bf16 number (spacing 2^-8 to 2^-7 of a value).  Chains of 2048 rows would
    give eight times as many; the bound is three and a half times."""
    T, H, d, r_k, r_v, N = 4, 16, 128, 288, 480, 500
    g = torch.Generator(device=DEV).manual_seed(17)
    rand = lambda *s: torch.rand(s, generator=g, device=DEV) + 0.5
    geom = lla.Geometry(T, H, d, r_k, r_v)
    pages = -(-N // 64)
    pool = torch.zeros(pages * lla.lla_cache_2d_block_bytes(geom), dtype=torch.uint8, device=DEV)
    x = rand(T, N, H, d).to(torch.bfloat16)
    w = [rand(T * H * d, r).to(torch.bfloat16) for r in (r_k, r_v)]
    mu = -rand(T * H * d) if with_mu else None
    lla.lla_encode_2d(geom, lla.Codec(w[0], w[1], None, None, mu, mu), lla.Cache(pool, pages, None, 1), x, x,
                      torch.arange(N, device=DEV))
    s = x.permute(1, 0, 2, 3).reshape(N, -1).double() - (mu.double() if with_mu else 0)
    wrong = 0
    for wa, got in zip(w, unpack_head(pool.cpu(), 1, r_k, r_v, "bf16", list(range(pages)), N, 0)):
        want = (s @ wa.double()).to(torch.bfloat16)
        wrong += int((torch.from_numpy(got).to(DEV) != want.double()).sum())
    assert wrong <= 3e-4 * N * (r_k + r_v), wrong


@pytest.mark.parametrize("d,r_k,r_v,lens,with_mu", [(72, 40, 56, [20, 3], True), (128, 100, 100, [300], True),
                                                    (40, 18, 30, [130], False)])
def test_encode_bf16_on_the_cuda_cores(lla, d, r_k, r_v, lens, with_mu):
    # what the tensor-core kernels leave: head widths that are not multiples of 32 (64 for prompts), and prompts
    # whose ranks are neither multiples of 8 nor small
    _encode_and_compare(lla, 4, 3, d, r_k, r_v, "bf16", "bf16", lens, with_mu, 19)


def test_encode_layers_equals_per_layer_calls_on_the_cuda_cores(lla):
    T, H, d, r_k, r_v, L, N = 4, 2, 72, 40, 56, 3, 16
    g = torch.Generator(device=DEV).manual_seed(20)
    rand = lambda *s: torch.randn(s, generator=g, device=DEV).to(torch.bfloat16)
    geom = lla.Geometry(T, H, d, r_k, r_v)
    bb, slots = lla.lla_cache_block_bytes(geom), torch.arange(N, device=DEV)
    codecs = [lla.Codec(rand(H, T * d, r_k), rand(H, T * d, r_v), None, None, rand(H, T * d).float() if l == 1 else None)
              for l in range(L)]
    x = [[rand(T, N, H, d) for _ in range(L)] for _ in range(2)]
    pools = [[torch.full((bb,), 0xFF, dtype=torch.uint8, device=DEV) for _ in range(L)] for _ in range(2)]
    caches = [[lla.Cache(p, 1, None, 1) for p in ps] for ps in pools]
    lla.lla_encode_layers(geom, codecs, caches[0], x[0], x[1], slots)
    for l in range(L):
        lla.lla_encode(geom, codecs[l], caches[1][l], x[0][l], x[1][l], slots)
    torch.cuda.synchronize()
    assert lla.lla_get_device_error() == 0
    for a, b in zip(*pools):
        assert torch.equal(a, b)


@pytest.mark.parametrize("N,r_k,r_v", [(20, 96, 160), (200, 96, 160), (200, 18, 30)])
@pytest.mark.parametrize("axis", ["k", "v"])
def test_encode_with_mu_of_one_axis(lla, axis, N, r_k, r_v):
    H, d, T = 2, 128, 4
    g = torch.Generator(device=DEV).manual_seed(21)
    rand = lambda *s: torch.randn(s, generator=g, device=DEV)
    geom = lla.Geometry(T, H, d, r_k, r_v)
    pages = -(-N // 64)
    pool = torch.zeros(pages * lla.lla_cache_block_bytes(geom), dtype=torch.uint8, device=DEV)
    w = {a: (rand(H, T * d, r) * (T * d) ** -0.5).to(torch.bfloat16) for a, r in (("k", r_k), ("v", r_v))}
    x = {a: rand(T, N, H, d).to(torch.bfloat16) for a in "kv"}
    mu = rand(H, T * d)
    codec = lla.Codec(w["k"], w["v"], None, None, mu if axis == "k" else None, mu if axis == "v" else None)
    lla.lla_encode(geom, codec, lla.Cache(pool, pages, None, 1), x["k"], x["v"], torch.arange(N, device=DEV))
    torch.cuda.synchronize()
    assert lla.lla_get_device_error() == 0
    pool_cpu = pool.cpu()
    for h in range(H):
        for a, got in zip("kv", unpack_head(pool_cpu, H, r_k, r_v, "bf16", list(range(pages)), N, h)):
            want = oracle.encode(f64(x[a])[:, :, h], f64(mu[h]) if a == axis else None, f64(w[a][h]))
            assert_parity(got, want, "bf16", f"{a} head {h}", io="bf16")
