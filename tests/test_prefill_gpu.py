"""GPU parity of lla_prefill_attn (causal pass-2 prefill, App. A and App. J) against the oracle.

The cache is filled by lla_encode; the oracle runs causal softmax attention over the explicitly
reconstructed K/V of every key (Eq. decode).  Two comparisons per (sequence, head):
  * against the oracle on its own latents (the full path, bf16 storage tolerance: max abs
    <= 2e-2 beyond the rounding of a bf16 output to its own format, relative L2 <= 5e-3; fp32
    storage: relative L2 <= 1e-5);
  * against the oracle fed the latents the GPU stored, so that only the attention kernel is
    under test (relative L2 <= 5e-3 with bf16 tensor-core operands, 1e-5 in fp32).
Cases reach both code paths (tcgen05 for bf16 storage at (96, 160), (192, 320) and (128, 128), and with
bf16 queries at (72, 120) and (18, 30); CUDA cores otherwise), prompts shorter than a page, on page and tile boundaries and across several query
tiles, fp32 and bf16 queries, with and without mu.
"""
import math

import numpy as np
import pytest
import torch

import oracle
from helpers import assert_parity, ensure_library, f64, rel_l2
from test_decode_gpu import Scene

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.fixture(scope="module")
def lla():
    ensure_library()
    from paper_2607_15456_gb300 import lla as m
    m.lla_clear_device_error()
    return m


def _prefill_case(lla, r_k, r_v, storage, io, lens, loop, with_mu, H=2, seed=0, tight=None):
    sc = Scene(lla, T=4, H=H, d=128, r_k=r_k, r_v=r_v, storage=storage, io=io, lens=lens,
               seed=seed, with_mu=with_mu, extra_tokens=0)
    W = sc.W
    N = sum(lens)
    dt = torch.bfloat16 if io == "bf16" else torch.float32
    q = W.normal((N, H, 128), seed, 60, loop, dtype=dt, device=DEV)
    out = torch.full_like(q, float("nan"))
    cu = torch.tensor(np.cumsum([0] + list(lens)), dtype=torch.int32, device=DEV)
    lla.lla_prefill_attn(sc.geom, sc.codec, sc.cache, cu, max(lens), loop, q, out)
    torch.cuda.synchronize()
    assert lla.lla_get_device_error() == 0
    got, q64 = f64(out), f64(q)
    w = sc.w64
    tight = tight or (1e-5 if storage == "fp32" else 5e-3)
    off = 0
    for b, L in enumerate(lens):
        for h in range(H):
            mk = None if w["mu_k"] is None else w["mu_k"][h]
            mv = None if w["mu_v"] is None else w["mu_v"][h]
            args = (w["w_up_k"][h], w["w_up_v"][h], mk, mv, q64[off:off + L, h], sc.scale)
            ref = oracle.prefill(loop, sc.ck[b, h], sc.cv[b, h], *args)
            assert_parity(got[off:off + L, h], ref, storage, f"prefill b{b} h{h}", io=io,
                          output_rounding=True)
            gk, gv = sc.gpu_latents(b, h)
            ref2 = oracle.prefill(loop, gk, gv, *args)
            err = rel_l2(got[off:off + L, h], ref2)
            assert err <= tight, (b, h, err)
        off += L
    return got


@pytest.mark.parametrize("io", ["bf16", "fp32"])
def test_prefill_tensor_core_ragged_prompts(lla, io):
    # 1 token; one page minus one; exactly one page; one more; two tiles plus; three tiles
    _prefill_case(lla, 96, 160, "bf16", io, [1, 63, 64, 65, 130, 300], 2, True)


def test_prefill_tensor_core_rho2_ranks(lla):
    # r_v = 320: the PV product is split in two N = 160 halves
    _prefill_case(lla, 192, 320, "bf16", "bf16", [200, 129], 0, False)


def test_prefill_tensor_core_full_rank(lla):
    _prefill_case(lla, 128, 128, "bf16", "bf16", [257], 1, True)


def test_prefill_long_prompt_rescales(lla):
    # 1500 keys: many pages per tile, so row maxima grow and O is rescaled in TMEM
    _prefill_case(lla, 96, 160, "bf16", "bf16", [1500], 3, False, H=1, seed=5)


def test_prefill_tensor_core_ranks_in_parts(lla):
    # r = (72, 120): not multiples of 32, served in three bf16 parts
    _prefill_case(lla, 72, 120, "bf16", "bf16", [70, 5], 1, False)


@pytest.mark.parametrize("r_k,r_v,io,tight", [(72, 120, "fp32", 1e-5), (18, 30, "fp32", 1e-5), (40, 56, "fp32", 1e-5),
                                              (40, 56, "bf16", 2 ** -8)])
def test_prefill_cuda_core_ranks(lla, r_k, r_v, io, tight):
    # bf16 storage on the CUDA cores: fp32 queries at the ranks that take parts, and any other ranks
    _prefill_case(lla, r_k, r_v, "bf16", io, [140, 70, 5], 1, True, tight=tight)


def test_prefill_fp32_storage(lla):
    _prefill_case(lla, 96, 160, "fp32", "fp32", [90, 33], 0, True)


def test_prefill_rejects_bad_context(lla):
    # a prompt longer than max_len is flagged on the device; nothing is written for it
    sc = Scene(lla, T=4, H=1, d=128, r_k=96, r_v=160, storage="bf16", io="bf16", lens=[100],
               seed=9, extra_tokens=0)
    q = torch.zeros((100, 1, 128), dtype=torch.bfloat16, device=DEV)
    out = torch.zeros_like(q)
    cu = torch.tensor([0, 100], dtype=torch.int32, device=DEV)
    lla.lla_clear_device_error()
    lla.lla_prefill_attn(sc.geom, sc.codec, sc.cache, cu, 64, 0, q, out)
    torch.cuda.synchronize()
    assert lla.lla_get_device_error() & 0x2  # LLA_DEVERR_CONTEXT
    lla.lla_clear_device_error()


def _rising_scores_case(lla, r_k, r_v, H, lens, seed, tol):
    """Row maxima that rise from page to page: token i's keys are scaled by 1 + i / 64, so the running
    maximum passes the rescale threshold (2^8) every page or two, in some rows of a warp and not in
    others."""
    from paper_2607_15456_gb300 import workloads as W
    sc = Scene(lla, T=4, H=H, d=128, r_k=r_k, r_v=r_v, storage="bf16", io="bf16", lens=lens, seed=seed,
               with_mu=True, extra_tokens=0)
    N = sum(lens)
    grow = torch.cat([1 + torch.arange(L, device=DEV) / 64 for L in lens]).view(1, N, 1, 1)
    x = [(W.normal((4, N, H, 128), seed, 70 + i, dtype=torch.float32, device=DEV) * (grow if i == 0 else 1)).to(torch.bfloat16)
         for i in range(2)]
    slots = torch.cat([sc.pt.slots(b, range(L)) for b, L in enumerate(lens)]).to(DEV)
    lla.lla_encode(sc.geom, sc.codec, sc.cache, x[0].contiguous(), x[1].contiguous(), slots)
    q = W.normal((N, H, 128), seed, 72, device=DEV)
    out = torch.full_like(q, float("nan"))
    cu = torch.tensor(np.cumsum([0] + list(lens)), dtype=torch.int32, device=DEV)
    lla.lla_prefill_attn(sc.geom, sc.codec, sc.cache, cu, max(lens), 1, q, out)
    torch.cuda.synchronize()
    assert lla.lla_get_device_error() == 0
    got, q64, w, off = f64(out), f64(q), sc.w64, 0
    for b, L in enumerate(lens):
        for h in range(H):
            gk, gv = sc.gpu_latents(b, h)
            ref = oracle.prefill(1, gk, gv, w["w_up_k"][h], w["w_up_v"][h], w["mu_k"][h], w["mu_v"][h],
                                 q64[off:off + L, h], sc.scale)
            err = rel_l2(got[off:off + L, h], ref)
            assert err <= tol, (b, h, err)
        off += L


def test_prefill_rising_scores_one_tile_per_cta(lla):
    # the two softmax groups take a tile's pages in turn and hand the running maximum on.  At (72, 120)
    # q~ and the softmax weights are sums of three bf16 parts: bf16 outputs are then as exact as their
    # own rounding (2^-9 relative) however large the scores
    _rising_scores_case(lla, 72, 120, 2, [700, 321], 31, 2 ** -9 + 1e-4)


def test_prefill_rising_scores_two_tiles_per_cta(lla):
    # 5 pairs of tiles x 13 prompts x 16 heads = 1040: each group owns a tile.  q~ is rounded to bf16
    # (2^-9 / sqrt 3 of each term, so 1.1e-3 sigma of a score whose sigma reaches 1 + 1030 / 64 = 17, of
    # which the few keys that share a row's weight see sqrt 2) and so is every weight (2^-9)
    _rising_scores_case(lla, 96, 160, 16, [1030, 500, 385, 384, 257, 256, 255, 129, 128, 127, 64, 63, 1], 32,
                        1.1e-3 * 17 * 2 ** 0.5 + 2 ** -8)


@pytest.mark.parametrize("r_k,r_v,io", [(96, 160, "bf16"), (96, 160, "fp32"), (128, 128, "bf16")])
def test_prefill_two_tiles_per_cta(lla, r_k, r_v, io):
    # 5 pairs x 13 prompts x 16 heads = 1040: second tiles that are empty, one row, part of a page, full
    _prefill_case(lla, r_k, r_v, "bf16", io, [1025, 520, 513, 512, 448, 385, 384, 383, 130, 129, 128, 64, 1], 2, True,
                  H=16, seed=6)


@pytest.mark.parametrize("H,lens", [(2, [1, 63, 64, 65, 130, 300]), (1, [900])])
def test_prefill_rows_without_16_byte_words(lla, H, lens):
    # (18, 30): pages and W_up rows go through the producer warps' registers; more pages than stages
    _prefill_case(lla, 18, 30, "bf16", "bf16", lens, 2, True, H=H, seed=7)


def test_prefill_rising_scores_rows_without_16_byte_words(lla):
    _rising_scores_case(lla, 18, 30, 2, [700, 321], 33, 2 ** -9 + 1e-4)


@pytest.mark.parametrize("r_k,r_v", [(72, 120), (18, 30)])
def test_prefill_in_parts_is_as_exact_as_the_cuda_cores(lla, r_k, r_v):
    """bf16 queries take the tensor cores with q~, weights and O / l in bf16 parts, the same queries in fp32 the
    CUDA cores in fp32.  A sum in the tensor core falls short by 2^-25 of itself per step on average; some 60
    steps (values and projection) over partial sums twice the result's size make 3.6e-6 of an output, which
    rounds one in 1500 (a spacing is 2^-8 to 2^-7) to another bf16 number.  Operands of 16 bits instead of 24
    would move one in 550; the bound is one in 1000."""
    lens, H = [200, 130, 64, 1], 8
    sc = Scene(lla, T=4, H=H, d=128, r_k=r_k, r_v=r_v, storage="bf16", io="bf16", lens=lens, seed=34, with_mu=True,
               extra_tokens=0)
    q = sc.W.normal((sum(lens), H, 128), 34, 72, device=DEV)
    cu = torch.tensor(np.cumsum([0] + lens), dtype=torch.int32, device=DEV)
    out, ref = torch.empty_like(q), torch.empty(q.shape, device=DEV)
    lla.lla_prefill_attn(sc.geom, sc.codec, sc.cache, cu, max(lens), 1, q, out)
    lla.lla_prefill_attn(sc.geom, sc.codec, sc.cache, cu, max(lens), 1, q.float(), ref)
    torch.cuda.synchronize()
    assert lla.lla_get_device_error() == 0
    moved = (out != ref.to(torch.bfloat16)).float().mean().item()
    assert moved <= 1e-3, moved


def _stepped_scores_case(lla, r_k, r_v, H, lens):
    """Scores that step up every third page and are equal within a step: only coordinate 0 of the K latents is
    not zero, and it holds the step.  Even rows' steps are 16 in the exp2 domain, past the rescale threshold
    (8), odd rows' are 4.  A row's output is then the mean of the V latents of its last step, and of those
    before it by 2^-16 or 2^-4 a step, so that a page that is lost or counted twice moves it by 1 / 3 of a
    value.  The step itself is off by 2^-9 (q~ in bf16), which moves the weight of the steps before by 3 %
    of 1 / 16 at most; weights and outputs are rounded by up to 2^-8 each."""
    g = torch.Generator(device=DEV).manual_seed(35)
    geom, d, T = lla.Geometry(1, H, 128, r_k, r_v), 128, 1
    w_k = torch.zeros(H, T, d, r_k, device=DEV, dtype=torch.bfloat16)
    w_k[..., 0] = 1 / 128  # q~_0 is the mean of q
    w_v = torch.zeros(H, T, d, r_v, device=DEV, dtype=torch.bfloat16)
    w_v[:, 0, torch.arange(min(d, r_v)), torch.arange(min(d, r_v))] = 1  # o is the mean of the V latents
    codec = lla.Codec(None, None, w_k, w_v)
    pages = [-(-L // 64) for L in lens]
    table = torch.full((len(lens), max(pages)), -1, dtype=torch.int32, device=DEV)
    perm = torch.randperm(sum(pages), generator=g, device=DEV).to(torch.int32)
    e = 8 if r_k % 8 == 0 else 2
    pool = torch.full((sum(pages), H, 64 * (r_k + r_v)), float("nan"), device=DEV, dtype=torch.bfloat16)
    cv, o = [], 0
    for b, n in enumerate(pages):
        blk = perm[o:o + n]
        table[b, :n] = blk
        o += n
        v = torch.randn(n, H, 64, r_v, generator=g, device=DEV).to(torch.bfloat16)
        k = torch.zeros(n, H, r_k // e, 64, e, device=DEV, dtype=torch.bfloat16)
        k[:, :, 0, :, 0] = (torch.arange(n, device=DEV) // 3).view(n, 1, 1).to(torch.bfloat16)
        pool[blk.long()] = torch.cat([k.reshape(n, H, -1), v.reshape(n, H, -1)], 2)
        cv.append(v.permute(1, 0, 2, 3).reshape(H, n * 64, r_v)[:, :lens[b]].double())
    N = sum(lens)
    step = torch.tensor([16.0, 4.0], device=DEV)[torch.arange(N, device=DEV) % 2]
    q = (step * math.log(2) * math.sqrt(d)).view(N, 1, 1).expand(N, H, d).to(torch.bfloat16).contiguous()
    out = torch.full_like(q, float("nan"))
    cu = torch.tensor(np.cumsum([0] + list(lens)), dtype=torch.int32, device=DEV)
    lla.lla_prefill_attn(geom, codec, lla.Cache(pool, sum(pages), table, max(pages)), cu, max(lens), 0, q, out)
    torch.cuda.synchronize()
    assert lla.lla_get_device_error() == 0
    off, cols = 0, min(d, r_v)
    for b, L in enumerate(lens):
        i = torch.arange(L, device=DEV)
        s = (i // 192).double()[None] * (q[off:off + L, 0, 0].double() / math.sqrt(d))[:, None]
        p = torch.softmax(s.masked_fill(i[None] > i[:, None], -math.inf), 1)
        ref = (p @ cv[b])[..., :cols].permute(1, 0, 2)
        err = (out[off:off + L, :, :cols].double() - ref).abs()
        # per output: its own rounding and the weights' (2^-8 each, of the values' weighted size), and 3 % of what
        # the steps before the last contribute to odd rows (1 / 16 of their size at most)
        size = (p @ cv[b].abs())[..., :cols].permute(1, 0, 2)
        bound = size * (2 * 2 ** -8 + 0.03 / 16) + 1e-6
        assert (err <= bound).all(), (b, (err / bound).max().item())
        off += L


@pytest.mark.parametrize("r_k,r_v,H,lens", [
    (96, 160, 2, [1000, 577]),                                    # one tile per CTA: the groups take turns
    (192, 320, 2, [700]),
    (72, 120, 2, [700, 321]),                                     # three bf16 parts
    (18, 30, 2, [700, 321]),
    (96, 160, 16, [1030, 1000, 900, 770, 500, 257, 129, 63]),     # 5 pairs x 8 x 16 = 640: two tiles per CTA
    (128, 128, 16, [1030, 1000, 900, 770, 500, 257, 129, 63]),
])
def test_prefill_stepped_scores(lla, r_k, r_v, H, lens):
    _stepped_scores_case(lla, r_k, r_v, H, lens)
