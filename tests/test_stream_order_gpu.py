"""Stream order of programmatically launched kernels: whatever input of a call the kernel just before it on
the stream writes, the codec's among them, is read as written.

The writer is lla_decode_attn, which lets its dependents launch before it has written its output; each call is
compared bit for bit with the same call after a synchronisation.
"""
import pytest
import torch

from test_decode_gpu import DEV, Scene, lla  # noqa: F401  (lla is a fixture)

pytestmark = pytest.mark.gpu


def _writer(lla, numel, io):
    """(write, out): write() enqueues a decode of numel / 256 sequences (2 heads) into out, zeroed before."""
    B = numel // 256
    assert B * 256 == numel
    sc = Scene(lla, H=2, io=io, lens=[300] * B, seed=91)
    q, ck, cv, out = sc.decode(0, pass1=True)
    lens = torch.tensor(sc.lens, dtype=torch.int32, device=DEV)

    def write():
        out.zero_()
        torch.cuda.synchronize()
        lla.lla_decode_attn(sc.geom, sc.codec, sc.cache, lens, 300, 0, q, ck, cv, out, sc.ws)

    return write, out.view(-1)


@pytest.mark.parametrize("r", [64, 18])
@pytest.mark.parametrize("what", ["w_down_k", "w_down_v", "mu_k"])
def test_step_encode_after_the_kernel_that_writes_its_codec(lla, what, r):
    H, d, N = 2, 128, 16
    write, buf = _writer(lla, H * d if what == "mu_k" else H * d * r, "fp32" if what == "mu_k" else "bf16")
    g = torch.Generator(device=DEV).manual_seed(92)
    geom = lla.Geometry(1, H, d, r, r)
    t = {n: torch.randn(H, d, r, generator=g, device=DEV).to(torch.bfloat16) for n in ("w_down_k", "w_down_v")}
    t["mu_k"] = None
    t[what] = buf
    codec = lla.Codec(t["w_down_k"], t["w_down_v"], None, None, t["mu_k"], None)
    x = torch.randn(1, N, H, d, generator=g, device=DEV).to(torch.bfloat16)
    slots = torch.arange(N, device=DEV)

    def encode(settle):
        pool = torch.zeros(lla.lla_cache_block_bytes(geom), dtype=torch.uint8, device=DEV)
        write()
        if settle:
            torch.cuda.synchronize()
        lla.lla_encode(geom, codec, lla.Cache(pool, 1, None, 1), x, x, slots)
        torch.cuda.synchronize()
        return pool

    want = encode(True)
    for _ in range(4):
        assert torch.equal(encode(False), want)
    assert lla.lla_get_device_error() == 0


@pytest.mark.parametrize("entry", ["loops", "2d"])
def test_shared_latent_decode_after_the_kernel_that_writes_its_codec(lla, entry):
    """W_up^K [H][T][d][r] (loops) or [T][H][d][r] (LLA-2D) of one loop, written just before the call."""
    H, d, r_k, r_v, B = 2, 128, 96, 160, 3
    write, buf = _writer(lla, H * d * r_k, "bf16")
    g = torch.Generator(device=DEV).manual_seed(93)
    rand = lambda *s: torch.randn(s, generator=g, device=DEV).to(torch.bfloat16)
    geom = lla.Geometry(1, H, d, r_k, r_v)
    codec = lla.Codec(None, None, buf, rand(H * d * r_v))
    two_d = entry == "2d"
    bb = (lla.lla_cache_2d_block_bytes if two_d else lla.lla_cache_block_bytes)(geom)
    pool = rand(B * bb // 2)
    cache = lla.Cache(pool, B, torch.arange(B, dtype=torch.int32, device=DEV).view(B, 1), 1)
    lens = torch.full((B,), 60, dtype=torch.int32, device=DEV)
    q = rand(1, B, H, d)
    size = lla.lla_decode_2d_workspace_size if two_d else lla.lla_decode_loops_workspace_size
    ws = torch.empty(size(geom, B), dtype=torch.uint8, device=DEV)

    def decode(settle):
        out = torch.empty_like(q)
        write()
        if settle:
            torch.cuda.synchronize()
        if two_d:
            lla.lla_decode_attn_2d(geom, codec, cache, lens, 64, 0, q[0], None, None, out[0], ws)
        else:
            lla.lla_decode_attn_loops(geom, codec, cache, lens, 64, q, None, None, out, ws)
        torch.cuda.synchronize()
        return out

    want = decode(True)
    for _ in range(4):
        assert torch.equal(decode(False), want)
    assert lla.lla_get_device_error() == 0
