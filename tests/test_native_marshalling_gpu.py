"""The two marshallings of the binding on real CUDA tensors: the native one (csrc/lla_binding.cpp) takes every
ordinary call, gives what the Python one gives bit for bit, and leaves to Python a call with one unusual
argument."""
import inspect

import pytest
import torch

from helpers import ensure_library

pytestmark = pytest.mark.gpu

DEV = "cuda"
T, H, D, B, L, BASE, DR = 2, 2, 128, 3, 70, 10000.0, 32


@pytest.fixture(scope="module")
def lla():
    ensure_library()
    from paper_2607_15456_gb300 import lla as m
    m.lla_clear_device_error()
    return m


class Call:
    """Arguments of one small call of lla.lla_<name>; `outputs` are the tensors it writes."""

    def __init__(self, lla, name):
        g = torch.Generator(device=DEV).manual_seed(18)
        rand = lambda *s, dt=torch.bfloat16: torch.randn(s, generator=g, device=DEV).to(dt)
        self.name, two_d = name, name.endswith("2d")
        geom = lla.Geometry(T, H, D, 96, 160)
        lead = (T * H * D,) if two_d else (H, T * D)
        up = (T, H, D) if two_d else (H, T, D)
        codec = lla.Codec(rand(*lead, 96), rand(*lead, 160), rand(*up, 96), rand(*up, 160), rand(*lead, dt=torch.float32),
                          rand(*lead, dt=torch.float32))
        per = 2
        table = torch.randperm(B * per, generator=g, device=DEV).to(torch.int32).view(B, per)
        bb = (lla.lla_cache_2d_block_bytes if two_d else lla.lla_cache_block_bytes)(geom)
        pool = rand(B * per * bb // 2)
        cache = lla.Cache(pool, B * per, table, per)
        n = B * L
        q = rand(T, B, H, D) if name == "decode_attn_loops" else rand(n if "prefill" in name else B, H, D)
        pos = torch.arange(L, device=DEV)
        slots = torch.cat([table[b].long()[pos // 64] * 64 + pos % 64 for b in range(B)])
        size = {"decode_attn": lambda: lla.lla_decode_workspace_size(geom, B),
                "decode_attn_rope": lambda: lla.lla_decode_workspace_size(geom, B),
                "decode_attn_loops": lambda: lla.lla_decode_loops_workspace_size(geom, B),
                "decode_attn_2d": lambda: lla.lla_decode_2d_workspace_size(geom, B),
                "decode_attn_decoupled": lambda: lla.lla_decode_decoupled_workspace_size(geom, DR, B),
                "prefill_attn_rope": lambda: lla.lla_prefill_rope_workspace_size(geom, B, L)}
        x_k, x_v = rand(T, n, H, D), rand(T, n, H, D)
        layers = name == "encode_layers"
        have = dict(geom=geom, codec=codec, cache=cache, codecs=[codec], caches=[cache], x_k=[x_k] if layers else x_k,
                    x_v=[x_v] if layers else x_v, slot_mapping=slots, max_ctx=L, max_len=L, loop=1, rope_base=BASE,
                    rope_pairing=0, d_rope=DR, rope_pool=rand(B * per * 64 * DR), q=q, out=torch.zeros_like(q),
                    context_lens=torch.full((B,), L, dtype=torch.int32, device=DEV),
                    cu_seqlens=torch.arange(0, n + 1, L, dtype=torch.int32, device=DEV), q_rope=rand(B, H, DR),
                    cur_k=rand(*q.shape), cur_v=rand(*q.shape), cur_k_rope=rand(B, DR), stream=None,
                    workspace=torch.zeros(size[name](), dtype=torch.uint8, device=DEV) if name in size else None)
        self.args = {p: have[p] for p in inspect.signature(getattr(lla, "lla_" + name)).parameters}
        self.outputs = [pool, have["out"]]

    def native(self, lla, **change):
        """What the native function of the module answers."""
        return getattr(lla._native(), self.name)(*{**self.args, **change}.values())

    def run(self, lla):
        getattr(lla, "lla_" + self.name)(**self.args)
        torch.cuda.synchronize()
        assert lla.lla_get_device_error() == 0
        res = [t.clone() for t in self.outputs]
        self.outputs[1].zero_()
        return res


NAMES = ["encode", "encode_2d", "encode_layers", "decode_attn", "decode_attn_2d", "decode_attn_loops", "decode_attn_rope",
         "decode_attn_decoupled", "prefill_attn", "prefill_attn_rope"]


@pytest.mark.parametrize("name", NAMES)
def test_both_marshallings_give_the_same(lla, name, monkeypatch):
    call = Call(lla, name)
    pool = call.outputs[0].clone()
    assert call.native(lla) == 0  # an ordinary call is taken
    native = call.run(lla)
    call.outputs[0].copy_(pool)
    monkeypatch.setattr(lla, "_native_module", lla._Absent())
    for a, b in zip(native, call.run(lla)):
        assert torch.equal(a, b)


class Subclass(torch.Tensor):
    pass


@pytest.mark.parametrize("name", NAMES)
def test_tensor_subclasses_are_left_to_python_and_parameters_are_taken(lla, name):
    call = Call(lla, name)
    key = "slot_mapping" if "encode" in name else "q"
    assert call.native(lla, **{key: call.args[key].as_subclass(Subclass)}) is None
    if name != "encode_layers":
        cd = call.args["codec"]
        cd.w_up_k = torch.nn.Parameter(cd.w_up_k)
        assert call.native(lla) == 0


@pytest.mark.parametrize("field,value", [("T", 2 ** 40), ("T", -2 ** 40), ("d", "128"), ("scale", 1), ("storage", 3),
                                         ("H", 2.0), ("r_k", True)])
def test_unusual_geometry_is_left_to_python(lla, field, value):
    call = Call(lla, "decode_attn")
    assert call.native(lla) == 0
    setattr(call.args["geom"], field, value)
    assert call.native(lla) is None


@pytest.mark.parametrize("change", [dict(max_ctx=2 ** 40), dict(loop="1"), dict(q="x"), dict(workspace=None),
                                    dict(context_lens=7), dict(stream=2 ** 70)])
def test_unusual_arguments_of_a_decode_are_left_to_python(lla, change):
    call = Call(lla, "decode_attn")
    assert call.native(lla, **change) is None


@pytest.mark.parametrize("dtype", [torch.float16, torch.float64])
def test_other_types_are_left_to_python_which_refuses_them(lla, dtype):
    call = Call(lla, "decode_attn")
    call.args["q"] = call.args["q"].to(dtype)
    assert call.native(lla) is None
    with pytest.raises(ValueError, match="unsupported dtype"):
        call.run(lla)
