"""What the binding accepts and refuses, without a GPU: nothing here gets as far as a launch."""
import ctypes as C

import pytest
import torch

A = 1 << 20      # a made-up, 16-byte aligned device address: never dereferenced here


@pytest.fixture(scope="module")
def rac():
    from paper_2608_04991_b200 import build, binding
    build.build()
    binding.load()
    return binding


def decode(rac, cfg, payload=A, T=16, ref_base=A, step=A, X_hat=A, stream=0):
    rac.rac_decode_reconstruct(cfg, payload, T, ref_base, 16, None, None, None, step, X_hat, A, stream=stream)


@pytest.mark.parametrize("kw,exc,text", [
    (dict(payload="x"), TypeError, "payload: expected a torch tensor, an address or None"),
    (dict(step=1.5), TypeError, "step: expected a torch tensor"),
    (dict(X_hat=torch.zeros(4, dtype=torch.bfloat16)), ValueError, "X_hat: must be a CUDA tensor"),
    (dict(T="many"), ValueError, "invalid literal"),
    (dict(T=None), TypeError, "int"),
])
def test_arguments_that_are_refused(rac, kw, exc, text):
    with pytest.raises(exc, match=text):
        decode(rac, rac.CodecCfg(4096, 128, 4, 0), **kw)


def test_configuration_types_are_told_apart(rac):
    with pytest.raises(TypeError):
        decode(rac, rac.IndexCfg(100))
    with pytest.raises(TypeError):
        decode(rac, None)
    with pytest.raises(TypeError):
        rac.rac_index_reset(rac.CodecCfg(4096, 128, 4, 0), A, 1 << 30, stream=0)


def test_addresses_and_numbers_reach_the_library(rac):
    cfg = rac.CodecCfg(4096, 128, 4, 0)
    for kw, code in [(dict(payload=None), -1), (dict(payload=A + 2), -2), (dict(T=-1), -1), (dict(T=17), -1)]:
        with pytest.raises(rac.RacError) as e:
            decode(rac, cfg, **kw)
        assert e.value.code == code
    with pytest.raises(rac.RacError) as e:
        decode(rac, rac.CodecCfg(4096, 100, 4, 0))
    assert e.value.code == -1 and "rac_decode_reconstruct" in str(e.value)
    decode(rac, cfg, T=0)                        # a no-op
    decode(rac, cfg, T=True and 0)


def test_prepared_call_checks_like_the_plain_one(rac):
    cfg = rac.CodecCfg(4096, 128, 4, 0)
    call = rac.prepare(rac.rac_decode_reconstruct, cfg, A + 2, 16, A, 16, None, None, None, A, A, A, stream=0)
    with pytest.raises(rac.RacError) as e:
        call()
    assert e.value.code == -2
    with pytest.raises(TypeError):
        call(1)
    none = rac.prepare(rac.rac_decode_reconstruct, cfg, A, 0, A, 16, None, None, None, A, A, A, stream=0)
    assert none() is None


class _Stream:
    """What torch.cuda.Stream is to ctypes."""
    _as_parameter_ = C.c_void_p(0x7000)


def test_streams_are_addresses_or_what_ctypes_takes_for_one(rac):
    cfg = rac.CodecCfg(4096, 128, 4, 0)
    assert hasattr(torch.cuda.Stream, "_as_parameter_")
    for stream in (0, 0x7000, True, _Stream(), C.c_void_p(0x7000), C.c_void_p(None), C.pointer(C.c_int(3))):
        decode(rac, cfg, T=0, stream=stream)
        rac.prepare(rac.rac_decode_reconstruct, cfg, A, 0, A, 16, None, None, None, A, A, A, stream=stream)()
    assert rac._stream_address(_Stream()) == 0x7000 and rac._stream_address(C.c_void_p(None)) == 0
    for stream in (3.7, torch.tensor(5), C.c_int64(5), object()):
        with pytest.raises((TypeError, C.ArgumentError)):
            decode(rac, cfg, T=0, stream=stream)


@pytest.mark.parametrize("cfg", [b"\0" * 36, bytearray(36), (C.c_int32 * 9)(4096, 128, 4), torch.zeros(9, dtype=torch.int32).numpy()])
def test_other_buffers_of_the_size_of_a_configuration_are_refused(rac, cfg):
    with pytest.raises(TypeError):
        decode(rac, cfg, T=0)
    with pytest.raises(TypeError):
        rac.rac_index_reset(memoryview(cfg)[:16] if isinstance(cfg, (bytes, bytearray)) else cfg, A, 1 << 30, stream=0)
    with pytest.raises(TypeError):
        rac.prepare(rac.rac_decode_reconstruct, cfg, A, 0, A, 16, None, None, None, A, A, A, stream=0)

    class Named(rac.CodecCfg):
        pass
    decode(rac, Named(4096, 128, 4, 0), T=0)


def test_prepared_call_shows_what_it_was_given(rac):
    args = (rac.CodecCfg(4096, 128, 4, 0), A, 0, A, 16, None, None, None, A, A, A)
    call = rac.prepare(rac.rac_decode_reconstruct, *args, stream=0)
    assert call.keepalive == (args, {"stream": 0}) and call.keepalive[0][0] is args[0]


def test_numbers_are_whatever_float_and_int_take(rac):
    def steps(clip, T=0):
        rac.rac_calibrate_steps(rac.CodecCfg(4096, 128, 4, 0), None, T, None, 0, None, None, None, clip, None, None, None, 0, None, stream=0)
    for clip, T in ((3, 0), (3.0, "0"), ("3.0", 0.9), (torch.tensor(3.0), torch.tensor(0))):
        with pytest.raises(rac.RacError) as e:      # marshalled; the library then misses the tables
            steps(clip, T)
        assert e.value.code == -1
    for clip in (None, "three", object()):
        with pytest.raises((TypeError, ValueError)):
            steps(clip)


def test_extension_module_by_itself_raises(rac):
    """Imported without binding.load(): an error, not a crash."""
    import subprocess
    import sys
    code = ("import torch\nfrom paper_2608_04991_b200 import _native as n\n"
            "try:\n    n.rac_index_reset(b'', 0, 0, 0)\nexcept RuntimeError as e:\n    print(e)")
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=rac.LIB_PATH.rsplit("/", 2)[0])
    assert out.returncode == 0 and "binding.load()" in out.stdout
