"""Host side of the C ABI over a stand-in for the CUDA runtime (fake_cuda.cpp):
what a workspace answers after calls that do not match or that failed half-way.
No GPU: launches are counted, not run."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2608_05780_gb300 import _binding as B
from paper_2608_05780_gb300.build import CSRC, INCLUDE, nvcc
from test_capi_host import FAKE, _args

EINVAL, ECUDA, ENOMEM, ESTATE = -1, -4, -5, -8


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-DEVISEL_BUILD_ID=\"fake\"", "-I" + INCLUDE,
                    "-I" + CSRC, "-I" + cuda, os.path.join(here, "fake_cuda.cpp"),
                    os.path.join(CSRC, "evisel_capi.cpp"), "-o", out, "-Wl,-z,defs",
                    "-Wl,-Bsymbolic"], check=True)   # its own cuda* calls, also where torch has loaded the runtime
    lib = ctypes.CDLL(out)
    lib.evisel_last_error.restype = ctypes.c_char_p
    lib.fake_fail.argtypes = [ctypes.c_char_p, ctypes.c_int]
    lib.evisel_free.argtypes = [ctypes.c_void_p]
    return lib


MAP = ctypes.c_void_p(FAKE)


def _topp(lib, ws, args, block=16):
    return lib.evisel_topp_mask(ctypes.byref(args), block, ctypes.c_float(0.9), MAP, None, None, ctypes.byref(ws))


def _coarse(lib, ws, args, block=16):
    return lib.evisel_coarse_evidence(ctypes.byref(args), ws, block, MAP, MAP, MAP, MAP, MAP, 0, None)


# Two videos of 640 tokens in all, and descriptions with the same total that
# differ in one thing each.
BUILT = dict(cu=[0, 340, 640], n_vis=[256, 256], npf=16, hq=4, hkv=2, d=64)


@pytest.mark.parametrize("over", [
    dict(n_vis=[256, 128]), dict(n_vis=[128, 256]), dict(n_vis=[320, 288]), dict(n_vis=[0, 0]),
    dict(cu=[0, 320, 640]), dict(cu=[0, 640], n_vis=[512]), dict(cu=[0, 340, 640, 640], n_vis=[256, 256, 0]),
    dict(npf=64), dict(npf=8), dict(hq=8), dict(hkv=1), dict(hkv=4), dict(d=128), dict(block=32)])
def test_coarse_map_refuses_another_description_than_the_builders(fake, over):
    """The builder's upload holds the videos' rows and columns: the scratch and
    the maps of a call are sized from its own arguments, so these must be the
    builder's, by value, or the kernels would write past them."""
    ws = ctypes.c_void_p(None)
    built, keep0 = _args(**BUILT)
    assert _topp(fake, ws, built) == 0
    assert _coarse(fake, ws, built) == 0
    n = fake.fake_calls(b"coarse")
    over = dict(over)
    block = over.pop("block", 16)
    other, keep1 = _args(**{**BUILT, **over})
    assert _coarse(fake, ws, other, block) == EINVAL
    assert fake.fake_calls(b"coarse") == n       # refused before any launch
    again, keep2 = _args(**BUILT)                # other arrays, the same values
    assert _coarse(fake, ws, again) == 0
    fake.evisel_free(ws)


@pytest.mark.parametrize("name", [b"cudaMalloc", b"cudaMallocHost", b"cudaMemcpyAsync", b"encode", b"topp"])
def test_coarse_map_is_refused_after_a_builder_call_that_failed(fake, name):
    """A failed rebuild leaves no builder state to read, neither the old call's
    (its buffer may be gone) nor its own."""
    ws = ctypes.c_void_p(None)
    built, keep0 = _args(**BUILT)
    assert _topp(fake, ws, built) == 0
    # (1,000 videos of one row tile each outgrow the buffers of the first call)
    larger, keep1 = _args(cu=list(range(0, 1001 * 32, 32)), n_vis=[16] * 1000, npf=16, hq=4, hkv=2, d=64)
    fake.fake_fail(name, 0)
    assert _topp(fake, ws, larger) in (ENOMEM, ECUDA)
    n = fake.fake_calls(b"coarse")
    for args in (built, larger):
        assert _coarse(fake, ws, args) == ESTATE
    assert fake.fake_calls(b"coarse") == n
    assert _topp(fake, ws, built) == 0 and _coarse(fake, ws, built) == 0
    fake.evisel_free(ws)


@pytest.mark.parametrize("text_evidence", [0, 1])
@pytest.mark.parametrize("name,after", [
    (b"probe_attn", 0), (b"attn_combine", 0), (b"text_evidence", 0), (b"encode", 0), (b"encode", 3), (b"encode", 4),
    (b"encode", 5)])
def test_no_evidence_after_a_probe_that_failed(fake, name, after, text_evidence):
    """A probe call that fails at any of its launches or descriptors leaves
    nothing to hand out, neither its own half nor an older call's sums, whether
    it ran on the plan at hand or on a new one."""
    def probe(ws, args):
        args.text_evidence = text_evidence
        return fake.evisel_probe_attention(ctypes.byref(args), None, ctypes.byref(ws))

    def reduce(ws):
        return fake.evisel_evidence_reduce(ws, MAP, MAP, MAP, MAP, 0, None)

    late = text_evidence and (name == b"text_evidence" or after >= 4)   # then the evidence call's own
    # 128 key tiles and two text tiles: split kv ranges, so the combine runs too
    n = 128 * 64
    row_ptr, cols = np.arange(129), np.arange(128)
    built, keep0 = _args(cu=[0, n + 100], n_vis=[n], row_ptr=row_ptr, col_idx=list(cols))
    other, keep1 = _args(cu=[0, n + 99], n_vis=[n], row_ptr=row_ptr, col_idx=list(cols))
    for args in (built, other):
        ws = ctypes.c_void_p(None)
        assert probe(ws, built) == 0 and reduce(ws) == 0
        fake.fake_fail(name, after)
        if late:
            assert probe(ws, args) == 0
            fake.fake_fail(name, max(after - 4, 0))
            assert reduce(ws) == ECUDA and reduce(ws) == 0
        else:
            assert probe(ws, args) == ECUDA
            runs = fake.fake_calls(b"evidence")
            assert reduce(ws) == ESTATE
            assert fake.fake_calls(b"evidence") == runs
            assert probe(ws, args) == 0 and reduce(ws) == 0
        fake.evisel_free(ws)
