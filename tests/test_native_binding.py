"""The native path of the forward entry points against their ctypes path: same results, same refusals."""
import gc

import numpy as np
import pytest
import torch

from paper_2401_14110_b200 import binding as lba
from paper_2401_14110_b200 import build as lba_build
from paper_2401_14110_b200 import synth, code_domain_formats, ORDER_SEQUENTIAL as SEQ, ORDER_CHUNKED as CHK

P, A12 = code_domain_formats(7, 4)


@pytest.fixture(autouse=True)
def _leave_no_tensors():
    # raised exceptions keep frames, and their tensors, until the next collection: not into a test that counts memory
    yield
    gc.collect()


def test_irregular_calls_are_left_to_ctypes():
    lba.load_library()
    a, one = torch.zeros(4, 16, dtype=torch.uint8), torch.ones(1)
    assert lba._native.gemm(a, a, one, one, None, P, A12, CHK, 16, None, None) is None          # not on the GPU
    assert lba._native.gemm(None, a, one, one, None, P, A12, CHK, 16, None, None) is None       # not a tensor
    assert lba._native.gemm(a, a, one, one, None, P, A12, CHK, 16) is None                      # too few arguments
    assert lba._native.conv2d(a, a, one, one, None, [1, 1], (0, 0), P, A12, CHK, 16, None, None) is None


@pytest.fixture
def reloaded():
    """The binding as a fresh process finds it; the library as it was loaded afterwards."""
    lib, native, path = lba.load_library(), lba._native, lba.TORCH_LIB_PATH
    lba._lib = lba._native = None
    yield
    lba._lib, lba._native, lba.TORCH_LIB_PATH = lib, native, path


def _without_native():
    with pytest.warns(RuntimeWarning, match="ctypes"):
        lba.load_library()
    assert lba._native is None
    assert "q=floor_fast" in lba.describe_plan(64, 64, 576, P, A12, CHK, 16)
    a, one = torch.zeros(4, 16, dtype=torch.uint8), torch.ones(1)
    with pytest.raises(TypeError):                      # reached the checks of the ctypes path
        lba.lba_gemm(a, a, one, one, None, P, A12, CHK, 16)


def test_without_the_native_module_calls_go_through_ctypes(reloaded, tmp_path):
    lba.TORCH_LIB_PATH = str(tmp_path / "lba_torch.so")
    _without_native()


def test_a_native_module_that_cannot_be_imported_is_left_out(reloaded, tmp_path):
    (tmp_path / "lba_torch.so").write_bytes(b"not a shared library")
    lba.TORCH_LIB_PATH = str(tmp_path / "lba_torch.so")
    _without_native()


def test_a_native_module_of_another_torch_is_left_out_and_rebuilt(reloaded, monkeypatch):
    assert lba_build._carries(lba_build.TORCH_LIB, lba_build.torch_tag())
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    _without_native()
    assert not lba_build._carries(lba_build.TORCH_LIB, lba_build.torch_tag())    # a build now compiles it anew


def test_a_failed_build_of_the_native_module_leaves_the_library(monkeypatch):
    def fail(force):
        raise RuntimeError("no compiler")
    monkeypatch.setattr(lba_build, "build_torch", fail)
    monkeypatch.setattr(lba_build, "_sources", lambda: [])
    monkeypatch.setattr(lba_build, "_stale", lambda target, sources: False)
    with pytest.warns(UserWarning, match="no compiler"):
        assert lba_build.build() == lba_build.LIB


@pytest.mark.gpu
def test_forward_calls_without_the_native_module(reloaded, tmp_path):
    a, one = synth.random_codes((20, 48), 1).to("cuda:0"), torch.ones(1, device="cuda:0")
    want = lba.lba_gemm(a, a, one, one, None, P, A12)
    lba._lib = lba._native = None
    lba.TORCH_LIB_PATH = str(tmp_path / "lba_torch.so")
    with pytest.warns(RuntimeWarning):
        got = lba.lba_gemm(a, a, one, one, None, P, A12)
    assert lba._native is None and torch.equal(got.view(torch.int32), want.view(torch.int32))


@pytest.mark.gpu
def test_native_and_ctypes_paths_agree():
    dev = "cuda:0"
    one, sb, bias = torch.ones(1, device=dev), torch.rand(37, device=dev), torch.rand(37, device=dev)
    a, b = synth.random_codes((3, 21, 48), 1).to(dev), synth.random_codes((3, 37, 48), 2).to(dev)
    x, w = synth.random_codes((2, 9, 11, 16), 3).to(dev), synth.random_codes((37, 3, 2, 16), 4).to(dev)
    here = torch.cuda.current_stream()
    for order in (SEQ, CHK):
        for pf, af in ((P, A12), (P.as_tuple(), A12.as_tuple())):
            calls = [(lba.lba_gemm, (a[0], b[0], one, sb, bias, pf, af, order, 16)),
                     (lba.lba_gemm_batched, (a, b, one, sb, None, pf, af, order, 16)),
                     (lba.lba_gemm_batched, (a, b[1], one, one, bias, pf, af, order, 16)),
                     (lba.lba_conv2d, (x, w, one, sb, bias, (2, 1), (1, 0), pf, af, order, 16))]
            for f, args in calls:
                want = f(*args, stream=here)            # an explicit stream is the ctypes path's
                assert lba._native is not None and torch.equal(f(*args).view(torch.int32), want.view(torch.int32))
                out = torch.empty_like(want)
                assert f(*args, out=out) is out and torch.equal(out.view(torch.int32), want.view(torch.int32))
    side = torch.cuda.Stream()
    side.wait_stream(here)
    with torch.cuda.stream(side):                       # the current stream is the one that is used
        got = lba.lba_gemm(a[0], b[0], one, sb, bias, P, A12, CHK, 16)
    side.synchronize()
    assert torch.equal(got.view(torch.int32), lba.lba_gemm(a[0], b[0], one, sb, bias, P, A12, CHK, 16, stream=here).view(torch.int32))


@pytest.mark.gpu
def test_parameters_are_regular_operands():
    dev = "cuda:0"
    a, b = synth.random_codes((21, 48), 1).to(dev), synth.random_codes((37, 48), 2).to(dev)
    x, w = synth.random_codes((2, 9, 11, 16), 3).to(dev), synth.random_codes((37, 3, 2, 16), 4).to(dev)
    one, sb, bias = torch.ones(1, device=dev), torch.rand(37, device=dev), torch.rand(37, device=dev)
    par = lambda t: torch.nn.Parameter(t, requires_grad=t.is_floating_point())
    for f, native, args in ((lba.lba_gemm, "gemm", (a, b, one, sb, bias, P, A12, CHK, 16)),
                            (lba.lba_gemm_batched, "gemm_batched", (a[None], b, one, sb, bias, P, A12, SEQ, 16)),
                            (lba.lba_conv2d, "conv2d", (x, w, one, sb, bias, (1, 1), (0, 0), P, A12, CHK, 16))):
        want = f(*args)
        got = getattr(lba._native, native)(*(par(t) if isinstance(t, torch.Tensor) else t for t in args), None, None)
        assert type(got) is torch.Tensor and not got.requires_grad
        assert torch.equal(got.view(torch.int32), want.view(torch.int32))


@pytest.mark.gpu
def test_what_was_refused_stays_refused():
    dev = "cuda:0"
    one = torch.ones(1, device=dev)
    a, b = synth.random_codes((8, 32), 1).to(dev), synth.random_codes((8, 48), 2).to(dev)
    with pytest.raises(ValueError):
        lba.lba_gemm(a, b, one, one, None, P, A12)
    with pytest.raises(TypeError):
        lba.lba_gemm(a, synth.random_codes((8, 64), 2).to(dev)[:, ::2], one, one, None, P, A12)  # not contiguous
    with pytest.raises(TypeError):
        lba.lba_gemm(a.float(), a, one, one, None, P, A12)
    with pytest.raises(TypeError):
        lba.lba_gemm(a, a, one.cpu(), one, None, P, A12)
    with pytest.raises(lba.LbaError):
        lba.lba_gemm(a, a, torch.ones(3, device=dev), one, None, P, A12)        # scale length
    with pytest.raises(lba.LbaError):
        lba.lba_gemm(a, a, one, one, None, P, A12, 7, 16)                       # order
    # arguments of other types go on being accepted
    want = lba.lba_gemm(a, a, one, one, None, P, A12).view(torch.int32)
    for args in ((torch.nn.Parameter(a, requires_grad=False), a, one, one, None, P, A12, True),
                 (a, a, one, one, None, list(P.as_tuple()), A12, CHK, np.int64(16))):
        assert torch.equal(lba.lba_gemm(*args).view(torch.int32), want)
    x, w = a.view(1, 1, 8, 32), a.view(8, 1, 1, 32)
    assert torch.equal(lba.lba_conv2d(x, w, one, one, None, [1, 1], [0, 0], P, A12).view(8, 8).view(torch.int32), want)


@pytest.mark.gpu
def test_regular_calls_are_made_by_the_native_functions():
    # called directly, for an entry point goes on through ctypes where they return None
    dev = "cuda:0"
    one, sb, bias = torch.ones(1, device=dev), torch.rand(37, device=dev), torch.rand(37, device=dev)
    a, b = synth.random_codes((3, 21, 48), 1).to(dev), synth.random_codes((3, 37, 48), 2).to(dev)
    x, w = synth.random_codes((2, 9, 11, 16), 3).to(dev), synth.random_codes((37, 3, 2, 16), 4).to(dev)
    here, side = torch.cuda.current_stream(), torch.cuda.Stream()
    lba.load_library()
    native = lba._native
    for order in (SEQ, CHK):
        for pf, af in ((P, A12), (P.as_tuple(), A12.as_tuple())):
            for f, direct, args in ((lba.lba_gemm, native.gemm, (a[0], b[0], one, sb, bias, pf, af, order, 16)),
                                    (lba.lba_gemm_batched, native.gemm_batched, (a, b, one, sb, None, pf, af, order, 16)),
                                    (lba.lba_gemm_batched, native.gemm_batched, (a, b[1], one, one, bias, pf, af, order, 16)),
                                    (lba.lba_conv2d, native.conv2d, (x, w, one, sb, bias, (2, 1), (1, 0), pf, af, order, 16))):
                want = f(*args, stream=here).view(torch.int32)
                out = torch.empty_like(want).view(torch.float32)
                assert direct(*args, out, None) is out
                side.wait_stream(here)
                with torch.cuda.stream(side):
                    on_side = direct(*args, None, None)
                side.synchronize()
                for got in (out, direct(*args, None, None), on_side):
                    assert type(got) is torch.Tensor and torch.equal(got.view(torch.int32), want)
