"""The C ABI without a GPU: the library loads, exports every declared symbol, and rejects bad arguments
on the host before anything is enqueued."""
import ctypes as C
import os
import re

import numpy as np
import pytest
import torch

from paper_2401_14110_b200 import binding as lba
from paper_2401_14110_b200 import FLAG_INPUT_M4E3, LbaFormat, code_domain_formats, m4e3_input_formats, ORDER_CHUNKED as CHK, ORDER_SEQUENTIAL as SEQ

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_functions():
    text = open(os.path.join(ROOT, "include", "lba.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(lba_[a-z0-9_]+)\s*\(", text)))


def test_library_exports_every_declared_symbol():
    lib = lba.load_library()
    names = _declared_functions()
    assert "lba_gemm" in names and "lba_conv2d" in names and len(names) >= 10
    for name in names:
        assert getattr(lib, name) is not None
    assert sorted(lba.EXPORTS) == names
    assert lib.lba_version() == 1
    assert lib.lba_status_string(0) == b"ok"


def test_plan_selection_by_format_and_order():
    p, a = code_domain_formats(7, 4)
    assert "q=floor_fast" in lba.describe_plan(64, 64, 576, p, a, SEQ, 16)
    assert "order=seq" in lba.describe_plan(64, 64, 576, p, a, SEQ, 16)
    assert "order=chunk16" in lba.describe_plan(64, 64, 576, p, a, CHK, 16)
    assert "order=chunk_slab" in lba.describe_plan(64, 64, 576, p, a, CHK, 32)
    assert "order=chunk_any" in lba.describe_plan(64, 64, 576, p, a, CHK, 5)
    assert "order=seq" in lba.describe_plan(64, 64, 576, p, a, CHK, 576)       # one chunk == sequential
    assert "q=floor_full" in lba.describe_plan(64, 64, 576, LbaFormat(7, 4, 12), LbaFormat(7, 4, 10), CHK, 16)
    assert "q=floor_full" in lba.describe_plan(64, 64, 576, *code_domain_formats(4, 4), CHK, 16)
    assert "q=rne_full" in lba.describe_plan(64, 64, 576, *code_domain_formats(7, 4, rounding=1), CHK, 16)
    assert "q=rne_wide" in lba.describe_plan(64, 64, 576, LbaFormat(23, 8, 127, 1), LbaFormat(23, 8, 127, 1), SEQ, 16)
    assert "pq=none" in lba.describe_plan(64, 64, 576, p, a, CHK, 16)                # the product flush is reachable
    assert "pq=fused" in lba.describe_plan(64, 64, 576, *code_domain_formats(8, 6), CHK, 16)
    assert "pq=fused" in lba.describe_plan(64, 64, 576, *code_domain_formats(7, 4, flags=0), SEQ, 16)
    assert "pq=cut" in lba.describe_plan(64, 64, 576, *code_domain_formats(5, 6), CHK, 16)
    assert "load=conv_vec" in lba.describe_plan(64, 64, 576, p, a, CHK, 16, is_conv=True)
    assert "load=any" in lba.describe_plan(64, 64, 147, p, a, CHK, 16, is_conv=True, vec_ok=False)


@pytest.mark.parametrize("prod,acc,order,chunk,status", [
    (LbaFormat(0, 4, 8), LbaFormat(7, 4, 8), SEQ, 16, -3),
    (LbaFormat(7, 9, 8), LbaFormat(7, 4, 8), SEQ, 16, -3),
    (LbaFormat(7, 4, 500), LbaFormat(7, 4, 8), SEQ, 16, -3),
    (LbaFormat(7, 4, 8, 3), LbaFormat(7, 4, 8, 3), SEQ, 16, -3),
    (LbaFormat(7, 4, 8, 0), LbaFormat(7, 4, 8, 1), SEQ, 16, -3),          # mixed rounding rules
    (LbaFormat(22, 8, 127, 1), LbaFormat(22, 8, 127, 1), SEQ, 16, -3),    # nearest-even with M = 22
    (LbaFormat(7, 4, 8), LbaFormat(7, 4, 8), 2, 16, -4),
    (LbaFormat(7, 4, 8), LbaFormat(7, 4, 8), CHK, 0, -4),
])
def test_rejected_arguments(prod, acc, order, chunk, status):
    with pytest.raises(lba.LbaError) as e:
        lba.describe_plan(8, 8, 8, prod, acc, order, chunk)
    assert e.value.status == status


def test_host_side_checks_run_before_any_cuda_call():
    lib = lba.load_library()
    p, a = code_domain_formats(7, 4)
    pf, af = lba._fmt(p), lba._fmt(a)
    # null operands, negative sizes, bad scale lengths: all refused without touching a device
    assert lib.lba_gemm(None, None, None, 1, None, 1, None, 4, 4, 4, C.byref(pf), C.byref(af), 0, 16, None, None) == -1
    assert lib.lba_gemm(None, None, None, 1, None, 1, None, -1, 4, 4, C.byref(pf), C.byref(af), 0, 16, None, None) == -2
    fake = C.c_void_p(256)
    assert lib.lba_gemm(fake, fake, fake, 3, fake, 1, None, 4, 4, 4, C.byref(pf), C.byref(af), 0, 16, fake, None) == -5
    assert lib.lba_conv2d(fake, fake, fake, 1, fake, 1, None, 1, 2, 2, 3, 4, 5, 5, 1, 1, 0, 0, C.byref(pf),
                          C.byref(af), 0, 16, fake, None) == -2
    assert lib.lba_gemm_host_workspace_bytes(4, 4, 16, 1, 1, 0) == 256 * 5
    assert lib.lba_set_tile_override(9) == -2 and lib.lba_set_tile_override(-1) == 0


def test_host_variants_refuse_shapes_whose_byte_counts_would_wrap():
    # M*K, N*K and 4*M*N are formed in size_t inside the host-buffer variants: a shape for which one of them does
    # not fit must come back as an error code (and a workspace size of 0), never as a small wrapped size
    lib = lba.load_library()
    p, a = code_domain_formats(7, 4)
    pf, af = lba._fmt(p), lba._fmt(a)
    fake = C.c_void_p(256)
    huge = 1 << 62
    assert lib.lba_gemm_host_workspace_bytes(huge, 1, 4, 1, 1, 0) == 0          # M*K = 2^64
    assert lib.lba_gemm_host_workspace_bytes(1 << 31, 1 << 31, 16, 1, 1, 0) == 0  # 4*M*N = 2^64
    assert lib.lba_gemm_host_workspace_bytes(1 << 20, 1 << 20, 16, 1, 1, 0) > 0   # 4 TiB: large, but it fits
    for (M, N, K) in ((huge, 1, 4), (1 << 31, 1 << 31, 16), (4, 4, 1 << 31)):
        assert lib.lba_gemm_host(fake, fake, fake, 1, fake, 1, None, M, N, K, C.byref(pf), C.byref(af), 1, 16, fake, fake,
                                 C.c_size_t(1 << 40), None) == -2
        assert lib.lba_gemm_host_static(fake, fake, fake, 1, fake, 1, None, M, N, K, C.byref(pf), C.byref(af), 1, 16, fake,
                                        None) in (-2, -8)
    # convolution: the output byte count is guarded the same way
    assert lib.lba_conv2d_host_workspace_bytes(1 << 20, 1, 1, 1, 1 << 20, 1, 1, 1, 1, 0, 0, 1, 1, 0) > 0
    assert lib.lba_conv2d_host_workspace_bytes(1 << 30, 1, 1, 1, 1 << 30, 1, 1, 1, 1, 0, 0, 1, 1, 0) == 0     # 4*M*C_out = 2^62


def test_tile_choice_follows_the_measured_order():
    # the host's tile model is fitted to measurements on B200 (148 SMs is also what the model assumes without a device):
    # these are the shapes it was fitted and checked on, with the tile that measured fastest
    f, r = code_domain_formats(7, 4), code_domain_formats(7, 4, rounding=1)
    tile = lambda shape, fm, order: lba.describe_plan(*shape, *fm, order, 16).split(" q=")[0]
    assert tile((8192, 8192, 8192), f, CHK) == "tile=128x128x16 micro=8x8"       # full SMs, floor: the 8x8 micro-tile
    assert tile((8192, 8192, 8192), f, SEQ) == "tile=128x128x16 micro=8x8"
    assert tile((8192, 8192, 8192), r, CHK) == "tile=64x64x16 micro=4x8"         # nearest-even, chunk 16: 64x64 is 12 % faster
    assert tile((4096, 768, 768), f, CHK) == "tile=64x64x16 micro=4x8"           # BERT linears: not the 32x32 tile
    assert tile((25088, 128, 1152), f, CHK) == "tile=64x64x16 micro=4x8"         # ResNet-18 layer2
    assert tile((1568, 512, 4608), f, CHK) == "tile=64x64x16 pair micro=4x8"     # layer4: two CTAs per tile
    assert tile((1568, 512, 4608), f, SEQ) == "tile=32x32x16 micro=4x4"          # no chunks to share in sequential order
    assert tile((32, 1000, 512), f, CHK) == "tile=32x32x16 micro=4x4"            # the classifier


def test_describe_plan_for_batched_calls():
    # 384 problems of 128x128 fill the SMs with 64x64 tiles; one such problem alone would get the 32x32 tile
    f = code_domain_formats(7, 4)
    assert lba.describe_plan(128, 128, 64, *f, CHK, 16).startswith("tile=32x32x16")
    assert lba.describe_plan(128, 128, 64, *f, CHK, 16, batch=384).startswith("tile=64x64x16 micro=4x8")
    with pytest.raises(lba.LbaError):
        lba.describe_plan(128, 128, 64, *f, CHK, 16, batch=0)


@pytest.mark.parametrize("fmts", [code_domain_formats(7, 4), code_domain_formats(4, 4), code_domain_formats(7, 4, rounding=1),
                                  code_domain_formats(12, 5, rounding=1)], ids=["floor", "cut", "nearest", "nearest_generic"])
@pytest.mark.parametrize("order,chunk", [(SEQ, 16), (CHK, 16), (CHK, 24), (CHK, 32)])
def test_wide_outputs_get_a_tile_that_can_be_launched(fmts, order, chunk):
    # a grid has at most 65535 columns of CTAs: up to 65535 * 128 columns there is a tile that fits, beyond there is none
    for N in (16 * 65535 + 1, 32 * 65535, 32 * 65535 + 1, 64 * 65535, 64 * 65535 + 1, 128 * 65535):
        for M in (1, 17, 80, 96, 280):
            for K in (64, 17):
                plan = lba.describe_plan(M, N, K, *fmts, order, chunk, vec_ok=K % 16 == 0)
                assert int(re.findall(r"grid=\d+x(\d+)", plan)[-1]) <= 65535, (M, N, K, plan)
    with pytest.raises(lba.LbaError) as e:
        lba.describe_plan(4, 128 * 65535 + 1, 64, *fmts, order, chunk)
    assert e.value.status == -2


def test_wide_outputs_of_the_fixed_point_kernel_are_refused_by_the_plan_too():
    f = LbaFormat(16, 0, -4, 0, 0)
    assert "q=fixed" in lba.describe_plan(4, 64 * 65535, 64, f, f)
    with pytest.raises(lba.LbaError) as e:
        lba.describe_plan(4, 64 * 65535 + 1, 64, f, f)
    assert e.value.status == -2


@pytest.mark.parametrize("box", [np.array, torch.tensor, np.int32, float], ids=["array", "tensor", "int32", "float"])
def test_format_fields_are_read_by_value_at_every_call(box):
    p, a = code_domain_formats(7, 4)
    plan = lambda f: lba.describe_plan(512, 512, 512, f, a)
    f = [box(v) for v in p.as_tuple()]
    assert plan(f) == plan(p) == plan(LbaFormat(*f)) == plan(tuple(f))
    if hasattr(f[0], "fill_"):
        f[0].fill_(4)     # the same object, another value
    else:
        f[0] = box(4)
    assert "pq=cut" in plan(f) and "pq=cut" in plan(LbaFormat(*f)) and "pq=none" in plan(p)


WIDE = LbaFormat(23, 8, 127, 1, 0)
FASTEST = [   # formats, order, chunk, shape, the tile that measured fastest (us against the next one)
    (code_domain_formats(12, 5, 1), SEQ, 16, (2048, 1024, 1024), "32x32"),    # 2080, 2278
    (code_domain_formats(12, 5, 1), SEQ, 16, (4096, 4096, 512), "128x64"),    # 7161, 7923
    (code_domain_formats(12, 5, 1), CHK, 16, (4096, 4096, 512), "128x64"),    # 7416, 8443
    (code_domain_formats(12, 5, 1), CHK, 24, (512, 512, 512), "32x32"),       # 156, 289
    ((WIDE, WIDE), CHK, 16, (3000, 1500, 1008), "64x64"),                     # 389, 405
    ((WIDE, WIDE), CHK, 24, (25088, 128, 256), "64x64"),                      # 92, 94
    (code_domain_formats(7, 4), CHK, 32, (25088, 128, 256), "64x64"),         # 97, 100
    (code_domain_formats(7, 4), CHK, 16, (2048, 1024, 1024), "64x64"),        # 242, 244; the 128x128 tile 254
    (code_domain_formats(7, 4), SEQ, 16, (12288, 128, 64), "64x64"),          # 14.3, 15.5
    (code_domain_formats(4, 4), SEQ, 16, (512, 512, 512), "32x32"),           # 32.8; the chain kernel 42
    (code_domain_formats(4, 4), SEQ, 16, (64, 4096, 2048), "32x32"),          # 124; the chain kernel 158
    (code_domain_formats(4, 4), CHK, 16, (64, 4096, 2048), "32x32"),          # 132; the split kernels 138
]


@pytest.mark.parametrize("fmts,order,chunk,shape,tile", FASTEST, ids=lambda v: str(v) if isinstance(v, (str, int)) else "")
def test_tile_choice_knows_each_kernel(fmts, order, chunk, shape, tile):
    plan = lba.describe_plan(*shape, *fmts, order, chunk)
    assert plan.startswith(f"tile={tile}x16 micro") and "by=" not in plan


M4E3 = m4e3_input_formats(7, 4)
RUNS = [   # formats, order, shape, convolution, what runs (us; with weights scaled per channel where two figures stand; the next one)
    (code_domain_formats(7, 4), SEQ, (128, 1000, 512), False, "chain16x16"),          # 20.5, 20.8; 32x32 22.6, 39.4
    (code_domain_formats(7, 4), SEQ, (256, 512, 4608), True, "chain16x16"),           # 171; 32x32 189
    (code_domain_formats(7, 4), SEQ, (49, 2048, 512), True, "chain16x16"),            # 21.6; 32x32 26.0
    (code_domain_formats(7, 4), SEQ, (16, 8192, 4096), False, "chain16x16"),          # 152, 153; 32x32 173, 249
    (code_domain_formats(7, 4), SEQ, (379, 3296, 144), False, "tile=32x32"),          # 22.7, 27.2; 64x64 25.7, 34.1
    (code_domain_formats(7, 4), SEQ, (3136, 128, 64), True, "tile=32x32"),            # 6.5; 64x64 8.1
    (code_domain_formats(4, 4), SEQ, (256, 512, 2304), True, "chain16x16"),           # 100; 32x32 118
    (M4E3, SEQ, (128, 1000, 512), False, "chain16x16"),                               # 24.1; 32x32 28.8
    (code_domain_formats(4, 4), CHK, (1931, 96, 2016), False, "split16x16"),          # 90; 32x32 112
    (M4E3, CHK, (1931, 96, 2016), False, "split16x16"),                               # 94; 32x32 115
    (code_domain_formats(10, 5, 1), SEQ, (64, 4096, 2048), False, "chain16x16"),      # 141, 143; 32x32 156, 165
    (code_domain_formats(10, 5, 1), SEQ, (2048, 1024, 1024), False, "tile=32x32"),    # 310, 322; 128x64 343, 357; 128x128 358, 377
    (code_domain_formats(10, 5, 1), SEQ, (4096, 4096, 4096), False, "tile=64x64"),    # 8950, 9130; 128x128 10200, 10540
]


@pytest.mark.parametrize("fmts,order,shape,conv,what", RUNS, ids=lambda v: str(v) if isinstance(v, (str, int)) else "")
def test_tile_choice_by_the_times_of_the_present_kernels(fmts, order, shape, conv, what):
    plan = lba.describe_plan(*shape, *fmts, order, 16, is_conv=conv, vec_ok=shape[2] % 16 == 0)
    assert (plan.partition(" by=")[2] or plan).startswith(what)


@pytest.mark.parametrize("fmts", [code_domain_formats(7, 4), code_domain_formats(10, 6), code_domain_formats(4, 4), code_domain_formats(10, 5, 1)],
                         ids=["floor", "fused", "cut", "nearest"])
@pytest.mark.parametrize("order,chunk", [(SEQ, 16), (CHK, 16), (CHK, 24), (CHK, 32)])
def test_tile_choice_of_a_convolution_with_few_channels(fmts, order, chunk):
    # 4 images of 64 x 64 x 24 through 64 3x3 filters: 128x64 is 3 to 11 % faster than 64x64 in every mode
    assert lba.describe_plan(16384, 64, 216, *fmts, order, chunk, is_conv=True, vec_ok=False).startswith("tile=128x64x16")
    # the ResNet stem, batch 1: 64x64 or 32x32 tiles fill the SMs
    assert lba.describe_plan(12544, 64, 147, *fmts, order, chunk, is_conv=True, vec_ok=False).startswith(("tile=64x64x16", "tile=32x32x16"))


def test_plan_names_the_small_kernel_that_runs():
    by = lambda shape, fm, order, chunk=16, **kw: lba.describe_plan(*shape, *fm, order, chunk, **kw).partition(" by=")[2]
    formats = {"none": [code_domain_formats(7, 4), code_domain_formats(10, 5, 1), code_domain_formats(10, 6), code_domain_formats(10, 7, 1)],
               "cut": [code_domain_formats(4, 4), code_domain_formats(4, 4, 1)], "cut_sat": [(LbaFormat(5, 4, 4), LbaFormat(7, 4, 6))]}
    for pq, several in formats.items():   # M10E6 and M10E7 are fused in the packed kernel, which has that variant
        for f in several:
            # a small problem gets the small kernels by itself, whatever the mode; one that fills the SMs does not
            assert by((64, 64, 576), f, CHK) == f"split16x16(micro=2x4,grid=4x4,pq={pq})"
            assert by((32, 1000, 512), f, CHK) == f"split16x16(micro=2x4,grid=2x63,pq={pq})"      # the classifier
            assert by((64, 64, 576), f, SEQ) == f"chain16x16(micro=1x2,grid=4x4,pq={pq})"
            assert by((49, 512, 4608), f, SEQ, is_conv=True) == f"chain16x16(micro=1x2,grid=4x32,pq={pq})"
            assert by((4096, 4096, 4096), f, CHK) == by((4096, 4096, 4096), f, SEQ) == by((64, 64, 576), f, CHK, 32) == ""
    assert by((512, 768, 768), code_domain_formats(7, 4), CHK) == "split32x32(micro=4x8,grid=16x24,pq=none)"


def test_cuts_too_short_for_the_operand_scales_run_without_a_clamp():
    # x (1 + 2^(23 - M)) must fit 24 bits beside x's own: M >= 3 on E4M3 bytes, M >= 4 on M4E3.  Below that the product is cut by
    # itself; only one that can saturate (R_OF_prod <= 448^2, 248^2) is clamped too
    import bench
    a = code_domain_formats(7, 4)[1]
    for order, chunk in ((SEQ, 16), (CHK, 16), (CHK, 32)):
        for flags, fits, bias in ((1, 3, 14), (1 | FLAG_INPUT_M4E3, 4, 15)):   # biases at which nothing of 2 bits and more saturates
            for man, more, want in ((fits, 0, "cut"), (fits - 1, 0, "cut_any"), (2, 0, "cut_any"), (2, 4, "cut_sat")):
                plan = lba.describe_plan(4096, 4096, 4096, LbaFormat(man, 5, bias + more, 0, flags), a, order, chunk)
                assert re.search(r"pq=(\w+)", plan)[1] == want and bench.mode_of(plan) == "floor_" + want, (man, more, plan)
    assert bench.min_issue_slots("floor_cut_any", 0) == 3.0


def test_benchmark_mix_is_that_of_the_kernel_that_runs():
    import bench
    mode = lambda shape, f, order: bench.mode_of(lba.describe_plan(*shape, *f, order, 16), acc_man_bits=f[1].man_bits)
    small, large = (64, 64, 576), (4096, 4096, 4096)
    assert mode(large, code_domain_formats(10, 6), CHK) == "floor_fused" and mode(small, code_domain_formats(10, 6), CHK) == "floor"
    assert mode(large, code_domain_formats(7, 4, 1), CHK) == "rne_bf16" and mode(large, code_domain_formats(7, 4, 1), SEQ) == "rne"
    assert mode(large, code_domain_formats(5, 5, 1), CHK) == "rne_cut" and mode(large, code_domain_formats(12, 5, 1), CHK) == "generic"
    # two packed instructions cut a pair: half of FMUL2, FFMA2, FMUL2, FFMA2 per MAC; a chunk adds the fold's FADD2, cut and
    # clamp (2.5) and saves the first step's FFMA2 and cut (1.5)
    assert bench.min_issue_slots("rne", 0) == 2.0 and bench.min_issue_slots("rne", 16) == 2.0625
    assert bench.min_issue_slots("floor", 16) == 2.0625 and bench.min_issue_slots("floor", 32) == 2 + 2.5 / 32
    assert all(bench.clocks_per_warp_mac(m, c)[0] >= bench.min_issue_slots(m, c) for m in bench.MIX for c in (0, 16, 24))
