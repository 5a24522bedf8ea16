"""Kernel variants at the sizes where they can go wrong, against the CPU oracle, bit for bit.  Needs a B200."""
import gc

import numpy as np
import pytest
import torch

from oracle import lba_oracle as orc
from paper_2401_14110_b200 import binding as lba
from paper_2401_14110_b200 import synth
from paper_2401_14110_b200 import (FLAG_INPUT_M4E3, LbaFormat, code_domain_formats, m4e3_input_formats, ORDER_SEQUENTIAL as SEQ,
                                   ORDER_CHUNKED as CHK)

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def check_gemm(A, B, prod, acc, order, chunk=16, what=""):
    one = torch.ones(1)
    got = lba.lba_gemm(A.to(DEV), B.to(DEV), one.to(DEV), one.to(DEV), None, prod, acc, order, chunk)
    want = orc.gemm(A.numpy(), B.numpy(), one.numpy(), one.numpy(), None, prod.as_tuple(), acc.as_tuple(), order, chunk)
    assert (got.cpu().numpy().view(np.uint32) == want.view(np.uint32)).all(), what


@pytest.mark.parametrize("rounding", [0, 1])
@pytest.mark.parametrize("man", [1, 3, 4, 5, 6, 7, 8, 10])
def test_rounding_cuts_of_every_width(man, rounding):
    # product and sum cut to `man` bits, in both orders, E4M3 and M4E3 bytes; dense codes and Gaussian data; every tile,
    # for by itself the shape runs in the small-problem kernels, whose cuts are not those of the packed kernel
    for exp in (4, 5, 6):
        for make, dense in ((code_domain_formats, synth.random_codes((70, 112), 3)),
                            (m4e3_input_formats, torch.arange(70 * 112).mul(37).to(torch.uint8).reshape(70, 112))):
            prod, acc = make(man, exp, rounding)
            B = dense.flip(0).roll(5, 1)[:67].contiguous()
            a, b, one = dense.to(DEV), B.to(DEV), torch.ones(1)
            for order, tiles in ((SEQ, (-1, 0, 1, 2, 3, 10)), (CHK, (-1, 0, 1, 2, 3, 5, 6, 7))):
                want = orc.gemm(dense.numpy(), B.numpy(), one.numpy(), one.numpy(), None, prod.as_tuple(), acc.as_tuple(), order, 16)
                for tile in tiles:
                    lba.set_tile_override(tile)
                    try:
                        plan = lba.describe_plan(70, 67, 112, prod, acc, order, 16)
                        got = lba.lba_gemm(a, b, one.to(DEV), one.to(DEV), None, prod, acc, order, 16).cpu().numpy()
                    finally:
                        lba.set_tile_override(-1)
                    what = f"{make.__name__} M{man}E{exp} r{rounding} order {order} tile {tile}: {plan}"
                    assert (got.view(np.uint32) == want.view(np.uint32)).all(), what
                    if 0 <= tile < 4:
                        assert plan.startswith("tile=" + ("128x128", "128x64", "64x64", "32x32")[tile]) and "by=" not in plan, what
                    elif tile == 5:
                        assert (" pair " in plan) == (rounding == 0), what
                    elif tile > 5:
                        assert ({6: "by=split16x16", 7: "by=split32x32", 10: "by=chain16x16"}[tile] in plan) == ("kernel=packed" in plan), what
                    if rounding == 0:
                        assert "kernel=packed" in plan, what


@pytest.mark.parametrize("K", [1, 15, 16, 17, 31, 33, 130])
def test_rows_at_every_byte_address(K):
    # operands that start at every offset from a 16-byte boundary, at the very end of their storage, K around whole blocks
    prod, acc = code_domain_formats(7, 4)
    M, N = 5, 35
    one = torch.ones(1, device=DEV)
    for off in range(16):
        A, B = synth.random_codes((M, K), 100 + off), synth.random_codes((N, K), 200 + off)
        store = [torch.full((off + t.numel(),), 0x7F, dtype=torch.uint8, device=DEV) for t in (A, B)]
        a, b = [s[off:].view(t.shape).copy_(t) for s, t in zip(store, (A, B))]
        for order in (SEQ, CHK):
            got = lba.lba_gemm(a, b, one, one, None, prod, acc, order, 16).cpu().numpy()
            want = orc.gemm(A.numpy(), B.numpy(), np.ones(1, np.float32), np.ones(1, np.float32), None, prod.as_tuple(),
                            acc.as_tuple(), order, 16)
            assert (got.view(np.uint32) == want.view(np.uint32)).all(), (off, order)


SMALL_FORMATS = {
    "m7e4": code_domain_formats(7, 4), "m4e4": code_domain_formats(4, 4), "m10e6": code_domain_formats(10, 6),
    "m7e4_rne": code_domain_formats(7, 4, 1), "m10e5_rne": code_domain_formats(10, 5, 1), "m4e4_rne": code_domain_formats(4, 4, 1),
    "m7e4_m4e3": m4e3_input_formats(7, 4), "m7e4_low_top": (LbaFormat(7, 4, 4), LbaFormat(7, 4, 6)),
}


@pytest.mark.parametrize("tile", [6, 7, 10])
@pytest.mark.parametrize("name", list(SMALL_FORMATS))
def test_small_problem_kernels(tile, name):
    # edges of the tiles, one to many rounds of chunks, short last chunk and round, saturating data; all loaders
    prod, acc = SMALL_FORMATS[name]
    order = CHK if tile < 10 else SEQ
    one = torch.ones(1)
    lba.set_tile_override(tile)
    try:
        for (M, N, K) in ((1, 1, 17), (16, 32, 32), (33, 47, 127), (5, 100, 128), (40, 17, 144), (31, 33, 1040), (2, 64, 1039)):
            A, B = synth.random_codes((M, K), 7 * M + K), synth.random_codes((N, K), 11 * N + K)
            if K == 1040:
                A, B = A & 0x7F, B & 0x7F
                A[:, 600:] |= 0x80
            by = lba.describe_plan(M, N, K, prod, acc, order, 16, vec_ok=K % 16 == 0).partition(" by=")[2]
            assert by.startswith({6: "split16x16(", 7: "split32x32(", 10: "chain16x16("}[tile]), by
            sa, sb, bias = torch.linspace(0.5, 1.5, M), torch.linspace(0.01, 0.02, N), torch.linspace(-1, 1, N)
            got = lba.lba_gemm(A.to(DEV), B.to(DEV), sa.to(DEV), sb.to(DEV), bias.to(DEV), prod, acc, order, 16).cpu().numpy()
            want = orc.gemm(A.numpy(), B.numpy(), sa.numpy(), sb.numpy(), bias.numpy(), prod.as_tuple(), acc.as_tuple(), order, 16)
            assert (got.view(np.uint32) == want.view(np.uint32)).all(), (M, N, K)
        x, w = synth.random_codes((2, 5, 7, 32), 1), synth.random_codes((19, 3, 3, 32), 2)
        got = lba.lba_conv2d(x.to(DEV), w.to(DEV), one.to(DEV), one.to(DEV), None, (2, 1), (1, 1), prod, acc, order, 16).cpu().numpy()
        want = orc.conv2d(x.numpy(), w.numpy(), one.numpy(), one.numpy(), None, (2, 1), (1, 1), prod.as_tuple(), acc.as_tuple(), order, 16)
        assert (got.view(np.uint32) == want.view(np.uint32)).all()
        A, B = synth.random_codes((3, 20, 48), 5), synth.random_codes((3, 35, 48), 6)
        got = lba.lba_gemm_batched(A.to(DEV), B.to(DEV), one.to(DEV), one.to(DEV), None, prod, acc, order, 16).cpu().numpy()
        for z in range(3):
            want = orc.gemm(A[z].numpy(), B[z].numpy(), one.numpy(), one.numpy(), None, prod.as_tuple(), acc.as_tuple(), order, 16)
            assert (got[z].view(np.uint32) == want.view(np.uint32)).all()
    finally:
        lba.set_tile_override(-1)


@pytest.mark.parametrize("name,fmts", [
    ("plain", code_domain_formats(7, 4)), ("fused", code_domain_formats(10, 6)), ("cut", code_domain_formats(4, 4)),
    ("product_wider", (LbaFormat(7, 4, -2), LbaFormat(5, 4, -4))), ("flush_not_shared", (LbaFormat(7, 4, -2), LbaFormat(7, 4, 0))),
    ("no_acc_flush", (LbaFormat(7, 4, -2), LbaFormat(7, 4, -4, 0, 0))), ("saturating", (LbaFormat(7, 4, 12), LbaFormat(7, 4, 10))),
    ("rne", code_domain_formats(7, 4, 1)), ("rne_cut", code_domain_formats(4, 4, 1)),
    # M4E3 bytes, whose products are the widest (10 bits)
    ("m4e3_cut", m4e3_input_formats(7, 4)), ("m4e3_fused", m4e3_input_formats(9, 4)),
    ("m4e3_flush", (LbaFormat(9, 4, -3, 0, 5), LbaFormat(9, 4, -5))), ("m4e3_cut_flush", (LbaFormat(6, 4, -3, 0, 5), LbaFormat(7, 4, -5))),
    ("m4e3_product_wider", (LbaFormat(9, 4, -3, 0, 5), LbaFormat(7, 4, -5))),
    ("m4e3_rne_flush", (LbaFormat(9, 4, -3, 1, 5), LbaFormat(9, 4, -5, 1))), ("m4e3_rne_cut", m4e3_input_formats(7, 4, 1))], ids=lambda v: v if isinstance(v, str) else "")
@pytest.mark.parametrize("tile", [0, 2, 5])
def test_first_step_of_a_chunk(tile, name, fmts):
    # chunks whose first product is tiny, short or large: the step that may leave out the mask and one multiplication
    A, B = synth.random_codes((65, 80), 5), synth.random_codes((70, 80), 6)
    A[:40, ::16] = torch.arange(40, dtype=torch.uint8)[:, None]      # subnormal and small codes
    B[:30, ::16] = torch.arange(1, 31, dtype=torch.uint8)[:, None]
    lba.set_tile_override(tile)
    try:
        check_gemm(A, B, *fmts, CHK, what=name)
        check_gemm(A[:, :77].contiguous(), B[:, :77].contiguous(), *fmts, CHK, what=name)
    finally:
        lba.set_tile_override(-1)


@pytest.mark.parametrize("tile", [2, 7])
@pytest.mark.parametrize("name", ["m7e4", "m4e4", "m10e6"])
def test_mask_passes_on_both_tiles(tile, name):
    # edges of the tiles, words of the masks cut short, saturating data
    prod, acc = SMALL_FORMATS[name]
    t, a = prod.as_tuple(), acc.as_tuple()
    lba.set_tile_override(tile)
    try:
        for (M, N, K) in ((1, 1, 1), (33, 31, 40), (65, 70, 545), (30, 100, 528)):
            A, B = synth.random_codes((M, K), 3 * M + K), synth.random_codes((N, K), 5 * N + K)
            if K == 545:
                A, B = A & 0x7F, B & 0x7F
            g = lambda x: x.cpu().numpy().view(np.uint32)
            for order in (SEQ, CHK):
                for kind, e1, e2 in ((lba.STE_OF, 0.0, 0.0), (lba.STE_DIFF, 4.0, 2.0 ** -7)):
                    m1, m2 = lba.lba_gemm_ste_mask(A.to(DEV), B.to(DEV), prod, acc, order, 16, kind, e1, e2)
                    w1, w2 = orc.gemm_ste_mask(A.numpy(), B.numpy(), t, a, order, 16, kind, e1, e2)
                    assert (g(m1) == w1).all() and (m2 is None or (g(m2) == w2).all()), (M, N, K, order, kind)
            last = lba.lba_gemm_last_overflow(A.to(DEV), B.to(DEV), prod, acc).cpu().numpy()
            assert (last == orc.gemm_last_overflow(A.numpy(), B.numpy(), t, a)).all(), (M, N, K)
    finally:
        lba.set_tile_override(-1)


@pytest.mark.parametrize("tile", [2, 7])
@pytest.mark.parametrize("name", ["m7e4", "m4e4"])
@pytest.mark.parametrize("chunk", [7, 24, 32, 40])
def test_mask_passes_of_other_chunk_lengths_on_both_tiles(tile, name, chunk):
    # the scalar kernels: chunks that end inside a slab, a slab that holds several, short last chunks and words
    prod, acc = SMALL_FORMATS[name]
    t, a = prod.as_tuple(), acc.as_tuple()
    lba.set_tile_override(tile)
    try:
        for (M, N, K) in ((1, 1, 1), (33, 31, 48), (65, 70, 301), (30, 100, 272)):
            A, B = synth.random_codes((M, K), 3 * M + K), synth.random_codes((N, K), 5 * N + K)
            if K == 301:
                A, B = A & 0x7F, B & 0x7F
            for kind, e1, e2 in ((lba.STE_OF, 0.0, 0.0), (lba.STE_DIFF, 4.0, 2.0 ** -7)):
                got = lba.lba_gemm_ste_mask(A.to(DEV), B.to(DEV), prod, acc, CHK, chunk, kind, e1, e2)
                want = orc.gemm_ste_mask(A.numpy(), B.numpy(), t, a, CHK, chunk, kind, e1, e2)
                for g, w in zip(got, want):
                    assert (g.cpu().numpy().view(np.uint32) == w).all(), (M, N, K, kind)
    finally:
        lba.set_tile_override(-1)


@pytest.mark.parametrize("man", [1, 2, 3, 4, 6, 8])
@pytest.mark.parametrize("wa", ["e4m3", "m4e3"])
def test_floor_cut_inside_the_operand_scales(wa, man):
    # every pair of codes as the only product of a chain, at the first step of a chunk, inside one and in the second slab: the cut
    # that A's scales carry, down to the shortest mantissa they can (E4M3: 3 bits, M4E3: 4) and below, with the product
    # flush in reach and not.  (E4M3 products have 8 bits: M = 8 is no cut.)
    for bias in (-6, 0):
        prod = LbaFormat(man, 5, bias, 0, 1 | (FLAG_INPUT_M4E3 if wa == "m4e3" else 0))
        acc = LbaFormat(man, 5, bias - 2)
        for pos in (0, 5, 18):
            A = torch.zeros(256, 20, dtype=torch.uint8)
            A[:, pos] = torch.arange(256, dtype=torch.uint8)
            if wa == "e4m3":
                A[127, pos] = A[255, pos] = 0  # NaN codes
            for tile in (0, 2, 3) if pos == 0 else (2,):
                lba.set_tile_override(tile)
                try:
                    for order in (SEQ, CHK):
                        check_gemm(A, A, prod, acc, order, what=f"{wa} M{man} bias {bias} step {pos} tile {tile}")
                finally:
                    lba.set_tile_override(-1)


@pytest.mark.parametrize("order,chunk", [(SEQ, 16), (CHK, 16), (CHK, 32)])
@pytest.mark.parametrize("prod,acc", [(LbaFormat(2, 5, 14), LbaFormat(2, 5, 12)),
                                      (LbaFormat(3, 6, 47, 0, 1 | FLAG_INPUT_M4E3), LbaFormat(3, 6, 45))], ids=["e4m3", "m4e3"])
def test_short_cuts_without_saturation(prod, acc, order, chunk):
    # mantissas that A's scales cannot carry, of products that cannot saturate: every tile and loader, and the overflow masks
    assert "pq=cut_any" in lba.describe_plan(4096, 4096, 4096, prod, acc, order, chunk)
    fmts = prod.as_tuple(), acc.as_tuple()
    one, any_code = torch.ones(1), lambda *shape: synth.random_codes(shape, sum(shape))
    gemms = [(any_code(70, K), any_code(67, K)) for K in (33, 112)]
    convs = [(any_code(2, 9, 7, C), any_code(67, 3, 3, C)) for C in (3, 16)]
    want = [orc.gemm(a.numpy(), b.numpy(), one.numpy(), one.numpy(), None, *fmts, order, chunk) for a, b in gemms]
    want += [orc.conv2d(x.numpy(), w.numpy(), one.numpy(), one.numpy(), None, (1, 1), (1, 1), *fmts, order, chunk) for x, w in convs]
    d = one.to(DEV)
    for tile in (-1, 0, 1, 2, 3) + ((5,) if order == CHK and chunk == 16 else ()):
        lba.set_tile_override(tile)
        try:
            got = [lba.lba_gemm(a.to(DEV), b.to(DEV), d, d, None, prod, acc, order, chunk) for a, b in gemms]
            got += [lba.lba_conv2d(x.to(DEV), w.to(DEV), d, d, None, (1, 1), (1, 1), prod, acc, order, chunk) for x, w in convs]
        finally:
            lba.set_tile_override(-1)
        for g, w in zip(got, want):
            assert (g.cpu().numpy().view(np.uint32) == w.view(np.uint32)).all(), (tile, w.shape)
    if prod.flags == 1 and chunk == 16:
        for a, b in gemms:
            w1, w2 = orc.gemm_ste_mask(a.numpy(), b.numpy(), *fmts, order, chunk, orc.STE_OF, 0.0, 0.0)
            for tile in (2, 7):
                lba.set_tile_override(tile)
                try:
                    masks = lba.lba_gemm_ste_mask(a.to(DEV), b.to(DEV), prod, acc, order, chunk, lba.STE_OF)
                finally:
                    lba.set_tile_override(-1)
                for g, w in zip(masks, (w1, w2)):
                    assert (g is None) == (w is None) and (g is None or (g.cpu().numpy().view(np.uint32) == w).all())


@pytest.mark.parametrize("order", [SEQ, CHK])
@pytest.mark.parametrize("shape", [(33, 64, 64), (700, 640, 64)])
def test_launches_keep_stream_order(shape, order):
    # launches that may be set up while the one before them drains: each call reads what the call before it wrote (its sums
    # as the bias, its buffer as the output of the call after next), in a stream and replayed from a graph
    M, N, K = shape
    prod, acc = code_domain_formats(7, 4)
    a, b, one = synth.random_codes((M, K), 1).to(DEV), synth.random_codes((N, K), 2).to(DEV), torch.ones(1, device=DEV)
    bufs = [torch.zeros(M, N, device=DEV) for _ in range(2)]

    def chain(steps, sync):
        for t in range(steps):
            lba.lba_gemm(a, b, one, one, bufs[t % 2].view(-1)[-N:], prod, acc, order, 16, out=bufs[(t + 1) % 2])
            if sync:
                torch.cuda.synchronize()
        return bufs[steps % 2].clone()

    def reset():
        for t in bufs:
            t.zero_()

    want = chain(40, True)
    for _ in range(5):
        reset()
        assert torch.equal(chain(40, False), want)
    reset()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = chain(40, False)
    for _ in range(3):
        reset()
        graph.replay()
        assert torch.equal(got, want)
    torch.cuda.synchronize()
    del graph, got
    gc.collect()


def test_launches_of_small_problems_leave_their_successors_evenly_spread():
    # a call behind a call of another kernel, or of its own, takes what it takes alone.  Where waiting CTAs settle on the room that
    # running ones happen to leave, the pairs below take 1.3 to 2.4 times as long; evenly spread, 1.0 times
    prod, acc = code_domain_formats(7, 4)
    one, cell = torch.ones(1, device=DEV), torch.zeros(1, device=DEV)

    def call(M, N, K, order, tile):
        a, b, out = synth.random_codes((M, K), 1).to(DEV), synth.random_codes((N, K), 2).to(DEV), torch.empty(M, N, device=DEV)

        def run():
            lba.set_tile_override(tile)
            lba.lba_gemm(a, b, one, one, None, prod, acc, order, 16, out=out)
        return run

    def time(*calls):
        graph, best = torch.cuda.CUDAGraph(), float("inf")
        for f in calls:
            f()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            for _ in range(20):
                for f in calls:
                    f()
        graph.replay()
        start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        for _ in range(5):
            start.record()
            graph.replay()
            stop.record()
            torch.cuda.synchronize()
            best = min(best, start.elapsed_time(stop) * 1e3 / 20)
        return best

    try:
        chain, split = call(32, 1000, 512, SEQ, 10), call(32, 1000, 512, CHK, 6)
        wider, packed = call(64, 1000, 512, CHK, 6), call(2368, 256, 512, CHK, 2)
        deep = call(128, 1000, 512, SEQ, 10)
        alone = {f: time(f) for f in (chain, split, wider, packed)}
        for f, g in ((chain, split), (wider, packed), (split, packed)):
            assert time(f, g) < 1.25 * (alone[f] + alone[g])
        assert time(deep) < 1.15 * time(deep, cell.zero_)
    finally:
        lba.set_tile_override(-1)
        gc.collect()


@pytest.mark.parametrize("how", ["stream", "two streams", "graph"])
def test_kernels_of_every_kind_keep_their_order(how):
    # every ordered pair of kernels one behind the other: a call adds the tail of what the call before it or the one before that
    # wrote (its bias) and writes over what the mask pass behind it still reads; the masks become operands through a PyTorch kernel
    one = torch.ones(1, device=DEV)
    codes = torch.empty(700 * 64, dtype=torch.uint8, device=DEV)
    first = synth.random_codes((700 * 64,), 1).to(DEV)
    w640, w64 = synth.random_codes((640, 64), 2).to(DEV), synth.random_codes((64, 64), 3).to(DEV)
    wconv = synth.random_codes((64, 3, 3, 16), 4).to(DEV)
    bufs = [torch.empty(700 * 640, device=DEV) for _ in range(3)]
    mask1, mask2 = torch.empty(80, 2, 64, dtype=torch.int32, device=DEV), torch.empty(80, 1, 64, dtype=torch.int32, device=DEV)
    floor, cut, near, generic = (code_domain_formats(7, 4), code_domain_formats(4, 4), code_domain_formats(7, 4, 1),
                                 code_domain_formats(12, 5, 1))

    def gemm(M, w, fmts, order, tile, chunk=16):
        def run(bias, out):
            lba.set_tile_override(tile)
            lba.lba_gemm(codes[:M * 64].view(M, 64), w, one, one, bias(len(w)), *fmts, order, chunk, out=out(M, len(w)))
        return run

    def conv(bias, out):
        lba.set_tile_override(-1)
        lba.lba_conv2d(codes[:2 * 9 * 11 * 16].view(2, 9, 11, 16), wconv, one, one, bias(64), (1, 1), (1, 1), *floor, CHK, 16,
                       out=out(2, 9, 11, 64))

    def masks(ste, order):
        def run(last, oldest):
            lba.set_tile_override(-1)
            lba.lba_gemm_ste_mask(last[:80 * 16].view(torch.uint8).view(80, 64), oldest[:64 * 16].view(torch.uint8).view(64, 64), *floor, order,
                                  16, ste, 4.0, 2.0 ** -7, mask1, mask2 if order == CHK else None)
        return run

    def glue(last, oldest):
        torch.bitwise_and(mask1.view(torch.uint8).view(-1)[:codes.numel()], 0x77, out=codes[:80 * 2 * 64 * 4])

    forward = [gemm(33, w64, floor, SEQ, 10), gemm(33, w64, near, CHK, 6), gemm(65, w64, cut, CHK, 7), gemm(700, w640, floor, CHK, 2),
               gemm(700, w640, cut, SEQ, 0), gemm(300, w640, floor, CHK, 5), gemm(130, w64, near, SEQ, 3), gemm(130, w64, generic, CHK, -1, 24),
               conv]
    others = [masks(lba.STE_OF, CHK), masks(lba.STE_OF, SEQ), masks(lba.STE_DIFF, CHK), masks(lba.STE_DIFF, SEQ), glue]
    kinds = forward + others
    steps = [k for f in kinds for g in kinds for k in (f, g)]
    sides = [torch.cuda.Stream(), torch.cuda.Stream()] if how == "two streams" else None

    def chain(sync):
        lens, t = [64 * 64] * 3, 0
        codes.copy_(first)
        mask1.zero_()
        mask2.zero_()
        for b in bufs:
            b.zero_()
        for i, step in enumerate(steps):
            if step in others:
                step(bufs[t % 3], bufs[(t + 1) % 3])
            else:
                source = (t - i % 2) % 3

                def out(*shape):
                    lens[(t + 1) % 3] = int(np.prod(shape))
                    return bufs[(t + 1) % 3][:lens[(t + 1) % 3]].view(shape)
                step(lambda n: bufs[source][lens[source] - n:lens[source]], out)
                t += 1
            if sync:
                torch.cuda.synchronize()
            elif sides:
                sides[1 - i % 2].wait_stream(torch.cuda.current_stream())
                torch.cuda.set_stream(sides[1 - i % 2])
        return [x.clone() for x in (*bufs, mask1, mask2, codes)]

    def same(got):
        return all(torch.equal(g.view(torch.uint8), w.view(torch.uint8)) for g, w in zip(got, want))

    home = torch.cuda.current_stream()
    try:
        want = chain(True)
        if how == "graph":
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                got = chain(False)
            for _ in range(3):
                graph.replay()
                torch.cuda.synchronize()
                assert same(got)
            del graph
        else:
            for _ in range(3):
                got = chain(False)
                torch.cuda.set_stream(home)
                torch.cuda.synchronize()
                assert same(got)
    finally:
        torch.cuda.set_stream(home)
        lba.set_tile_override(-1)
        gc.collect()
