"""The GEMM of few rows (output channels on the MMA's rows, tokens on its columns, K ranges split over clusters, activations
quantized inside): bit for bit the results of the tile form, which the parity tests hold to the oracle.  Both add the same
terms in the same order: int8 sums are exact however a K range is split, e4m3 ones are never split."""
import threading

import pytest
import torch
from cuda.bindings import driver

from paper_2507_14811_b200 import binding as B
from paper_2507_14811_b200.layer import SegQuantLinear

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
BF16, F32 = torch.bfloat16, torch.float32
TILE_FORM, ROWS_FORM = 9, 8


def make(M, K, N, kb, nb, dual, code, x_dtype):
    g = torch.Generator(device=DEV).manual_seed(M + K + N)
    layer = SegQuantLinear(torch.randn((N, K), generator=g, device=DEV) * 0.02, torch.randn((N,), generator=g, device=DEV), kb, nb, dual, code)
    X = torch.randn((M, K), generator=g, device=DEV).to(x_dtype)
    layer.calibrate(X * 0.9)                             # the largest inputs are clipped
    return layer, X


def gemm(layer, codes, y_dtype, dump=False):
    c_pos, c_neg = codes
    if layer.dual:
        return B.segquant_dualscale_gemm(c_pos, c_neg, layer.Wq, layer.seg, layer.code, layer.s_pos, layer.s_neg, layer.s_w,
                                         layer.bias, layer.workspace, y_dtype=y_dtype, dump_acc=dump)
    return B.segquant_seglinear_gemm(c_pos, layer.Wq, layer.seg, layer.code, layer.s_pos, layer.s_w, layer.bias, layer.workspace,
                                     y_dtype=y_dtype, dump_acc=dump)


TILE_THREADS, ROWS_THREADS = 384, 320


def gemm_forms(fn):
    """Block sizes of the GEMM kernels that fn launches, from the nodes of a graph it is captured into (nothing runs)."""
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.stream(stream):
        graph.capture_begin(capture_error_mode="relaxed")
        fn()
        graph.capture_end()
    raw = driver.CUgraph(graph.raw_cuda_graph())
    err, _, count = driver.cuGraphGetNodes(raw)
    err, nodes, _ = driver.cuGraphGetNodes(raw, count)
    assert err == driver.CUresult.CUDA_SUCCESS
    threads = []
    for node in nodes:
        if driver.cuGraphNodeGetType(node)[1] == driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            err, params = driver.cuGraphKernelNodeGetParams(node)
            assert err == driver.CUresult.CUDA_SUCCESS
            threads.append(params.blockDimX)
    return [t for t in threads if t in (TILE_THREADS, ROWS_THREADS)]


@pytest.mark.parametrize("case", [
    # M, K, N, kb, nb, x, y: one 16-code step; a K tail; one channel past a tile; every token count around 8 and 16; segments
    # inside a K-block and across the cut of a split K range; more segments than CTAs; N-bounds anywhere; several token tiles
    (1, 16, 8, [0, 16], [0, 8], BF16, BF16),
    (7, 1040, 136, [0, 1040], [0, 136], F32, BF16),
    (9, 2064, 264, [0, 32, 96, 1056, 2064], [0, 1, 130, 264], BF16, F32),
    (17, 528, 1000, [0, 160, 528], [0, 328, 1000], F32, F32),
    (40, 1152, 96, [0, 64, 128, 192, 256, 1024, 1152], [0, 96], BF16, BF16),
    (128, 384, 72, [0, 384], [0, 40, 72], BF16, F32),
    (250, 640, 392, [0, 320, 640], [0, 392], BF16, BF16),
])
@pytest.mark.parametrize("code,dual", [("int8", True), ("int8", False), ("e4m3", True), ("e4m3", False)])
def test_every_shape_equals_the_tile_form(case, code, dual):
    M, K, N, kb, nb, x_dtype, y_dtype = case
    layer, X = make(M, K, N, kb, nb, dual, code, x_dtype)
    codes = B.segquant_quantize_act(X, layer.seg, layer.s_pos, layer.s_neg, code)
    try:
        B.segquant_set_tuning(segment_mode=TILE_FORM)
        ref, ref_acc = gemm(layer, codes, y_dtype, dump=True)
        splits = (1, 2, 4, 8, 1, 8) if code == "int8" else (1,) * 6          # e4m3: one CTA has the whole K range
        for (rows, tokens), split in zip(((0, 0), (128, 8), (32, 16), (64, 256), (96, 32), (128, 128), (32, 8)), (0, *splits)):
            B.segquant_set_tuning(rows, tokens, split, ROWS_FORM)        # shapes that do not fit run the tile form
            kblocks, t = (K + 127) // 128, min(tokens or 8, M)
            columns = 2 * ((t + 7) // 8 * 8) if dual else (t + 15) // 16 * 16
            fits = split <= kblocks and columns <= 256
            held = (kblocks + max(split, 1) - 1) // max(split, 1) * 128 * (columns + t * X.element_size())   # codes and inputs of a CTA
            Y = torch.full((M + 1, N), 7.0, dtype=y_dtype, device=DEV)
            n = B.segquant_launch_count()
            layer.forward(X, Y[:M])                                      # quantized inside
            inside = B.segquant_launch_count() == n + 1
            assert inside if fits and held <= 100 * 1024 else fits or not inside
            assert gemm_forms(lambda: gemm(layer, codes, y_dtype, dump=True)) == [ROWS_THREADS if fits else TILE_THREADS]
            y, acc = gemm(layer, codes, y_dtype, dump=True)
            layer.check_status()
            shape = (rows, tokens, split)
            assert torch.equal(Y[:M], ref) and torch.equal(y, ref) and torch.equal(acc, ref_acc), shape
            assert torch.equal(gemm(layer, codes, y_dtype), ref) and bool(torch.all(Y[M:] == 7.0)), shape
    finally:
        B.segquant_set_tuning()


@pytest.mark.parametrize("dual", [True, False])
@pytest.mark.parametrize("M,K,N,kb", [(1, 4096, 264, [0, 4096]), (5, 1056, 1000, [0, 96, 1056]), (100, 512, 136, [0, 512])])
def test_per_token_scales(M, K, N, kb, dual):
    P = len(kb) - 1
    g = torch.Generator(device=DEV).manual_seed(5)
    seg, ws = B.SegTable(kb, [0, N]), B.new_workspace(DEV)
    s_pos, s_neg, c_pos, c_neg = B.segquant_quantize_per_row(torch.randn((M, K), generator=g, device=DEV), seg, dual)
    s_w, _, w, _ = B.segquant_quantize_per_row(torch.randn((N, K), generator=g, device=DEV), seg, False, bits=4)
    bias = torch.randn((N,), generator=g, device=DEV)
    run = lambda: B.segquant_w4a8_gemm(c_pos, c_neg, w, seg, s_pos, s_neg, s_w, bias, ws, y_dtype=F32)
    try:
        B.segquant_set_tuning(segment_mode=TILE_FORM)
        ref = run()
        for shape in ((0, 0, 0), (32, 8, 1), (128, 32, 8), (64, 16, 2)):
            B.segquant_set_tuning(*shape, ROWS_FORM)
            assert torch.equal(run(), ref), shape
            assert gemm_forms(run) == [ROWS_THREADS if shape[2] <= (K + 127) // 128 else TILE_THREADS], shape
    finally:
        B.segquant_set_tuning()
    B.check_device_status(ws)


@pytest.mark.parametrize("scale", [2.0 ** -90, 2.0 ** 105])
@pytest.mark.parametrize("code,dual", [("int8", True), ("int8", False), ("e4m3", True)])
def test_scales_outside_the_fast_quantizer(scale, code, dual):
    layer, X = make(6, 288, 40, [0, 288], [0, 40], dual, code, F32)
    X = X * scale
    layer.calibrate(X)
    outs = []
    try:
        for mode in (TILE_FORM, ROWS_FORM):
            B.segquant_set_tuning(segment_mode=mode)
            outs.append(layer.forward(X, y_dtype=F32))
    finally:
        B.segquant_set_tuning()
    assert torch.equal(*outs)


def test_output_in_place_of_the_input():
    """X is read before Y is written wherever the two share memory."""
    layer, X = make(24, 256, 256, [0, 256], [0, 256], True, "int8", F32)
    ref = layer.forward(X, y_dtype=F32)
    n = B.segquant_launch_count()
    layer.forward(X.clone(), y_dtype=F32)
    assert B.segquant_launch_count() == n + 1                            # apart, this layer is one launch
    Y = X.clone()
    layer.forward(Y, Y)
    assert torch.equal(Y, ref)


@pytest.mark.parametrize("M,K,kb", [(8, 1024, [0, 1024]), (8, 1056, [0, 320, 1056]), (256, 256, [0, 256]), (256, 288, [0, 96, 288])])
@pytest.mark.parametrize("code,dual", [("int8", True), ("int8", False), ("e4m3", True), ("e4m3", False)])
def test_scales_from_the_calibration_in_front(M, K, kb, code, dual):
    """A layer that quantizes inside, queued right behind the calibration that writes its scales, with and without another
    such layer between the two, eagerly, from a plan and in a graph: what it gives after a synchronization."""
    layer, X = make(M, K, 136, kb, [0, 136], dual, code, BF16)
    other, X_other = make(16, 512, 64, [0, 512], [0, 64], True, "int8", BF16)
    g = torch.Generator(device=DEV).manual_seed(1)
    batches = [torch.randn((40000, K), generator=g, device=DEV).to(BF16) * s for s in (1.0, 3.0)]
    X_cal = torch.empty_like(batches[0])
    calibrate = lambda batch: B.segquant_calib_scales_static(batch, layer.seg, code, False, dual, s_pos=layer.s_pos, s_neg=layer.s_neg)

    def spoil():
        for s in (layer.s_pos, layer.s_neg) if dual else (layer.s_pos,):
            s.fill_(1e3)

    try:
        B.segquant_set_tuning(segment_mode=ROWS_FORM)
        Y, Y_plan, Y_other = (torch.empty((m, n), dtype=BF16, device=DEV) for m, n in ((M, 136), (M, 136), (16, 64)))
        plan = layer.plan(X, Y_plan)
        want = []
        for batch in batches:
            calibrate(batch)
            torch.cuda.synchronize()
            want.append(layer.forward(X).clone())
        assert not torch.equal(*want)
        n = B.segquant_launch_count()
        layer.forward(X, Y)
        plan.run()
        assert B.segquant_launch_count() == n + 2                        # one launch each
        torch.cuda.synchronize()
        for between in (False, True):
            got = []
            for i in range(6):
                torch.cuda._sleep(400_000)                               # the calls below are queued before the first one starts
                for run, out in ((lambda: layer.forward(X, Y), Y), (plan.run, Y_plan)):
                    spoil()
                    calibrate(batches[i % 2])
                    if between:
                        other.forward(X_other, Y_other)
                    run()
                    got.append((i % 2, out.clone()))
            assert all(torch.equal(out, want[i]) for i, out in got), between

        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(stream):
            with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
                spoil()
                calibrate(X_cal)
                layer.forward(X, Y)
                spoil()
                calibrate(X_cal)
                other.forward(X_other, Y_other)
                plan.run()
        torch.cuda.current_stream().wait_stream(stream)
        for i in range(6):
            X_cal.copy_(batches[i % 2])
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(Y, want[i % 2]) and torch.equal(Y_plan, want[i % 2])
    finally:
        B.segquant_set_tuning()
    layer.check_status()


@pytest.mark.parametrize("code,dual", [("int8", True), ("int8", False), ("e4m3", True)])
def test_infinite_inputs(code, dual):
    layer, X = make(24, 288, 40, [0, 96, 288], [0, 40], dual, code, F32)
    X[::3, ::7], X[1::3, ::5] = float("inf"), -float("inf")
    outs = []
    try:
        for mode in (TILE_FORM, ROWS_FORM):
            B.segquant_set_tuning(segment_mode=mode)
            outs.append(layer.forward(X, y_dtype=F32))
            outs.append(layer.forward(X.clamp(torch.finfo(F32).min, torch.finfo(F32).max), y_dtype=F32))
    finally:
        B.segquant_set_tuning()
    assert all(torch.equal(o, outs[0]) for o in outs) and bool(torch.all(outs[0].isfinite()))


@pytest.mark.parametrize("M,K,kb,x_dtype", [(5, 528, [0, 528], BF16), (40, 1152, [0, 64, 96, 1152], F32), (256, 256, [0, 256], BF16)])
def test_symmetric_code_range(M, K, kb, x_dtype):
    """A negative bound of -127 (SQ_FLAG_QMIN_SYM), with inputs that a bound of -128 would not clip to it."""
    layer, X = make(M, K, 136, kb, [0, 136], True, "int8", x_dtype)
    layer.flags = B.SQ_FLAG_QMIN_SYM
    layer.calibrate(X * 0.9)
    _, c_neg = B.segquant_quantize_act(X, layer.seg, layer.s_pos, layer.s_neg, "int8", layer.flags)
    _, c_128 = B.segquant_quantize_act(X, layer.seg, layer.s_pos, layer.s_neg, "int8")
    assert not bool(torch.any(c_neg == 0x80)) and bool(torch.any(c_128 == 0x80))
    outs = []
    try:
        for mode, launches in ((TILE_FORM, 2), (ROWS_FORM, 1)):
            B.segquant_set_tuning(segment_mode=mode)
            n = B.segquant_launch_count()
            outs.append(layer.forward(X, y_dtype=F32))
            assert B.segquant_launch_count() == n + launches
    finally:
        B.segquant_set_tuning()
    assert torch.equal(*outs)


@pytest.mark.parametrize("tuning,form", [({}, ROWS_THREADS), ({"segment_mode": ROWS_FORM}, ROWS_THREADS), ({"stages": 4}, TILE_THREADS),
                                         ({"tile_n": 64}, TILE_THREADS), ({"cta_group": 1}, TILE_THREADS),
                                         ({"segment_mode": TILE_FORM}, TILE_THREADS)])
def test_tuning_words_keep_the_tile_form(tuning, form):
    """Any of them asks for the tile form, whose dimensions they are, in the GEMM alone and in a layer call."""
    layer, X = make(2, 8192, 640, [0, 8192], [0, 640], True, "int8", BF16)
    codes = B.segquant_quantize_act(X, layer.seg, layer.s_pos, layer.s_neg, "int8")
    ref = gemm(layer, codes, BF16)
    try:
        B.segquant_set_tuning(**tuning)
        Y = layer.forward(X)
        y = gemm(layer, codes, BF16)
        assert gemm_forms(lambda: layer.forward(X)) == gemm_forms(lambda: gemm(layer, codes, BF16)) == [form]
    finally:
        B.segquant_set_tuning()
    assert torch.equal(Y, ref) and torch.equal(y, ref)


@pytest.mark.parametrize("M,K,N,P,code,dual,form", [
    (4, 4992, 424, 13, "e4m3", True, TILE_THREADS), (4, 2496, 424, 13, "e4m3", True, ROWS_THREADS),    # blocks that K-segments cut
    (101, 8448, 1008, 22, "e4m3", False, TILE_THREADS), (38, 3520, 1880, 22, "int8", True, ROWS_THREADS),
    (42, 8016, 8936, 1, "int8", False, TILE_THREADS), (31, 10192, 3392, 2, "int8", False, ROWS_THREADS),    # weights read per token tile
])
def test_layers_that_the_tile_form_takes_in_less_time(M, K, N, P, code, dual, form):
    layer, X = make(M, K, N, [K * p // P // 32 * 32 for p in range(P)] + [K], [0, N], dual, code, BF16)
    codes = B.segquant_quantize_act(X, layer.seg, layer.s_pos, layer.s_neg, code)
    Y = gemm(layer, codes, BF16)
    assert gemm_forms(lambda: gemm(layer, codes, BF16)) == [form]
    try:
        B.segquant_set_tuning(segment_mode=TILE_FORM)
        assert torch.equal(gemm(layer, codes, BF16), Y)
    finally:
        B.segquant_set_tuning()


def test_streams_and_host_threads():
    """Layers of few rows, split over clusters and not, from two host threads with streams, buffers and workspaces of their
    own: kernels of both share SMs, tensor memory and what the library keeps; every thread has its own layer shapes."""
    sizes = [(8, 4096, 264, "int8"), (250, 256, 768, "int8"), (40, 1152, 392, "e4m3"), (1, 8192, 136, "int8")]
    work = [[make(M + t, K, N, [0, K // 64 * 32, K], [0, N], True, code, BF16) for M, K, N, code in sizes] for t in range(2)]
    want = [[layer.forward(X).clone() for layer, X in w] for w in work]
    torch.cuda.synchronize()
    failed = []

    def call(t):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                plans = [(layer.plan(X, y), y) for layer, X in work[t] for y in [torch.empty_like(layer.forward(X))]]
                for _ in range(60):
                    got = [layer.forward(X) for layer, X in work[t]]
                    for plan, _ in plans:
                        plan.run()
                torch.cuda.current_stream().synchronize()
                if not all(torch.equal(g, w) and torch.equal(y, w) for g, (_, y), w in zip(got, plans, want[t])):
                    failed.append(t)
        except Exception as e:
            failed.append(repr(e))

    threads = [threading.Thread(target=call, args=(t,)) for t in range(2)]
    for thread in threads:
        thread.start()
    for thread in threads:
        thread.join()
    assert not failed
    for w in work:
        for layer, _ in w:
            layer.check_status()
