"""The bit-stream kernels (code widths other than 4 bits; feature counts, strides and selected counts that are
multiples of nothing) and the group kernels against the shape-generic kernels, which the parity tests pin to the oracle:
payload bytes and FP32 / BF16 sums bit for bit.  The shapes sit where the layout can go wrong: rows of 32 bits and a
little more, a last group of 1 to 7 slots, stages of 4 rows and tiles of 8 with one row less or more, a run of rows that
starts inside a word, panels of 64 groups with one group more, the row kernel's last shape (640 groups, 384 selected
features) and the panel kernel's first, one and two groups a lane.  Some of the smaller shapes are the group kernels' or
the shape-generic quantiser's by size."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2411_07942_b200 import binding, synth  # noqa: E402

import gpu_util as gu  # noqa: E402

CASES = [  # N, T, E, k, bits, row padding, bias
    (1, 1, 33, 1, 2, 0, False), (2, 7, 17, 0, 2, 0, True), (3, 8, 65, 1, 3, 3, True), (2, 9, 130, 2, 4, 0, False),
    (2, 33, 1033, 8, 4, 0, True), (4, 16, 1024 + 51, 51, 4, 0, False), (4, 67, 5120, 51, 4, 64, True),
    (8, 40, 2304, 36, 4, 0, False), (8, 129, 4608, 72, 8, 0, True), (5, 31, 5120, 80, 5, 8, False),
    (3, 65, 1041, 17, 7, 0, True), (3, 24, 1047, 23, 6, 1, False), (16, 50, 832, 13, 5, 0, True),
    (33, 18, 520, 9, 4, 0, False), (64, 70, 264, 8, 8, 0, True), (2, 20, 8192, 128, 8, 0, False), (2, 11, 16384, 9, 8, 0, False),
    (4, 147, 5120, 0, 8, 0, True), (3, 297, 2048, 33, 6, 64, True), (4, 5, 1024, 380, 4, 0, True), (2, 149, 4096, 400, 4, 8, False),
    (1, 2, 64, 7, 7, 0, True), (4, 595, 512, 40, 2, 0, False),
    (1, 300, 5121, 5000, 4, 0, False), (2, 600, 200, 3, 3, 0, False), (1, 2500, 1000, 15, 4, 0, True),
    # five to eight devices on the row kernel: its narrowest and widest rows and one group more or less, more than 96 selected
    (5, 33, 1296, 17, 4, 0, True), (8, 149, 1272, 8, 3, 0, False), (8, 31, 2600, 40, 8, 8, True), (6, 20, 2608, 40, 6, 0, False),
    (7, 13, 2312, 105, 5, 0, True), (8, 150, 2304, 0, 2, 0, False),
]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    gu.ensure_lib()


@pytest.mark.parametrize("N,T,E,k,bits,pad,with_bias", CASES)
def test_stream_kernels_equal_generic(N, T, E, k, bits, pad, with_bias):
    rng = np.random.default_rng(E + T)
    T += -(-(1 << 18) // (8 * E)) * 8
    w = synth.Workload("stream", N, T, E, 0.7, max(1, E // 100), 20.0, 200.0, 1, 8, E + 7 * T + bits)
    scale = synth.column_scales(w)
    t = binding.Tpq(N, E, bits=bits)
    gu.calibrate_both(t, [synth.calibration_np(w, i, scale=scale) for i in range(N)])
    bias = torch.from_numpy(rng.standard_normal(E).astype(np.float32)).cuda() if with_bias else None
    ys = []
    for i in range(N):
        wide = torch.full((T, E + pad), float("nan"), dtype=torch.bfloat16, device="cuda")
        wide[:, :E] = gu.dev_bf16(synth.activations_np(w, i, T, scale=scale)).view(torch.bfloat16).view(T, E)
        ys.append(wide)
    # the selector's set, one run that ends inside a group, and both ends of the feature range
    start = int(rng.integers(0, E - k + 1))
    sets = [None, list(range(start, start + k)), sorted(set(range(k // 2)) | set(range(E - (k - k // 2), E)))]
    for hp in sets if k else [None]:
        t.select_features(k) if hp is None else t.set_features(hp)
        P = t.payload_bytes(T)
        got = {}
        for path in (binding.PATH_GENERIC, binding.PATH_AUTO):
            t.set_option(binding.TPQ_OPT_KERNEL_PATH, path)
            guarded = [gu.guarded(P) for _ in range(N)]
            ptrs = [v.data_ptr() for _, v in guarded]
            t.quantize_pack_batch(0, [y.data_ptr() for y in ys], T, ptrs, P, row_stride=E + pad)
            outs = []
            for dt, size in ((binding.TPQ_OUT_FP32, 4), (binding.TPQ_OUT_BF16, 2)):
                whole, out = gu.guarded(T * (E + pad) * size)
                t.dequant_reduce(ptrs, T, out.data_ptr(), dt, out_row_stride=E + pad, bias_ptr=bias.data_ptr() if with_bias else None)
                torch.cuda.synchronize()
                assert gu.guards_intact(whole, T * (E + pad) * size)
                outs.append(out.cpu().numpy())
            assert t.device_status() == 0
            assert all(gu.guards_intact(whole, P) for whole, _ in guarded)
            got[path] = ([v.cpu().numpy() for _, v in guarded], outs)
        for a, b in zip(got[binding.PATH_GENERIC], got[binding.PATH_AUTO]):
            for x, y in zip(a, b):
                assert np.array_equal(x, y), (hp, np.nonzero(x != y)[0][:8])
    t.close()


@pytest.mark.parametrize("N,T,E,k,bits,pad,with_bias", [
    (4, 300, 512, 8, 3, 0, True), (3, 37, 64, 8, 2, 8, False), (2, 9, 11264, 176, 5, 0, False), (2, 5, 9216, 144, 7, 16, True),
    (2, 3, 32768, 512, 8, 0, True), (2, 1, 131072, 2048, 2, 8, False), (16, 60, 2048, 32, 6, 0, False), (17, 130, 256, 248, 8, 0, False)])
def test_group_kernels_equal_generic(N, T, E, k, bits, pad, with_bias):
    """Other code widths where the group kernels quantise: narrow rows, rows too long for the ring or of two groups a lane; the
    two longest are also theirs to reduce."""
    test_stream_kernels_equal_generic(N, T, E, k, bits, pad, with_bias)


@pytest.mark.parametrize("T,E,k,bits,n_dst", [(1000, 512, 8, 3, 1), (1900, 1024, 16, 5, 3), (70, 8192, 128, 8, 1), (1500, 8192, 128, 7, 2),
                                              (40, 16384, 256, 6, 2)])
def test_pushes_through_the_group_kernels(T, E, k, bits, n_dst):
    """The quantise, copy and publish form of a push: every destination and word, against the shape-generic quantiser."""
    t = binding.Tpq(1, E, bits=bits)
    g = torch.Generator(device="cuda").manual_seed(T + E)
    y = (torch.randn((T + 16, E), generator=g, device="cuda") * 2).to(torch.bfloat16)
    t.calibrate_ranges(0, y.data_ptr(), 1, 16)
    torch.cuda.synchronize()
    t.select_features(k)
    P = t.payload_bytes(T)
    want = torch.zeros(P, dtype=torch.uint8, device="cuda")
    t.set_option(binding.TPQ_OPT_KERNEL_PATH, binding.PATH_GENERIC)
    t.quantize_pack(0, y.data_ptr(), T, want.data_ptr(), P)
    t.set_option(binding.TPQ_OPT_KERNEL_PATH, binding.PATH_AUTO)
    bufs = [gu.guarded(P) for _ in range(n_dst)]
    words = torch.zeros(n_dst, dtype=torch.int32, device="cuda")
    t.quantize_pack_push(0, y.data_ptr(), T, [v.data_ptr() for _, v in bufs], [words.data_ptr() + 4 * d for d in range(n_dst)], P, 11)
    torch.cuda.synchronize()
    assert t.device_status() == 0 and bool((words == 11).all())
    for whole, v in bufs:
        assert gu.guards_intact(whole, P) and torch.equal(v, want)
    t.close()


@pytest.mark.parametrize("E,k,bits", [(5121, 51, 4), (16385, 3, 2), (1033, 16, 8), (5121, 5000, 4), (65, 1, 3)])
def test_rows_that_bulk_copies_cannot_fetch(E, k, bits):
    """The tile kernel and the shape-generic one share these shapes by size: token counts on both sides of the line, tiles of
    less than 4 and less than 8 rows, one shard and three."""
    N = 3
    g = torch.Generator(device="cuda").manual_seed(E + bits)
    t = binding.Tpq(N, E, bits=bits)
    c = torch.randn((32, E), generator=g, device="cuda").to(torch.bfloat16)
    for i in range(N):
        t.calibrate_ranges(i, c.data_ptr(), 1, 32)
    torch.cuda.synchronize()
    t.select_features(k)
    for T in (1, 4, 5, 64, 167, 601, 2049 if E < 6000 else 900):
        ys = [(1.5 * torch.randn((T, E), generator=g, device="cuda")).to(torch.bfloat16) for _ in range(N)]
        P = t.payload_bytes(T)
        got = []
        for path, n in ((binding.PATH_GENERIC, 1), (binding.PATH_AUTO, 1), (binding.PATH_AUTO, N)):
            t.set_option(binding.TPQ_OPT_KERNEL_PATH, path)
            bufs = [gu.guarded(P) for _ in range(N)]
            for i in range(0, N, n):
                t.quantize_pack_batch(i, [y.data_ptr() for y in ys[i:i + n]], T, [v.data_ptr() for _, v in bufs[i:i + n]], P)
            torch.cuda.synchronize()
            assert t.device_status() == 0 and all(gu.guards_intact(w, P) for w, _ in bufs)
            got.append([v for _, v in bufs])
        for other in got[1:]:
            assert all(torch.equal(a, b) for a, b in zip(got[0], other)), T
    t.close()


def _kernels(call):
    from torch.profiler import ProfilerActivity, profile

    with profile(activities=[ProfilerActivity.CUDA], acc_events=True) as p:
        call()
        torch.cuda.synchronize()
    return " ".join(e.name for e in p.events())


@pytest.mark.parametrize("N,T,E,k,bits,quantiser,reducer", [
    (3, 37, 512, 8, 3, "quantize_stream<", "dequant_stream_rows<"), (6, 9, 520, 16, 8, "quantize_stream<", "dequant_stream<"),
    (2, 3, 32768, 512, 8, "quantize_groups<", "dequant_groups<"), (2, 5, 16, 8, 2, "quantize_groups<", "dequant_groups<"),
    (2, 3, 512, 8, 4, "quantize_tiled<", "dequant_rows<")])
def test_forced_path_runs_no_generic_kernel(N, T, E, k, bits, quantiser, reducer):
    """Path 2 at sizes that the automatic choice leaves to the shape-generic reduction: every width's own kernels, and the
    same bytes and sums as path 1."""
    t = binding.Tpq(N, E, bits=bits)
    g = torch.Generator(device="cuda").manual_seed(E + bits)
    ys = [(2 * torch.randn((T, E), generator=g, device="cuda")).to(torch.bfloat16) for _ in range(N)]
    for i in range(N):
        t.calibrate_ranges(i, ys[i].data_ptr(), 1, T)
    torch.cuda.synchronize()
    t.select_features(k)
    P = t.payload_bytes(T)
    got = []
    for path, kernels in ((binding.PATH_GENERIC, ("quantize_generic", "dequant_generic")), (binding.PATH_TILED, (quantiser, reducer))):
        t.set_option(binding.TPQ_OPT_KERNEL_PATH, path)
        pls = [torch.zeros(P, dtype=torch.uint8, device="cuda") for _ in range(N)]
        out = torch.empty((T, E), dtype=torch.float32, device="cuda")
        ptrs = [p.data_ptr() for p in pls]
        assert kernels[0] in _kernels(lambda: t.quantize_pack_batch(0, [y.data_ptr() for y in ys], T, ptrs, P))
        assert kernels[1] in _kernels(lambda: t.dequant_reduce(ptrs, T, out.data_ptr(), binding.TPQ_OUT_FP32))
        assert t.device_status() == 0
        got.append([*pls, out])
    assert all(torch.equal(a, b) for a, b in zip(*got))
    t.close()


@pytest.mark.parametrize("N,T,E,k,bits,pad,with_bias", [
    (2, 40, 5128, 8, 3, 0, True), (2, 40, 5128, 7, 4, 0, True), (3, 9, 2048, 384, 8, 0, False), (3, 9, 2048, 385, 4, 8, False),
    (6, 40, 1040, 8, 5, 0, True), (7, 41, 1033, 8, 4, 0, False), (5, 80, 8712, 136, 2, 0, False)])
def test_stream_kernels_at_the_limits_of_a_kernel(N, T, E, k, bits, pad, with_bias):
    """640 and 641 groups, 384 and 385 selected features (row kernel, panel kernel), two panels of 64 groups and one group
    more, whole and of one slot; the ring's last shapes of two groups a lane."""
    test_stream_kernels_equal_generic(N, T, E, k, bits, pad, with_bias)


@pytest.mark.parametrize("bits", [2, 3, 4, 5, 6, 7, 8])
def test_every_pattern_at_every_width(bits):
    """All BF16 patterns (steps of 1 and 0.37: exact ties, values far past the clamps, infinities) through the pipelined
    quantiser (rows of 256 and of 264 features with 9 selected, which the other kernels cannot take at 4 bits), bit-exact
    against the oracle; and with the NaN patterns as the shape-generic kernel has them."""
    orc = oracle.c()
    allp = np.arange(65536, dtype=np.uint32).astype(np.uint16)
    nan = ((allp & 0x7F80) == 0x7F80) & ((allp & 0x007F) != 0)
    for E, hp in ((256, []), (264, list(range(100, 109)))) if bits != 4 else ((264, list(range(100, 109))),):
        T = 65536 // E + 1
        steps = np.array([1.0, 0.37], np.float32)
        t = binding.Tpq(2, E, bits=bits)
        M = np.repeat((steps * np.float32((2 ** bits - 1) / 2))[:, None], E, axis=1)
        t.set_ranges(-M, M, np.ones(2, np.int64))
        t.set_features(hp)
        _, inv = t.get_scales()
        P = t.payload_bytes(T)
        for with_nan in (False, True):
            y = np.resize(allp if with_nan else allp[~nan], (T, E))
            d = gu.dev_bf16(y)
            for i in range(2):
                got = []
                for path in (binding.PATH_GENERIC, binding.PATH_AUTO):
                    t.set_option(binding.TPQ_OPT_KERNEL_PATH, path)
                    whole, view = gu.guarded(P)
                    t.quantize_pack(i, d.data_ptr(), T, view.data_ptr(), P)
                    torch.cuda.synchronize()
                    assert gu.guards_intact(whole, P)
                    got.append(view.cpu().numpy())
                assert np.array_equal(*got), (E, i)
                if not with_nan:
                    assert np.array_equal(got[1], orc.quantize_pack(y, np.asarray(hp, np.int32), inv[i], bits)), (E, i)
        t.set_option(binding.TPQ_OPT_KERNEL_PATH, binding.PATH_AUTO)
        assert "quantize_stream<" in _kernels(lambda: t.quantize_pack(0, d.data_ptr(), T, view.data_ptr(), P))
        t.close()


@pytest.mark.parametrize("bits", [2, 3, 4, 5, 8])
def test_groups_with_many_selected_features(bits):
    """3 to 8 selected features in one group of 8 beside groups with fewer, and a warp with 32 and with 33 of them: payloads
    of the pipelined quantisers (at 4 bits the one for multiples of 8 too, by the set's size) against the generic kernel."""
    N, T, E = 2, 23, 1024
    w = synth.Workload("holes", N, T, E, 0.7, 10, 20.0, 200.0, 1, 8, 5 + bits)
    scale = synth.column_scales(w)
    t = binding.Tpq(N, E, bits=bits)
    gu.calibrate_both(t, [synth.calibration_np(w, i, scale=scale) for i in range(N)])
    ys = [gu.dev_bf16(synth.activations_np(w, i, T, scale=scale)) for i in range(N)]
    group = lambda g, n: [8 * g + (3 * i + g) % 8 for i in range(n)]  # n features of a group, not its first ones
    sets = [group(0, n) + group(1, 2) + group(31, 1) + group(63, n) for n in range(3, 9)]
    sets += [group(2, 8) + group(3, 8) + group(9, 8) + group(30, n) for n in (8, 7)] + [group(2, 8) + group(3, 8) + group(9, 8) + group(30, 8) + group(11, 1)]
    sets += [s + group(100, -len(s) % 8) for s in sets]   # sizes that are multiples of 8 as well
    for hp in map(sorted, sets):
        t.set_features(hp)
        P = t.payload_bytes(T)
        got = []
        for path in (binding.PATH_GENERIC, binding.PATH_AUTO):
            t.set_option(binding.TPQ_OPT_KERNEL_PATH, path)
            pls = [torch.zeros(P, dtype=torch.uint8, device="cuda") for _ in range(N)]
            t.quantize_pack_batch(0, [y.data_ptr() for y in ys], T, [p.data_ptr() for p in pls], P)
            torch.cuda.synchronize()
            assert t.device_status() == 0
            got.append([p.cpu().numpy() for p in pls])
        for a, b in zip(*got):
            assert np.array_equal(a, b), hp
    t.close()


def _row_case(N, rows, short, E, k, bits, pad, split=False):
    """A context with an arbitrary set (both ends of the feature range in it), its payloads (shape-generic quantiser) and T: `rows`
    to a block of the row kernel, the last block `short` rows less."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    T = rows * (sms // 2 if split else sms) - short
    rng = np.random.default_rng(E + T + k)
    g = torch.Generator(device="cuda").manual_seed(E + T + k)
    t = binding.Tpq(N, E, bits=bits)
    M = rng.lognormal(0, 1, (N, E)).astype(np.float32)
    t.set_ranges(-M, M, np.ones(N, np.int64))
    ends = sorted({0, E - 1, E - k - 1, E - k} & set(range(E)))[:k]
    t.set_features(sorted(ends + rng.permutation(sorted(set(range(E)) - set(ends)))[:k - len(ends)].tolist()))
    P = t.payload_bytes(T)
    t.set_option(binding.TPQ_OPT_KERNEL_PATH, binding.PATH_GENERIC)
    pls = [torch.zeros(P, dtype=torch.uint8, device="cuda") for _ in range(N)]
    for i in range(N):
        y = (torch.randn((T, E), generator=g, device="cuda") * 2).to(torch.bfloat16)
        t.quantize_pack(i, y.data_ptr(), T, pls[i].data_ptr(), P)
    return t, T, pls


@pytest.mark.parametrize("N,rows,short,E,k,bits,pad,with_bias,split", [
    # rows of a block: whole stages, a short first or last one, more stages than the ring has, a last block with fewer;
    # selected: none, one (its last values lie in the last rows of several blocks), more than the auxiliary threads, the most
    (1, 9, 3, 1024, 7, 4, 0, True, False), (2, 14, 5, 2048, 1, 3, 8, False, False), (3, 7, 2, 1032, 105, 8, 0, True, False),
    (3, 30, 1, 640, 3, 4, 64, False, False), (4, 6, 4, 5120, 80, 2, 0, True, False), (4, 21, 7, 512, 384, 5, 0, False, False),
    (4, 2, 1, 1024, 1, 7, 0, True, False), (5, 5, 1, 2304, 37, 6, 0, True, False), (5, 14, 0, 1792, 0, 3, 8, False, False),
    (6, 30, 11, 1808, 105, 8, 0, True, False), (6, 8, 3, 2048, 2, 4, 0, False, False), (7, 5, 2, 2600, 41, 5, 0, True, False),
    (7, 18, 5, 2312, 384, 7, 0, False, False), (8, 14, 1, 2304, 36, 4, 0, True, False), (8, 30, 3, 1304, 1, 8, 8, False, False),
    (6, 4, 2, 2608, 40, 6, 0, True, True), (6, 16, 3, 4608, 105, 8, 8, False, True), (7, 14, 5, 5120, 384, 5, 0, True, True),
    (8, 14, 2, 4608, 72, 8, 0, True, True), (8, 9, 0, 5120, 51, 4, 0, False, True), (8, 2, 1, 3008, 1, 8, 0, True, True),
    (8, 15, 5, 4608, 0, 6, 8, False, True)])
def test_row_kernel_stages(N, rows, short, E, k, bits, pad, with_bias, split):
    """The bit-stream row kernel for one to eight devices, one and two blocks to a run of rows, against the shape-generic kernel,
    bit for bit."""
    t, T, pls = _row_case(N, rows, short, E, k, bits, pad, split)
    bias = torch.randn(E, generator=torch.Generator(device="cuda").manual_seed(k), device="cuda")
    ptrs = [p.data_ptr() for p in pls]
    for dt, size in ((binding.TPQ_OUT_FP32, 4), (binding.TPQ_OUT_BF16, 2)):
        got = []
        for path in (binding.PATH_GENERIC, binding.PATH_AUTO):
            t.set_option(binding.TPQ_OPT_KERNEL_PATH, path)
            whole, out = gu.guarded(T * (E + pad) * size)
            call = lambda: t.dequant_reduce(ptrs, T, out.data_ptr(), dt, out_row_stride=E + pad, bias_ptr=bias.data_ptr() if with_bias else None)
            if path == binding.PATH_AUTO:
                assert "dequant_stream_rows<" in _kernels(call)
            else:
                call()
            torch.cuda.synchronize()
            assert t.device_status() == 0 and gu.guards_intact(whole, T * (E + pad) * size)
            got.append(out)
        assert torch.equal(*got)
    t.close()


@pytest.mark.parametrize("N,rows,short,E,k,bits,split", [(4, 3, 1, 1024, 3, 4, False), (2, 7, 0, 2048, 1, 3, False), (6, 5, 2, 2304, 35, 4, False),
                                                         (8, 9, 1, 4608, 5, 8, True)])
def test_row_kernel_on_payloads_written_by_the_call_ahead(N, rows, short, E, k, bits, split):
    """Steps in one stream over the same payload buffers, all queued when the first one starts: each sum is of its own step's
    payloads, to the last value (the BF16 values end inside 16 bytes)."""
    t, T, pls = _row_case(N, rows, short, E, k, bits, 0, split)
    assert T * k % 8
    g = torch.Generator(device="cuda").manual_seed(T)
    steps = [[(torch.randn((T, E), generator=g, device="cuda") * 2).to(torch.bfloat16) for _ in range(N)] for _ in range(4)]
    ptrs, P = [p.data_ptr() for p in pls], t.payload_bytes(T)
    got = []
    for path in (binding.PATH_GENERIC, binding.PATH_AUTO):
        t.set_option(binding.TPQ_OPT_KERNEL_PATH, path)
        outs = [torch.empty((T, E), dtype=torch.float32, device="cuda") for _ in steps]
        side = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(1 << 20)
        for ys, out in zip(steps, outs):
            t.quantize_pack_batch(0, [y.data_ptr() for y in ys], T, ptrs, P, stream=side.cuda_stream)
            t.dequant_reduce(ptrs, T, out.data_ptr(), binding.TPQ_OUT_FP32, stream=side.cuda_stream)
            if path == binding.PATH_GENERIC:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert t.device_status() == 0
        got.append(outs)
    assert all(torch.equal(a, b) for a, b in zip(*got))
    t.close()


@pytest.mark.parametrize("N,T,E,k,bits,reducer", [
    # five to eight devices: one group too few; 160 to 199 groups up to 16 rows an SM and above, by width; from 200 on
    (8, 300, 1280, 15, 4, "dequant_stream<"), (7, 2368, 1408, 22, 3, "dequant_stream_rows<"), (7, 2369, 1408, 22, 3, "dequant_stream<"),
    (5, 2369, 1408, 22, 7, "dequant_stream<"), (6, 2369, 1408, 22, 5, "dequant_stream_rows<"), (5, 2369, 1408, 22, 8, "dequant_stream_rows<"),
    (5, 2369, 1624, 22, 2, "dequant_stream_rows<"),
    # two blocks to a run of rows: where the panel kernel's blocks fill one wave and need two, the most rows, too few devices
    (8, 740, 2624, 41, 3, "dequant_stream<"), (8, 888, 2624, 41, 3, "dequant_stream_rows<"), (8, 1184, 5120, 80, 8, "dequant_stream_rows<"),
    (8, 1185, 5120, 80, 8, "dequant_stream<"), (5, 64, 4608, 72, 3, "dequant_stream<")])
def test_which_reduction_serves_a_call(N, T, E, k, bits, reducer):
    """The rule's lines for five to eight devices (148 SMs), each side the same sums as the shape-generic kernel."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the lines are stated for 148 SMs")
    t, _, pls = _row_case(N, 1, 148 - T, E, k, bits, 0)
    ptrs, got = [p.data_ptr() for p in pls], []
    for path in (binding.PATH_GENERIC, binding.PATH_AUTO):
        t.set_option(binding.TPQ_OPT_KERNEL_PATH, path)
        out = torch.empty((T, E), dtype=torch.float32, device="cuda")
        names = _kernels(lambda: t.dequant_reduce(ptrs, T, out.data_ptr(), binding.TPQ_OUT_FP32))
        assert (reducer if path == binding.PATH_AUTO else "dequant_generic") in names
        assert t.device_status() == 0
        got.append(out)
    assert torch.equal(*got)
    t.close()
