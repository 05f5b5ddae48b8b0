"""Kernels and dispatch branches at the sizes where they can go wrong (tile and stage edges,
remainders, the ends of their ranges), bit for bit against the oracle."""

import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_1401_8288_gb300 import synth, xcorr

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return t


@pytest.mark.parametrize("variant", [4, 5, 6, 10])
@pytest.mark.parametrize("n_sta,n_chan,n_time", [(8, 3, 129), (32, 9, 300), (72, 2, 65), (136, 2, 257)])
def test_adding_launch_of_the_fused_kernel(torch, variant, n_sta, n_chan, n_time):
    """A second and third execute add into sums that are there: full and ragged tiles, odd row
    alignments, packed channels, and (variant 10) the time-split form."""
    x = synth.uniform_ci4(3 * n_time, n_chan, n_sta, seed=n_sta + n_time, lo=-8, hi=7)
    xd = torch.from_numpy(x).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="ci4", engine="tensor") as plan:
        plan.set_tuning(variant, 0, 2, 0)
        for k in range(3):
            plan.execute(xd[k * n_time:(k + 1) * n_time].clone())
        got = plan.dump().cpu().numpy()
        plan.sync()
    assert np.array_equal(got.astype(np.int64), oracle.correlate(oracle.FMT_CI4, x))


# ------------------------------------------------ the CTA-pair kernel over its ring of planes ---
# Two or more 128-input tiles: every tile count's grouping (an odd one leaves a CTA without a row
# tile, transposed tile pairs), input counts that end inside a tile and inside 16, samples that end
# inside a stage (64 / 32), a chunk (512 / 256 / 384) and an exact window, few and many channels.
PAIR_SIZES = [(65, 2, 40), (128, 3, 300), (129, 1, 1), (130, 3, 65), (169, 5, 513), (192, 2, 385), (200, 3, 700), (256, 2, 1100), (320, 1, 130),
              (331, 2, 96)]


def draw(fmt, n_time, n_chan, n_sta, seed):
    if fmt == "ci4":
        return synth.uniform_ci4(n_time, n_chan, n_sta, seed=seed, lo=-8, hi=7)
    if fmt == "ci8":
        return synth.uniform_ci8(n_time, n_chan, n_sta, seed=seed)
    return synth.gaussian_cf32(n_time, n_chan, n_sta, seed=seed)


def placed(torch, x, offset):
    """x on the device, its first byte `offset` bytes past a 16-byte boundary."""
    flat = torch.from_numpy(np.ascontiguousarray(x)).view(torch.uint8).reshape(-1).cuda()
    buf = torch.zeros(flat.numel() + 64, dtype=torch.uint8, device="cuda")
    buf[offset:offset + flat.numel()] = flat
    assert buf.data_ptr() % 16 == 0
    return buf


def check(fmt, got, x, n_in):
    want = oracle.correlate({"ci4": oracle.FMT_CI4, "ci8": oracle.FMT_CI8, "cf32": oracle.FMT_CF32}[fmt], x)
    if fmt != "cf32":
        assert np.array_equal(got.astype(np.int64), want)
        return
    # the float path's tolerance: 1e-6 of sqrt(V_ii V_jj) per entry
    i = np.arange(n_in)
    autos = want[:, i * (i + 1) // 2 + i, 0]
    ii, jj = np.tril_indices(n_in)
    scale = np.sqrt(autos[:, ii] * autos[:, jj])
    err = np.abs((got[..., 0] - want[..., 0]) + 1j * (got[..., 1] - want[..., 1]))
    assert (err <= 1e-6 * scale).all()


@pytest.mark.parametrize("fmt", ["ci4", "ci8", "cf32"])
@pytest.mark.parametrize("n_sta,n_chan,n_time", PAIR_SIZES)
def test_pair_ring_kernel(torch, fmt, n_sta, n_chan, n_time):
    x = draw(fmt, n_time, n_chan, n_sta, seed=n_sta + n_time)
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor") as plan:
        plan.set_tuning(0, 0, 1, 1)
        out = torch.full((n_chan, plan.info["n_pairs"], 2), -1, device="cuda",
                         dtype=torch.float32 if fmt == "cf32" else torch.int32)
        plan.execute_dump(torch.from_numpy(x).cuda(), out)
        plan.sync()
    check(fmt, out.cpu().numpy(), x, 2 * n_sta)


@pytest.mark.parametrize("fmt,offset", [("ci4", 1), ("ci4", 6), ("ci8", 3), ("ci8", 2), ("cf32", 4), ("cf32", 8)])
@pytest.mark.parametrize("n_sta", [160, 135, 129, 192])
def test_pair_ring_kernel_reads_any_alignment(torch, fmt, offset, n_sta):
    x = draw(fmt, 150, 3, n_sta, seed=offset)
    buf = placed(torch, x, offset)
    with xcorr.Plan(n_sta, 3, 150, fmt=fmt, engine="tensor") as plan:
        xcorr.xcorr_execute(plan.handle, buf.data_ptr() + offset, 150, torch.cuda.current_stream().cuda_stream)
        got = plan.dump().cpu().numpy()
        plan.sync()
    check(fmt, got, x, 2 * n_sta)


@pytest.mark.parametrize("fmt,n_chan,n_time", [("ci4", 200, 600), ("ci8", 130, 300), ("cf32", 60, 800)])
def test_pair_ring_kernel_refills_its_ring(torch, fmt, n_chan, n_time):
    """More chunks than ring slots, over three adding executes of different lengths."""
    n_sta = 129
    x = draw(fmt, 2 * n_time + 40, n_chan, n_sta, seed=11)
    parts = [x[:n_time], x[n_time:n_time + 40], x[n_time + 40:]]
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor") as plan:
        plan.set_tuning(0, 0, 1, 1)
        for part in parts:
            plan.execute(torch.from_numpy(np.ascontiguousarray(part)).cuda())
        got = plan.dump().cpu().numpy()
        plan.sync()
    check(fmt, got, x, 2 * n_sta)


@pytest.mark.parametrize("fmt", ["ci8", "cf32"])
def test_pair_ring_kernel_in_graphs_and_on_two_streams(torch, fmt):
    """A captured execute replays on new data; two plans on two streams do not wait for each other."""
    n_sta, n_chan, n_time = 136, 4, 200
    xs = [draw(fmt, n_time, n_chan, n_sta, seed=s) for s in (1, 2)]
    xd = [torch.from_numpy(x).cuda() for x in xs]
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt) as plan, xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt) as other:
        out = plan.execute_dump(xd[0])
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        buf = xd[0].clone()
        with torch.cuda.graph(graph):
            plan.execute_dump(buf, out)
        for k in (1, 0):
            buf.copy_(xd[k])
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            check(fmt, out.cpu().numpy(), xs[k], 2 * n_sta)
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        outs = [torch.zeros_like(out) for _ in range(2)]
        torch.cuda.synchronize()
        for _ in range(5):
            for k, pl in enumerate((plan, other)):
                pl.execute_dump(xd[k], outs[k], stream=streams[k])
        torch.cuda.synchronize()
        plan.sync()
        other.sync()
        for k in range(2):
            check(fmt, outs[k].cpu().numpy(), xs[k], 2 * n_sta)


def test_pair_ring_kernel_float_edges(torch):
    """Windows past the drain's fast range (powers 2^90 apart), an all-zero input, one NaN."""
    n_sta, n_chan, n_time = 130, 2, 500
    x = synth.gaussian_cf32(n_time, n_chan, n_sta, seed=3)
    x[:, :, 5] *= np.float32(2.0**50)
    x[:, :, 9] *= np.float32(2.0**-40)
    x[:, 1, 40, 1] = 0
    clean = oracle.correlate(oracle.FMT_CF32, x)
    x[450, 0, 100, 0, 1] = np.nan
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="cf32") as plan:
        got = plan.execute_dump(torch.from_numpy(x).cuda()).cpu().numpy()
        plan.sync()
    n_in = 2 * n_sta
    ii, jj = np.tril_indices(n_in)
    bad = np.zeros((n_chan, ii.size), dtype=bool)
    bad[0] = (ii == 200) | (jj == 200)
    assert np.array_equal(np.isnan(got[..., 0]), bad) and np.array_equal(np.isnan(got[..., 1]), bad)
    i = np.arange(n_in)
    autos = clean[:, i * (i + 1) // 2 + i, 0]
    scale = np.sqrt(autos[:, ii] * autos[:, jj])
    err = np.abs((got[..., 0] - clean[..., 0]) + 1j * (got[..., 1] - clean[..., 1]))
    assert (err[~bad] <= 1e-6 * scale[~bad]).all()


# ------------------------------------------- int8 samples decoded on chip, on CTA pairs ---
@pytest.mark.parametrize("n_sta,n_chan,n_time", [(4, 3, 1), (4, 20, 33), (32, 5, 511), (60, 2, 513), (64, 90, 70), (68, 2, 1024),
                                                 (128, 3, 1025), (132, 2, 31), (200, 2, 600), (256, 1, 1600), (324, 2, 64)])
def test_int8_decoded_on_chip(torch, n_sta, n_chan, n_time):
    """Input counts that are a multiple of 8 (and end inside a half-tile), samples that end inside a
    stage (32) and a window (512), full-scale codes, three executes that add up."""
    x = synth.uniform_ci8(3 * n_time, n_chan, n_sta, seed=n_sta)
    x[:n_time, 0] = -128
    x[n_time:, 0, 0, 0] = 127
    xd = torch.from_numpy(x).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="ci8", engine="tensor") as plan:
        for k in range(3):
            plan.execute(xd[k * n_time:(k + 1) * n_time].clone())
        got = plan.dump().cpu().numpy()
        plan.sync()
        one = plan.execute_dump(xd[n_time:2 * n_time].clone()).cpu().numpy()
        plan.sync()
    check("ci8", got, x, 2 * n_sta)
    check("ci8", one, x[n_time:2 * n_time], 2 * n_sta)


# ------------------------------------------------ launches that start over the previous one's tail --
@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time", [("ci4", 4, 8, 64), ("ci8", 6, 8, 64), ("ci4", 32, 16, 300), ("ci4", 160, 128, 200),
                                                     ("ci8", 64, 16, 200), ("ci8", 160, 128, 100)])
@pytest.mark.parametrize("captured", [False, True])
def test_back_to_back_launches_see_the_previous_writes(torch, fmt, n_sta, n_chan, n_time, captured):
    """Eight executes into one accumulator, each on a buffer that the stream has just rewritten (by a
    kernel of the same stream, and once by a joined one), then the dump: short and long launches."""
    x = draw(fmt, 8 * n_time, n_chan, n_sta, seed=7 * n_sta + n_time)
    xd = torch.from_numpy(x).cuda()
    buf = torch.zeros_like(xd[:n_time])
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt) as plan:
        out = torch.empty((n_chan, plan.info["n_pairs"], 2), dtype=torch.int32, device="cuda")

        def passes():
            for k in range(8):
                part = xd[k * n_time:(k + 1) * n_time]
                if k == 3:  # written on another stream, joined by events
                    side = torch.cuda.Stream()
                    side.wait_stream(torch.cuda.current_stream())
                    with torch.cuda.stream(side):
                        torch.add(part, 0, out=buf)
                    torch.cuda.current_stream().wait_stream(side)
                else:
                    torch.add(part, 0, out=buf)
                plan.execute(buf)
            plan.dump(out=out)

        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            if captured:
                passes()
                graph = torch.cuda.CUDAGraph()
                stream.synchronize()
                with torch.cuda.graph(graph, stream=stream):
                    passes()
                out.zero_()
                graph.replay()
                graph.replay()
            else:
                passes()
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        plan.sync()
    assert np.array_equal(got.astype(np.int64), oracle.correlate(oracle.FMT_CI4 if fmt == "ci4" else oracle.FMT_CI8, x))


# ------------------------------------------- rows copied to 16-byte units before the on-chip decode ---
@pytest.mark.parametrize("fmt", ["ci4", "ci8"])
@pytest.mark.parametrize("n_sta,n_chan,n_time", [(1, 1, 1), (1, 40, 130), (3, 5, 257), (4, 33, 128), (5, 300, 64), (9, 7, 1030), (23, 6, 129),
                                                 (29, 9, 1100), (31, 2, 40), (33, 3, 300), (61, 4, 515), (65, 3, 129), (135, 2, 200), (131, 40, 90)])
def test_padded_rows(torch, fmt, n_sta, n_chan, n_time):
    """Every remainder of a row by 16 bytes, single samples, packed and split small layouts; stores,
    then an adding execute of a shorter block, from a base address off its 16-byte boundary."""
    x = draw(fmt, n_time + 3, n_chan, n_sta, seed=n_sta + n_time)
    bufs = [placed(torch, x[:n_time], 0), placed(torch, x[n_time:], 5)]
    with xcorr.Plan(n_sta, n_chan, max(n_time, 3), fmt=fmt, engine="tensor") as plan:
        stream = torch.cuda.current_stream().cuda_stream
        for variant in (None, 4, 5, 6, 10) if fmt == "ci4" else (None,):
            if variant is not None:
                plan.set_tuning(variant, 0, 2, 0)
            xcorr.xcorr_execute(plan.handle, bufs[0].data_ptr(), n_time, stream)
            xcorr.xcorr_execute(plan.handle, bufs[1].data_ptr() + 5, 3, stream)
            got = plan.dump().cpu().numpy()
            plan.sync()
            check(fmt, got, x, 2 * n_sta)


@pytest.mark.parametrize("offset", list(range(16)))
@pytest.mark.parametrize("fmt,n_sta", [("ci4", 69), ("ci8", 33), ("ci4", 72)])
def test_padded_rows_from_any_address(torch, fmt, n_sta, offset):
    x = draw(fmt, 70, 3, n_sta, seed=offset)
    buf = placed(torch, x, offset)
    with xcorr.Plan(n_sta, 3, 70, fmt=fmt, engine="tensor") as plan:
        xcorr.xcorr_execute(plan.handle, buf.data_ptr() + offset, 70, torch.cuda.current_stream().cuda_stream)
        got = plan.dump().cpu().numpy()
        plan.sync()
    check(fmt, got, x, 2 * n_sta)


@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time,spare", [("ci4", 69, 40, 3000, 1 << 22), ("ci8", 69, 40, 1500, 1 << 22),
                                                           ("ci8", 33, 3, 9000, 1 << 18), ("ci8", 129, 4, 700, 1)])
def test_padded_rows_in_pieces(torch, fmt, n_sta, n_chan, n_time, spare):
    """A memory limit that leaves room for a few channels, or for a part of one channel's samples."""
    n_in = 2 * n_sta
    x = draw(fmt, n_time, n_chan, n_sta, seed=3)
    budget = n_chan * n_in * (n_in + 1) // 2 * 8 + 256 + spare
    for _ in range(40):  # (the least that a plan needs beside its accumulator is the library's to say)
        try:
            plan = xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor", hbm_budget_bytes=budget)
            break
        except xcorr.XcorrError:
            budget += 1 << 18
    with plan:
        assert plan.info["device_bytes"] <= budget
        for _ in range(2):
            plan.execute(torch.from_numpy(x).cuda())
        got = plan.dump().cpu().numpy()
        plan.sync()
    check(fmt, got, np.concatenate([x, x]), n_in)


@pytest.mark.parametrize("fmt,n_sta", [("ci4", 75), ("ci4", 13), ("ci8", 75)])
def test_padded_rows_in_graphs_and_tuned(torch, fmt, n_sta):
    n_chan, n_time = 6, 150
    xs = [draw(fmt, n_time, n_chan, n_sta, seed=s) for s in (1, 2)]
    buf = torch.from_numpy(xs[0]).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor") as plan:
        plan.autotune(buf)
        out = plan.execute_dump(buf)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            plan.execute_dump(buf, out)
        for k in (1, 0):
            buf.copy_(torch.from_numpy(xs[k]))
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            check(fmt, out.cpu().numpy(), xs[k], 2 * n_sta)
        plan.sync()


# --------------------------------------------- float input of one tile: any address, shared blocks ---
@pytest.mark.parametrize("n_sta,n_chan,n_time,offset", [(1, 1, 1, 0), (1, 3, 385, 4), (4, 16, 384, 0), (7, 5, 800, 8), (9, 30, 383, 12), (16, 19, 1153, 0),
                                                        (33, 38, 769, 0), (61, 2, 1536, 4), (64, 9, 100, 0), (64, 76, 400, 0), (63, 77, 390, 8),
                                                        (64, 160, 385, 0)])
@pytest.mark.parametrize("variant", [0, 1, 2])
def test_float_one_tile(torch, variant, n_sta, n_chan, n_time, offset):
    """Clusters of 8, 4, 2 and single CTAs per tile, columns that end inside a slice of 16, windows that
    end inside a stage, every 4-byte address; a store, then an adding execute; equal in two runs."""
    x = draw("cf32", n_time, n_chan, n_sta, seed=n_sta + n_time)
    buf = placed(torch, x, offset)
    got = []
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="cf32") as plan:
        plan.set_tuning(variant, 0, 2, 0)
        for _ in range(2):
            for _ in range(2):
                xcorr.xcorr_execute(plan.handle, buf.data_ptr() + offset, n_time, torch.cuda.current_stream().cuda_stream)
            got.append(plan.dump().cpu().numpy())
            plan.sync()
    assert np.array_equal(got[0], got[1])
    check("cf32", got[0], np.concatenate([x, x]), 2 * n_sta)


@pytest.mark.parametrize("value", [np.nan, np.inf, 1e-40])
def test_float_one_tile_edges(torch, value):
    """One non-finite or subnormal sample: its input's visibilities, and no other's."""
    n_sta, n_chan, n_time = 19, 4, 800
    x = draw("cf32", n_time, n_chan, n_sta, seed=5)
    x[401, 2, 7, 1, 0] = value
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="cf32") as plan:
        got = plan.execute_dump(torch.from_numpy(x).cuda()).cpu().numpy()
        plan.sync()
    ii, jj = np.tril_indices(2 * n_sta)
    hit = np.zeros(got.shape[:2], dtype=bool)
    if not np.isfinite(value):
        hit[2] = (ii == 15) | (jj == 15)
        assert not np.isfinite(got[hit]).any()
        x[401, 2, 7, 1, 0] = 0
    want = oracle.correlate(oracle.FMT_CF32, x)
    autos = want[:, np.arange(2 * n_sta) * (np.arange(2 * n_sta) + 3) // 2, 0]
    scale = np.sqrt(autos[:, ii] * autos[:, jj])
    err = np.abs((got[..., 0] - want[..., 0]) + 1j * (got[..., 1] - want[..., 1]))
    assert (err[~hit] <= 1e-6 * scale[~hit]).all()


@pytest.mark.parametrize("shape", [3, 4, 5])
@pytest.mark.parametrize("subs", [[(8, 1, 1), (8, 9, 200), (16, 5, 129), (24, 3, 300), (32, 3, 64)],
                                  [(8, 700, 70), (24, 151, 33), (40, 30, 260), (72, 40, 100), (32, 2, 1000), (64, 200, 20)]])
def test_batch_packs_channels(torch, shape, subs):
    """Channel groups that end inside a tile, beside subarrays that pack nothing; fewer and more items
    than SMs, so that the dealing has short last rounds."""
    xs = [draw("ci4", t, c, s, seed=s + c + t) for s, c, t in subs]
    batch = xcorr.Batch(subs)
    batch.set_variant(shape)
    outs = batch.execute([torch.from_numpy(x).cuda() for x in xs])
    batch.sync()
    for x, out in zip(xs, outs):
        check("ci4", out.cpu().numpy(), x, 2 * x.shape[2])
    batch.close()


@pytest.mark.parametrize("n_groups", [0, 1, 3, 8])
@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time", [("ci4", 128, 9, 300), ("ci4", 37, 70, 700), ("ci8", 64, 11, 130), ("ci8", 70, 130, 400),
                                                     ("ci8", 101, 10, 129), ("ci4", 131, 64, 1500), ("ci4", 1, 3, 5)])
def test_host_to_host_in_groups(torch, fmt, n_sta, n_chan, n_time, n_groups):
    """Channel groups of every on-chip route: whole rows, rows that are padded, int8; twice, on new data."""
    for seed in (1, 2):
        x = draw(fmt, n_time, n_chan, n_sta, seed=seed)
        with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor") as plan:
            out = plan.execute_dump_host(torch.from_numpy(x).pin_memory(), n_groups=n_groups)
            plan.sync()
        check(fmt, out.numpy(), x, 2 * n_sta)


@pytest.mark.parametrize("variant", [4, 5, 6])
@pytest.mark.parametrize("n_sta,n_chan,n_time", [(64, 5, 1088), (64, 5, 1089), (72, 170, 1152), (136, 30, 2049), (64, 320, 2300)])
def test_epilogue_of_short_and_long_items(torch, variant, n_sta, n_chan, n_time):
    """Both numbers of epilogue warps on either side of their lines, storing then adding; several items a CTA."""
    x = draw("ci4", n_time, n_chan, n_sta, seed=n_time)
    xd = torch.from_numpy(x).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="ci4", engine="tensor") as plan:
        plan.set_tuning(variant, 0, 2, 0)
        plan.execute(xd)
        plan.execute(xd[:n_time // 2].contiguous())
        got = plan.dump().cpu().numpy()
        plan.sync()
    check("ci4", got, np.concatenate([x, x[:n_time // 2]]), 2 * n_sta)


def test_batch_of_long_items(torch):
    subs = [(64, 30, 2500), (16, 40, 3000), (72, 50, 2100)]
    xs = [draw("ci4", t, c, s, seed=s + c + t) for s, c, t in subs]
    batch = xcorr.Batch(subs)
    outs = batch.execute([torch.from_numpy(x).cuda() for x in xs])
    batch.sync()
    for x, out in zip(xs, outs):
        check("ci4", out.cpu().numpy(), x, 2 * x.shape[2])
    batch.close()


@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time", [("ci4", 1, 1, 3), ("ci4", 9, 5, 70), ("ci8", 65, 3, 40), ("cf32", 1, 1, 9), ("cf32", 33, 5, 400)])
def test_wide_dump_into_a_new_buffer(torch, fmt, n_sta, n_chan, n_time):
    """The buffer a wide dump makes itself holds what adding to zeros gives (odd and even pair counts),
    also where the allocator hands out memory that held other numbers."""
    x = torch.from_numpy(draw(fmt, n_time, n_chan, n_sta, seed=2)).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt) as plan:
        zeros = torch.zeros((n_chan, plan.info["n_pairs"], 2), dtype=torch.float64 if fmt == "cf32" else torch.int64, device="cuda")
        plan.execute(x)
        plan.dump(out=zeros, reset=False, wide=True)
        torch.full_like(zeros, -7)
        torch.cuda.synchronize()
        assert torch.equal(plan.dump(wide=True), zeros) and plan.samples == n_time
        torch.full_like(zeros, -7)
        assert torch.equal(plan.execute_dump(x, wide=True), zeros)
        empty = plan.dump(wide=True)  # nothing integrated since the reset
        assert not empty.any() and plan.samples == 0
        plan.sync()


@pytest.mark.parametrize("n_sta,n_chan,n_time", [(64, 153, 2700), (72, 60, 4001), (64, 40, 3300), (136, 12, 4100), (61, 155, 2900), (100, 70, 4000),
                                                 (64, 228, 2817), (64, 229, 2817), (40, 76, 4225), (40, 38, 2049)])
@pytest.mark.parametrize("variant", [4, 10])
def test_last_wave_split_over_the_idle_sms(torch, variant, n_sta, n_chan, n_time):
    """Whole tiles, then parts of the last ones added into cleared channels; one part of one stage, part
    counts that leave a short last part, launches that are a last wave altogether; then an adding
    execute. Twice into a buffer that held other numbers."""
    x = draw("ci4", n_time, n_chan, n_sta, seed=n_sta + n_time)
    xd = torch.from_numpy(x).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="ci4", engine="tensor") as plan:
        plan.set_tuning(variant, 0, 2, 0)
        out = torch.full((n_chan, plan.info["n_pairs"], 2), -5, dtype=torch.int32, device="cuda")
        for _ in range(2):
            plan.execute_dump(xd, out)
        check("ci4", out.cpu().numpy(), x, 2 * n_sta)
        plan.execute(xd)
        plan.execute(xd[:100].contiguous())
        got = plan.dump().cpu().numpy()
        plan.sync()
    check("ci4", got, np.concatenate([x, x[:100]]), 2 * n_sta)


@pytest.mark.parametrize("n_sta,n_chan,n_time,offset", [(4, 500, 385, 0), (1, 700, 400, 4), (10, 301, 800, 0), (16, 333, 400, 8), (25, 200, 769, 0),
                                                        (32, 155, 300, 12), (8, 64, 1024, 0)])
def test_float_channels_side_by_side(torch, n_sta, n_chan, n_time, offset):
    """Packed tiles: a last group that is not full, single and shared tiles; a store, then an adding
    execute; a non-finite sample reaches its own channel's visibilities only."""
    x = draw("cf32", n_time, n_chan, n_sta, seed=n_sta + n_time)
    buf = placed(torch, x, offset)
    stream = torch.cuda.current_stream().cuda_stream
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="cf32") as plan:
        for _ in range(2):
            xcorr.xcorr_execute(plan.handle, buf.data_ptr() + offset, n_time, stream)
        check("cf32", plan.dump().cpu().numpy(), np.concatenate([x, x]), 2 * n_sta)
        c = n_chan // 2 + 1
        bad = torch.from_numpy(x).cuda()
        clean = plan.execute_dump(bad).cpu().numpy()
        bad[n_time - 1, c, 0, 1, 0] = float("nan")
        got = plan.execute_dump(bad).cpu().numpy()
        plan.sync()
    ii, jj = np.tril_indices(2 * n_sta)
    hit = np.zeros(got.shape[:2], dtype=bool)
    hit[c] = (ii == 1) | (jj == 1)
    assert np.isnan(got[hit]).all() and np.array_equal(got[~hit], clean[~hit])


@pytest.mark.parametrize("n_sta,n_chan,n_time", [(64, 1500, 1), (72, 700, 40), (100, 500, 128), (136, 120, 300)])
def test_eight_epilogue_warps_item_after_item(torch, n_sta, n_chan, n_time):
    """Many short items a CTA whose row corrections differ as far as codes allow (every input at another
    level, another one in the next channel), storing and adding: a row's correction is read by two
    warps, of which one may be an item behind."""
    rng = np.random.default_rng(n_sta)
    level = rng.integers(0, 256, size=(1, n_chan, n_sta, 2), dtype=np.uint8)
    x = np.broadcast_to(level, (n_time, n_chan, n_sta, 2)).copy()
    xd = torch.from_numpy(x).cuda()
    want = oracle.correlate(oracle.FMT_CI4, x)
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="ci4", engine="tensor") as plan:
        plan.set_tuning(4, 0, 2, 0)
        for _ in range(5):
            for _ in range(3):
                plan.execute(xd)
            assert np.array_equal(plan.dump().cpu().numpy().astype(np.int64), 3 * want)
        plan.sync()


def least_budget(n_sta, n_chan, n_time, fmt):
    """The smallest memory limit that a plan is made with, from the error of one that is too small."""
    with pytest.raises(RuntimeError, match="plan needs") as err:
        xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor", hbm_budget_bytes=1)
    return int(str(err.value).split("plan needs ")[1].split()[0])


@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time", [("cf32", 129, 60, 800), ("cf32", 256, 33, 500), ("cf32", 150, 90, 385), ("ci4", 129, 200, 600),
                                                     ("ci4", 256, 70, 1100)])
@pytest.mark.parametrize("more", [0, 3])
def test_pair_ring_kernel_at_its_least_ring(torch, fmt, n_sta, n_chan, n_time, more):
    """A ring cut to one step of a batch by the memory limit (and to a little more): many batches, each
    slot refilled again and again; a store, then an adding execute."""
    budget = least_budget(n_sta, n_chan, n_time, fmt)
    chunk = 384 * 6 * 2 if fmt == "cf32" else 512 * 2
    x = draw(fmt, n_time, n_chan, n_sta, seed=n_sta)
    xd = torch.from_numpy(x).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor",
                    hbm_budget_bytes=budget + more * chunk * 256 * ((2 * n_sta + 255) // 256)) as plan:
        plan.set_tuning(0, 0, 1, 1)
        for _ in range(2):
            plan.execute(xd)
        got = plan.dump().cpu().numpy()
        plan.sync()
    check(fmt, got, np.concatenate([x, x]), 2 * n_sta)


def test_pair_ring_kernel_waits_alike_in_every_run(torch):
    """Unpack warps that find their slot still read, or just read, in every batch: the same bits each
    time, and a plan that reports no failure."""
    n_sta, n_chan, n_time = 140, 120, 385
    x = torch.from_numpy(draw("cf32", n_time, n_chan, n_sta, seed=3)).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="cf32", hbm_budget_bytes=least_budget(n_sta, n_chan, n_time, "cf32")) as plan:
        first = plan.execute_dump(x)
        for _ in range(30):
            assert torch.equal(plan.execute_dump(x), first)
        plan.sync()
    check("cf32", first.cpu().numpy(), x.cpu().numpy(), 2 * n_sta)


@pytest.mark.parametrize("n_sta,n_chan,n_time", [(8, 16, 256), (32, 64, 1024), (29, 5, 700)])
def test_split_launches_into_an_output_off_its_pairs(torch, n_sta, n_chan, n_time):
    """Launches whose every tile is split in time clear the output and add 4-byte integers: an output that
    is aligned to those only is as good as any."""
    x = draw("ci4", n_time, n_chan, n_sta, seed=n_time)
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="ci4", engine="tensor") as plan:
        plan.set_tuning(10, 0, 2, 0)
        n = n_chan * plan.info["n_pairs"] * 2
        buf = torch.full((n + 2,), -9, dtype=torch.int32, device="cuda")
        for _ in range(2):
            plan.execute_dump(torch.from_numpy(x).cuda(), buf[1:n + 1])
        plan.sync()
    got = buf.cpu().numpy()
    assert got[0] == -9 and got[-1] == -9
    check("ci4", got[1:-1].reshape(n_chan, -1, 2), x, 2 * n_sta)


@pytest.mark.parametrize("n_sta,n_chan,n_time,planes", [(8, 152, 4096, True), (9, 78, 1014, True), (4, 395, 2567, True), (32, 512, 1024, True),
                                                        (64, 4, 4096, True), (68, 48, 256, True), (64, 64, 1024, False),
                                                        (128, 152, 1024, False), (31, 304, 1024, False)])
def test_int8_route(torch, n_sta, n_chan, n_time, planes):
    """int8 plans decode on chip or go through planes, whichever is faster at their size: an unpack and
    an X launch a group, or one launch (two where rows are padded)."""
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="ci8", engine="tensor") as plan:
        info = plan.query()
    assert info["kernels_per_execute"] == (2 * info["tuning"]["groups"] if planes else 1 if n_sta % 4 == 0 else 2)


@pytest.mark.parametrize("n_sta,n_chan,n_time,offset", [(1, 152, 257, 0), (5, 100, 400, 2), (8, 160, 383, 0), (8, 160, 384, 1), (12, 305, 129, 0),
                                                        (32, 153, 769, 0), (33, 80, 385, 16), (64, 3, 1500, 0), (65, 48, 200, 0), (66, 49, 33, 8)])
def test_int8_through_planes(torch, n_sta, n_chan, n_time, offset):
    """Windows, stages and 16-byte units that do not end evenly, all-(-128) samples among them; a store,
    an adding execute of a few samples (by whichever route), then a graph's replay and host memory."""
    x = draw("ci8", n_time, n_chan, n_sta, seed=n_sta + n_time)
    x[:, n_chan // 2] = -128
    buf = placed(torch, x, offset)
    stream = torch.cuda.current_stream().cuda_stream
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="ci8", engine="tensor") as plan:
        for variant, groups in ((0, 0), (1, 3), (2, 8)):
            plan.set_tuning(variant, groups, 2, 0)
            xcorr.xcorr_execute(plan.handle, buf.data_ptr() + offset, n_time, stream)
            xcorr.xcorr_execute(plan.handle, buf.data_ptr() + offset, 30, stream)
            check("ci8", plan.dump().cpu().numpy(), np.concatenate([x, x[:30]]), 2 * n_sta)
        out = torch.empty((n_chan, plan.info["n_pairs"], 2), dtype=torch.int32, device="cuda")
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            xcorr.xcorr_execute_dump(plan.handle, buf.data_ptr() + offset, n_time, out.data_ptr(), True,
                                     xcorr.XCORR_DUMP_RESET, torch.cuda.current_stream().cuda_stream)
        out.fill_(7)
        graph.replay()
        check("ci8", out.cpu().numpy(), x, 2 * n_sta)
        host = plan.execute_dump_host(torch.from_numpy(x).pin_memory())
        plan.sync()
        check("ci8", host.numpy(), x, 2 * n_sta)


@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time,ring", [("cf32", 128, 16, 256, False), ("cf32", 128, 16, 1024, False), ("cf32", 65, 8, 4096, False),
                                                          ("cf32", 256, 64, 2048, True), ("cf32", 256, 256, 1024, True), ("ci4", 128, 100, 1024, False),
                                                          ("ci4", 169, 97, 1500, True), ("ci4", 65, 16, 256, False)])
def test_route_of_two_or_more_tiles(torch, fmt, n_sta, n_chan, n_time, ring):
    """The ring's one launch, or an unpack and an X launch a group through all planes."""
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor") as plan:
        plan.set_tuning(0, 0, 2, 1)
        info = plan.query()
    assert info["kernels_per_execute"] == (1 if ring else 2 * info["tuning"]["groups"])


@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time,offset", [("cf32", 65, 90, 800, 0), ("cf32", 75, 100, 1100, 4), ("cf32", 169, 60, 900, 0),
                                                            ("cf32", 331, 30, 800, 8), ("cf32", 200, 70, 1153, 0), ("ci4", 65, 200, 1100, 0),
                                                            ("ci4", 169, 120, 1600, 3), ("ci4", 136, 160, 1300, 0), ("ci4", 260, 80, 1031, 8)])
def test_ring_where_all_planes_do_not_fit(torch, fmt, n_sta, n_chan, n_time, offset):
    """The ring under a limit that all planes pass: odd tile counts, inputs that end inside a tile, rows
    and addresses off 16 bytes, a last chunk that is not full; a store, then a shorter adding execute."""
    x = draw(fmt, n_time, n_chan, n_sta, seed=n_sta)
    buf = placed(torch, x, offset)
    stream = torch.cuda.current_stream().cuda_stream
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor", hbm_budget_bytes=least_budget(n_sta, n_chan, n_time, fmt) + (1 << 20)) as plan:
        plan.set_tuning(0, 0, 2, 1)
        assert plan.query()["kernels_per_execute"] == 1
        xcorr.xcorr_execute(plan.handle, buf.data_ptr() + offset, n_time, stream)
        xcorr.xcorr_execute(plan.handle, buf.data_ptr() + offset, n_time - 77, stream)
        got = plan.dump().cpu().numpy()
        plan.sync()
    check(fmt, got, np.concatenate([x, x[:n_time - 77]]), 2 * n_sta)


@pytest.mark.parametrize("n_sta,n_chan,max_time", [(72, 16, 16777215), (128, 1024, 300000)])
def test_plans_of_very_long_executes(torch, n_sta, n_chan, max_time):
    """4-bit plans whose longest execute has more ring places than short ones ever need."""
    n_time = 700
    x = draw("ci4", n_time, n_chan, n_sta, seed=n_sta)
    xd = torch.from_numpy(x).cuda()
    with xcorr.Plan(n_sta, n_chan, max_time, fmt="ci4") as plan:
        for unfused in (0, 1):
            plan.set_tuning(4, 0, 2, unfused)
            plan.execute(xd)
            plan.execute(xd[:65].contiguous())
            got = plan.dump().cpu().numpy()
            plan.sync()
            if unfused == 0:
                check("ci4", got, np.concatenate([x, x[:65]]), 2 * n_sta)
                first = got
            else:
                assert np.array_equal(got, first)


@pytest.mark.parametrize("n_sta,n_chan,n_time", [(64, 5, 400), (50, 3, 385), (8, 9, 768), (65, 4, 300)])
def test_float_plan_takes_its_planes_and_no_more(torch, n_sta, n_chan, n_time):
    """The limit that planes of all channels (twelve bytes a sample of rows of a multiple of 16), one
    exponent a window and input, the accumulator and the status words need."""
    pad = (2 * n_sta + 15) // 16 * 16
    windows = (n_time + 383) // 384
    need = n_chan * (n_sta * (2 * n_sta + 1) * 8 + 12 * n_time * pad + 2 * windows * pad) + 256
    x = draw("cf32", n_time, n_chan, n_sta, seed=n_sta)
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="cf32", hbm_budget_bytes=need) as plan:
        assert plan.query()["device_bytes"] <= need
        got = plan.execute_dump(torch.from_numpy(x).cuda()).cpu().numpy()
        plan.sync()
    check("cf32", got, x, 2 * n_sta)


@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time", [("ci4", 169, 24, 513), ("ci4", 65, 1, 100), ("ci4", 99, 40, 700), ("ci4", 136, 3, 130), ("cf32", 65, 1, 100),
                                                     ("cf32", 256, 48, 2048), ("ci8", 65, 3, 100), ("ci8", 201, 9, 1000)])
def test_plan_at_the_limit_of_all_its_planes(torch, fmt, n_sta, n_chan, n_time):
    """Whatever the route, a plan is made where planes of all channels, the accumulator, the exponents
    and the status words fit, and it stays within that."""
    pad = (2 * n_sta + 15) // 16 * 16
    bytes_per = {"ci4": 2, "ci8": 4, "cf32": 12}[fmt]
    need = n_chan * (n_sta * (2 * n_sta + 1) * 8 + bytes_per * n_time * pad) + 256
    if fmt == "cf32":
        need += n_chan * 2 * pad * ((n_time + 383) // 384)
    x = draw(fmt, n_time, n_chan, n_sta, seed=n_sta)
    xd = torch.from_numpy(x).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor", hbm_budget_bytes=need) as plan:
        assert plan.query()["device_bytes"] <= need
        for unfused in (0, 1):
            plan.set_tuning(4, 0, 2, unfused)
            got = plan.execute_dump(xd).cpu().numpy()
            plan.sync()
            check(fmt, got, x, 2 * n_sta)


FIRST_PLANS = r"""
import threading
import numpy as np, torch
import oracle
from paper_1401_8288_gb300 import synth, xcorr
xcorr.load()
torch.zeros(1, device="cuda")
sizes = [("cf32", 20, 9, 800), ("cf32", 64, 12, 400), ("ci8", 64, 20, 300), ("ci8", 130, 9, 200), ("cf32", 130, 8, 500), ("cf32", 8, 40, 900)]
makers = {"ci8": (synth.uniform_ci8, oracle.FMT_CI8), "cf32": (synth.gaussian_cf32, oracle.FMT_CF32)}
xs = [makers[f][0](t, c, s, seed=k) for k, (f, s, c, t) in enumerate(sizes)]
xd = [torch.from_numpy(x).cuda() for x in xs]
torch.cuda.synchronize()
got, meet = [None] * len(sizes), threading.Barrier(len(sizes))
def work(k):
    f, s, c, t = sizes[k]
    stream = torch.cuda.Stream()
    meet.wait()
    with torch.cuda.stream(stream):
        plan = xcorr.Plan(s, c, t, fmt=f, engine="tensor")
        out = plan.execute_dump(xd[k])
        plan.sync()
        got[k] = out.cpu().numpy()
threads = [threading.Thread(target=work, args=(k,)) for k in range(len(sizes))]
[t.start() for t in threads]
[t.join() for t in threads]
for k, (f, s, c, t) in enumerate(sizes):
    want = oracle.correlate(makers[f][1], xs[k])
    if f == "ci8":
        assert np.array_equal(got[k].astype(np.int64), want), sizes[k]
    else:
        i = np.arange(2 * s)
        autos = want[:, i * (i + 1) // 2 + i, 0]
        ii, jj = np.tril_indices(2 * s)
        err = np.abs((got[k][..., 0] - want[..., 0]) + 1j * (got[k][..., 1] - want[..., 1]))
        assert (err <= 1e-6 * np.sqrt(autos[:, ii] * autos[:, jj])).all(), sizes[k]
print("alike")
"""


def test_first_plans_of_several_threads(torch):
    """The first plans of a process, made and run by threads that start together."""
    r = subprocess.run([sys.executable, "-c", FIRST_PLANS], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("alike"), r.stdout + r.stderr


def kernels_of(torch, call):
    """Kernel nodes of a captured call."""
    import ctypes
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    rt = ctypes.CDLL("libcudart.so.13")
    n = ctypes.c_size_t()
    raw = ctypes.c_void_p(graph.raw_cuda_graph())
    assert rt.cudaGraphGetNodes(raw, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(raw, nodes, ctypes.byref(n)) == 0
    kinds = []
    for node in nodes:
        kind = ctypes.c_int()
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    return kinds.count(0)  # cudaGraphNodeTypeKernel


@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time,variant", [
    ("ci4", 8, 16, 256, 10), ("ci4", 32, 64, 1024, 10), ("ci4", 64, 40, 3300, 4), ("ci4", 64, 153, 2700, 4), ("ci4", 64, 153, 2700, 0),
    ("ci4", 128, 16, 700, 7), ("ci4", 29, 5, 700, 10), ("ci4", 70, 20, 4100, 4), ("ci4", 16, 3, 40000, 10), ("ci4", 20, 3, 40000, 4),
    ("ci8", 64, 20, 300, 0), ("ci8", 33, 200, 300, 0), ("ci8", 70, 20, 1024, 0), ("cf32", 64, 20, 800, 0), ("cf32", 130, 100, 300, 0),
    ("cf32", 256, 64, 2048, 0)])
def test_kernels_per_execute(torch, fmt, n_sta, n_chan, n_time, variant):
    """The count that the plan gives is what a storing execute launches."""
    x = torch.zeros((n_time * n_chan * n_sta * 2 * {"ci4": 1, "ci8": 2, "cf32": 8}[fmt],), dtype=torch.uint8, device="cuda")
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor") as plan:
        plan.set_tuning(variant, 0, 2, 0)
        out = torch.empty((n_chan, plan.info["n_pairs"], 2), dtype=torch.float32 if fmt == "cf32" else torch.int32, device="cuda")

        def call():
            xcorr.xcorr_execute_dump(plan.handle, x.data_ptr(), n_time, out.data_ptr(), True, xcorr.XCORR_DUMP_RESET,
                                     torch.cuda.current_stream().cuda_stream)

        call()
        plan.sync()
        assert kernels_of(torch, call) == plan.query()["kernels_per_execute"]


@pytest.mark.parametrize("n_sta,n_chan,n_time", [(4, 60, 400), (16, 200, 800), (32, 300, 385)])
def test_autotune_of_packed_float_channels(torch, n_sta, n_chan, n_time):
    """Packed channels have one launch shape: the tuner does not choose among names for it."""
    x = torch.from_numpy(draw("cf32", n_time, n_chan, n_sta, seed=1)).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="cf32") as plan:
        for _ in range(4):
            plan.set_tuning(2, 0, 2, 0)
            shape, ms = plan.autotune(x)
            assert shape["stage_variant"] == 0 and ms > 0
        check("cf32", plan.execute_dump(x).cpu().numpy(), x.cpu().numpy(), 2 * n_sta)
        plan.sync()


@pytest.mark.parametrize("wide", [False, True])
def test_execute_dump_without_memory_for_the_output(torch, wide, monkeypatch):
    """A call that cannot make its output has not integrated the samples."""
    n_sta, n_chan, n_time = 8, 3, 100
    x = torch.from_numpy(draw("ci4", n_time, n_chan, n_sta, seed=1)).cuda()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt="ci4") as plan:
        with monkeypatch.context() as m:
            m.setattr(plan._torch, "empty", lambda *a, **k: (_ for _ in ()).throw(torch.OutOfMemoryError("no memory")))
            with pytest.raises(torch.OutOfMemoryError):
                plan.execute_dump(x, wide=wide)
        assert plan.query()["samples_integrated"] == 0
        got = plan.execute_dump(x, wide=wide).cpu().numpy()
        plan.sync()
    check("ci4", got, x.cpu().numpy(), 2 * n_sta)


@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time,n_groups", [("ci8", 64, 20, 300, 0), ("ci8", 70, 20, 300, 3), ("ci4", 37, 20, 300, 8), ("cf32", 20, 5, 100, 0)])
def test_host_executes_are_timed(torch, fmt, n_sta, n_chan, n_time, n_groups):
    """Host-to-host executes of int8, float and padded rows leave their durations, each once."""
    x = torch.from_numpy(draw(fmt, n_time, n_chan, n_sta, seed=1)).pin_memory()
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor") as plan:
        xcorr.xcorr_profile_enable(plan.handle, 4)
        for k in range(3):
            plan.execute_dump_host(x, n_groups=n_groups)
            plan.execute_dump(x.cuda())
        plan.sync()
        read = xcorr.xcorr_profile_read(plan.handle, 4)
        xcorr.xcorr_profile_enable(plan.handle, 0)
    assert len(read) == 4 and all(0 <= unpack < 10 and 0 < span < 10 for unpack, span in read)


@pytest.mark.parametrize("n_groups", [0, 1, 5])
@pytest.mark.parametrize("pinned", [(True, True), (False, False), (True, False), (False, True)])
@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time", [("ci4", 64, 40, 4000), ("ci4", 37, 70, 700), ("ci8", 64, 40, 1000), ("ci8", 9, 64, 5000), ("ci8", 8, 64, 4096),
                                                     ("cf32", 20, 9, 100)])
def test_host_memory_that_is_not_pinned(torch, fmt, n_sta, n_chan, n_time, pinned, n_groups):
    """Pageable memory on either side; int8 whose chains allow few groups, and through planes in one piece."""
    x = draw(fmt, n_time, n_chan, n_sta, seed=n_time)
    xt = torch.from_numpy(x)
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor") as plan:
        shape, dtype = (n_chan, plan.info["n_pairs"], 2), torch.float32 if fmt == "cf32" else torch.int32
        out = torch.full(shape, 3, dtype=dtype, pin_memory=pinned[1])
        plan.execute_dump_host(xt.pin_memory() if pinned[0] else xt, out, n_groups=n_groups)
        plan.sync()
    check(fmt, out.numpy(), x, 2 * n_sta)


@pytest.mark.parametrize("fmt,n_sta,n_chan,n_time,offset,rows,least", [
    ("ci8", 19, 90, 2500, 0, 76 * 256, 30), ("ci8", 21, 90, 2500, 0, 76 * 1100, 10), ("ci8", 64, 40, 1500, 2, 40 * 1100, 4), ("ci8", 20, 2, 300, 3, 128, 12),
    ("ci8", 131, 30, 1400, 0, 25 * 1030, 8), ("ci4", 65, 3, 80000, 0, 3 * 40000, 6), ("ci4", 65, 60, 2600, 0, 50 * 1600, 6), ("ci4", 72, 40, 2600, 5, 40 * 1850, 4)])
def test_long_padded_rows_in_pieces_of_samples(torch, fmt, n_sta, n_chan, n_time, offset, rows, least):
    """Memory for fewer samples of a wave's channels than there are: pieces along time that add into the
    first, whole stages or the fused kernel's blocks, with short last ones in both directions."""
    row = (2 * n_sta * (1 if fmt == "ci4" else 2) + 15) // 16 * 16
    budget = n_chan * n_sta * (2 * n_sta + 1) * 8 + 256 + 8192 + rows * row
    x = draw(fmt, n_time, n_chan, n_sta, seed=rows)
    buf = placed(torch, x, offset)
    stream = torch.cuda.current_stream().cuda_stream
    with xcorr.Plan(n_sta, n_chan, n_time, fmt=fmt, engine="tensor", hbm_budget_bytes=budget) as plan:
        if offset == 0:
            assert plan.query()["kernels_per_execute"] >= least
        for _ in range(2):
            xcorr.xcorr_execute(plan.handle, buf.data_ptr() + offset, n_time, stream)
        got = plan.dump().cpu().numpy()
        plan.sync()
    check(fmt, got, np.concatenate([x, x]), 2 * n_sta)
