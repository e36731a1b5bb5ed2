"""The lane-private counting paths at the sizes where their splits change,
against the oracle, bit-exact."""
import os
import subprocess
import sys
import time

import numpy as np
import pytest
import torch

import oracle
import paper_1011_0235_gb300 as hl
import synth
from tests.gpu_util import dev, pattern_dev, u32

pytestmark = pytest.mark.gpu
SEED = synth.SEED_BASE


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_ok):
    from paper_1011_0235_gb300 import build

    build.build()
    hl.lib()


STEP = 16 << 10  # bytes of one load per thread of a CTA


@pytest.mark.parametrize("n", [STEP * c + d for c in (1, 2, 4, 8, 16, 32, 64) for d in (-1, 0, 1)] +
                         [STEP * 64 + 127, 3 << 20, 152 * 4 * STEP - 5])
def test_oneshot_cluster_and_grid_splits(n):
    """One-shot calls on both sides of every cluster size and of the longest
    input that one cluster counts, at an aligned and an odd address; the
    output buffer holds rubbish before the call."""
    x = synth.host(n + 77, synth.mixture([0.3, 0.7], [10, 200], [2, 40]), SEED + 91, n)
    xd = dev(x)
    pat = pattern_dev(oracle.default_pattern(960))
    for off in (0, 77):
        ref = oracle.hist_u32(x[off:off + n])
        out = torch.full((256,), -7, dtype=torch.int32, device="cuda")
        assert np.array_equal(u32(hl.hist_plain(xd[off:off + n], out)), ref), off
        out.fill_(9)
        assert np.array_equal(u32(hl.hist_adaptive(xd[off:off + n], pat, out)), ref), off


@pytest.mark.parametrize("widest", [1, 2, 8, 15, 16])
@pytest.mark.parametrize("n", [0, 1, 143, STEP, STEP + 1, 2 * STEP + 77, 8 * STEP, 8 * STEP + 1, 16 * STEP, 64 * STEP - 3,
                               64 * STEP, 64 * STEP + 1])
def test_oneshot_where_wide_clusters_cannot_be_placed(n, widest):
    """Short one-shot calls on a part of a GPU that places clusters of at most
    `widest` CTAs: the inputs of a wider one are counted by a plain grid, on
    both sides of every limit, at an aligned and an odd address."""
    x = synth.host(n + 77, synth.mixture([0.3, 0.7], [10, 200], [2, 40]), SEED + 93, n)
    xd = dev(x)
    s = torch.cuda.current_stream().cuda_stream
    for off in (0, 77):
        out = torch.full((256,), -7, dtype=torch.int32, device="cuda")
        assert hl.lib().hist_plain_test_cluster(xd.data_ptr() + off, n, widest, out.data_ptr(), s) == 0
        assert np.array_equal(u32(out), oracle.hist_u32(x[off:off + n])), off


def test_oneshot_cluster_hook_rejects_bad_widths():
    out, s = hl.empty_hist(), torch.cuda.current_stream().cuda_stream
    for widest in (0, 17, 1 << 31):
        assert hl.lib().hist_plain_test_cluster(out.data_ptr(), 100, widest, out.data_ptr(), s) == hl._abi.EINVAL


def test_first_call_of_a_process_is_captured():
    """The device's widest cluster is asked for by the first call, which may
    be a captured one."""
    prog = """
import numpy as np, torch
import paper_1011_0235_gb300 as hl
x = torch.full((300_001,), 9, dtype=torch.uint8, device="cuda")
out, s = hl.empty_hist(), torch.cuda.Stream()
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=s):
    hl.hist_plain(x, out)
for _ in range(2):
    out.zero_()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    h = hl.as_u32(out)
    assert h[9] == 300_001 and h.sum() == 300_001
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", prog], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("n", [5000, 300_001, 5_000_011])
def test_oneshot_chain_replayed_from_a_graph(n):
    """Count, pattern and degeneracy chained on one stream behind the kernel
    that writes the pixels (which lets its successor start early), captured
    and replayed over new pixels."""
    xd = torch.empty(n, dtype=torch.uint8, device="cuda")
    out, pat = hl.empty_hist(), hl.empty_pattern()
    laws = [synth.normal(100, 20), synth.degenerate(7, 0.6), synth.uniform()]
    s = torch.cuda.Stream()
    res = None
    with torch.cuda.stream(s):
        def step():
            hl.hist_plain(xd, out)
            hl.binning_pattern(out, 1500, pat)
            return hl.degeneracy(out, 450)
        step()
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            res = step()
        for k, law in enumerate(laws):
            synth.device_fill_early(xd.data_ptr(), n, law, SEED + 92, k * n, s.cuda_stream)
            g.replay()
            s.synchronize()
            ref = oracle.hist_u32(synth.host(n, law, SEED + 92, k * n))
            assert np.array_equal(u32(out), ref), k
            assert bytes(pat.cpu().numpy()) == oracle.binning_pattern(ref, 1500).to_bytes(), k
            arg, m, t = oracle.degeneracy(ref.astype(np.uint64))
            assert hl.degeneracy_to_host(res) == (arg, m, t, oracle.switch(ref.astype(np.uint64), 450)), k


@pytest.mark.parametrize("n", [700, 400_003, 3_000_017])
def test_calls_behind_a_copy_in_a_graph(n):
    """One-shot, batch and stream launches captured behind a memcpy that writes
    their pixels (work that is no kernel), replayed over new pixels."""
    src = torch.empty(n, dtype=torch.uint8, device="cuda")
    xd = torch.empty(n, dtype=torch.uint8, device="cuda")
    mid = torch.empty(n, dtype=torch.uint8, device="cuda")
    out = hl.empty_hist()
    rows = torch.empty((2, 256), dtype=torch.int32, device="cuda")
    ptrs = torch.tensor([xd.data_ptr(), xd.data_ptr() + 5], dtype=torch.int64, device="cuda")
    szs = torch.tensor([n, min(n - 5, 3000)], dtype=torch.int64, device="cuda")
    st = hl.Stream(mode=hl.MODE_AUTO)
    push_out = torch.empty(256, dtype=torch.int32, device="cuda")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        def step():
            xd.copy_(src)
            hl.hist_plain(xd, out)
            mid.copy_(xd)
            assert hl.lib().hist_batch(ptrs.data_ptr(), szs.data_ptr(), 2, rows.data_ptr(), None, s.cuda_stream) == 0
            mid.copy_(xd)
            st.push(xd, push_out)
        src.zero_()
        step()
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            step()
        for k, law in enumerate([synth.normal(60, 9), synth.uniform(), synth.degenerate(3, 0.9)]):
            x = synth.host(n, law, SEED + 97, k * n)
            src.copy_(torch.from_numpy(x))
            g.replay()
            s.synchronize()
            ref = oracle.hist_u32(x)
            assert np.array_equal(u32(out), ref) and np.array_equal(u32(push_out), ref), k
            got = u32(rows).reshape(2, 256)
            assert np.array_equal(got[0], ref), k
            assert np.array_equal(got[1], oracle.hist_u32(x[5:5 + min(n - 5, 3000)])), k
    st.close()


def _sample_flag(x, addr, theta=450):
    """The switch from a chunk's sample: 256 evenly spaced 16-byte vectors
    from the first 16-byte boundary of its address, or the whole chunk."""
    head = min((16 - addr % 16) % 16, x.size)
    nvec = (x.size - head) // 16
    if nvec >= 256:
        v = (np.arange(256, dtype=np.int64) * nvec) // 256
        x = x[(head + 16 * v)[:, None] + np.arange(16)[None, :]].reshape(-1)
    return oracle.switch(oracle.hist_u32(x).astype(np.uint64), theta) if x.size else 0


# sizes around the sample's (256 vectors after a head of up to 15 bytes), of
# whole small chunks, and of chunks cut between CTAs
@pytest.mark.parametrize("sizes,cuts", [
    ([4095, 4096, 4097, 4110, 4111, 4112, 5000, 8191] * 12, [0, 1, 2, 5, 40, 96]),
    ([65_536, 70_001, 262_144, 262_145, 17, 0, 4096, 33_333] * 10, [0, 1, 3, 30, 80]),
    ([1_300_003, 2_000_000, 65_536, 1 << 20, 5, 900_001] * 3, [0, 2, 3, 18]),
])
@pytest.mark.parametrize("overlap", [False, True])
def test_recounted_is_the_samples_misjudgements(sizes, cuts, overlap):
    """AUTO pushes of one, two and many chunks whose largest bin is near the
    threshold, so that a chunk's sample and the chunk itself often disagree:
    recounted equals the disagreements of a host model of the sample (of
    every chunk but a push's last), the outputs, patterns and switches the
    oracle's, whichever of them runs in a group, in one CTA or in several."""
    rng = np.random.default_rng(len(sizes) + overlap)
    chunks = []
    for c, n in enumerate(sizes):
        x = rng.integers(0, 256, n).astype(np.uint8)
        x[rng.random(n) < 0.4475 + 0.003 * rng.standard_normal()] = c % 200
        chunks.append(x)
    offs, pos = [], 0
    for c, n in enumerate(sizes):
        pos += int(rng.integers(0, 40))
        offs.append(pos)
        pos += n
    buf = np.zeros(pos + 16, np.uint8)
    for o, ch in zip(offs, chunks):
        buf[o:o + ch.size] = ch
    bd = dev(buf)
    outs = torch.full((len(sizes), 256), -1, dtype=torch.int32, device="cuda")
    st = hl.Stream(mode=hl.MODE_AUTO, overlap=overlap)
    ref = oracle.StreamOracle(8192)
    expect = 0
    for lo, hi in zip(cuts[:-1], cuts[1:]):
        st.push_many(np.uint64(bd.data_ptr()) + np.array(offs[lo:hi], dtype=np.uint64),
                     np.array(sizes[lo:hi], dtype=np.uint64),
                     np.array([outs[j].data_ptr() for j in range(lo, hi)], dtype=np.uint64))
        recs = [ref.push(chunks[j]) for j in range(lo, hi)]
        for j in range(lo, hi - 1):
            exact = oracle.switch(oracle.hist_u32(chunks[j]).astype(np.uint64), 450)
            expect += int(_sample_flag(chunks[j], bd.data_ptr() + offs[j]) != exact)
        s = st.state()
        assert bytes(s.pattern) == ref.pattern.to_bytes() and s.flag == ref.flag
        assert s.last_kernel == recs[-1].kernel
        assert s.recounted == expect, (lo, hi)
    got = u32(outs.reshape(-1)).reshape(len(sizes), 256)
    for j, ch in enumerate(chunks):
        assert np.array_equal(got[j], oracle.hist_u32(ch)), j
    assert np.array_equal(np.array(s.totals, np.uint64), ref.totals) and s.status == 0
    st.close()


@pytest.mark.parametrize("mode,overlap,window", [(hl.MODE_AUTO, False, 1), (hl.MODE_PLAIN, True, 1),
                                                 (hl.MODE_ADAPTIVE, False, 1), (hl.MODE_AUTO, True, 2)])
def test_single_pushes_around_the_one_cta_limit(mode, overlap, window):
    """Pushes of one chunk on both sides of the largest that one CTA counts
    alone, at every alignment, without an output now and then, between pushes
    of several chunks: outputs and the state after each push are the oracle's."""
    rng = np.random.default_rng(11 + mode)
    sizes = [0, 1, 15, 143, 4097, 16_384, 65_536, 65_537, 131_071, 131_072, 131_073, 200_000]
    x = rng.integers(0, 256, 500_000, dtype=np.uint8)
    x[rng.random(x.size) < 0.46] = 9
    xd = dev(x)
    st = hl.Stream(mode=mode, overlap=overlap, window=window)
    ref = oracle.StreamOracle(oracle.BUDGET_MAX, mode=mode, window=window)
    outs = torch.full((3 * len(sizes), 256), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for i in range(3 * len(sizes)):
        n, off = sizes[(5 * i) % len(sizes)], int(rng.integers(0, 299_000))
        st.push_ptr(xd.data_ptr() + off, n, None if i % 5 == 4 else outs[i].data_ptr())
        rec = ref.push(x[off:off + n])
        if i % 7 == 6:
            st.push_many([xd.data_ptr() + 3, xd.data_ptr() + 40_000], [30_001, 140_000])
            ref.push(x[3:30_004])
            rec = ref.push(x[40_000:180_000])
        if i % 3 == 2:
            s = st.state()
            assert bytes(s.pattern) == ref.pattern.to_bytes() and bytes(s.last_pattern) == rec.pattern.to_bytes(), i
            assert s.flag == ref.flag and s.last_kernel == rec.kernel and s.chunks == ref.chunks and s.status == 0
            assert np.array_equal(np.array(s.last_hist, np.uint32), rec.hist)
            assert np.array_equal(np.array(s.totals, np.uint64), ref.totals)
        got = None if i % 5 == 4 else u32(outs[i])
        if i % 7 != 6 and got is not None:
            assert np.array_equal(got, rec.hist), (i, n)
    st.close()


def _sample_hist(x, addr):
    """A chunk's sample (_sample_flag) as a histogram, and its pixels' weight."""
    head = min((16 - addr % 16) % 16, x.size)
    nvec = (x.size - head) // 16
    if nvec < 256:
        return oracle.hist_u32(x), np.float32(1.0 if x.size else 0.0)
    v = (np.arange(256, dtype=np.int64) * nvec) // 256
    y = x[(head + 16 * v)[:, None] + np.arange(16)[None, :]].reshape(-1)
    return oracle.hist_u32(y), np.float32(x.size) / np.float32(4096)


# pushes of as many chunks as one window a CTA takes, one more, and so on for
# four and eight windows a CTA, windows shorter and longer than the pushes
@pytest.mark.parametrize("mode,window,pushes", [
    (hl.MODE_AUTO, 256, [1, 2, 152, 153, 305]),
    (hl.MODE_AUTO, 100, [304, 305, 608]),
    (hl.MODE_AUTO, 165, [609, 7, 152]),
    (hl.MODE_AUTO, 5, [152, 153, 305, 609]),
    (hl.MODE_ADAPTIVE, 7, [1, 2, 3, 400, 1]),
    (hl.MODE_PLAIN, 256, [3, 200, 2, 1]),
])
def test_windows_of_long_pushes(mode, window, pushes):
    """The window, the switches and, in AUTO mode, the windows whose switch
    their samples misjudge (a host model in FP32 and the chunks' order;
    windows within 1e-5 of the threshold count either way)."""
    rng = np.random.default_rng(window)
    count = sum(pushes)
    sizes = [int(n) for n in rng.choice([0, 700, 4111, 4200, 5000, 7001], count)]
    offs = np.cumsum([0] + [n + int(rng.integers(0, 20)) for n in sizes])[:-1]
    host = rng.integers(0, 256, int(offs[-1]) + sizes[-1] + 16).astype(np.uint8)
    for o, n in zip(offs, sizes):
        x = host[o:o + n]
        x[rng.random(n) < 0.4475 + 0.01 * rng.standard_normal()] = 9
    bd = dev(host)
    outs = torch.full((count, 256), -1, dtype=torch.int32, device="cuda")
    st = hl.Stream(mode=mode, window=window)
    ref = oracle.StreamOracle(8192, mode=mode, window=window)
    low = high = done = 0
    sampled = []
    for push in pushes:
        lo, hi = done, done + push
        st.push_many(np.uint64(bd.data_ptr()) + offs[lo:hi].astype(np.uint64), np.array(sizes[lo:hi], dtype=np.uint64),
                     np.array([outs[j].data_ptr() for j in range(lo, hi)], dtype=np.uint64))
        for j in range(lo, hi):
            x = host[offs[j]:offs[j] + sizes[j]]
            rec = ref.push(x)
            sampled.append(_sample_hist(x, bd.data_ptr() + int(offs[j])))
            if mode != hl.MODE_AUTO or j + 1 == hi:
                continue
            f = np.zeros(256, np.float32)
            for s, w in sampled[-window:]:
                f = (s.astype(np.float64) * np.float64(w) + f).astype(np.float32)
            fm, fs = float(f.max()) * 1000.0, float(f.astype(np.float64).sum()) * 450.0
            near = abs(fm - fs) <= 1e-5 * fs
            wrong = int(fs > 0 and fm >= fs) != ref.flag
            low += wrong and not near
            high += wrong or near
        done = hi
        s = st.state()
        assert s.flag == ref.flag and s.last_kernel == rec.kernel and s.status == 0
        assert low <= s.recounted <= high, push
        assert np.array_equal(st.window().cpu().numpy().view(np.uint64), ref.mw)
    assert np.array_equal(u32(outs).reshape(count, 256), np.stack([oracle.hist_u32(host[o:o + n]) for o, n in zip(offs, sizes)]))
    if mode == hl.MODE_AUTO and window < 10:
        assert low > 0
    st.close()


def test_a_captured_push_replayed():
    """Pushes of one and of two chunks captured into a graph and replayed over
    new pixels: totals, the last two patterns and the switch follow the
    replays."""
    n = 100_001
    xd = torch.empty(2 * n, dtype=torch.uint8, device="cuda")
    for count in (1, 2):
        st = hl.Stream(budget=960)
        ref = oracle.StreamOracle(960)
        s = torch.cuda.Stream()
        first = [synth.host(n, synth.uniform(), SEED + 95, k) for k in range(count)]
        with torch.cuda.stream(s):
            def push():
                st.push_many([xd.data_ptr() + k * n for k in range(count)], [n] * count)
            xd[:count * n].copy_(dev(np.concatenate(first)))
            push()
            for x in first:
                ref.push(x)
            s.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                push()
            for r in range(5):
                chunks = [synth.host(n, synth.normal(30 + 20 * r, 3 + r) if (r + k) % 2 else synth.degenerate(5, 0.7),
                                     SEED + 96 + r, k * n) for k in range(count)]
                xd[:count * n].copy_(dev(np.concatenate(chunks)))
                g.replay()
                s.synchronize()
                for x in chunks:
                    rec = ref.push(x)
            t = st.state()
        assert np.array_equal(np.array(t.totals, np.uint64), ref.totals)
        assert bytes(t.pattern) == ref.pattern.to_bytes() and bytes(t.last_pattern) == rec.pattern.to_bytes()
        assert t.flag == ref.flag and t.last_kernel == rec.kernel and t.chunks == ref.chunks
        st.close()


def _batch(sizes, seed, spread, out_shift=0):
    """hist_batch on random images of these sizes, at every alignment; the
    output rows start out_shift words into a buffer of rubbish."""
    rng = np.random.default_rng(seed)
    offs, pos = [], 0
    for n in sizes:
        pos += int(rng.integers(0, spread))
        offs.append(pos)
        pos += n
    x = rng.integers(0, 256, pos + 16, dtype=np.uint8)
    x[rng.random(pos + 16) < 0.3] = 77
    xd = dev(x)
    ptrs = torch.tensor([xd.data_ptr() + o for o in offs], dtype=torch.int64, device="cuda")
    szs = torch.tensor(list(sizes), dtype=torch.int64, device="cuda")
    buf = torch.full((len(sizes) * 256 + out_shift,), -5, dtype=torch.int32, device="cuda")
    out = buf[out_shift:]
    rc = hl.lib().hist_batch(ptrs.data_ptr(), szs.data_ptr(), len(sizes), out.data_ptr(), None,
                             torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    got = u32(out).reshape(len(sizes), 256)
    for i, (o, n) in enumerate(zip(offs, sizes)):
        assert np.array_equal(got[i], oracle.hist_u32(x[o:o + n])), (i, n)
    assert (buf[:out_shift] == -5).all()


@pytest.mark.parametrize("name,sizes,out_shift", [
    # on both sides of the warps', the groups' and the whole-image limits
    ("edges", [0, 1, 15, 16, 127, 128, 143, 4095, 4096, 4097, 131_071, 131_072, 131_073, 500_000] * 40, 1),
    ("edges of more", [0, 1, 15, 16, 127, 128, 143, 4095, 4096, 4097, 131_071, 131_072, 131_073, 250_000] * 80, 1),
    # the most images of a few, and one more
    ("most", [1 + (i * 977) % 9000 for i in range(1024)], 0),
    ("not few", [1 + (i * 977) % 9000 for i in range(1025)], 0),
    # a few images, all cut between CTAs
    ("few", [300_000, 131_072, 70_001, 5000, 4096, 3], 0),
    # one range holds hundreds of tiny images (many windows of 64) between
    # pieces of large ones
    ("long", [20_000_000] + [9] * 700 + [5000] * 300 + [30_000_001] + [0] * 100 + [4097] * 200, 3),
    # more images than one launch takes, tiny and not (and the rest few)
    ("many", [100 + 37 * (i % 300) for i in range(4096 + 70)], 2),
    ("empty", [0, 0, 0], 0),
    ("one", [1], 0),
])
def test_batch_lane_launches(name, sizes, out_shift):
    """The default batch's two launches against the oracle, image by image:
    sizes around every limit of their rule, outputs at any word."""
    _batch(sizes, 17, 40, out_shift)


@pytest.mark.parametrize("depth,window,overlap", [(2, 1, False), (4, 5, False), (3, 1, True)])
def test_host_chunks_pinned_registered_and_pageable(depth, window, overlap):
    """Chunks read in place (pinned, registered: at every alignment, to the
    range's last byte) and staged ones (pageable) in turn with device chunks,
    sizes around the limits of the launch's grid, several in flight; the
    buffers are rewritten when the stream has passed their pushes."""
    rng = np.random.default_rng(depth)
    big = 3 << 20
    pinned = torch.empty(20 << 20, dtype=torch.uint8, pin_memory=True).numpy()
    page = np.zeros((20 << 20) + 4096, np.uint8)
    first = -page.ctypes.data % 4096
    reg, plain = page[first:first + (20 << 20)], np.zeros(20 << 20, np.uint8)
    assert int(torch.cuda.cudart().cudaHostRegister(reg.ctypes.data, reg.size, 0)) == 0
    st = hl.Stream(window=window, overlap=overlap)
    st.attach_staging(big, depth)
    ref = oracle.StreamOracle(oracle.BUDGET_MAX)
    sizes = [1, 100, 4097, 32768, 65536 + 1, 16 * 32768 - 1, 16 * 32768 + 129, 1 << 20, 2_000_003, big, 0]
    outs = torch.full((66, 256), -1, dtype=torch.int32, device="cuda")
    hists, rec, keep = [], None, []
    for i in range(66):
        if i % 22 == 0:  # the buffers from their ends down
            torch.cuda.current_stream().synchronize()
            end = {id(b): b.size for b in (pinned, reg, plain)}
            for b in (pinned, reg, plain):
                b[:] = 0
        n, where = sizes[i % len(sizes)], (pinned, reg, pinned, plain, None)[int(rng.integers(0, 5))]
        data = rng.integers(0, 256, n, dtype=np.uint8)
        data[rng.random(n) < rng.choice([0.0, 0.45, 0.9])] = 31
        if where is None:
            keep.append(dev(data) if n else torch.empty(0, dtype=torch.uint8, device="cuda"))
            st.push(keep[-1], outs[i])
        else:
            at = end[id(where)] - n
            end[id(where)] = at - int(rng.integers(0, 300))
            where[at:at + n] = data
            st.push_host(where.ctypes.data + at, n, outs[i].data_ptr())
        rec = ref.push(data)
        hists.append(rec.hist)
    win = st.window().cpu().numpy().view(np.uint64)
    torch.cuda.synchronize()
    s = st.state()
    assert np.array_equal(u32(outs).reshape(66, 256), np.stack(hists))
    assert np.array_equal(win, np.sum(np.stack(hists[-window:]).astype(np.uint64), axis=0))
    assert np.array_equal(np.array(s.totals, np.uint64), ref.totals) and s.status == 0 and s.chunks == 66
    assert bytes(s.pattern) == ref.pattern.to_bytes() and s.flag == ref.flag and s.last_kernel == rec.kernel
    st.close()
    assert int(torch.cuda.cudart().cudaHostUnregister(reg.ctypes.data)) == 0


@pytest.mark.parametrize("mode", [hl.MODE_AUTO, hl.MODE_PLAIN, hl.MODE_ADAPTIVE])
@pytest.mark.parametrize("window", [1, 2, 5])
def test_switch_of_host_chunks_over_a_window(window, mode):
    """The switch and the kernel of chunks pushed from pinned and from pageable
    memory follow the window's histogram: the window's switch differs from
    the last chunk's on the way."""
    rng = np.random.default_rng(window)
    sizes = [30_000, 70_001, 140_000, 300_007]
    top = max(sizes)
    pinned = torch.empty(top, dtype=torch.uint8, pin_memory=True).numpy()
    plain = np.zeros(top, np.uint8)
    st = hl.Stream(mode=mode, window=window)
    st.attach_staging(top, 2)
    ref = oracle.StreamOracle(oracle.BUDGET_MAX, mode=mode, window=window)
    single = oracle.StreamOracle(oracle.BUDGET_MAX, mode=mode)
    out = torch.empty(256, dtype=torch.int32, device="cuda")
    differ = 0
    for i in range(24):
        n = sizes[(i * 7 + i // 4) % 4]
        data = rng.integers(0, 256, n, dtype=np.uint8)
        if i // 3 % 2:
            data[rng.random(n) < 0.8] = 31
        where = plain if i % 5 == 2 else pinned
        where[:n] = data
        st.push_host(where.ctypes.data, n, out.data_ptr())
        rec = ref.push(data)
        single.push(data)
        s = st.state()  # (the stream has passed the push)
        differ += ref.flag != single.flag
        assert np.array_equal(u32(out), rec.hist), i
        assert s.flag == ref.flag and s.last_kernel == rec.kernel and s.status == 0, i
        assert np.array_equal(st.window().cpu().numpy().view(np.uint64), ref.mw), i
    assert (differ > 0) == (window > 1)
    st.close()


@pytest.mark.parametrize("overlap", [False, True])
@pytest.mark.parametrize("mode", [hl.MODE_AUTO, hl.MODE_ADAPTIVE])
def test_early_pushes_after_captured_and_replayed_ones(mode, overlap):
    """A captured push advances the stream's launch numbers without a launch,
    and its replay sets the device's number back: pushes that start early
    behind both (from pinned memory, and with overlap from the device) are
    exact and no wait of theirs runs out."""
    rng = np.random.default_rng(5 + mode)
    n = 700_001
    st = hl.Stream(mode=mode, overlap=overlap)
    st.attach_staging(n, 2)
    ref, rec, count = oracle.StreamOracle(oracle.BUDGET_MAX, mode=mode), None, 0
    pinned = torch.empty(n, dtype=torch.uint8, pin_memory=True)
    chunks = [rng.integers(0, 256, n - 1000 * k, dtype=np.uint8) for k in range(4)]
    for k, c in enumerate(chunks):
        c[rng.random(c.size) < (0.0, 0.9, 0.44, 0.5)[k]] = 31
    on = [dev(c) for c in chunks]
    pinned.copy_(torch.from_numpy(chunks[0]))
    out = torch.full((256,), -1, dtype=torch.int32, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()

    def live(k):
        st.push(on[k], out)
        return chunks[k]

    def host(k):
        st.push_host(pinned.data_ptr(), n, out.data_ptr())
        return chunks[0]

    def replay(k):
        g.replay()
        return chunks[1]

    with torch.cuda.stream(s):
        for captured, steps in ((1, [host, live]), (6, [host, live, host]), (1, [live] * 6 + [replay, host]),
                                (5, [replay, replay, live, live, replay, host, host, live])):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                for _ in range(captured):
                    st.push(on[1], out)
            for i, step in enumerate(steps):
                data = step(i % 4)
                for _ in range(captured if step is replay else 1):
                    rec = ref.push(data)
                    count += 1
                s.synchronize()
                assert np.array_equal(u32(out), rec.hist), (captured, i)
                state = st.state()
                assert state.status == 0 and state.chunks == count, (captured, i)
            # the same steps without a look between them
            for i, step in enumerate(steps):
                data = step(i % 4)
                for _ in range(captured if step is replay else 1):
                    rec = ref.push(data)
                    count += 1
            s.synchronize()
            state = st.state()
            assert np.array_equal(u32(out), rec.hist) and state.status == 0 and state.chunks == count
            assert np.array_equal(np.array(state.totals, np.uint64), ref.totals)
            assert bytes(state.pattern) == ref.pattern.to_bytes() and state.flag == ref.flag
            assert state.last_kernel == rec.kernel
            # and after a resume, with the graph from before it
            st.set_state(state)
            for step in (replay, host, live):
                data = step(1)
                for _ in range(captured if step is replay else 1):
                    rec = ref.push(data)
                    count += 1
            s.synchronize()
            state = st.state()
            assert np.array_equal(u32(out), rec.hist) and state.status == 0 and state.chunks == count
            assert np.array_equal(np.array(state.totals, np.uint64), ref.totals)
    st.close()


@pytest.mark.parametrize("overlap", [False, True])
def test_captured_push_longer_than_the_rings(overlap):
    """Five launches of 1024 chunks on two CTAs, captured and replayed: in each
    a large chunk is cut between the CTAs, and the fifth launch's uses the ring
    slot of the first's."""
    rng = np.random.default_rng(77)
    big, small, launches = 40 << 20, 100, 5
    x = rng.integers(0, 256, big + launches, dtype=np.uint8)
    x[rng.random(x.size) < 0.3] = 200
    xd = dev(x)
    ptrs, sizes = [], []
    for k in range(launches * 1024):
        launch, j = divmod(k, 1024)
        ptrs.append(xd.data_ptr() + (launch if j == 512 else 13 * k % 1_000_000))
        sizes.append(big if j == 512 else small)
    outs = torch.full((launches, 256), -1, dtype=torch.int32, device="cuda")
    rows = [outs[k // 1024].data_ptr() if k % 1024 == 512 else None for k in range(len(ptrs))]
    st = hl.Stream(mode=hl.MODE_ADAPTIVE, grid=2, overlap=overlap)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            st.push_many(ptrs, sizes, rows)
        want = np.stack([oracle.hist_u32(x[k:k + big]) for k in range(launches)])
        total = want.astype(np.uint64).sum(axis=0)
        for p, n in zip(ptrs, sizes):
            if n == small:
                at = p - xd.data_ptr()
                total += np.bincount(x[at:at + n], minlength=256).astype(np.uint64)
        for r in range(3):
            outs.fill_(-1)
            g.replay()
            s.synchronize()
            assert np.array_equal(u32(outs).reshape(launches, 256), want), r
            state = st.state()
            assert state.status == 0 and state.chunks == (r + 1) * len(ptrs)
            assert np.array_equal(np.array(state.totals, np.uint64), (r + 1) * total)
    st.close()


@pytest.mark.parametrize("sizes", [
    [0, 1, 15, 16, 17, 19, 20, 255, 4079, 4080, 4095, 4096, 4097, 4100, 4111, 4112, 5000] * 4,
    [3000 + 401 * k for k in range(300)] + [2_000_003, 4096 * 256 + 1],
])
def test_regimes_behind_a_copy(sizes):
    """Classification behind the counting launches, right after a copy wrote
    the images and before another reads the regimes, images at every
    alignment: the oracle's regimes and histograms, three times over."""
    rng = np.random.default_rng(len(sizes))
    offs = np.concatenate(([0], np.cumsum([n + 1 + k % 16 for k, n in enumerate(sizes)])))[:-1] + 3
    host = np.zeros((3, int(offs[-1]) + sizes[-1] + 64), np.uint8)
    for r in range(3):
        for k, (o, n) in enumerate(zip(offs, sizes)):
            x = rng.integers(0, 256, n) if (k + r) % 3 == 0 else np.clip(rng.normal(128, 8 if k % 2 else 25, n), 0, 255)
            if (k + r) % 3 == 1:
                x[rng.random(n) < rng.choice([0.4, 0.45, 0.95])] = 77
            host[r, o:o + n] = x
    src, x = dev(host), torch.zeros(host.shape[1], dtype=torch.uint8, device="cuda")
    ptrs = torch.tensor([x.data_ptr() + int(o) for o in offs], dtype=torch.int64).cuda()
    sz = torch.tensor(sizes, dtype=torch.int64).cuda()
    out = torch.empty((3, len(sizes), 256), dtype=torch.int32, device="cuda")
    reg = torch.empty(len(sizes), dtype=torch.uint8, device="cuda")
    regs = torch.empty((3, len(sizes)), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    s = torch.cuda.current_stream().cuda_stream
    for r in range(3):
        x.copy_(src[r])
        assert hl.lib().hist_batch_regimes(ptrs.data_ptr(), sz.data_ptr(), len(sizes), out[r].data_ptr(), reg.data_ptr(),
                                           None, s) == 0
        regs[r].copy_(reg)
    got, greg = u32(out).reshape(3, len(sizes), 256), regs.cpu().numpy()
    for r in range(3):
        for k, (o, n) in enumerate(zip(offs, sizes)):
            im = host[r, o:o + n]
            assert np.array_equal(got[r, k], oracle.hist_u32(im)), (r, k, n)
            assert greg[r, k] == oracle.batch_regime(im), (r, k, n)


@pytest.mark.parametrize("mode,budget", [(hl.MODE_AUTO, 8192), (hl.MODE_PLAIN, 960), (hl.MODE_ADAPTIVE, 2048)])
def test_server_requests_around_the_groups_limit(mode, budget):
    """Requests around the sizes at which a batch's paths change (empty, inside
    a line, the groups' largest, cut between CTAs), at every alignment, three
    rounds of one per stream: outputs and each stream's state equal the
    oracle's."""
    sizes = [0, 1, 127, 143, 4096, 70_001, 262_143, 262_144, 262_145, 600_007, 3_000_001, 9_000_000] * 6
    rng = np.random.default_rng(budget)
    srv = hl.Server(streams=len(sizes), mode=mode, pattern_budget=budget, max_batch=64)
    refs = [oracle.StreamOracle(budget, mode=mode) for _ in sizes]
    x = rng.integers(0, 256, max(sizes) + 300, dtype=np.uint8)
    x[rng.random(x.size) < 0.46] = 9  # near the switch's threshold
    xd = dev(x)
    for rnd in range(3):
        outs = torch.full((len(sizes), 256), -1, dtype=torch.int32, device="cuda")
        offs = rng.integers(0, 300, len(sizes))
        torch.cuda.synchronize()
        for i, n in enumerate(sizes):
            srv.submit_ptr(i, xd.data_ptr() + int(offs[i]), n, outs[i].data_ptr(), i)
        srv.drain(20000)
        got = u32(outs).reshape(len(sizes), 256)
        for i, n in enumerate(sizes):
            rec = refs[i].push(x[offs[i]:offs[i] + n])
            assert np.array_equal(got[i], rec.hist), (rnd, i, n)
            s = srv.stream_state(i)
            assert bytes(s.pattern) == refs[i].pattern.to_bytes() and bytes(s.last_pattern) == rec.pattern.to_bytes()
            assert s.flag == refs[i].flag and s.last_kernel == rec.kernel and s.chunks == rnd + 1
            assert np.array_equal(np.array(s.totals, np.uint64), refs[i].totals)
    srv.close()


@pytest.mark.parametrize("streams,max_batch,max_inflight", [(1, 256, 4), (3, 1, 8), (3, 7, 4), (5, 1024, 8), (40, 64, 2)])
def test_server_long_queues_of_few_streams(streams, max_batch, max_inflight):
    """More queued requests than streams: a stream's next request is launched
    while the last one may still be writing its record.  Some requests write
    where an earlier one of their stream wrote, or read what it wrote: the
    outputs, the completions' order and the states are those of the stream's
    order."""
    rng = np.random.default_rng(streams * 1000 + max_batch)
    x = rng.integers(0, 256, 2_000_000, dtype=np.uint8)
    x[rng.random(x.size) < 0.46] = 9  # near the switch's threshold
    xd = dev(x)
    for mode in (hl.MODE_AUTO, hl.MODE_ADAPTIVE, hl.MODE_PLAIN):
        srv = hl.Server(streams=streams, mode=mode, max_batch=max_batch, max_inflight=max_inflight)
        refs = [oracle.StreamOracle(oracle.BUDGET_MAX, mode=mode) for _ in range(streams)]
        count = 400
        outs = torch.full((count, 256), -1, dtype=torch.int32, device="cuda")
        host = np.full((count, 256), 0xffffffff, np.uint32)
        rows = [[] for _ in range(streams)]  # each stream's output rows
        last = [None] * streams
        torch.cuda.synchronize()
        for i in range(count):
            s = int(rng.integers(0, streams))
            row, n, off = i, int(rng.choice([0, 5, 1000, 30_000, 200_000, 500_000])), int(rng.integers(0, 1_000_000))
            ptr, data = xd.data_ptr() + off, x[off:off + n]
            k = int(rng.integers(0, 12))
            if k == 0 and rows[s]:  # over an earlier output
                row = rows[s][-1]
            elif k == 1 and rows[s]:  # from an earlier output, from inside it to its end
                at = rows[s][-int(rng.integers(1, min(4, len(rows[s])) + 1))]
                ptr, n = outs[at].data_ptr() + 100, 924
                data = np.ascontiguousarray(host[at]).view(np.uint8)[100:].copy()
            last[s] = refs[s].push(data)
            host[row] = last[s].hist
            rows[s].append(row)
            srv.submit_ptr(s, ptr, n, outs[row].data_ptr(), i)
        order = [[] for _ in range(streams)]
        got = 0
        t0 = time.monotonic()
        while got < count:
            assert time.monotonic() - t0 < 20
            for c in srv.poll():
                order[c.stream].append(c.tag)
                got += 1
        srv.drain(20000)
        assert all(o == sorted(o) for o in order)
        assert np.array_equal(u32(outs).reshape(count, 256), host)
        for s in range(streams):
            if last[s] is None:
                continue
            st = srv.stream_state(s)
            assert bytes(st.pattern) == refs[s].pattern.to_bytes()
            assert bytes(st.last_pattern) == last[s].pattern.to_bytes()
            assert np.array_equal(np.array(st.last_hist, np.uint32), last[s].hist)
            assert np.array_equal(np.array(st.totals, np.uint64), refs[s].totals)
            assert st.flag == refs[s].flag and st.last_kernel == last[s].kernel and st.chunks == refs[s].chunks
        srv.close()
