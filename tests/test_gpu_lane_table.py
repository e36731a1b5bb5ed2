"""The lane-private counting paths at the sizes where their splits change,
against the oracle, bit-exact."""
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
