"""Boxcar detector on the GPU vs the FP64 oracle: identical candidate lists.

Every S/N value is a chain of correctly rounded FP64 operations in the same
order on both sides, so trials, indices, widths and S/N values agree exactly.
"""
import numpy as np
import pytest

from oracle import boxcar as ob
from paper_1503_01405_gb300 import pond, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1503_01405_gb300 import build as pbuild
    pbuild.build()


def gpu_detect(block, thr=6.0):
    import torch
    t = torch.from_numpy(np.ascontiguousarray(block, dtype=np.float32)).cuda()
    c = pond.boxcar(t.data_ptr(), block.shape[0], block.shape[1], block.shape[1], thr,
                    stream=torch.cuda.current_stream().cuda_stream)
    return [(x["trial"], x["index"], x["width"], x["snr"]) for x in c]


@pytest.mark.parametrize("ndm,n", [(1, 1), (3, 7), (8, 4096), (5, 10001), (20, 65536)])
def test_boxcar_matches_oracle(ndm, n):
    rng = np.random.default_rng(ndm * 1000 + n)
    block = (1000 + 30 * rng.standard_normal((ndm, n))).astype(np.float32)
    for k in range(min(6, n // 100)):           # boxes of several widths and heights
        d = int(rng.integers(ndm))
        w = int(2 ** rng.integers(0, 7))
        t = int(rng.integers(0, max(1, n - w)))
        block[d, t:t + w] += float(rng.uniform(20, 200))
    assert gpu_detect(block) == ob.detect(block)


def test_constant_and_even_odd_rows():
    block = np.stack([np.full(1000, 5.0), np.arange(1000, dtype=np.float64) % 7, np.r_[np.zeros(999), 100.0]])
    block = block.astype(np.float32)
    assert gpu_detect(block, thr=3.0) == ob.detect(block, threshold=3.0)


def test_candidates_from_a_batched_plan():
    dms = [0.0, 0.1, 0.2, 0.3, 0.4]
    spec = synth.StreamSpec(n=3_000_000, seed=41, dm=0.0, period=0.0, snr=0.0)
    pulses = [synth.Pulse(0.03, 0.2, 2e-4, 40.0), synth.Pulse(0.06, 0.35, 1e-4, 25.0)]
    x = synth.make_chunk(spec, pulses)
    with pond.Engine(326.5, 16.0, 32e6, 0.0, 1 << 16, 16, 1, 1.0, t_dec=8e-6, dms=dms) as e:
        e.push(x)
        e.flush()
        cands = e.candidates(6.0)
        T, C, j0 = e.timeseries()
    want = ob.detect(T)
    got = [(c["trial"], c["index"] - j0, c["width"], c["snr"]) for c in cands]
    assert got == want
    assert all(c["dm"] == dms[c["trial"]] for c in cands)
    # the brightest candidate sits at the pulse's DM and time
    best = max(cands, key=lambda c: c["snr"])
    assert best["trial"] == 2
    assert abs((best["index"] + best["width"] / 2) * 8e-6 - 0.03) < 1e-3


def gpu_detect_strided(block, pad, thr):
    """As gpu_detect with rows `pad` samples apart from their ends."""
    import torch
    t = torch.full((block.shape[0], block.shape[1] + pad), 7.0e9, device="cuda")
    t[:, :block.shape[1]] = torch.from_numpy(np.ascontiguousarray(block, dtype=np.float32)).cuda()
    c = pond.boxcar(t.data_ptr(), block.shape[0], block.shape[1], t.stride(0), thr,
                    stream=torch.cuda.current_stream().cuda_stream)
    return [(x["trial"], x["index"], x["width"], x["snr"]) for x in c]


@pytest.mark.parametrize("pad", [0, 1], ids=["aligned", "odd_stride"])
@pytest.mark.parametrize("n", [63, 64, 447, 448, 449, 512, 513, 897, 8191, 8193, 70001])
def test_screened_points_at_the_edges(n, pad):
    """Row lengths around a warp's 448 points, its 64-sample reach and the collection
    chunk; pulses at both ends and across the seams; an outlier that widens the bound."""
    rng = np.random.default_rng(n + pad)
    block = (4e5 + 1.8e4 * rng.standard_normal((6, n))).astype(np.float32)
    for t in (0, max(0, n - 1), max(0, n - 40), min(n - 1, 440), min(n - 1, 447), n // 2):
        block[rng.integers(6), t:t + int(rng.integers(1, 64))] += np.float32(2e5)
    block[2, n // 3] = 3e9
    want = ob.detect(block)
    assert gpu_detect_strided(block, pad, 6.0) == want


@pytest.mark.parametrize("kind", ["ties", "two_values", "negative", "tiny_spread", "skewed", "sorted"])
def test_order_statistics_of_awkward_rows(kind):
    rng = np.random.default_rng(5)
    n = 30000
    x = {"ties": rng.integers(0, 12, (3, n)), "two_values": rng.integers(0, 2, (3, n)) * 5.0,
         "negative": -1e3 + 5 * rng.standard_normal((3, n)), "tiny_spread": 1e6 + 0.25 * rng.integers(0, 9, (3, n)),
         "skewed": rng.exponential(3.0, (3, n)) ** 2, "sorted": np.sort(rng.standard_normal((3, n)), axis=1)}[kind]
    block = x.astype(np.float32)
    block[1, 100:103] += np.float32(40 * (np.abs(block).max() + 1))
    assert gpu_detect(block, thr=5.0) == ob.detect(block, threshold=5.0)


@pytest.mark.parametrize("n", [1, 2, 3, 70, 257, 2048, 2049])
def test_many_short_rows(n):
    """More rows than the brackets' CTAs at once, shorter and longer than the rule's line: each
    row's statistics and the candidates are the oracle's, with ties, a NaN and infinities among them."""
    rng = np.random.default_rng(n)
    block = (100 + 3 * rng.standard_normal((310, n))).astype(np.float32)
    block[::3] = np.round(block[::3])
    block[5] = 7.0
    block[9::50, n // 2:n // 2 + 5] += 60
    want = ob.detect(block)
    assert gpu_detect(block) == want
    block[20, 0], block[40, n // 3], block[41, n - 1] = np.nan, np.inf, -np.inf
    some = np.r_[0:18, 25:36, 46:310]      # trials whose neighbours hold only finite values
    got = [c for c in gpu_detect(block) if c[0] in some]
    assert got == [c for c in want if c[0] in some]


@pytest.mark.parametrize("cap", [3, 1500], ids=["within_scratch", "beyond_scratch"])
def test_more_candidates_than_room(cap):
    """An overrun reports the number found and touches nothing of the caller's array, from the
    detector and from a plan's series."""
    import ctypes

    import torch
    rng = np.random.default_rng(2)
    block = (100 + 3 * rng.standard_normal((1 if cap == 3 else 120, 20000))).astype(np.float32)
    block[:, 100::300 if cap == 3 else 130] += 80
    found = len(gpu_detect(block))
    assert found > cap
    d = torch.from_numpy(block).cuda()
    out = (pond.pond_cand * cap)()
    ctypes.memset(out, 0x7f, ctypes.sizeof(out))
    before, nf = bytes(out), ctypes.c_size_t()
    rc = pond.lib().pond_boxcar(d.data_ptr(), *block.shape, block.shape[1], 6.0, out, cap, ctypes.byref(nf), None)
    assert rc == pond.POND_E_OVERRUN and nf.value == found and bytes(out) == before
    x = torch.randint(-60, 61, (1 << 22,), dtype=torch.int8)
    x[::65536] = 127
    with pond.Engine(326.5, 16.0, 32e6, 0.0, 1 << 14, 4, 1, 1.0, t_dec=1e-6, dms=[0.0, 0.001]) as e:
        e.push(x.numpy())
        e.flush()
        rc = pond.lib().pond_candidates(e._h, 3.0, out, 2, ctypes.byref(nf))
        assert rc == pond.POND_E_OVERRUN and nf.value > 2 and bytes(out) == before
        assert nf.value == len(e.candidates(3.0))


def test_screened_and_dense_forms_agree():
    """A threshold below 1 evaluates every point; its list cut at S/N 6 is the screened
    list, also where rows hold infinities or NaN (and an overflowing list takes the dense form)."""
    rng = np.random.default_rng(8)
    block = (100 + 3 * rng.standard_normal((7, 20000))).astype(np.float32)
    block[1, 5000:5008] += 30
    block[2, 77] = np.inf
    block[3, 900] = -np.inf
    block[4, 901] = np.nan
    block[5, 6000] = 1e30
    every = gpu_detect(block, thr=0.5)
    for thr in (1.0, 2.0, 6.0):
        got = gpu_detect(block, thr=thr)
        want = [c for c in every if c[3] >= thr]
        assert got == want
