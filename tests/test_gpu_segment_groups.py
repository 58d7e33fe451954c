"""Launches over groups of segments: a stream pushed at once (whole groups), one
segment at a time, and in ragged pieces gives the same series and profile bit for
bit, and both match the oracle; the fold's window form is checked where its cases
differ (several bin edges per window, bins shorter than a lane's run, periods
shorter than a window, a phase model that runs forwards or turns round)."""
import numpy as np
import pytest

from oracle import pcd
from paper_1503_01405_gb300 import pond, synth

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / np.linalg.norm(b))


def engine(x, cuts, nfft, nchan, dm, nbins, period, t_dec, phase=None, **kw):
    with pond.Engine(326.5, 16.0, 32e6, dm, nfft, nchan, nbins, period, t_dec=t_dec, phase_model=phase, **kw) as e:
        a = 0
        for c in cuts:
            e.push(x[a:a + c])
            a += c
        e.flush()
        s, h, _ = e.profile()
        T, C, j0 = e.timeseries()
    return s, h, T, C, j0


CASES = [  # log2 nfft, nchan, bins, period, t_dec, segments
    (14, 4, 64, 0.0123, 61.44e-6, 21),    # four passes, more segments than one group holds
    (16, 1, 1024, 0.00311, 4e-6, 9),      # one channel, 48 samples per bin: an edge in most lanes' runs
    (16, 1, 4096, 0.00311, 61.44e-6, 9),  # 12 samples per bin: several edges per run
    (16, 1, 32, 2.9e-5, 61.44e-6, 9),     # a period (464 samples) shorter than a window
    (18, 8, 100, 0.0371, 33e-6, 7),       # three passes; series samples straddle segments
    (20, 16, 256, 0.0371, 300e-6, 5),     # a series sample of 300 channel samples (one warp each)
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"nfft2^{c[0]}_nch{c[1]}_bins{c[2]}_P{c[3]}")
def test_groups_are_exact(case):
    logn, nchan, nbins, period, t_dec, nseg = case
    nfft, dm = 1 << logn, 0.04 if nchan > 1 else 0.001
    p = pcd.make_plan(326.5, 16.0, 32e6, dm, nfft, nchan, nbins, period, t_dec)
    n = nfft + (nseg - 1) * p.S + p.S // 3 + 77
    x = synth.make_stream(synth.StreamSpec(n=n, seed=logn, dm=dm, period=period, snr=40.0, duty=0.05))
    whole = engine(x, [n], nfft, nchan, dm, nbins, period, t_dec)
    single = engine(x, [p.S] * (n // p.S) + [n % p.S], nfft, nchan, dm, nbins, period, t_dec)
    rng, cuts = np.random.default_rng(logn), []
    while sum(cuts) < n:
        cuts.append(int(min(n - sum(cuts), rng.integers(1, 3 * nfft))))
    ragged = engine(x, cuts, nfft, nchan, dm, nbins, period, t_dec)
    timed = engine(x, [n], nfft, nchan, dm, nbins, period, t_dec, timing=True)   # one segment per launch
    for other in (single, ragged, timed):
        assert all(np.array_equal(a, b) for a, b in zip(whole[:4], other[:4])) and whole[4] == other[4]
    r = pcd.run(p, x)
    assert np.array_equal(whole[1], r.prof_hits) and np.array_equal(whole[3], r.ts_counts) and whole[4] == r.ts_first
    assert rel(whole[0], r.prof_sum) <= 1e-5 and rel(whole[2], r.ts) <= 1e-5


MODELS = [  # (t_ref, coefficients)
    (0.01, [0.25, 80.0, -30.0]),                    # spin-down, forwards
    (0.02, [0.4, 0.5, 40.0]),                       # turns round inside the stream
    (-3.0, [0.1, 200.0, 0.5, -0.01, 1e-4]),         # long lever arm
    (0.0, [0.75]),                                  # one bin for ever
]


@pytest.mark.parametrize("model", MODELS, ids=["spin", "turn", "lever", "constant"])
def test_phase_model_windows(model):
    nfft, nchan, nbins, dm = 1 << 16, 2, 128, 0.01
    p = pcd.make_plan(326.5, 16.0, 32e6, dm, nfft, nchan, nbins, 0.01, 61.44e-6, phase=model)
    x = synth.make_stream(synth.StreamSpec(n=12 * nfft + 999, seed=3, dm=dm, period=0.01, snr=40.0, duty=0.05))
    s, h, T, C, j0 = engine(x, [len(x)], nfft, nchan, dm, nbins, 0.01, 61.44e-6, phase=model)
    r = pcd.run(p, x)
    assert np.array_equal(h, r.prof_hits) and rel(s, r.prof_sum) <= 1e-5
