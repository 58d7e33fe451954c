"""GPU parity of the passes with 64 values per thread against the FP64 oracle, at
every column and row length that takes them and at the neighbouring geometry
that does not (a partly filled tile).  Tolerances as for the radix-16 passes:
an FP32 transform of 2^18 .. 2^24 points with FP64-built twiddles stays within
a few 1e-7 relative L2, and the project's bar for voltages is 1e-5."""
import numpy as np
import pytest

from oracle import pcd
from paper_1503_01405_gb300 import pond, synth

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / np.linalg.norm(b))


GEOMETRIES = [  # log2 nfft, sub-channels, column length R2, groups per column set
    (19, 8),    # R2 512, half a tile per column set
    (20, 16),   # R2 512, one group
    (21, 16),   # R2 1024, two groups
    (22, 32),   # R2 1024, four groups
    (23, 32),   # R2 2048, eight groups
    (24, 64),   # R2 2048, sixteen groups
]


@pytest.mark.parametrize("volt", [False, True], ids=["power", "voltages"])
@pytest.mark.parametrize("bw", [16.0, -16.0], ids=["upper", "inverted"])
@pytest.mark.parametrize("geo", GEOMETRIES, ids=lambda g: f"nfft2^{g[0]}_nch{g[1]}")
def test_three_pass_geometries(geo, bw, volt):
    logn, nchan = geo
    if volt and logn == 24:
        pytest.skip("the 2^24 voltages are covered at the full size")
    nfft, dm, period, nbins = 1 << logn, 0.02 * 2 ** (logn - 19), 0.0371, 128
    p = pcd.make_plan(326.5, bw, 32e6, dm, nfft, nchan, nbins, period, 61.44e-6)
    x = synth.make_stream(synth.StreamSpec(n=nfft + p.S + p.S // 3 + 77, seed=logn, dm=dm, period=period, snr=40.0,
                                           duty=0.05, bw=bw))
    with pond.Engine(326.5, bw, 32e6, dm, nfft, nchan, nbins, period, want_voltages=volt) as e:
        e.push(x)
        e.flush()
        s, h, _ = e.profile()
        T, C, j0 = e.timeseries()
        V = e.voltages()[0] if volt else None
    r = pcd.run(p, x, want_voltages=volt)
    assert np.array_equal(h, r.prof_hits) and np.array_equal(C, r.ts_counts) and j0 == r.ts_first
    assert rel(s, r.prof_sum) <= 1e-5 and rel(T, r.ts) <= 1e-5
    if volt:
        assert V.shape == r.voltages.shape and rel(V, r.voltages) <= 1e-5


FOUR_PASS = [  # log2 nfft, sub-channels, inverse split Q1 x Q2 (rows of a tile: 8192 / (Q1 sub-channels))
    (19, 1),    # 512 x 512, sixteen rows
    (21, 1),    # 1024 x 1024, eight rows
    (21, 8),    # 512 x 256 (short columns), two rows of every sub-channel
    (22, 2),    # 1024 x 1024
    (22, 16),   # 512 x 256, one row of every sub-channel
    (23, 2),    # 2048 x 1024
    (24, 1),    # 2048 x 4096
    (23, 8),    # 1024 x 512, the chirp table read in runs of four bins
    (23, 32),   # 256 x 512, runs of one bin: no table
]


@pytest.mark.parametrize("chirp", [pond.POND_CHIRP_AUTO, pond.POND_CHIRP_ANCHORS], ids=["table", "anchors"])
@pytest.mark.parametrize("geo", FOUR_PASS, ids=lambda g: f"nfft2^{g[0]}_nch{g[1]}")
def test_four_pass_geometries(geo, chirp):
    """The four-pass inverse at line lengths of 512 and more, its chirp from the
    per-bin table or the anchors, powers and voltages."""
    logn, nchan = geo
    if chirp == pond.POND_CHIRP_ANCHORS and logn > 22:
        pytest.skip("the anchor form is covered at the smaller lengths")
    nfft, dm, period, nbins = 1 << logn, 0.02 * 2 ** (logn - 19), 0.0371, 128
    p = pcd.make_plan(326.5, -16.0, 32e6, dm, nfft, nchan, nbins, period, 61.44e-6)
    x = synth.make_stream(synth.StreamSpec(n=nfft + p.S + p.S // 3 + 77, seed=logn + nchan, dm=dm, period=period,
                                           snr=40.0, duty=0.05, bw=-16.0))
    out = {}
    for volt in (False, True):
        with pond.Engine(326.5, -16.0, 32e6, dm, nfft, nchan, nbins, period, want_voltages=volt, chirp=chirp,
                         schedule=pond.POND_SCHEDULE_FOUR_PASS) as e:
            e.push(x)
            e.flush()
            out[volt] = e.profile()[:2] + e.timeseries()
            V = e.voltages()[0] if volt else None
    for a, b in zip(out[False], out[True]):
        assert np.array_equal(a, b)
    s, h, T, C, j0 = out[True]
    r = pcd.run(p, x, want_voltages=True)
    assert np.array_equal(h, r.prof_hits) and np.array_equal(C, r.ts_counts) and j0 == r.ts_first
    assert rel(s, r.prof_sum) <= 1e-5 and rel(T, r.ts) <= 1e-5
    assert V.shape == r.voltages.shape and rel(V, r.voltages) <= 1e-5
