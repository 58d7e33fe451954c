"""Series longer than the device ring from one push: the same as from many short
pushes, sample for sample, whatever the number of FFT lengths in the plan, and also where
one segment's series alone is longer than the ring's usual size."""
import numpy as np
import pytest

from paper_1503_01405_gb300 import pond

pytestmark = pytest.mark.gpu


def noise(n):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    return torch.randint(-60, 61, (n,), generator=g, device="cuda", dtype=torch.int8)


def series(e, x, piece):
    e.reset()
    for a in range(0, len(x), piece):
        e.push_tensor(x[a:a + piece])
    e.flush()
    return e.timeseries()


def test_one_push_longer_than_the_ring():
    x = noise(36_000_003)       # 9M series samples of two channel samples
    with pond.Engine(326.5, 16.0, 32e6, 0.001, 1 << 18, 1, 64, 0.0371, t_dec=125e-9) as e:
        whole, parts = series(e, x, len(x)), series(e, x, 5_000_000)
        assert whole[2] == parts[2] and len(whole[0]) > 1 << 23
        assert np.array_equal(whole[1], parts[1]) and np.array_equal(whole[0], parts[0])
        # the detector searches undrained samples on the device: refused when a push has left only some there
        e.reset()
        e.push_tensor(x)
        with pytest.raises(pond.PondError) as err:
            e.candidates(8.0)
        assert err.value.name == "OVERRUN"


def test_one_push_longer_than_the_ring_at_two_lengths():
    x = noise(100_000_000)      # 0.78M samples per trial
    # 2^24 points do not reach over the last trial's overlap; 2^25 have no three-pass form
    with pond.Engine(326.5, 16.0, 32e6, 0.0, 1 << 24, 64, 1, 1.0, t_dec=4e-6, dms=[0.0, 0.47, 150.0],
                     nfft_choices=(1 << 24, 1 << 25), autotune=True) as e:
        if len(e.tuning()) < 2:
            pytest.skip("the tuner chose one length")
        whole, parts = series(e, x, len(x)), series(e, x, 20_000_000)
    assert whole[2] == parts[2] and whole[0].shape[1] > 1 << 19
    assert np.array_equal(whole[1], parts[1]) and np.array_equal(whole[0], parts[0])


def test_segment_longer_than_the_usual_ring():
    """2^23 channel samples in a segment; 63 ns samples pair up to 126 ns ones."""
    x = noise((1 << 24) + 4001)
    out = []
    for t_dec in (63e-9, 126e-9):
        with pond.Engine(326.5, 16.0, 32e6, 0.001, 1 << 24, 1, 64, 0.0371, t_dec=t_dec) as e:
            out.append(series(e, x, len(x)))
    (T1, C1, j1), (T2, C2, j2) = out
    lo, hi = 2 * (j2 + 1) - j1, 2 * (j2 + len(T2) - 1) - j1      # whole 126 ns samples inside both
    assert len(T1) > 1 << 22 and len(T2) > 3
    assert np.array_equal(C1[lo:hi].reshape(-1, 2).sum(1), C2[1:-1])
    pairs = T1[lo:hi].reshape(-1, 2).sum(1)
    # at most two FP32 additions on either side, each to 2^-24
    assert np.linalg.norm(pairs - T2[1:-1]) <= 2.4e-7 * np.linalg.norm(T2[1:-1])
