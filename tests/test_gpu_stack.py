"""GPU parity of the phase-model fold and pulse stacks (PONDER Sec. 3.4 fold with a
predicted period, Sec. 4 single-pulse stack) against the FP64 oracle, through the
C ABI.  Phases, rotations and bins are decided with the same FP64 operations on
both sides and every cell adds its samples in sample order, so sums and hits are
compared bit for bit."""
import numpy as np
import pytest

from oracle import stack as st
from paper_1503_01405_gb300 import pond

pytestmark = pytest.mark.gpu

MODELS = [  # (t_ref, coefficients), dt, g0, nbins
    (st.spin_model(0.7145, 4e-6, 0.0123, 0.3), 61.44e-6, 12345, 256),
    ((2.5, np.array([0.3, 7.0, -0.02, 1e-4])), 1e-4, 0, 64),
    (st.spin_model(0.0331, 0.0, 0.0, 0.0), 4e-6, 777, 1024),
]


@pytest.mark.parametrize("model", MODELS, ids=["spin_down", "cubic", "crab_like"])
@pytest.mark.parametrize("mode,n_sub", [(st.ROTATION, 0), (st.SUBINT, 9973), (st.SUBINT, 1 << 22)],
                         ids=["rotation", "subint", "one_subint"])
def test_stack_matches_oracle_bit_for_bit(model, mode, n_sub):
    import torch
    (t_ref, c), dt, g0, nbins = model
    y = np.random.default_rng(7).normal(10.0, 3.0, 300_001).astype(np.float32)
    S_ref, H_ref, q0_ref = st.stack(y, g0, dt, c, t_ref, nbins, mode, n_sub)
    S, H, q0 = pond.fold_stack(torch.from_numpy(y).cuda(), g0, dt, c, t_ref, nbins, mode, n_sub)
    assert q0 == q0_ref and S.shape == S_ref.shape
    assert np.array_equal(H, H_ref)
    assert np.array_equal(S, S_ref)


def test_stack_errors_and_empty_series():
    import torch
    y = torch.ones(1000, dtype=torch.float32, device="cuda")
    with pytest.raises(pond.PondError) as ei:           # phase running backwards
        pond.fold_stack(y, 0, 1e-3, [0.0, 5.0, -10.0], 0.0, 16)
    assert ei.value.name == "ARG"
    S, H, _ = pond.fold_stack(y[:0], 0, 1e-3, [0.0, 5.0], 0.0, 16)
    assert S.shape == (0, 16) and H.shape == (0, 16)
    import ctypes
    rows, q0 = ctypes.c_int64(), ctypes.c_int64()
    c = np.array([0.0, 5.0])
    rc = pond.lib().pond_fold_stack(y.data_ptr(), 1000, 0, 1e-3, c.ctypes.data, 2, 0.0, 16, 0, 0, None, None, 2,
                                    ctypes.byref(rows), ctypes.byref(q0), None)
    assert rc == pond.POND_E_OVERRUN and rows.value == 5


@pytest.mark.parametrize("n", [1, 2, 31, 33, 257, 5000])
@pytest.mark.parametrize("period_samples", [0.37, 3.0, 700.3], ids=["undersampled", "coarse", "fine"])
@pytest.mark.parametrize("mode,n_sub", [(st.ROTATION, 0), (st.SUBINT, 1), (st.SUBINT, 100)])
def test_stack_key_tables_and_searches(n, period_samples, mode, n_sub):
    """Short series and key counts from far below to far above the samples' (the
    table of starts and the search), bit for bit."""
    import torch
    dt, nbins = 1e-3, 4096 if period_samples < 1 else 37
    c = np.array([0.2, 1.0 / (period_samples * dt), 1e-3])
    y = np.random.default_rng(n).normal(10.0, 3.0, n).astype(np.float32)
    S_ref, H_ref, q0_ref = st.stack(y, 5, dt, c, 0.1, nbins, mode, n_sub)
    S, H, q0 = pond.fold_stack(torch.from_numpy(y).cuda(), 5, dt, c, 0.1, nbins, mode, n_sub)
    assert q0 == q0_ref and np.array_equal(H, H_ref) and np.array_equal(S, S_ref)


@pytest.mark.parametrize("n", [16383, 32769, 65535, 131073, 262145, 524287, 600_001])
@pytest.mark.parametrize("period_samples,nbins", [(30.0, 64), (11629.3, 1024)], ids=["keys_per_sample", "samples_per_key"])
def test_stack_run_lengths(n, period_samples, nbins):
    """Series lengths around each run length's line, bit for bit."""
    import torch
    dt = 1e-3
    c = np.array([0.2, 1.0 / (period_samples * dt), 1e-4])
    y = np.random.default_rng(n).normal(10.0, 3.0, n).astype(np.float32)
    S_ref, H_ref, q0_ref = st.stack(y, 5, dt, c, 0.1, nbins, st.SUBINT, 50_000)
    S, H, q0 = pond.fold_stack(torch.from_numpy(y).cuda(), 5, dt, c, 0.1, nbins, st.SUBINT, 50_000)
    assert q0 == q0_ref and np.array_equal(H, H_ref) and np.array_equal(S, S_ref)


@pytest.mark.parametrize("nbins", [64, 4096], ids=["table", "search"])
def test_overlapping_calls_keep_their_own_verdict(nbins):
    """Calls on two streams, one with a model that runs forwards and one whose model
    turns round: each gets its own answer, the forward one the oracle's bit for bit."""
    import threading

    import torch
    n, dt, rounds = 60_001, 1e-3, 100
    y = np.random.default_rng(3).normal(10.0, 3.0, n).astype(np.float32)
    per = 40.0 if nbins == 64 else 0.4      # samples per rotation: under and over eight keys per sample
    good = np.array([0.2, 1.0 / (per * dt), 1e-3])
    turns = np.array([0.2, 1.0 / (per * dt), -1.0 / (per * dt) / (n * dt)])    # the derivative is zero half-way
    ref = st.stack(y, 5, dt, good, 0.0, nbins, st.SUBINT, 997)
    d = torch.from_numpy(y).cuda()
    torch.cuda.synchronize()
    bad = []

    def forwards():
        s = torch.cuda.Stream()
        for _ in range(rounds):
            try:
                S, H, q0 = pond.fold_stack(d, 5, dt, good, 0.0, nbins, st.SUBINT, 997, stream=s)
            except pond.PondError as e:
                bad.append(f"refused: {e}")
                return
            if q0 != ref[2] or not np.array_equal(H, ref[1]) or not np.array_equal(S, ref[0]):
                bad.append("wrong stack")
                return

    def turned():
        s = torch.cuda.Stream()
        for _ in range(rounds):
            try:
                pond.fold_stack(d, 5, dt, turns, 0.0, nbins, st.SUBINT, 997, stream=s)
            except pond.PondError as e:
                if e.name != "ARG":
                    bad.append(str(e))
                    return
            else:
                bad.append("a model that turns round was accepted")
                return

    threads = [threading.Thread(target=f) for f in (forwards, turned, forwards, turned)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
