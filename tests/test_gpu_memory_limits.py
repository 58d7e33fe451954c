"""Calls at scratch limits: buffers that only make a call faster are done without when
device memory is short, and results stay the same.

The shortage is made on the host: a preloaded library stands in for the runtime's
allocation calls of a child process and answers with an out-of-memory error once
the bytes it has handed out would exceed a budget."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.gpu

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <pthread.h>
#include <stddef.h>
static pthread_mutex_t mu = PTHREAD_MUTEX_INITIALIZER;
static int armed;
static size_t budget, live, peak;
static struct { void *p; size_t n; } held[8192];
static int nheld;
static void *real(const char *name) {
  static void *lib;
  if (!lib) lib = dlopen("libcudart.so.13", RTLD_LAZY);
  return dlsym(lib ? lib : RTLD_NEXT, name);
}
void shim_arm(size_t n) { pthread_mutex_lock(&mu); armed = 1; budget = n; live = peak = 0; nheld = 0; pthread_mutex_unlock(&mu); }
size_t shim_disarm(void) { armed = 0; return peak; }
static int fits(size_t n) { return !armed || (live + n <= budget && nheld < 8192); }
static void took(void *p, size_t n) {
  if (!armed) return;
  held[nheld].p = p;
  held[nheld++].n = n;
  live += n;
  if (live > peak) peak = live;
}
static void gave(void *p) {
  pthread_mutex_lock(&mu);
  if (armed && p)
    for (int i = 0; i < nheld; ++i)
      if (held[i].p == p) {
        live -= held[i].n;
        held[i] = held[--nheld];
        break;
      }
  pthread_mutex_unlock(&mu);
}
int cudaMalloc(void **p, size_t n) {
  int (*f)(void **, size_t) = real("cudaMalloc"), e;
  pthread_mutex_lock(&mu);
  if (!fits(n)) {
    f(p, (size_t)1 << 60);   /* sets the runtime's last error */
    *p = 0;
    e = 2;
  } else if (!(e = f(p, n))) took(*p, n);
  pthread_mutex_unlock(&mu);
  return e;
}
int cudaMallocFromPoolAsync(void **p, size_t n, void *pool, void *st) {
  int (*f)(void **, size_t, void *, void *) = real("cudaMallocFromPoolAsync"), e;
  pthread_mutex_lock(&mu);
  if (!fits(n)) {
    f(p, (size_t)1 << 60, pool, st);
    *p = 0;
    e = 2;
  } else if (!(e = f(p, n, pool, st))) took(*p, n);
  pthread_mutex_unlock(&mu);
  return e;
}
int cudaFree(void *p) { gave(p); return ((int (*)(void *))real("cudaFree"))(p); }
int cudaFreeAsync(void *p, void *st) { gave(p); return ((int (*)(void *, void *))real("cudaFreeAsync"))(p, st); }
int cudaMemGetInfo(size_t *fr, size_t *tot) {
  int e = ((int (*)(size_t *, size_t *))real("cudaMemGetInfo"))(fr, tot);
  if (!e && armed && *fr > budget - live) *fr = budget - live;
  return e;
}
"""
NO_LIMIT = 1 << 50


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    d = tmp_path_factory.mktemp("shim")
    (d / "shim.c").write_text(SHIM)
    so = d / "shim.so"
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-w", "-o", str(so), str(d / "shim.c"), "-ldl", "-lpthread"],
                   check=True)
    from paper_1503_01405_gb300 import build
    build.build()
    return str(so)


@pytest.mark.parametrize("case", ["stack_without_table", "trials_without_words", "segments_one_by_one",
                                  "four_pass_without_table",
                                  "boxcar_without_lists"])
def test_short_of_memory(shim, case):
    r = subprocess.run([sys.executable, os.path.abspath(__file__), case], cwd=ROOT, text=True, capture_output=True,
                       timeout=300, env=dict(os.environ, LD_PRELOAD=shim, SHIM=shim))
    assert r.returncode == 0 and "ok" in r.stdout.split(), r.stdout[-2000:] + r.stderr[-2000:]


class Budget:
    """Allocations of the block may hold n bytes at most; .peak afterwards."""
    lib = None

    def __init__(self, n=NO_LIMIT):
        if Budget.lib is None:
            Budget.lib = ctypes.CDLL(os.environ["SHIM"])
            Budget.lib.shim_disarm.restype = ctypes.c_size_t
        self.n = n

    def __enter__(self):
        Budget.lib.shim_arm(ctypes.c_size_t(self.n))
        return self

    def __exit__(self, *a):
        self.peak = Budget.lib.shim_disarm()


def stack_without_table():
    """pond_fold_stack needs no memory of its own: without the table of key starts the
    cells search, in the same order."""
    import torch

    from paper_1503_01405_gb300 import pond
    n, dt, nbins = 200_003, 1e-3, 64
    c = np.array([0.2, 100.0, 1e-3])         # ten samples a rotation: 6.4 keys a sample
    y = torch.from_numpy(np.random.default_rng(1).normal(10.0, 3.0, n).astype(np.float32)).cuda()
    S_ref, H_ref, q_ref = pond.fold_stack(y, 3, dt, c, 0.0, nbins)
    S = torch.zeros(S_ref.shape, dtype=torch.float64, device="cuda")
    H = torch.zeros(H_ref.shape, dtype=torch.int64, device="cuda")
    rows, q0 = ctypes.c_int64(), ctypes.c_int64()
    torch.cuda.synchronize()
    with Budget(0):
        rc = pond.lib().pond_fold_stack(y.data_ptr(), n, 3, dt, c.ctypes.data, 3, 0.0, nbins, 0, 0, S.data_ptr(),
                                        H.data_ptr(), S.shape[0], ctypes.byref(rows), ctypes.byref(q0), None)
    torch.cuda.synchronize()
    assert rc == pond.POND_OK, pond.lib().pond_last_error()
    assert q0.value == q_ref and np.array_equal(S.cpu().numpy(), S_ref) and np.array_equal(H.cpu().numpy(), H_ref)


def samples(n):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x = torch.randn(n, generator=g, device="cuda").mul_(20.0).clamp_(-127, 127).to(torch.int8)
    torch.cuda.synchronize()
    return x


def engine(x, budget, *args, **kw):
    """Outputs of one stream through an engine made under the budget, and the peak of its allocations."""
    from paper_1503_01405_gb300 import pond
    with Budget(budget) as b:
        with pond.Engine(326.5, 16.0, 32e6, *args, **kw) as e:
            e.push_tensor(x)
            e.flush()
            out = list(e.timeseries())
            if not kw.get("dms"):
                out += e.profile()[:2]
    return out, b.peak


def same(a, b):
    return len(a) == len(b) and all(np.array_equal(p, q) for p, q in zip(a, b))


def trials_without_words():
    """The anchor form over several trials per launch (blocks of three and of two) and the
    per-trial form without the trials' phase words: the same series."""
    from paper_1503_01405_gb300 import pond
    nfft, ndm = 1 << 20, 8
    x = samples(5 * nfft + 1234)
    args = (0.0, nfft, 16, 1, 1.0)
    words = ndm * (nfft // 2) * 4
    for mode in (pond.POND_TRIALS_MULTI_ANCHOR, pond.POND_TRIALS_PER_TRIAL):
        kw = dict(t_dec=32e-6, dms=[0.31 + 0.0137 * d ** 1.3 for d in range(ndm)], trial_mode=mode, trials_per_launch=3)
        ref, peak = engine(x, NO_LIMIT, *args, **kw)
        out, less = engine(x, peak - words // 2, *args, **kw)
        assert less <= peak - words and same(out, ref), mode


def segments_one_by_one():
    """A single-DM plan without room for the buffers of a group of segments: the same outputs
    from one segment per launch."""
    nfft = 1 << 20
    x = samples(19 * nfft + 4321)
    args = (0.4, nfft, 16, 128, 0.0371)
    ref, peak = engine(x, NO_LIMIT, *args)
    slices = 15 * 2 * 2 * (nfft // 2) * 8      # 15 further segments, two slots, two spectra
    out, less = engine(x, peak - slices, *args)
    assert less <= peak - slices and same(out, ref)


def four_pass_without_table():
    """A four-pass plan without room for its per-bin chirp table takes the anchors."""
    from paper_1503_01405_gb300 import pond
    nfft = 1 << 21
    x = samples(3 * nfft + 99)
    args, kw = (0.3, nfft, 1, 128, 0.0371), dict(timing=True)      # one segment per launch
    ref, _ = engine(x, NO_LIMIT, *args, chirp=pond.POND_CHIRP_ANCHORS, **kw)
    _, peak = engine(x, NO_LIMIT, *args, **kw)
    out, less = engine(x, peak - nfft // 2 * 8, *args, **kw)
    assert less <= peak - nfft // 2 * 8 and same(out, ref)


def boxcar_without_lists():
    """The detector never needs more than the 9 bytes per series sample of its dense form and
    its candidate array: where too many points reach the threshold for the lists
    (0.9: not screened at all, 1.0: they overflow), and where the lists of short rows do not fit."""
    import torch

    from paper_1503_01405_gb300 import pond
    cap = 1 << 17
    for ndm, n, thr in ((48, 20_000, 0.9), (48, 20_000, 1.0), (1500, 700, 6.0)):
        g = torch.Generator(device="cuda")
        g.manual_seed(n)
        x = torch.randn((ndm, n), generator=g, device="cuda") * 3 + 10
        x[ndm // 2, n // 2:n // 2 + 8] += 9.0
        torch.cuda.synchronize()
        ref = pond.boxcar(x.data_ptr(), ndm, n, n, thr, cap)
        with Budget(9 * ndm * n + cap * ctypes.sizeof(pond.pond_cand) + ndm * 256 + 4096):
            got = pond.boxcar(x.data_ptr(), ndm, n, n, thr, cap)
        assert ref and got == ref, (ndm, n, thr, len(ref), len(got))


if __name__ == "__main__":
    sys.path.insert(0, ROOT)
    globals()[sys.argv[1]]()
    print("ok")
