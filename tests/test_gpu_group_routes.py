"""Routes of launches over several segments that plans without voltages take: N / S
pairs and single-channel streams cut so that segments lose their alignment, pushes
of several pieces from page-locked memory; and the training kernels on patches that
are not aligned for wide loads."""
import numpy as np
import pytest

from oracle import pcd
from paper_1503_01405_gb300 import pond, synth
from test_gpu_parity import CONFIGS, THREE_PASS, _stream, check, run_engine

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / np.linalg.norm(b))


def outputs(p, pushes, **kw):
    with pond.Engine(p.f0, p.bw, p.fs, p.dm, p.nfft, p.nchan, p.nbins, p.period, **kw) as e:
        for q in pushes:
            e.push_tensor(q) if hasattr(q, "is_cuda") else e.push(q)
        e.flush()
        s, h, _ = e.profile()
        return (s, h) + tuple(e.timeseries())


def same(a, b):
    return all(np.array_equal(u, v) for u, v in zip(a, b))


def cut(x, sizes):
    a = 0
    while a < len(x):
        n = sizes.pop(0) if sizes else len(x) - a
        yield x[a:a + n]
        a += n


@pytest.mark.parametrize("cfg", CONFIGS + THREE_PASS, ids=lambda c: f"N{c[0]}_c{c[1]}_dm{c[2]}_bw{c[3]}")
def test_grouped_plans_match_oracle(cfg):
    """The parity suite's plans without voltages, which launch groups of segments."""
    nfft, nchan, dm, bw, nbins, period = cfg
    p = pcd.make_plan(326.5, bw, 32e6, dm, nfft, nchan, nbins, period)
    x = _stream(p, seed=nfft + nchan, extra=17)
    check(run_engine(x, p, want_voltages=False, device_push=True), pcd.run(p, x), voltages=False)


@pytest.mark.parametrize("ch", [1, 2], ids=["one_channel", "pairs"])
@pytest.mark.parametrize("cfg", [(1 << 16, 16, 0.3, 16.0, 128, 0.033), (1 << 18, 8, 1.0, -16.0, 128, 0.03),
                                 (1 << 20, 16, 1.0, 16.0, 128, 0.03)],
                         ids=["four_pass", "three_pass", "three_pass_direct"])
def test_groups_of_unaligned_segments(cfg, ch):
    """Whole groups from one push (aligned, and at an address that no wide load allows) and from
    cuts at odd samples equal one segment per launch bit for bit, and the oracle."""
    import torch
    nfft, nchan, dm, bw, nbins, period = cfg
    p = pcd.make_plan(326.5, bw, 32e6, dm, nfft, nchan, nbins, period)
    spec = dict(n=nfft + 6 * p.S + 4321, dm=dm, period=period, snr=60.0, duty=0.05, bw=bw)
    halves = [synth.make_stream(synth.StreamSpec(seed=60 + i, **spec)) for i in range(ch)]
    x = np.stack(halves, 1).reshape(-1)
    kw = dict(input_channels=ch)
    d = torch.zeros(len(x) + 16, dtype=torch.int8, device="cuda")
    at = {}
    for ofs in (0, ch):                       # ch bytes on: neither 8- nor 2 ch-byte aligned
        d[ofs:ofs + len(x)] = torch.from_numpy(x).cuda()
        at[ofs] = outputs(p, [d[ofs:ofs + len(x)]], **kw)
    whole = at[0]
    d[:len(x)] = torch.from_numpy(x).cuda()
    odd = [ch * (nfft // 3 + 1), ch * (2 * nfft + 7), ch * 1]
    others = [at[ch], outputs(p, cut(d[:len(x)], list(odd)), **kw), outputs(p, cut(x, list(odd)), **kw),
              outputs(p, [d[:len(x)]], timing=True, **kw)]
    assert all(same(o, whole) for o in others)
    r = pcd.run(p, halves[0] if ch == 1 else pcd.adding_in_phase(x))
    assert np.array_equal(whole[1], r.prof_hits) and np.array_equal(whole[3], r.ts_counts) and whole[4] == r.ts_first
    assert rel(whole[0], r.prof_sum) <= 1e-5 and rel(whole[2], r.ts) <= 1e-5


@pytest.mark.parametrize("ch", [1, 2], ids=["one_channel", "pairs"])
def test_pinned_push_in_several_pieces(ch):
    """130 MiB and a few bytes from page-locked memory reach the device in several pieces, the
    first and the last short: bit for bit the outputs of one push from the device."""
    import torch
    p = pcd.make_plan(326.5, 16.0, 32e6, 1.0, 1 << 20, 16, 128, 0.03)
    n = (130 << 20) + ch * 5
    g = torch.Generator(device="cuda")
    g.manual_seed(ch)
    d = torch.randint(-60, 61, (n,), generator=g, device="cuda", dtype=torch.int8)
    h = torch.empty(n, dtype=torch.int8, pin_memory=True)
    h.copy_(d)
    want = outputs(p, [d], input_channels=ch)
    assert same(outputs(p, [h.numpy()], input_channels=ch), want)
    odd = list(cut(h.numpy(), [ch * 777_777]))      # the pieces of the second push start off every boundary
    assert same(outputs(p, odd, input_channels=ch), want)


@pytest.mark.parametrize("batch", [1, 5])
def test_training_on_unaligned_patches(batch):
    """The loss and gradient of patches two bytes off an eight-byte boundary are those of an
    aligned copy bit for bit."""
    import torch
    net = pond.Classifier(np.random.default_rng(2).normal(0, 0.1, pond.CNN_NPARAM).astype(np.float32), max_batch=batch)
    flat = torch.randn(batch * 32 * 256 + 1, device="cuda").to(torch.bfloat16)
    x = flat[1:].view(batch, 32, 256)
    assert x.data_ptr() % 8 == 2
    y = torch.arange(batch, device="cuda", dtype=torch.int32) % 4
    loss, grad = net.gradient(x, y)
    loss2, grad2 = net.gradient(x.clone(), y)
    net.close()
    assert loss == loss2 and np.array_equal(grad, grad2)


def test_pushes_of_a_running_stream_are_not_cut():
    """A 100 MiB push behind another one reaches the device in one piece: one launch, the
    copy, more than the same pushes from the device."""
    import torch
    p = pcd.make_plan(326.5, 16.0, 32e6, 26.8, 1 << 24, 64, 128, 0.03)
    sizes = [20 << 20, 100 << 20]
    h = torch.empty(max(sizes), dtype=torch.int8, pin_memory=True).zero_()
    d = h.cuda()
    launches = []
    for src in (d, h.numpy()):
        with pond.Engine(p.f0, p.bw, p.fs, p.dm, p.nfft, p.nchan, p.nbins, p.period) as e:
            for n in sizes:
                e.push_tensor(src[:n]) if src is d else e.push(src[:n])
            e.sync()
            launches.append(e.stats()["kernel_launches"])
    assert launches[1] == launches[0] + len(sizes)
