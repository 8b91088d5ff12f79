"""GPU semi-coherent sum (fstat_semicoherent) against the oracle.

Per segment the mixed-precision path meets |d2F| <= 1e-3 2F + 0.02, so the
sum over S segments is held to 1e-3 2F_sum + 0.02 S.  Cases: three segments
with an injection whose segment frequencies fall on bins (the sliding must
line the peaks up), four unequal segments over two sky positions, one
segment against fstat_compute (bitwise), and argument checks.
"""

import numpy as np
import pytest
import torch

import paper_2201_00451_gb300 as pkg
from oracle import semicoh, synth
from workloads import segment_slices, small_target, split_segments
from workloads.gen import template_grid

pytestmark = pytest.mark.gpu

REL, ABS = 1e-3, 0.02


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2201_00451_gb300 import build as fbuild

    fbuild.build()
    pkg.load()


def _plans(t, n_seg, x, precision=pkg.MIXED):
    segs = split_segments(t, n_seg)
    data = [[xx[a:a + n] for xx in x] for a, n in segment_slices(t, n_seg)]
    plans = []
    for s, d in zip(segs, data):
        p = pkg.FstatPlan.from_target(s, precision)
        for X in range(len(t.detectors)):
            p.set_data(X, d[X], t.sigmas[X])
        plans.append(p)
    return segs, data, plans


def _check(got, want, n_seg):
    excess = np.abs(got - want) - (REL * np.abs(want) + ABS * n_seg)
    assert excess.max() <= 0, excess.max()


def test_three_segments_line_up_an_injection():
    S, n_seg, dt, n_fft = 3, 6000, 1.0, 1 << 14
    df = 1.0 / (n_fft * dt)
    f1 = 3 * df / (n_seg * dt)
    f2 = 2.0 * df / (n_seg * dt) ** 2
    t = small_target(n_samples=S * n_seg, dt=dt, n_fft=n_fft, n_det=2, n_inj=1, rho2_range=(300.0, 300.0),
                     seed=91, f1dots=(f1,), f2dots=(f2,), dtype="c64")
    inj = t.injections[0]
    x = synth.make_data(t)
    segs, data, plans = _plans(t, S, x)
    tm = template_grid(((inj.alpha, inj.delta),), np.array([f1 - 2 * df / (n_seg * dt), f1, 0.0]),
                       np.array([0.0, f2]))
    got = pkg.semicoherent(plans, tm, t.t_reference).cpu().numpy()
    want = semicoh.semicoherent(segs, data, tm, t.t_reference)
    _check(got, want, S)
    k = int(np.where((tm["f1dot"] == f1) & (tm["f2dot"] == f2))[0][0])
    assert int(np.argmax(got[k])) == inj.bin_index
    for p in plans:
        p.close()


def test_unequal_segments_two_skies():
    S = 4
    t = small_target(n_samples=4 * 2500 + 777, dt=2.0, n_fft=1 << 13, n_det=2, n_inj=1, seed=92,
                     f1dots=(-2e-10, 0.0, 1e-10), f2dots=(0.0,), dtype="c64",
                     skies=((0.4, -0.3), (2.1, 0.5)))
    x = synth.make_data(t)
    segs, data, plans = _plans(t, S, x)
    tm = t.templates()[::-1].copy()      # unsorted: the library groups by sky
    got = pkg.semicoherent(plans, tm, t.t_reference).cpu().numpy()
    _check(got, semicoh.semicoherent(segs, data, tm, t.t_reference), S)
    for p in plans:
        p.close()


def test_one_segment_equals_compute():
    t = small_target(n_samples=5003, dt=2.0, n_fft=1 << 14, n_det=2, n_inj=1, seed=93,
                     f1dots=(-3e-10, 0.0), f2dots=(0.0, 1e-16), dtype="c64")
    x = synth.make_data(t)
    segs, data, plans = _plans(t, 1, x)
    tm = t.templates()
    got = pkg.semicoherent(plans, tm, t.t_reference)
    dense = plans[0].compute(tm)
    torch.cuda.synchronize()
    assert torch.equal(got, dense)
    plans[0].close()


def test_fp64_segments():
    S = 2
    t = small_target(n_samples=2 * 3001, dt=2.0, n_fft=1 << 13, n_det=2, n_inj=1, seed=94,
                     f1dots=(-1e-10, 0.0), f2dots=(0.0,), dtype="c128")
    x = synth.make_data(t)
    segs, data, plans = _plans(t, S, x, precision=pkg.FP64)
    tm = t.templates()
    got = pkg.semicoherent(plans, tm, t.t_reference).cpu().numpy()
    want = semicoh.semicoherent(segs, data, tm, t.t_reference)
    # FP64 arithmetic, float32 output sums
    assert np.max(np.abs(got - want) - (1e-6 * np.abs(want) + 1e-6)) <= 0
    for p in plans:
        p.close()


def test_argument_checks():
    t = small_target(n_samples=4000, dt=2.0, n_fft=1 << 13, n_det=1, seed=95, dtype="c64")
    x = synth.make_data(t)
    segs, data, plans = _plans(t, 2, x)
    tm = t.templates()
    with pytest.raises(pkg.FstatError):
        pkg.semicoherent([plans[0], plans[0]], tm, t.t_reference)
    with pytest.raises(pkg.FstatError):
        pkg.semicoherent(plans, tm, float("nan"))
    other = small_target(n_samples=2000, dt=2.0, n_fft=1 << 12, n_det=1, seed=95, dtype="c64")
    po = pkg.FstatPlan.from_target(other)
    po.set_data(0, synth.make_data(other)[0], other.sigmas[0])
    with pytest.raises(pkg.FstatError):
        pkg.semicoherent([plans[0], po], tm, t.t_reference)
    for p in plans + [po]:
        p.close()


def test_segments_with_different_splits_and_rows():
    # all segments use the first plan's intermediates one after the other, each in its
    # own layout: the sum equals the segments' own rows, slid and added in order
    S, n_seg, dt, n_fft = 3, 40_001, 1.0, 1 << 16
    t = small_target(n_samples=S * n_seg, dt=dt, n_fft=n_fft, n_det=2, seed=96, dtype="c64")
    rng = np.random.default_rng(96)
    x = [(rng.standard_normal(S * n_seg) + 1j * rng.standard_normal(S * n_seg)).astype(np.complex64) for _ in range(2)]
    segs, data, plans = _plans(t, S, x)
    df = 1.0 / (n_fft * dt)
    tm = np.zeros(5, dtype=pkg.TEMPLATE_DTYPE)
    tm["alpha"], tm["delta"] = 0.4, -0.3
    tm["f1dot"] = np.array([-3.0, -1.0, 0.0, 1.0, 2.0]) * df / (n_seg * dt)
    for p, n1, cb in zip(plans, (32, 2048, 512), (0, 2, 8)):
        p.set_split(n1)
        p.set_cta(0, cb, 0, 0)
    got = pkg.semicoherent(plans, tm, t.t_reference)
    want = torch.zeros_like(got)
    for s, (seg, p) in enumerate(zip(segs, plans)):
        rows = p.compute(tm)
        for i in range(len(tm)):
            k = semicoh.segment_shift(df, seg.t_reference - t.t_reference, float(tm["f1dot"][i]), 0.0)
            lo, hi = max(0, -k), min(n_fft, n_fft - k)
            want[i, lo:hi] += rows[i, lo + k:hi + k]
    torch.cuda.synchronize()
    assert torch.equal(got, want)
    for p in plans:
        p.close()
