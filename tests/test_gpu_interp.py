"""GPU parity of the step-(v) interpolator variants and half-widths.

Every kernel (tapered, untapered and periodic Dirichlet) at D = 4, 8, 16,
32 against the oracle: the per-sky resampled, weighted series G_a, G_b
(relative 2e-5 of their largest element, as for the default kernel) and
2F at |d2F| <= 1e-3 2F + 0.02 on a ragged two-detector case.
"""

import numpy as np
import pytest

import paper_2201_00451_gb300 as pkg
from oracle import resamp, synth
from workloads import small_target

pytestmark = pytest.mark.gpu

REL, ABS = 1e-3, 0.02


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2201_00451_gb300 import build as fbuild

    fbuild.build()
    pkg.load()


@pytest.mark.parametrize("interp", [pkg.INTERP_TAPERED, pkg.INTERP_UNTAPERED, pkg.INTERP_PERIODIC])
@pytest.mark.parametrize("dterms", [4, 8, 16, 32])
def test_interpolator_variants_match_oracle(interp, dterms):
    t = small_target(n_samples=5003, dt=2.0, n_fft=1 << 14, n_det=2, n_inj=1, rho2_range=(150.0, 150.0),
                     seed=60 + dterms, f1dots=(-3e-10, 0.0), f2dots=(0.0,), dtype="c64", dterms=dterms,
                     interp=interp)
    x = synth.make_data(t)
    a, d = t.skies[0]
    ref = resamp.sky_prep(t, x, a, d)
    tm = t.templates()
    with pkg.FstatPlan.from_target(t) as plan:
        for X in range(2):
            plan.set_data(X, x[X], t.sigmas[X])
        ga, gb, abcd = plan.export_sky(a, d)
        got = plan.compute(tm)
        plan.sync()
        got = got.cpu().numpy()
    scale = max(np.abs(ref["Ga"]).max(), np.abs(ref["Gb"]).max())
    assert np.abs(ga - ref["Ga"]).max() <= 2e-5 * scale
    assert np.abs(gb - ref["Gb"]).max() <= 2e-5 * scale
    for k, v in zip("ABCD", abcd):
        assert abs(v - ref[k]) <= 1e-10 * abs(ref[k]) + 1e-12
    want = resamp.fstat(t, x, tm)
    excess = np.abs(got - want) - (REL * np.abs(want) + ABS)
    assert excess.max() <= 0, excess.max()


# FP64: the nodes' cubics are exact to ~1e-11 of a, b (32 s), f_h t_m to ~1e-10
# radians; FP32 as above
@pytest.mark.parametrize("precision,tol", [(pkg.MIXED, 2e-5), (pkg.FP64, 1e-9)])
@pytest.mark.parametrize("dtype", ["c64", "c128", "both"])
@pytest.mark.parametrize("n,dt,dterms", [
    (17, 2.0, 2), (700, 4.0, 8), (1025, 1.0, 5), (4096, 0.5, 8), (40000, 1.0, 20), (600001, 0.5, 8)])
def test_series_lengths_and_node_steps_match_oracle(n, dt, dterms, dtype, precision, tol):
    # a node every 16, 32 and 64 samples; tap weights in the short- and the
    # long-series form, unrolled (D = 8) or not; one and several tiles per
    # block; whole steps of nodes and a cut one at the end
    t = small_target(n_samples=n, dt=dt, n_fft=1 << max(10, (n - 1).bit_length()), n_det=2, seed=n, dtype="c128",
                     dterms=dterms)
    rng = np.random.default_rng(n)
    x = [rng.standard_normal(n) + 1j * rng.standard_normal(n) for _ in range(2)]
    for X in range(2):
        if dtype == "c64" or (dtype == "both" and X == 0):
            x[X] = x[X].astype(np.complex64)
    # (delays of both signs at both ends: which samples of the last, cut step count)
    with pkg.FstatPlan.from_target(t, precision) as plan:
        for X in range(2):
            plan.set_data(X, x[X], t.sigmas[X])
        for a, d in (t.skies[0], (0.3, -0.6), (2.0, 0.4), (3.6, 0.2), (5.2, -0.1)):
            ref = resamp.sky_prep(t, [v.astype(np.complex128) for v in x], a, d)
            ga, gb, abcd = plan.export_sky(a, d)
            scale = max(np.abs(ref["Ga"]).max(), np.abs(ref["Gb"]).max())
            assert np.abs(ga - ref["Ga"]).max() <= tol * scale
            assert np.abs(gb - ref["Gb"]).max() <= tol * scale
            for k, v in zip("ABCD", abcd):
                assert abs(v - ref[k]) <= 1e-10 * abs(ref[k]) + 1e-12


@pytest.mark.parametrize("f_het,dt", [(490.0, 0.25), (490.0, 0.5), (490.0, 2.0), (2000.0, 0.5), (2000.0, 2.0)])
def test_heterodyne_phase_of_mixed_plans_at_high_frequencies(f_het, dt):
    # Step (iii) in mixed plans against FP64 plans: what a non-zero f_h adds to the
    # rms difference of G (at f_h = 0 only the taps' and the patterns' rounding is
    # left).  The phase: two FP32 roundings of at most a half turn (6e-8 rad rms
    # together) and node steps in units of 2^-32 cycles (at most 5e-8 rad); the
    # sine and cosine 6e-8, the rotation's products and sum 6e-8 each: 1.3e-7 in
    # all.  It must not grow with f_h or with the node spacing.
    n = 60001
    rng = np.random.default_rng(1)
    x = [(rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64) for _ in range(2)]
    rms = []
    for f in (0.0, f_het):
        t = small_target(n_samples=n, dt=dt, n_fft=1 << 16, n_det=2, seed=5, dtype="c64", f_het=f)
        g = []
        for precision in (pkg.MIXED, pkg.FP64):
            with pkg.FstatPlan.from_target(t, precision) as plan:
                for X in range(2):
                    plan.set_data(X, x[X], t.sigmas[X])
                ga, gb, _ = plan.export_sky(*t.skies[0])
                g.append(np.concatenate([ga, gb]))
        rms.append((np.abs(g[0] - g[1]) ** 2).mean() / (np.abs(g[1]) ** 2).mean())
    assert np.sqrt(max(0.0, rms[1] - rms[0])) <= 2e-7


@pytest.mark.parametrize("precision", [pkg.MIXED, pkg.FP64])
@pytest.mark.parametrize("n,dt", [(100, 0.5), (3001, 2.0), (20001, 0.25), (60001, 0.5), (40001, 1.0), (9001, 4.0), (4001, 8.0)])
def test_antenna_integrals_to_fp64_rounding(n, dt, precision):
    # A, B, C are doubles in both precisions.  Against the oracle's FP64 sums: the
    # patterns' angles round to ~2^-53 times a few turns on both sides (1e-15), the
    # interpolant through six nodes 32 s apart leaves 1e-15 of the largest pattern,
    # and sums of n <= 60001 positive terms round to well below n^(1/2) 2^-53 = 3e-14
    # (C: of products bounded by (A B)^(1/2)); 1e-13 in all.  Four nodes leave 6e-12.
    t = small_target(n_samples=n, dt=dt, n_fft=1 << max(10, (n - 1).bit_length()), n_det=2, seed=n, dtype="c64")
    x = [np.ones(n, np.complex64)] * 2
    with pkg.FstatPlan.from_target(t, precision) as plan:
        for X in range(2):
            plan.set_data(X, x[X], t.sigmas[X])
        for a, d in ((0.3, -0.6), (3.6, 0.2)):
            ref = resamp.sky_prep(t, [v.astype(np.complex128) for v in x], a, d)
            A, B, C, _ = plan.export_sky(a, d)[2]
            assert abs(A - ref["A"]) <= 1e-13 * ref["A"]
            assert abs(B - ref["B"]) <= 1e-13 * ref["B"]
            assert abs(C - ref["C"]) <= 1e-13 * np.sqrt(ref["A"] * ref["B"])
