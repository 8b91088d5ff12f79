"""Templates that share launches give what each gives alone.

A plan of up to 2^21 bins hands several templates of one sky position to one
launch of each transform pass; fstat_set_streams(1) makes it one per launch.
The arithmetic of a template is the same, so 2F, the band maxima and the
crossings have to be equal bit for bit, in every count of templates (one, fewer
than a launch holds, a launch and a rest), with sky positions interleaved.
"""

import numpy as np
import pytest

import paper_2201_00451_gb300 as pkg
from workloads import small_target

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2201_00451_gb300 import build as fbuild

    fbuild.build()
    pkg.load()


def bank(n, n_skies, span):
    tm = np.zeros(n, dtype=pkg.TEMPLATE_DTYPE)
    tm["alpha"] = np.array((0.4, 2.9, 5.0))[np.arange(n) % n_skies]
    tm["delta"] = np.array((0.2, -0.7, 1.1))[np.arange(n) % n_skies]
    tm["f1dot"] = np.linspace(-1.0, 1.0, n) * 40.0 / span ** 2
    return tm


@pytest.mark.parametrize("log2_n", [10, 13, 16, 17, 19, 21, 22])
@pytest.mark.parametrize("n_tmpl,n_skies", [(1, 1), (2, 1), (5, 1), (7, 3), (37, 1), (70, 2)])
def test_shared_launches_equal_single_ones(log2_n, n_tmpl, n_skies):
    if log2_n > 19 and n_tmpl > 37:
        pytest.skip("covered by the smaller lengths")
    n = (1 << log2_n) * 5 // 7
    t = small_target(n_samples=n, dt=2.0, n_fft=1 << log2_n, n_det=2, seed=log2_n, dtype="c64")
    rng = np.random.default_rng(n_tmpl)
    tm = bank(n_tmpl, n_skies, n * 2.0)
    got = []
    with pkg.FstatPlan.from_target(t) as plan:
        for X in range(2):
            x = rng.standard_normal((n, 2)).astype(np.float32).view(np.complex64)[:, 0]
            plan.set_data(X, x, t.sigmas[X])
        for streams in (0, 1):
            if streams:
                plan.set_streams(streams)
            two_f = plan.compute(tm)
            pk = plan.compute_peaks(tm, threshold=14.0, n_bands=4, capacity=n_tmpl << (log2_n - 2))
            assert int(pk["count"].item()) <= n_tmpl << (log2_n - 2)
            plan.sync()
            lst = np.sort(pkg.peaks_to_numpy(pk), order=("tmpl", "bin"))
            got.append((two_f.cpu().numpy(), lst, pk["band_max"].cpu().numpy(), pk["band_bin"].cpu().numpy()))
    assert np.all(np.isfinite(got[0][0]))
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("log2_n", [13, 18, 20])
@pytest.mark.parametrize("rows", [1, 2, 3, 4, 8, 12])
def test_ring_of_rows_keeps_the_last(log2_n, rows):
    import torch

    n = (1 << log2_n) * 5 // 7
    t = small_target(n_samples=n, dt=2.0, n_fft=1 << log2_n, n_det=2, seed=1, dtype="c64")
    rng = np.random.default_rng(rows)
    tm = bank(24, 1, n * 2.0)
    with pkg.FstatPlan.from_target(t) as plan, pkg.FstatBatch() as batch:
        for X in range(2):
            x = rng.standard_normal((n, 2)).astype(np.float32).view(np.complex64)[:, 0]
            plan.set_data(X, x, t.sigmas[X])
        want = plan.compute(tm)
        if rows in (1, 3):  # not shared among launches: in order over one stream
            plan.set_streams(1)
        out = torch.zeros((rows, t.n_fft), dtype=torch.float32, device="cuda")
        batch.add(plan, tm, out, out_rows=rows)
        batch.instantiate()
        batch.launch()
        torch.cuda.synchronize()
        for i in range(24 - rows, 24):
            assert torch.equal(out[i % rows], want[i])


@pytest.mark.parametrize("log2_n", [13, 18, 20])
@pytest.mark.parametrize("rows", [1, 3])
def test_ring_of_rows_that_the_streams_do_not_divide(log2_n, rows):
    # the default plan's own choice for these rings: one template per launch, a row
    # with one stream
    import torch

    n = (1 << log2_n) * 5 // 7
    t = small_target(n_samples=n, dt=2.0, n_fft=1 << log2_n, n_det=2, seed=1, dtype="c64")
    rng = np.random.default_rng(rows)
    tm = bank(24, 1, n * 2.0)
    with pkg.FstatPlan.from_target(t) as plan, pkg.FstatBatch() as batch:
        for X in range(2):
            x = rng.standard_normal((n, 2)).astype(np.float32).view(np.complex64)[:, 0]
            plan.set_data(X, x, t.sigmas[X])
        out = torch.zeros((rows, t.n_fft), dtype=torch.float32, device="cuda")
        batch.add(plan, tm, out, out_rows=rows)
        batch.instantiate()
        batch.launch()
        torch.cuda.synchronize()
        want = plan.compute(tm)
        for i in range(24 - rows, 24):
            assert torch.equal(out[i % rows], want[i])


def test_memory_follows_the_bank():
    # 2^18 bins: the series' buffers (50 000 samples: 3 MB with padding), tables and
    # four 4 MB intermediates, 24 MB in all; the 64 MB block only with a larger bank,
    # in place of the four, and results as before
    import torch

    n, n_fft = 50_000, 1 << 18
    t = small_target(n_samples=n, dt=2.0, n_fft=n_fft, n_det=2, seed=7, dtype="c64")
    rng = np.random.default_rng(7)
    x = rng.standard_normal((n, 2)).astype(np.float32).view(np.complex64)[:, 0]
    tm = bank(20, 1, n * 2.0)
    out = torch.zeros((20, n_fft), dtype=torch.float32, device="cuda")

    def held():
        torch.cuda.synchronize()
        return free0 - torch.cuda.mem_get_info()[0]

    def make():
        plan = pkg.FstatPlan.from_target(t)
        for X in range(2):
            plan.set_data(X, x, t.sigmas[X])
        plan.compute(tm[:4], out=out[:4])
        return plan

    make().close()  # (modules are loaded)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    with make() as plan:
        assert held() <= 24 << 20
        few = out[:4].clone()
        plan.compute(tm, out=out)
        assert (64 << 20) < held() <= (24 - 16 + 64) << 20
        assert torch.equal(out[:4], few)
        plan.sync()


def test_default_stream_count_shares_launches_again():
    t = small_target(n_samples=20_000, dt=2.0, n_fft=1 << 15, n_det=2, seed=8, dtype="c64")
    rng = np.random.default_rng(8)
    x = rng.standard_normal((20_000, 2)).astype(np.float32).view(np.complex64)[:, 0]
    tm = bank(16, 1, 40_000.0)
    launches = []
    with pkg.FstatPlan.from_target(t) as plan:
        for X in range(2):
            plan.set_data(X, x, t.sigmas[X])
        plan.compute(tm)  # (the per-sky work)
        for streams in (0, 1, 4):
            if streams:
                plan.set_streams(streams)
            before = plan.launches
            plan.compute(tm)
            launches.append(plan.launches - before)
        plan.sync()
    assert launches[0] < launches[1] and launches[2] == launches[0]


def test_a_captured_batch_keeps_its_intermediates():
    # a batch of two templates holds the plan's first intermediates; a later call
    # whose bank takes the larger block leaves them in place
    import torch

    n = 50_000
    t = small_target(n_samples=n, dt=2.0, n_fft=1 << 18, n_det=2, seed=9, dtype="c64")
    rng = np.random.default_rng(9)
    tm = bank(20, 1, n * 2.0)
    with pkg.FstatPlan.from_target(t) as plan, pkg.FstatBatch() as batch:
        for X in range(2):
            x = rng.standard_normal((n, 2)).astype(np.float32).view(np.complex64)[:, 0]
            plan.set_data(X, x, t.sigmas[X])
        out = torch.zeros((2, t.n_fft), dtype=torch.float32, device="cuda")
        batch.add(plan, tm[:2], out)
        batch.instantiate()
        want = plan.compute(tm)
        out.zero_()
        batch.launch()
        torch.cuda.synchronize()
        assert torch.equal(out, want[:2])
        plan.sync()


@pytest.mark.parametrize("log2_n,n1,n", [(21, 256, 600_001), (21, 256, 1_400_001), (20, 256, 1_000_003), (20, 1024, 700_001),
                                          (16, 32, 40_001)])
def test_staged_columns_and_row_counts_give_the_same_bits(log2_n, n1, n):
    # every distinct kernel of a split: pass A's columns staged where there is room
    # (0; 16 and 18 require it at 8192 and 4096 points) and straight into registers
    # (2), 1 to 8 rows per tile of pass B
    t = small_target(n_samples=n, dt=1.0, n_fft=1 << log2_n, n_det=2, seed=11, dtype="c64")
    rng = np.random.default_rng(11)
    tm = bank(3, 1, float(n))
    need = {13: 16, 12: 18}.get(log2_n - (n1.bit_length() - 1))
    got = []
    with pkg.FstatPlan.from_target(t) as plan:
        for X in range(2):
            x = rng.standard_normal((n, 2)).astype(np.float32).view(np.complex64)[:, 0]
            plan.set_data(X, x, t.sigmas[X])
        plan.set_split(n1)
        for va, cb in [(2, 0), (0, 0)] + ([(need, 0)] if need else []) + ([(2, c) for c in (1, 2, 4, 8)] if n1 >= 512 else []):
            plan.set_cta(0, cb, va, 0)
            got.append(plan.compute(tm).cpu().numpy())
        plan.sync()
    assert np.isfinite(got[0]).all()
    for g in got[1:]:
        assert np.array_equal(g, got[0])
