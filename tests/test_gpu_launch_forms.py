"""The launch forms that depend on sizes: the one-pass FFT of short signals at each of its lengths and with more signals
than CTAs, the band launches on both sides of the batch where they change; against the fp64 oracle, first and last row."""
import numpy as np
import pytest

import workloads as wl
from helpers import band_rel_errors, library_plan, oracle_layout, small_workload, snr_db, split_bands
from oracle import nsgt_oracle as orc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


def check_rows(w, batch):
    lay, plan = oracle_layout(w), library_plan(w)
    x = torch.randn(batch, w.valid_len, generator=torch.Generator().manual_seed(w.N + batch)).cuda()
    c = plan.analyse(x, valid_len=w.valid_len)
    y = plan.synthesise_adjoint(x, valid_len=w.valid_len)
    xr = plan.synthesise(y, valid_len=w.valid_len)
    rows = sorted({0, batch - 1})
    xs = orc.pad_signal(x[rows].cpu().numpy(), w.N)
    assert band_rel_errors(lay, c[rows].cpu().numpy(), orc.analyse(lay, xs)).max() <= TOL
    assert band_rel_errors(lay, y[rows].cpu().numpy(), orc.synthesise_adjoint(lay, xs)).max() <= TOL
    want = orc.synthesise(lay, split_bands(lay, y[rows].cpu().numpy().astype(np.complex128)))[..., :w.valid_len]
    got = xr[rows].cpu().numpy()
    assert (np.linalg.norm(got - want, axis=-1) / np.linalg.norm(want, axis=-1)).max() <= TOL
    plan.close()


@pytest.mark.parametrize("batch", [1, 2501])
@pytest.mark.parametrize("log_n", range(6, 14))
def test_one_pass_fft_lengths(log_n, batch):
    n = 1 << log_n
    check_rows(small_workload(f"short{n}", N=n, valid_len=n - 3, fs=float(n), fmin=max(3.0, n / 64.0), fmax=n / 2.0,
                              bins_per_octave=4, m_policy=wl.M_SMOOTH, channels=batch), batch)


# 24 bands per octave from short to long on either side of the few-items form; lengths with large prime factors (direct
# sums and chirp-z); a band long enough for 1024 threads
@pytest.mark.parametrize("batch", [1, 5, 9, 70])
@pytest.mark.parametrize("kw", [dict(N=1 << 15, valid_len=30001, bins_per_octave=24, m_policy=wl.M_SMOOTH),
                                dict(N=1 << 14, valid_len=1 << 14, bins_per_octave=6, m_policy=wl.M_MULT4),
                                dict(N=1 << 15, valid_len=1 << 15, bins_per_octave=12, fmax=11025.0, m_policy=wl.M_POW2)],
                         ids=lambda k: f"n{k['N']}_b{k['bins_per_octave']}_p{k['m_policy']}")
def test_band_launch_forms(kw, batch):
    check_rows(small_workload("forms", **{"fs": 44100.0, "fmin": 60.0, "fmax": 22050.0, "channels": batch, **kw}), batch)


def check_bands_of_length(M, width, policy, batch, N=1 << 15):
    """Two overlapping regular bands of M coefficients against numpy's FFT of the windowed, slot-placed spectrum; the round
    trip covers the synthesis form."""
    from paper_2609_29119_b200 import Plan
    centre = [N / 4.0 - 0.1 * M, N / 4.0 + 0.1 * M]
    plan = Plan.from_bands(float(N), N, centre, [width] * 2, m_policy=policy)
    rng = np.random.default_rng(M)
    x = rng.standard_normal((batch, N)).astype(np.float32)
    c = plan.analyse(torch.from_numpy(x).cuda())
    g, _ = plan.tables()
    X = np.fft.rfft(x.astype(np.float64))
    for bi in plan.bands():
        if bi.is_sideband:
            continue
        assert bi.M == M
        d = np.arange(bi.first_offset, bi.first_offset + bi.support)
        slots = np.zeros((batch, M), dtype=np.complex128)
        slots[:, d % M] = g[bi.table_offset:bi.table_offset + bi.support] * X[:, bi.centre_bin + d]
        want = np.fft.ifft(slots)
        got = c[:, bi.coeff_offset:bi.coeff_offset + M].cpu().numpy()
        assert (np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)).max() <= TOL
    y = plan.synthesise(c).cpu().numpy().astype(np.float64)
    assert (np.sum((y - x) ** 2, axis=1) / np.sum(x.astype(np.float64) ** 2, axis=1)).max() <= 1e-12
    plan.close()


@pytest.mark.parametrize("m", [33, 64 - 3, 127, 257, 509, 1021, 2039, 2053, 3191])
def test_lengths_with_a_large_prime_factor(m):
    """4 m coefficients, m prime or not 5-smooth, up to both sides of each convolution length."""
    check_bands_of_length(4 * m, 4 * m - 1.5, wl.M_MULT4, 3)


@pytest.mark.parametrize("batch", [1, 33])
@pytest.mark.parametrize("fill", [1.0, 0.52])
@pytest.mark.parametrize("M", [256, 512, 1024, 2048, 4096, 8192])
def test_power_of_two_lengths(M, fill, batch):
    """Full support and one that leaves nearly half of the slots empty; an odd number of items in CTAs that share several."""
    check_bands_of_length(M, fill * M - 1.5, wl.M_POW2, batch)


@pytest.mark.parametrize("batch", [1, 33])
@pytest.mark.parametrize("log_n, fill", [(15, 0.52), (17, 1.0)], ids=["alone", "beside_two_pass_bands"])
def test_longest_power_of_two_length(log_n, fill, batch):
    """16,384 coefficients, the longest that one CTA transforms; in the longer signal the sidebands take the two-pass kernels."""
    check_bands_of_length(1 << 14, fill * (1 << 14) - 1.5, wl.M_POW2, batch, N=1 << log_n)


# more bands over one bin than a word has bits for planes: another form of the cover words and of the inverse kernels
@pytest.mark.parametrize("batch", [1, 9])
@pytest.mark.parametrize("log_n", [12, 15])
def test_more_than_31_planes(log_n, batch):
    N = 1 << log_n
    centres = [210 + 10 * i for i in range(80)] + list(range(1010, N // 2 - 210, 150))
    w = small_workload("planes", N=N, fs=float(N), valid_len=N - 5, channels=batch, m_policy=wl.M_SMOOTH,
                       bands=tuple((float(c), 400.0) for c in centres))
    cover = np.zeros(N // 2 + 1, dtype=int)
    for c in centres:
        cover[c - 199:c + 200] += 1
    assert cover.max() > 31
    check_rows(w, batch)
    lay, plan = oracle_layout(w), library_plan(w)
    y = wl.make_cotangent(w, lay.coeff_count)[:1]
    got = plan.analyse_adjoint(torch.from_numpy(y).cuda(), valid_len=w.valid_len).cpu().numpy()
    want = orc.analyse_adjoint(lay, split_bands(lay, y.astype(np.complex128)))[..., :w.valid_len]
    assert np.linalg.norm(got - want) <= TOL * np.linalg.norm(want)
    plan.close()


def test_few_items_form_ends_where_its_ctas_are_no_longer_resident():
    """Two bands of 8,212 coefficients (convolution length 8,192: one CTA per SM, four per band and signal) and two sidebands
    split into four items (two CTAs per SM): 12 SMs per signal."""
    from paper_2609_29119_b200 import Plan
    N, M = 1 << 15, 8212
    plan = Plan.from_bands(float(N), N, [N / 4.0 - 0.1 * M, N / 4.0 + 0.1 * M], [M - 1.5] * 2, m_policy=wl.M_MULT4)
    assert [b.M for b in plan.bands()][1:3] == [M, M] and min(plan.band_info(0).M, plan.band_info(3).M) > 13500
    most = torch.cuda.get_device_properties(0).multi_processor_count // 12
    for batch, few in ((1, True), (most, True), (most + 1, False)):
        x = torch.zeros(batch, N, device="cuda")
        plan.set_timing(True)
        plan.synthesise(plan.analyse(x))
        torch.cuda.synchronize()
        names = {n.split("/")[1] for n, _ in plan.read_timing() if "/" in n}
        plan.set_timing(False)
        assert "chirp" in names and ("split" in names) == few and ("class4" in names) == (not few), (batch, names)
    plan.close()


# one signal: bands of 23,328 coefficients are split, and class 0 stays on the run-time planned kernel beside them
@pytest.mark.parametrize("log_n, fmax, split", [(17, 18000.0, True), (15, 22050.0, False)])
def test_short_class_beside_split_bands(log_n, fmax, split):
    w = small_workload("short_class", N=1 << log_n, valid_len=99225 if split else 1 << log_n, fs=44100.0, fmin=55.0, fmax=fmax, bins_per_octave=36, channels=1, m_policy=wl.M_SMOOTH)
    plan = library_plan(w)
    x = torch.from_numpy(wl.make_signal(w)).cuda()
    plan.set_timing(True)
    y = plan.synthesise(plan.analyse(x, valid_len=w.valid_len), valid_len=w.valid_len)
    torch.cuda.synchronize()
    names = {n for n, _ in plan.read_timing()}
    plan.set_timing(False)
    for d in ("bands_from_spectrum", "bands_to_spectrum"):
        assert (f"{d}/split" in names) == split and f"{d}/merged" in names
        assert (f"{d}/class0" if split else f"{d}/class0/smooth") in names
    assert snr_db(x.cpu().numpy(), y.cpu().numpy()).min() >= 120.0
    plan.close()


# more than 3,120 bands of one class: the list of their records is a large table, uploaded by itself (class 0; class 1 and the
# list of the one-launch form, on both sides of the batch where that form ends)
@pytest.mark.parametrize("n_bands, width, spacing, log_n, batch", [(4000, 32.0, 16, 17, 2), (3300, 200.0, 36, 18, 1), (3300, 200.0, 36, 18, 2)])
def test_plans_with_thousands_of_bands(n_bands, width, spacing, log_n, batch):
    N = 1 << log_n
    centres = [float(150 + spacing * i) for i in range(n_bands)]
    w = small_workload("many_bands", N=N, fs=float(N), valid_len=N, channels=batch, m_policy=wl.M_SMOOTH,
                       bands=tuple((c, width) for c in centres))
    lay, plan = oracle_layout(w), library_plan(w)
    assert plan.num_bands == n_bands + 2
    x = wl.make_signal(w)
    c = plan.analyse(torch.from_numpy(x).cuda())
    got, X = c.cpu().numpy(), orc.long_dft(orc.pad_signal(x, N))
    for i in (0, 1, 2, n_bands // 2, 3119, 3120, 3121, 3122, n_bands - 1, n_bands, n_bands + 1):
        n = np.arange(lay.bands[i].M) if lay.bands[i].M < 1000 else np.arange(0, lay.bands[i].M, 97)
        want = orc.analyse_band(lay, X, i, n)
        err = np.linalg.norm(got[:, lay.coeff_offsets[i] + n] - want, axis=-1) / np.linalg.norm(want, axis=-1)
        assert err.max() <= TOL, (i, err)
    assert snr_db(x, plan.synthesise(c).cpu().numpy()).min() >= 120.0
    plan.close()


# chained band kernels read what the kernel before the chain wrote, in buffers that the calls before have used too
@pytest.mark.parametrize("kw", [dict(N=1 << 14, valid_len=1 << 14, bins_per_octave=12, m_policy=wl.M_MULT4, channels=1),   # chirp-z, merged, short
                                dict(N=1 << 17, valid_len=99225, bins_per_octave=36, fmax=18000.0, m_policy=wl.M_SMOOTH, channels=3),   # split first
                                dict(N=1 << 16, valid_len=60001, bins_per_octave=24, m_policy=wl.M_POW2, channels=5)],
                         ids=lambda k: f"n{k['N']}_p{k['m_policy']}")
def test_chained_kernels_see_the_call_before(kw):
    """Round trips of changing signals through the same buffers, enqueued without a pause, equal bit for bit those that are
    waited for after every kernel."""
    w = small_workload("chain", **{"fs": 44100.0, "fmin": 60.0, "fmax": 22050.0, **kw})
    plan, steps = library_plan(w), 24
    xs = torch.randn(steps, w.channels, w.valid_len, generator=torch.Generator().manual_seed(5)).cuda()
    xs *= torch.logspace(-3, 3, steps, device="cuda")[:, None, None]
    c = torch.empty((w.channels, plan.coeff_count), dtype=torch.complex64, device="cuda")
    y, ws = torch.empty_like(xs[0]), plan.workspace(w.channels)
    want = []
    for x in xs:
        plan.analyse(x, valid_len=w.valid_len, out=c, ws=ws)
        torch.cuda.synchronize()
        plan.synthesise(c, valid_len=w.valid_len, out=y, ws=ws)
        torch.cuda.synchronize()
        want.append((c.clone(), y.clone()))
    got_c, got_y = torch.empty((steps,) + c.shape, dtype=c.dtype, device="cuda"), torch.empty_like(xs)
    for _ in range(3):
        for i in range(steps):
            plan.analyse(xs[i], valid_len=w.valid_len, out=got_c[0], ws=ws)      # one buffer for all: rewritten by every call
            plan.synthesise(got_c[0], valid_len=w.valid_len, out=got_y[i], ws=ws)
        for i in range(1, steps):
            plan.analyse(xs[i], valid_len=w.valid_len, out=got_c[i], ws=ws)
        torch.cuda.synchronize()
        assert all(torch.equal(got_y[i], want[i][1]) for i in range(steps))
        assert all(torch.equal(torch.view_as_real(got_c[i]), torch.view_as_real(want[i][0])) for i in range(1, steps))
    plan.close()
