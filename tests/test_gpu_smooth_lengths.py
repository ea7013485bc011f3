"""Every 5-smooth band length with a kernel of its own, in the forms that reach it: analysis against numpy's FFT of the windowed,
slot-placed spectrum, its adjoint against the transposed steps, and the round trip.  The launches are named, so that a test fails
where another kernel ran."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


def smooth(m):
    for f in (2, 3, 5):
        while m % f == 0:
            m //= f
    return m == 1


def lengths(lo, hi):
    """5-smooth multiples of 4 above lo up to hi."""
    return [m for m in range(lo // 4 * 4 + 4, hi + 1, 4) if smooth(m)]


def band_list(wanted, fill, N):
    """Bands of the wanted lengths between bands of the longest one, which keep the frame complete; long ones twice each, from
    one end of the spectrum to the other.  fill: part of the slots used."""
    longest, used = max(wanted), [max(m - 1.5 if m == max(wanted) else fill * (m - 1.5), 2.5) for m in wanted]
    if longest > 4096:
        widths = [w for w in used[::2] + used[1::2][::-1] for _ in range(2)]   # the longest in the middle
        return [float(c) for c in np.linspace(0.6 * widths[0], N / 2 - 0.6 * widths[-1], len(widths))], widths
    widths = [w for u in reversed(used) for w in (longest - 1.5, u)]
    centres = [1.1 * longest + longest / 12.0 * i for i in range(len(widths))]
    assert centres[-1] + longest < N / 2
    return centres, widths


def check_lengths(wanted, fill, N, batch, forms, policy=wl.M_SMOOTH):
    """forms: launches that have to be of these kernels, direction and class."""
    from paper_2609_29119_b200 import Plan
    longest = max(wanted)
    centres, widths = band_list(wanted, fill, N)
    plan = Plan.from_bands(float(N), N, centres, widths, m_policy=policy)
    have = {b.M for b in plan.bands()}
    assert fill < 1.0 or set(wanted) <= have
    rng = np.random.default_rng(longest)
    x = rng.standard_normal((batch, N)).astype(np.float32)
    xg = torch.from_numpy(x).cuda()
    plan.set_timing(True)
    plan.synthesise(plan.analyse(xg))
    torch.cuda.synchronize()
    names = {n.removesuffix("/smooth") for n, _ in plan.read_timing() if n.endswith("/smooth")}
    plan.set_timing(False)
    assert {f"bands_{direction}_spectrum/{cls}" for direction, cls in forms} <= names, names
    c = plan.analyse(xg)
    got, (g, _) = c.cpu().numpy(), plan.tables()
    rows = sorted({0, 1, batch // 2, batch - 1} & set(range(batch)))
    # the adjoint on other coefficients, sidebands (folded onto the half spectrum there) among them
    cbar = torch.randn(batch, plan.coeff_count, 2, generator=torch.Generator(device="cuda").manual_seed(longest), device="cuda")
    back = plan.analyse_adjoint(torch.view_as_complex(cbar))[rows].cpu().numpy()
    cbar = torch.view_as_complex(cbar)[rows].cpu().numpy().astype(np.complex128)
    X = np.fft.fft(x[rows].astype(np.float64))     # both halves: sidebands reach over bins 0 and N/2
    Z = np.zeros_like(X)
    for bi in plan.bands():
        d = np.arange(bi.first_offset, bi.first_offset + bi.support)
        window, own = g[bi.table_offset:bi.table_offset + bi.support], slice(bi.coeff_offset, bi.coeff_offset + bi.M)
        slots = np.zeros((len(rows), bi.M), dtype=np.complex128)
        slots[:, d % bi.M] = window * X[:, (bi.centre_bin + d) % N]
        want = np.fft.ifft(slots)
        err = np.linalg.norm(got[rows, own] - want, axis=1) / np.linalg.norm(want, axis=1)
        assert err.max() <= TOL, (bi.M, err.max())
        Z[:, (bi.centre_bin + d) % N] += window / bi.M * np.fft.fft(cbar[:, own])[:, d % bi.M]
    want = N * np.fft.ifft(Z).real
    assert (np.linalg.norm(back - want, axis=1) / np.linalg.norm(want, axis=1)).max() <= TOL
    y = plan.synthesise(c).cpu().numpy().astype(np.float64)
    assert (np.sum((y - x) ** 2, axis=1) / np.sum(x.astype(np.float64) ** 2, axis=1)).max() <= 1e-12
    plan.close()


def both(cls):
    return {("from", cls), ("to", cls)}


# 1 and 3 signals: the few-items form; 401, 1601, 4501: class kernels side by side, one, two and four units per CTA, the last one ragged
@pytest.mark.parametrize("batch", [1, 3, 401, 1601, 4501])
@pytest.mark.parametrize("fill", [1.0, 0.6])
def test_short_lengths(fill, batch):
    check_lengths(lengths(0, 128), fill, 1 << 11, batch, both("class0"))


@pytest.mark.parametrize("batch", [1, 37, 701])
def test_short_lengths_of_power_of_two_plans(batch):
    check_lengths([4, 8, 16, 32, 64, 128], 1.0, 1 << 11, batch, both("class0"), policy=wl.M_POW2)


# enough items for the side-by-side form: a CTA has one, two or four units, the last one ragged
@pytest.mark.parametrize("lo, hi, log_n, batch", [(128, 1024, 14, 101), (128, 1024, 14, 403), (128, 1024, 14, 701), (1024, 4096, 16, 17), (1024, 4096, 16, 53), (1024, 4096, 16, 113)])
@pytest.mark.parametrize("fill", [1.0, 0.6])
def test_middle_lengths(fill, lo, hi, log_n, batch):
    check_lengths(lengths(lo, hi), fill, 1 << log_n, batch, {("from", "class1" if hi == 1024 else "class2")})


# a CTA and nearly all of an SM's shared memory per item
@pytest.mark.parametrize("fill", [1.0, 0.9])
@pytest.mark.parametrize("part", range(3))
def test_long_lengths(part, fill):
    check_lengths(lengths(13500, 27648)[part::3], fill, 1 << 17, 8, both("class4"))
