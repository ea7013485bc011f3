"""Gradients through the differentiable wrappers against gradients assembled from the oracle's adjoints (Sec. 3.2):
for L = 1/2 ||S T x - t||^2 the gradient is T' S' (S T x - t); for a loss on the coefficients it is T' of the cotangent."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as wl
from helpers import library_plan, oracle_layout, small_workload, snr_db, split_bands
from oracle import nsgt_oracle as orc

pytestmark = pytest.mark.gpu

CASES = [
    small_workload("ad_n4096", N=4096, valid_len=4096, fs=22050.0, fmin=200.0, fmax=11025.0, bins_per_octave=24,
                   m_policy=wl.M_SMOOTH, channels=2),
    small_workload("ad_ragged", N=4096, valid_len=3001, fs=22050.0, fmin=200.0, fmax=11025.0, bins_per_octave=12,
                   m_policy=wl.M_MULT4, channels=2),
    small_workload("ad_multires", N=8192, valid_len=8192, fs=8192.0, fmin=100.0, fmax=4096.0, bins_per_octave=0,
                   m_policy=wl.M_POW2, channels=2, sections=((2, 4), (2, 8), (1, 16))),
]


@pytest.mark.parametrize("w", CASES, ids=lambda w: w.name)
def test_round_trip_loss_gradient_matches_oracle_adjoints(w):
    from paper_2609_29119_b200 import autograd as ad
    lay, plan = oracle_layout(w), library_plan(w)
    x = wl.make_signal(w)
    t = np.random.default_rng(w.seed + 1).standard_normal(x.shape).astype(np.float32)
    xd = torch.from_numpy(x).cuda().requires_grad_(True)
    c = ad.analyse(plan, xd, valid_len=w.valid_len)
    c.retain_grad()
    y = ad.synthesise(plan, c, valid_len=w.valid_len)
    loss = 0.5 * ((y - torch.from_numpy(t).cuda()) ** 2).sum()
    loss.backward()
    # oracle: residual r = S T x - t on the true samples (zero beyond), grad_c = S' r, grad_x = T' grad_c
    x64 = orc.pad_signal(x, w.N)
    r = orc.synthesise(lay, orc.analyse(lay, x64))
    r[..., w.valid_len:] = 0.0
    r[..., :w.valid_len] -= t
    gc = orc.synthesise_adjoint(lay, r)
    gx = orc.analyse_adjoint(lay, gc)[..., :w.valid_len]
    got_x = xd.grad.cpu().numpy()
    got_c = split_bands(lay, c.grad.cpu().numpy())
    assert min(snr_db(gx, got_x)) >= 100.0, snr_db(gx, got_x)     # 1e-5 relative
    for a, b in zip(got_c, gc):
        assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b)
    plan.close()


def test_coefficient_loss_gradient_and_padding_columns():
    """Loss on the coefficients of a strided, over-wide input: gradient = T'(cotangent) on the true samples, zero beyond."""
    from paper_2609_29119_b200 import autograd as ad
    w = CASES[1]
    lay, plan = oracle_layout(w), library_plan(w)
    x = wl.make_signal(w)
    wide = np.zeros((x.shape[0], w.valid_len + 17), dtype=np.float32)
    wide[:, :w.valid_len] = x
    xd = torch.from_numpy(wide).cuda().requires_grad_(True)
    m = wl.make_cotangent(w, lay.coeff_count)
    c = ad.analyse(plan, xd, valid_len=w.valid_len)
    loss = (c * torch.from_numpy(m).cuda().conj()).real.sum()     # <m, c>: cotangent is m
    loss.backward()
    want = orc.analyse_adjoint(lay, split_bands(lay, m.astype(np.complex128)))[..., :w.valid_len]
    got = xd.grad.cpu().numpy()
    assert np.all(got[:, w.valid_len:] == 0)
    assert min(snr_db(want, got[:, :w.valid_len])) >= 100.0
    plan.close()


def test_conjugate_and_negative_views_are_read_as_what_they_stand_for():
    """Tensors whose conjugation or negation is still to be computed (torch's conj and neg bits), as inputs and cotangents."""
    from paper_2609_29119_b200 import SliCQ
    from paper_2609_29119_b200 import autograd as ad
    w = CASES[0]
    plan = library_plan(w)
    x = torch.from_numpy(wl.make_signal(w)).cuda()
    m = torch.from_numpy(wl.make_cotangent(w, plan.coeff_count)).cuda()

    def same(a, b):
        a, b = (t.resolve_conj().resolve_neg() for t in (a, b))
        return torch.equal(torch.view_as_real(a), torch.view_as_real(b)) if a.is_complex() else torch.equal(a, b)
    neg_x, conj_m, neg_m = torch._neg_view(x), m.conj(), torch._neg_view(m)
    assert neg_x.is_neg() and conj_m.is_conj() and neg_m.is_neg() and torch._neg_view(conj_m).is_conj()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    for stream in (None, side):
        out_c, out_x = torch.empty_like(m), torch.empty_like(x)
        plan.analyse(neg_x, out=out_c, stream=stream)
        torch.cuda.synchronize()
        assert same(out_c, plan.analyse(-x))
        for view in (conj_m, neg_m, torch._neg_view(conj_m)):
            stored = view.resolve_conj().resolve_neg().clone()
            plan.synthesise(view, out=out_x, stream=stream)
            torch.cuda.synchronize()
            assert same(out_x, plan.synthesise(stored))
            plan.analyse_adjoint(view, out=out_x, stream=stream)
            torch.cuda.synchronize()
            assert same(out_x, plan.analyse_adjoint(stored))
    # cotangents and differentiable inputs
    xg, cg = x.clone().requires_grad_(True), m.clone().requires_grad_(True)
    c, y = ad.analyse(plan, xg), ad.synthesise(plan, cg)
    for view in (conj_m, neg_m):
        got, = torch.autograd.grad(c, xg, grad_outputs=view, retain_graph=True)
        assert same(got, plan.analyse_adjoint(view.resolve_conj().resolve_neg()))
    got, = torch.autograd.grad(y, cg, grad_outputs=neg_x, retain_graph=True)
    assert same(got, plan.synthesise_adjoint(-x))
    got, = torch.autograd.grad(ad.synthesise(plan, torch._neg_view(cg.conj())), cg, grad_outputs=x)
    assert same(got, (-plan.synthesise_adjoint(x)).conj().resolve_conj())
    # the sliced form, and outputs that are such views
    a, b = SliCQ(plan, w.channels, 512, 2), SliCQ(plan, w.channels, 512, 2)
    assert a.push(neg_x) == b.push(-x) == 2
    assert same(a.coeffs(1).clone(), b.coeffs(1).clone())
    for call in (lambda: plan.analyse(x, out=conj_m), lambda: plan.synthesise(m, out=neg_x), lambda: a.pull(neg_x)):
        with pytest.raises(AssertionError):
            call()
    a.close(); b.close(); plan.close()


def test_backward_runs_on_the_stream_of_the_forward_pass():
    """Forward passes on a side stream, backward calls from the default one, inputs that change from step to step: the same
    gradients as on one stream."""
    from paper_2609_29119_b200 import autograd as ad
    w = CASES[2]
    plan, one = library_plan(w), library_plan(w)
    side = torch.cuda.Stream()
    gen = torch.Generator(device="cuda").manual_seed(3)
    for _ in range(8):
        x = torch.randn(w.channels, w.valid_len, generator=gen, device="cuda")
        t = torch.randn(w.channels, w.valid_len, generator=gen, device="cuda")
        a, b = x.clone().requires_grad_(True), x.clone().requires_grad_(True)
        ((ad.synthesise(one, ad.analyse(one, a)) - t) ** 2).sum().backward()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            loss = ((ad.synthesise(plan, ad.analyse(plan, b)) - t) ** 2).sum()
        torch.cuda.current_stream().wait_stream(side)
        loss.backward()
        assert torch.equal(a.grad, b.grad)
        torch.cuda.synchronize()          # the next forward pass reuses the plan's workspace on the side stream
    plan.close(); one.close()


def test_what_the_wrappers_do_not_support_is_refused():
    """Forward-mode derivatives and function transforms raise instead of dropping the tangent or reading a wrapper's memory."""
    import torch.autograd.forward_ad as fwd
    from paper_2609_29119_b200 import autograd as ad
    w = CASES[0]
    plan = library_plan(w)
    x = torch.from_numpy(wl.make_signal(w)).cuda()
    m = torch.from_numpy(wl.make_cotangent(w, plan.coeff_count)).cuda()
    for f, t in ((lambda t: ad.analyse(plan, t), x), (lambda t: ad.synthesise(plan, t), m)):
        with fwd.dual_level():
            with pytest.raises(NotImplementedError):
                f(fwd.make_dual(t, torch.ones_like(t)))
            f(t)                                  # a tensor without a tangent is taken
        with pytest.raises(RuntimeError):
            torch.func.vmap(f)(t[None].repeat(2, 1, 1))
        with pytest.raises(RuntimeError):
            torch.func.jvp(f, (t,), (t,))
        with pytest.raises(RuntimeError):
            torch.func.grad(lambda t: f(t).abs().sum())(t)
    plan.close()
