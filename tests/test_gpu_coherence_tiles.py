"""The end of the coherence backward where its 64 x 128 blocks do not divide the tensor, over a batch,
with and without the gradients it may leave out, against the float64 oracle (rel-L2 1e-5)."""
import numpy as np
import pytest
import torch

import oracle as O
from synthetic import normal, sub_seed, to_c64, uniform

from conftest import rel_l2

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    import __graft_entry__ as g
    g.build()
    import paper_2411_18591_gb300 as T
    return T


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("ny,nx,pad,batch", [(12, 12, 2.667, 1), (12, 24, 2.667, 2), (32, 16, 2.0, 1)])
def test_coherence_backward_tiles(T, ny, nx, pad, batch):
    d, lam, z = 9e-6, 600e-9, 0.003
    shape = (batch, ny, nx, ny, nx)
    cplx = lambda seed, s: to_c64(normal(seed, s) + 1j * normal(sub_seed(seed, 1), s))
    seed = 7700 + ny * nx
    gamma, g = cplx(seed, shape), cplx(seed + 1, shape)
    mask, amp = cplx(seed + 2, (ny, nx)), uniform(seed + 3, (ny, nx), 0.5, 1.5).astype(np.float32)
    phi = uniform(seed + 4, (ny, nx), -np.pi, np.pi).astype(np.float32)
    e = np.exp(1j * phi.astype(np.float64))
    m = mask.astype(np.complex128) * amp * e
    mod = T.Modulation(mask=dev(mask), amplitude=dev(amp), phase=dev(phi))
    gp, ga = torch.zeros((ny, nx), device="cuda"), torch.zeros((ny, nx), device="cuda")
    gc = torch.zeros((ny, nx), dtype=torch.complex64, device="cuda")
    run = lambda **kw: T.top_propagate_coherence_backward(dev(g), d, d, lam, z, pad, mask=mod, **kw)
    gin = run(saved_in=dev(gamma), grad_phase=gp, grad_amplitude=ga, grad_mask=gc)
    assert torch.equal(gin, run())
    gp2 = torch.zeros_like(gp)
    assert run(saved_in=dev(gamma), grad_phase=gp2, want_grad_in=False) is None
    assert torch.equal(gp, gp2)
    g_m, ref = 0, []
    for b in range(batch):
        gg = O.propagate_coherence(g[b].astype(np.complex128), d, d, lam, z, pad, adjoint=True)
        g_m = g_m + O.grad_modulate_coherence(gamma[b].astype(np.complex128), m, gg)
        ref.append(gg * np.conj(m[:, :, None, None] * np.conj(m)[None, None]))
    assert rel_l2(gin.cpu().numpy(), np.stack(ref)) < TOL
    assert rel_l2(gp.cpu().numpy(), np.imag(np.conj(m) * g_m)) < TOL
    assert rel_l2(ga.cpu().numpy(), np.real(np.conj(mask.astype(np.complex128) * e) * g_m)) < TOL
    assert rel_l2(gc.cpu().numpy(), g_m * np.conj(amp * e)) < TOL
    out = T.top_propagate_coherence(dev(gamma), d, d, lam, z, pad, mask=mod)
    fwd = [O.propagate_coherence(O.modulate_coherence(x.astype(np.complex128), m), d, d, lam, z, pad) for x in gamma]
    assert rel_l2(out.cpu().numpy(), np.stack(fwd)) < TOL


def test_mask_gradient_sums_round_little(T):
    """The sums over a 64^4 tensor alone, against the same sums in float64 of the call's own grad_in. A term takes
    eight roundings (its products and the mask's values), the sums at most sixteen levels of rounding: in
    quadrature sqrt(24) times the rms of one, 2^-24 / sqrt 3."""
    n, d, lam, z = 64, 10e-6, 633e-9, 0.2
    g = torch.Generator(device="cuda").manual_seed(4)
    cplx = lambda: torch.randn((n,) * 4, generator=g, device="cuda", dtype=torch.complex64)
    gamma, grad = cplx(), cplx()
    phi = (torch.rand((n, n), generator=g, device="cuda") * 2 - 1) * np.pi
    gp = torch.zeros_like(phi)
    gin = T.top_propagate_coherence_backward(grad, d, d, lam, z, mask=T.Modulation(phase=phi), saved_in=gamma, grad_phase=gp)
    # dL/dphi(r) = sum_s Im(gin(r, s) conj(gamma(r, s))) - sum_s Im(gin(s, r) conj(gamma(s, r)))
    t = (gin.reshape(n * n, n * n).to(torch.complex128) * gamma.reshape(n * n, n * n).to(torch.complex128).conj()).imag
    ref = (t.sum(1) - t.sum(0)).reshape(n, n)
    assert float((gp - ref).norm() / ref.norm()) < np.sqrt(24 / 3) * 2.0 ** -24


@pytest.mark.parametrize("n,batch", [(16, 160), (16, 3), (32, 9)])
def test_batches_in_slices(T, n, batch):
    """A batch that the last pass cuts into slices of several tensors, with a shorter last one: every tensor's
    grad_in is that of a call of its own, and the mask gradient the sum over the batch (eight roundings a term, up
    to 24 levels of sums, as above)."""
    d, lam, z = 10e-6, 633e-9, 0.1
    g = torch.Generator(device="cuda").manual_seed(n + batch)
    cplx = lambda: torch.randn((batch,) + (n,) * 4, generator=g, device="cuda", dtype=torch.complex64)
    gamma, grad = cplx(), cplx()
    mod = T.Modulation(phase=(torch.rand((n, n), generator=g, device="cuda") * 2 - 1) * np.pi)
    gp = torch.zeros((n, n), device="cuda")
    gin = T.top_propagate_coherence_backward(grad, d, d, lam, z, mask=mod, saved_in=gamma, grad_phase=gp)
    ref = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    for b in range(batch):
        assert torch.equal(gin[b], T.top_propagate_coherence_backward(grad[b], d, d, lam, z, mask=mod)), b
        t = (gin[b].reshape(n * n, n * n).to(torch.complex128) * gamma[b].reshape(n * n, n * n).to(torch.complex128).conj()).imag
        ref += (t.sum(1) - t.sum(0)).reshape(n, n)
    assert float((gp - ref).norm() / ref.norm()) < np.sqrt(32 / 3) * 2.0 ** -24
