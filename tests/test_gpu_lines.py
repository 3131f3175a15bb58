"""The passes at the edges of their tiles and layouts: odd numbers of rows, rows that do not fill a
tile of four, paddings that fold both ends of a line, and every pairing of row plans that interleave
workspace lines (even thread groups) with ones that do not (25 threads a line) and with two- and
three-stage column plans. Forward and backward with modulations against the float64 oracle (rel-L2
1e-5, the propagation target), and a fused chain against its separate calls, bit for bit."""
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


def host(t):
    return t.cpu().numpy()


def cfield(seed, shape):
    return to_c64(normal(seed, shape) + 1j * normal(sub_seed(seed, 1), shape))


# padded sizes: 512 x 500, 500 x 512, 512 x 2048, 2048 x 512, 2000 x 512, 512 x 2000; then padding 2
CASES = [(341, 333, 1.5), (333, 341, 1.5), (341, 1365, 1.5), (1365, 341, 1.5), (1333, 341, 1.5), (341, 1333, 1.5),
         (250, 1024, 2.0), (1024, 250, 2.0), (250, 2048, 2.0), (2048, 250, 2.0), (500, 1000, 2.0), (16, 32, 2.0)]


@pytest.mark.parametrize("ny,nx,pad", CASES)
def test_tile_edges(T, ny, nx, pad):
    dy, dx, z, lams = 7e-6, 6e-6, 0.01, [500e-9, 640e-9]
    seed = 9000 + ny * 7 + nx
    x, g = cfield(seed, (2, ny, nx)), cfield(seed + 1, (2, ny, nx))
    phi = uniform(seed + 2, (ny, nx), -np.pi, np.pi).astype(np.float32)
    amp = uniform(seed + 3, (ny, nx), 0.5, 1.5).astype(np.float32)
    m = amp.astype(np.float64) * np.exp(1j * phi.astype(np.float64))
    pre = T.Modulation(phase=dev(phi), amplitude=dev(amp))
    radius = 0.4317 * min(ny * dy, nx * dx)
    post = T.Modulation(focal_length=0.2, radius=radius)
    pm = np.stack([O.circ(ny, nx, dy, dx, radius) * O.lens(ny, nx, dy, dx, l, 0.2) for l in lams])
    out = T.top_propagate(dev(x), dy, dx, lams, z, pad, pre=pre, post=post)
    ref = O.propagate(x.astype(np.complex128) * m, dy, dx, lams, z, pad)
    assert rel_l2(host(out), ref * pm) < TOL
    gp, ga = torch.zeros((ny, nx), device="cuda"), torch.zeros((ny, nx), device="cuda")
    gin = T.top_propagate_backward(dev(g), dy, dx, lams, z, pad, pre=pre, post=post, saved_in=dev(x), grad_phase=gp,
                                   grad_amplitude=ga)
    gy = O.propagate_adjoint(np.conj(pm) * g, dy, dx, lams, z, pad)
    gx, gm, gphi = O.grad_modulation(x.astype(np.complex128), m, gy)
    assert rel_l2(host(gin), gx) < TOL
    assert rel_l2(host(gp), gphi) < TOL
    # dM/dA = exp(i phi): sum_b Re(conj(g_y) exp(i phi) x)
    assert rel_l2(host(ga), np.real(gm * np.conj(np.exp(1j * phi.astype(np.float64))))) < TOL
    # a fused chain and its separate calls
    keep = torch.empty_like(out)
    y, inten = T.top_fused_chain(dev(x), dy, dx, lams, [T.Stage(z, keep=keep), T.Stage(0.5 * z, pre=pre)], pad,
                                 intensity_group=2)
    first = T.top_propagate(dev(x), dy, dx, lams, z, pad)
    assert torch.equal(keep, first)
    assert torch.equal(y, T.top_propagate(first, dy, dx, lams, 0.5 * z, pad, pre=pre))
    assert rel_l2(host(inten), (np.abs(host(y).astype(np.complex128)) ** 2).sum(0)) < TOL


# batches large enough for the row passes to move their tiles by copy, at every plan that does: whole and
# part-filled last tiles, one-field and grouped items, groups of different lengths
@pytest.mark.parametrize("ny,nx,batch", [(16, 256, 800), (250, 256, 48), (250, 512, 32), (16, 768, 256), (16, 1000, 160),
                                         (16, 1024, 264), (250, 1024, 16), (16, 2048, 128)])
def test_copied_tiles_match_direct_ones(T, ny, nx, batch):
    d, z, lam = 6e-6, 0.02, 600e-9
    gen = torch.Generator(device="cuda").manual_seed(ny * 3 + nx)
    x = torch.randn((batch, ny, nx), generator=gen, device="cuda", dtype=torch.complex64)
    phi = torch.rand((ny, nx), generator=gen, device="cuda") * 6 - 3
    pre = T.Modulation(phase=phi)
    stages = [T.Stage(z, pre=pre), T.Stage(0.5 * z, pre=T.Modulation(focal_length=0.3, radius=0.4 * nx * d))]
    out = T.top_propagate(x, d, d, lam, z, 2.0, pre=pre)
    group = 4
    y, inten = T.top_fused_chain(x, d, d, lam, stages, 2.0, intensity_group=group)
    gp, direct = torch.zeros_like(phi), torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    back = T.top_propagate_backward(x, d, d, lam, z, 2.0, pre=pre, saved_in=out, grad_phase=gp)
    for b in range(batch):
        assert torch.equal(out[b], T.top_propagate(x[b], d, d, lam, z, 2.0, pre=pre)[0]), b
        y1, i1 = T.top_fused_chain(x[b], d, d, lam, stages, 2.0, intensity_group=1)
        assert torch.equal(y[b], y1[0]), b
        g1 = torch.zeros_like(phi)
        assert torch.equal(back[b], T.top_propagate_backward(x[b], d, d, lam, z, 2.0, pre=pre, saved_in=out[b],
                                                             grad_phase=g1)), b
        direct += g1
    ref = (y.abs().double() ** 2).reshape(batch // group, group, ny, nx).sum(1)
    assert rel_l2(host(inten), host(ref)) < TOL
    assert rel_l2(host(gp), host(direct)) < TOL
