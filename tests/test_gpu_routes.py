"""Calls that take one of several routes through the passes, against calls of a field each (bit for bit) and
float64 sums, and what a pass may take where a route once held it up."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    import __graft_entry__ as g
    g.build()
    import paper_2411_18591_gb300 as T
    return T


def cfield(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.complex64)


@pytest.mark.parametrize("n,pad,batch,sets", [(61, 1.0, 1, 1), (61, 1.0, 40, 1), (61, 1.0, 16, 16), (61, 1.0, 17, 17),
                                              (61, 1.0, 6, 3), (1021, 2.0, 3, 3)])
def test_bluestein_tables(T, n, pad, batch, sets):
    """One transfer table for the call, a few in the launch, or a list in memory (also as a shared source's
    repeats), at single and split convolutions."""
    d = 6e-6
    x = cfield(n + batch, batch, n, n)
    zs = [0.02 + 0.003 * (b % sets) for b in range(batch)]
    lams = [5e-7 + 1e-8 * (b % sets) for b in range(batch)]
    each = [T.top_propagate(x[b].clone(), d, d, lams[b], zs[b], pad)[0] for b in range(batch)]
    out = T.top_propagate(x, d, d, lams[0] if sets == 1 else lams, zs[0] if sets == 1 else zs, pad)
    assert torch.equal(out, torch.stack(each))
    if sets > 1:
        out = T.top_propagate(x[:1].clone(), d, d, lams, zs, pad, input_repeat=batch)
        for b in range(batch):
            assert torch.equal(out[b], T.top_propagate(x[0].clone(), d, d, lams[b], zs[b], pad)[0])


@pytest.mark.parametrize("ny,nx,pad,batch", [(16, 16, 2.0, 3), (33, 32, 1.0, 2), (64, 64, 2.0, 2), (250, 256, 2.0, 2),
                                             (7, 1000, 2.0, 2), (1024, 1024, 2.0, 1), (16, 4096, 2.0, 1)])
def test_overlap_sums(T, ny, nx, pad, batch):
    """The overlap and power of every field against float64 sums of the field the call itself returns, at every
    shape of block (a sum of float64 products of float32 values: 1e-12 leaves 2^13 roundings of 2^-53)."""
    d = 6e-6
    x, t = cfield(ny, batch, ny, nx), cfield(nx + 1, ny, nx)
    overlap, power, field = T.top_propagate_overlap(x, t, d, d, 5e-7, 0.01, pad, keep_field=True)
    f, ref = field.to(torch.complex128), t.to(torch.complex128)
    want = (f * ref.conj()).sum((1, 2)) * d * d
    scale = float((f.abs().square().sum((1, 2)).sqrt() * ref.abs().square().sum().sqrt()).max()) * d * d
    assert float((overlap - want).abs().max()) < 1e-12 * scale
    want = f.abs().square().sum((1, 2)) * d * d
    assert float(((power - want) / want).abs().max()) < 1e-12


def inverse_rows_us(T, call, reps=6):
    """Device time of a call's inverse row passes, the least of `reps` calls."""
    from paper_2411_18591_gb300 import binding as B
    best = 1e9
    B.profile_enable(True)
    try:
        for _ in range(3):
            call()
        B.profile_read()
        for _ in range(reps):
            call()
            torch.cuda.synchronize()
            best = min(best, 1e3 * B.profile_read()["rows_inv"][0])
    finally:
        B.profile_enable(False)
    return best


@pytest.mark.parametrize("n,batch", [(1024, 8), (4096, 1)])
def test_overlap_sums_do_not_hold_the_pass(T, n, batch):
    """The overlap's inverse rows read one field more than plain ones (32 bytes a sample of padding 2 instead of
    24) and add up: at most five times as long (seven with a serial sum a block)."""
    d = 6e-6
    x, t = cfield(1, batch, n, n), cfield(2, n, n)
    plain = inverse_rows_us(T, lambda: T.top_propagate(x, d, d, 5e-7, 0.01, 2.0))
    assert inverse_rows_us(T, lambda: T.top_propagate_overlap(x, t, d, d, 5e-7, 0.01, 2.0)) < 5 * plain


# padded rows of 512 samples filled, of 512 with both ends of the line folded, of 2000 with odd numbers of rows
# (lines interleaved in pairs: the last box of a field is clipped), of 1024 filled
@pytest.mark.parametrize("ny,nx,pad,batch,group", [(512, 512, 1.0, 48, 3), (320, 320, 1.6, 64, 8), (333, 1333, 1.5, 16, 2),
                                                   (1024, 1024, 1.0, 16, 16)])
def test_copied_rows_at_other_paddings(T, ny, nx, pad, batch, group):
    """Row passes that move their tiles by copy, at paddings other than 2: fields, chains, weighted intensities of
    groups and the gradients of all three planes, against calls of a field each (which do not copy) bit for bit,
    the sums against float64 sums of theirs (a rounding of 2^-24 each, in quadrature)."""
    d, z, lam = 6e-6, 0.01, 600e-9
    g = torch.Generator(device="cuda").manual_seed(ny + nx)
    x, w = cfield(ny, batch, ny, nx), torch.rand(batch, generator=g, device="cuda") + 0.5
    planes = dict(phase=torch.rand((ny, nx), generator=g, device="cuda") * 6 - 3,
                  amplitude=torch.rand((ny, nx), generator=g, device="cuda") + 0.5, mask=cfield(nx, ny, nx))
    pre = T.Modulation(**planes)
    stages = [T.Stage(z, pre=pre), T.Stage(0.5 * z, pre=T.Modulation(phase=planes["phase"]))]
    new = lambda: {"grad_" + k: torch.zeros_like(v) for k, v in planes.items()}
    one = lambda b: x[b].clone()
    out = T.top_propagate(x, d, d, lam, z, pad, pre=pre)
    inten, kept = T.top_propagate_intensity(x, d, d, lam, z, pad, group=group, weights=w, pre=pre, keep_field=True)
    chain, _ = T.top_fused_chain(x, d, d, lam, stages, pad)
    grads = new()
    back = T.top_propagate_backward(x, d, d, lam, z, pad, pre=pre, saved_in=out, **grads)
    sums = {k: torch.zeros_like(v, dtype=torch.complex128 if v.is_complex() else torch.float64) for k, v in grads.items()}
    for b in range(batch):
        o = T.top_propagate(one(b), d, d, lam, z, pad, pre=pre)[0]
        assert torch.equal(out[b], o) and torch.equal(kept[b], o), b
        assert torch.equal(chain[b], T.top_fused_chain(one(b), d, d, lam, stages, pad)[0][0]), b
        g1 = new()
        assert torch.equal(back[b], T.top_propagate_backward(one(b), d, d, lam, z, pad, pre=pre, saved_in=o.clone(), **g1)), b
        for k in sums:
            sums[k] += g1[k]
    off = lambda a, ref: float((a - ref).norm() / ref.norm())
    for k in sums:
        assert off(grads[k], sums[k]) < batch ** 0.5 * 2.0 ** -24, k
    ref = (w.double()[:, None, None] * kept.to(torch.complex128).abs() ** 2).reshape(-1, group, ny, nx).sum(1)
    assert off(inten, ref) < (group + 4) ** 0.5 * 2.0 ** -24
    phase = torch.zeros_like(planes["phase"])
    only = T.Modulation(phase=planes["phase"])
    T.top_propagate_backward(x, d, d, lam, z, pad, pre=only, saved_in=out, grad_phase=phase)
    ref = torch.zeros_like(phase, dtype=torch.float64)
    for b in range(batch):
        g1 = torch.zeros_like(phase)
        T.top_propagate_backward(one(b), d, d, lam, z, pad, pre=only, saved_in=out[b].clone(), grad_phase=g1)
        ref += g1
    assert off(phase, ref) < batch ** 0.5 * 2.0 ** -24


@pytest.mark.parametrize("n,batch,pad,most", [(1024, 2, 2.0, 1.8), (1024, 8, 1.0, 4.5), (2048, 2, 1.0, 4.5)])
def test_gradient_epilogue_does_not_hold_the_pass(T, n, batch, pad, most):
    """The inverse rows with a phase gradient against plain ones: they read the saved field and the partial sums
    and write these besides (2.2, 6.7 and 6.7 times as long with the partials loaded slot by slot)."""
    d = 6e-6
    x, gx = cfield(1, batch, n, n), cfield(2, batch, n, n)
    gp, phase = torch.zeros((n, n), device="cuda"), torch.rand((n, n), device="cuda")
    plain = inverse_rows_us(T, lambda: T.top_propagate(x, d, d, 5e-7, 0.01, pad))
    back = inverse_rows_us(T, lambda: T.top_propagate_backward(gx, d, d, 5e-7, 0.01, pad, pre=T.Modulation(phase=phase),
                                                               saved_in=x, grad_phase=gp))
    assert back < most * plain


def test_first_noalloc_call_of_a_process_may_be_captured(T):
    """The look-up of the static scratch and the word beside it does not break a capture under way."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = """
import torch
import paper_2411_18591_gb300 as T
x = torch.randn(3, 512, 512, device="cuda", dtype=torch.complex64)
y, ref = torch.zeros_like(x), torch.zeros_like(x)
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    T.top_propagate_noalloc(x, 8e-6, 8e-6, 5e-7, 0.02, out=y)
graph.replay()
T.top_propagate_noalloc(x, 8e-6, 8e-6, 5e-7, 0.02, out=ref)
torch.cuda.synchronize()
T.check_waits()
T.check_waits(noalloc=True)
assert torch.equal(y, ref) and float(y.abs().sum()) > 0
"""
    run = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr[-2000:]
