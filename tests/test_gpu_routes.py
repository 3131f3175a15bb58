"""Calls whose fields take one of several routes through a kernel, against calls of a field each, bit for bit."""
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
