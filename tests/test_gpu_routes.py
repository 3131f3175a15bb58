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
