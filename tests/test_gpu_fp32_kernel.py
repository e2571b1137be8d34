"""The plain-FMA kernel where its tiling can go wrong: block remainders, numbers of terms (entries leave the
rounds of the residual sum block by block), launches of few chunks (several CTAs per chunk), features in slices, entries that are not finite."""
import numpy as np
import pytest
import torch

from oracle import gdn_oracle as orc
from paper_2606_06034_b200 import binding as gdn
from paper_2606_06034_b200 import inputs as gen

pytestmark = pytest.mark.gpu

TOL = 1e-5  # relative Frobenius error per chunk: sums of at most 128 fp32 terms (2^-24 each) with room for their growth


def _compare(inp, N=-1, S=-1):
    W, U, T = gdn.chunk_prepare(inp.K.cuda(), inp.V.cuda(), inp.beta.cuda(), inp.g.cuda(), inp.C, N, S)
    sl = gen.chunk_slices(inp, range(inp.n_chunks))
    ref = orc.chunk_prepare(*(np.stack([s[k] for s in sl]) for k in range(4)), None if N < 0 else N, None if S < 0 else S)
    n, C = inp.n_chunks, inp.C
    for got, want in zip((W.reshape(n, C, -1), U.reshape(n, C, -1), T.reshape(n, C, C)), ref):
        assert orc.rel_frobenius(got.double().cpu().numpy(), want).max() <= TOL


@pytest.mark.parametrize("C", [2, 7, 8, 9, 16, 17, 24, 25, 31, 32, 33, 47, 48, 49, 63, 64, 128])
@pytest.mark.parametrize("d_k,d_v", [(8, 72), (136, 128), (256, 40)])
def test_sizes(C, d_k, d_v):
    _compare(gen.make_inputs(1, 1, 3, 2 * C, C, d_k, d_v, seed=C + d_k, dtype=torch.float32))


@pytest.mark.parametrize("C", [32, 64, 128])
@pytest.mark.parametrize("N", [1, 3, 20])
@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 6, 9, 10, 12, 15])
def test_numbers_of_terms(C, N, S):
    """Correlated keys without decay, beta = 0.3: the series has not converged and every term shows."""
    inp = gen.make_inputs(1, 1, 1, C, C, 64, 64, seed=S, dtype=torch.float32, adversarial_heads="all")
    inp.beta.fill_(0.3)
    _compare(inp, N, S)


@pytest.mark.parametrize("n", [1, 37, 38, 74, 75])
@pytest.mark.parametrize("C,d_k,d_v", [(64, 128, 128), (64, 200, 72), (24, 64, 136), (128, 128, 64)])
def test_few_chunks(n, C, d_k, d_v):
    """One, two or four CTAs per chunk: the same bits, as every chunk of the launch is an independent problem."""
    inp = gen.make_inputs(1, 1, 1, n * C, C, d_k, d_v, seed=n, dtype=torch.float32)
    dev = [x.cuda() for x in (inp.K, inp.V, inp.beta, inp.g)]
    got = gdn.chunk_prepare(*dev, C)
    many = gdn.chunk_prepare(*(x.repeat(160, *[1] * (x.dim() - 1)) for x in dev), C)
    for a, b in zip(got, many):
        assert torch.equal(a[0], b[0]) and torch.equal(a[0], b[-1])
    _compare(inp)


@pytest.mark.parametrize("C,at", [(16, 8), (33, 14), (64, 24), (128, 45), (128, 64), (128, 74), (128, 101), (128, 127)])
@pytest.mark.parametrize("what", ["K", "V"])
def test_tokens_before_one_that_is_not_finite(C, at, what):
    inp = gen.make_inputs(1, 1, 1, C, C, 128, 128, seed=5, dtype=torch.float32)
    clean = gdn.chunk_prepare(inp.K.cuda(), inp.V.cuda(), inp.beta.cuda(), inp.g.cuda(), C)
    for value in (float("nan"), float("inf")):
        K, V = inp.K.clone(), inp.V.clone()
        (K if what == "K" else V)[0, 0, at, 3] = value
        W, U, T = gdn.chunk_prepare(K.cuda(), V.cuda(), inp.beta.cuda(), inp.g.cuda(), C)
        for got, want in ((W[0, 0, :at], clean[0][0, 0, :at]), (U[0, 0, :at], clean[1][0, 0, :at]), (T[0, 0, 0, :at], clean[2][0, 0, 0, :at])):
            assert torch.isfinite(got).all()
            assert (got - want).abs().max().item() <= 1e-5  # (the order of the sums differs)
        # and the entries of the inverse that no sum takes over that token: columns behind it
        assert torch.isfinite(T[0, 0, 0, :, at + 1:]).all()
        assert not torch.isfinite(U[0, 0, at]).all() and (what == "V" or not torch.isfinite(W[0, 0, at]).all())


@pytest.mark.parametrize("C,d", [(64, 96), (64, 72), (48, 200), (24, 40), (32, 136), (128, 96)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_calls_do_not_depend_on_what_ran_before(C, d, dtype):
    """Feature sizes that end inside a unit of columns (64, 32 for chunks up to 32), after a launch that has left zeros in the
    shared memory of every SM and after one that has left NaN: the same bits, and no second evaluation of the outputs (which takes
    four times as long at C = 128, twice at 64)."""
    inp = gen.make_inputs(1, 1, 1, 600 * C, C, d, d, seed=d, dtype=dtype)
    dev = [x.cuda() for x in (inp.K, inp.V, inp.beta, inp.g)]
    out, time = [], []
    for left in (0.0, float("nan")):
        fill = [torch.full((1, 1, 600 * C, 128), left, device="cuda") for _ in range(2)]
        runs = []
        for _ in range(9):
            gdn.chunk_prepare(*fill, dev[2], dev[3], C)
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            res = gdn.chunk_prepare(*dev, C)
            b.record()
            torch.cuda.synchronize()
            runs.append(a.elapsed_time(b))
        out.append(res)
        time.append(min(runs))
    for a, b in zip(*out):
        assert torch.equal(a, b)
    assert time[1] < 1.5 * time[0]


@pytest.mark.parametrize("variant", [gdn.GDN_FWDSUBST_ROWS, gdn.GDN_FWDSUBST_BLOCKED])
def test_forward_substitution_over_two_blocks_costs_its_terms(variant):
    """A column of 128 rows has four times the terms of one of 64 and there are as many columns, so the same tokens take about four
    times as long; two block matrices addressed entry by entry took twelve times."""
    time = []
    for C in (64, 128):
        inp = gen.make_inputs(1, 1, 1, 128000, C, 64, 64, seed=C)
        dev = [x.cuda() for x in (inp.K, inp.V, inp.beta, inp.g)]
        runs = []
        for _ in range(7):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            gdn.chunk_prepare(*dev, C, method="fwdsubst", variant=variant)
            b.record()
            torch.cuda.synchronize()
            runs.append(a.elapsed_time(b))
        time.append(min(runs))
    assert time[1] < 6 * time[0]


@pytest.mark.parametrize("C,method", [(17, "neumann"), (24, "neumann"), (25, "neumann"), (32, "neumann"), (23, "fwdsubst"), (32, "fwdsubst")])
@pytest.mark.parametrize("d_k,d_v", [(128, 128), (136, 72), (72, 200)])
@pytest.mark.parametrize("flags", [0, gdn.GDN_FLAG_K_L2NORM | gdn.GDN_FLAG_W_GATED])
def test_many_chunks_read_the_keys_again(C, method, d_k, d_v, flags):
    """Launches of more chunks than fit at once read K a second time for W: the bits of a launch of one chunk."""
    inp = gen.make_inputs(1, 1, 1, C, C, d_k, d_v, seed=C, dtype=torch.float32)
    dev = [x.cuda() for x in (inp.K, inp.V, inp.beta, inp.g)]
    one = gdn.chunk_prepare(*dev, C, method=method, flags=flags)
    many = gdn.chunk_prepare(*(x.repeat(1300, *[1] * (x.dim() - 1)) for x in dev), C, method=method, flags=flags)
    for a, b in zip(one, many):
        assert torch.equal(a.expand_as(b), b)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("C,method,flags", [(C, "neumann", f) for C in (17, 24, 32) for f in (
    0, gdn.GDN_FLAG_G_RAW, gdn.GDN_FLAG_G_RAW | gdn.GDN_FLAG_K_L2NORM | gdn.GDN_FLAG_W_GATED)] + [(32, "fwdsubst", 0)])
def test_keys_read_again_are_the_chunks_own(dtype, C, method, flags):
    """1080 different chunks in one launch (K read again) and the same batches in launches of 360 (K kept): the same bits. Grouped
    heads, several chunks per sequence, raw gates, features of an odd slice, both tensor types."""
    B, H_k, H_v, n = 36, 2, 6, 5
    r = torch.Generator(device="cuda").manual_seed(C + flags)
    rand = lambda *s: torch.randn(*s, generator=r, device="cuda")
    K = torch.nn.functional.normalize(rand(B, H_k, n * C, 136), dim=-1).to(dtype)
    V, beta = rand(B, H_v, n * C, 72).to(dtype), torch.sigmoid(rand(B, H_v, n * C))
    g = -torch.nn.functional.softplus(rand(B, H_v, n * C))
    if not flags & gdn.GDN_FLAG_G_RAW:
        g = g.view(B, H_v, n, C).cumsum(-1).view(B, H_v, n * C)
    many = gdn.chunk_prepare(K, V, beta, g, C, method=method, flags=flags)
    for b in range(0, B, 12):
        few = gdn.chunk_prepare(K[b:b + 12], V[b:b + 12], beta[b:b + 12], g[b:b + 12], C, method=method, flags=flags)
        for x, y in zip(many, few):
            assert torch.equal(x[b:b + 12], y)
    assert gdn.gdn_device_status() == gdn.GDN_OK
