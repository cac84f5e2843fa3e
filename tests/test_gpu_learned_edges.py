"""The learned-guess kernels at the edges of their tiles and ranges: one
sample, tile remainders, more tiles than pipelines; features of values that
the FP64 -> FP32 narrowing treats apart; statistics of a handful of samples
and targets outside the logarithm's fast range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2311_08927_gb300 import chad as CH  # noqa: E402
from paper_2311_08927_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_08927_gb300 import build
    build.build()


def _net(P, X):
    w = torch.split(P, [2048, 64, 4096, 64, 128, 2])
    bf = lambda t: t.to(torch.bfloat16).double()
    silu = torch.nn.functional.silu
    a = silu(X @ bf(w[0]).view(64, 32).T + w[1])
    a = silu(a @ bf(w[2]).view(64, 64).T + w[3])
    return a @ bf(w[4]).view(2, 64).T + w[5]


def _data(n, seed=3):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    P = 0.15 * torch.randn(CH.MLP_NPARAM, generator=g, device="cuda")
    X = torch.randn((n, 32), generator=g, device="cuda").to(torch.bfloat16)
    Y = torch.randn((n, 2), generator=g, device="cuda")
    return P, X, Y


# BF16 activations: 2^-9 relative per unit, 64 units of two layers; the
# gradient adds the BF16 rounding of dZ.  1e-2 as for the whole batches.
@pytest.mark.parametrize("tiles,extra", [(0, 1), (0, 127), (1, 0), (1, 1), (152, 1), (304, 5), (608, 77)])
def test_forward_and_gradient_at_tile_edges(tiles, extra):
    n = 128 * tiles + extra
    P, X, Y = _data(n)
    bits = X.view(torch.int16)
    out = torch.empty((n, 2), device="cuda")
    CH.chad_mlp_forward(bits, P, out)
    Pd = P.double().requires_grad_()
    ref = _net(Pd, X.double())
    assert (out - ref).norm() <= 1e-2 * ref.norm()
    loss = (ref - Y.double()).square().sum(1).mean()
    (g_ref,) = torch.autograd.grad(loss, Pd)
    grad, lv = torch.zeros_like(P), torch.zeros(1, device="cuda")
    scratch = torch.empty(CH.mlp_grad_scratch_bytes(n) // 4 + 1, device="cuda")
    CH.chad_mlp_grad(bits, Y, P, grad, lv, scratch)
    again = torch.zeros_like(P)
    CH.chad_mlp_grad(bits, Y, P, again, lv, scratch)
    assert torch.equal(grad, again)
    assert abs(lv.item() - loss.item()) <= 1e-2 * loss.item()
    for a, b in zip(torch.split(grad.double(), [2048, 64, 4096, 64, 128, 2]),
                    torch.split(g_ref, [2048, 64, 4096, 64, 128, 2])):
        assert (a - b).norm() <= 1e-2 * b.norm() + 1e-3 * g_ref.norm()


@pytest.mark.parametrize("aligned", [True, False])
def test_features_of_special_values(aligned):
    """log10 of the float nearest each state: halfway cases round to even,
    below the floor, zero, negative and NaN give the floor, an infinity (or
    a double beyond the float range) an infinity."""
    half = 1.0 + 2.0 ** -24
    special = [0.0, -1.0, np.nan, 1e-300, 1e-20, 9.9e-21, 1.17e-38, 2.0 ** -126, half, 1.0 + 3 * 2.0 ** -24,
               np.nextafter(half, 2), np.nextafter(half, 0), 1e-7, 25.0, 3e38, 3.5e38, 1e300, np.inf]
    n = len(special)
    y = np.ones((I.NS, n))
    y[0], y[28] = special, special
    T = np.linspace(250.0, 390.0, n)
    norm = torch.zeros(64, device="cuda")
    norm[32:] = 1.0
    buf = torch.zeros(n * 32 + 8, dtype=torch.int16, device="cuda")
    X = buf[:n * 32].view(n, 32) if aligned else buf[1:n * 32 + 1].view(n, 32)
    CH.chad_mlp_features(torch.from_numpy(y).cuda(), torch.from_numpy(T).cuda(), norm, X)
    got = X.clone().view(torch.bfloat16).float().cpu().numpy()
    with np.errstate(all="ignore"):
        f = np.fmax(y.astype(np.float32), np.float32(1e-20)).astype(np.float64)
        ref = np.concatenate([np.log10(f), T[None].astype(np.float32) * 0.01]).T
    assert np.array_equal(np.isinf(got[:, :30]), np.isinf(ref))
    ok = np.isfinite(ref)
    # BF16's unit roundoff with its 8 significant bits is 2^-8; the float
    # logarithm's last place comes on top
    assert np.all(np.abs(got[:, :30][ok] - ref[ok]) <= 2.0 ** -8 * np.abs(ref[ok]) + 1e-7)
    assert np.all(got[:, 30:] == 0)


@pytest.mark.parametrize("n", [2, 3, 127, 129, 1025, 200_003])
def test_statistics_of_few_and_many_samples(n):
    rng = np.random.default_rng(n)
    y = I.x_ss()[:, None] * np.exp(0.3 * rng.standard_normal((I.NS, n)))
    y[5] = y[5, 0]                       # a constant feature: std at its floor
    y[6] = 10.0 ** rng.uniform(-30, 30, n)
    T = rng.uniform(303.15, 313.15, n)
    SH = 10.0 ** rng.uniform(-300, 2, n)
    h = 10.0 ** rng.uniform(-10, 0, n)
    SH[0] = 5e-324                       # subnormal: the general logarithm
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    sc = torch.empty(CH.mlp_prep_scratch_bytes() // 8 + 1, dtype=torch.float64, device="cuda")
    norm = torch.empty(64, device="cuda")
    CH.chad_mlp_feature_norm(d(y), d(T), norm, sc)
    f = np.vstack([np.log10(np.maximum(y.astype(np.float32), np.float32(1e-20))).astype(np.float64),
                   (T.astype(np.float32) * np.float32(0.01)).astype(np.float64)])
    nm = norm.cpu().numpy()
    sd = np.maximum(f.std(1, ddof=1), 1e-6)
    np.testing.assert_allclose(nm[:30], f.mean(1), rtol=2e-6, atol=2e-7)
    # the float logarithm's last place (6e-8 of up to 20) against the spread
    np.testing.assert_allclose(nm[32:62], 1.0 / sd, rtol=1e-5 + np.max(2e-6 / sd[sd > 1e-5]))
    Y, on = torch.empty((n, 2), device="cuda"), torch.empty(4, device="cuda")
    CH.chad_mlp_targets(d(SH), d(h), Y, on, sc)
    t = np.vstack([np.log10(SH), np.log10(h)])
    o = on.cpu().numpy()
    np.testing.assert_allclose(o[:2], t.mean(1), rtol=1e-6, atol=1e-6)
    np.testing.assert_allclose(o[2:], t.std(1, ddof=1), rtol=1e-5)
    ref = (t.T.astype(np.float32) - o[:2]) / o[2:]
    np.testing.assert_allclose(Y.cpu().numpy(), ref, rtol=1e-5, atol=1e-5)


# The standard deviation of n values moves by at most the largest error of one
# of them: log10f's two last places of the largest value (equal values carry
# equal errors; the temperature's float product has none).  The FP64 joins of
# sum and sum of squares round at most a hundred times by 1.1e-16 of the mean
# square (some 30 roundings in each of b, a and mu), the float results by 6e-8.
@pytest.mark.parametrize("n", [300, 100_003])
@pytest.mark.parametrize("spread", [0.0, 2e-6, 1e-5, 1e-4])
def test_statistics_of_nearly_constant_features(n, spread):
    rng = np.random.default_rng(n)
    centre = np.linspace(-0.1, 0.1, I.NS)
    centre[:5] = [0.0, 1e-3, 0.05, np.log10(0.866), np.log10(I.x_ss()[I.SIDX["X_aa"]])]
    y = 10.0 ** (centre[:, None] + spread * rng.standard_normal((I.NS, n)))
    T = 308.15 + 100.0 * spread * rng.standard_normal(n)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    sc = torch.empty(CH.mlp_prep_scratch_bytes() // 8 + 1, dtype=torch.float64, device="cuda")
    norm = torch.empty(64, device="cuda")

    def check(T):
        CH.chad_mlp_feature_norm(d(y), d(T), norm, sc)
        f = np.vstack([np.log10(y.astype(np.float32).astype(np.float64)),
                       (T.astype(np.float32) * np.float32(0.01)).astype(np.float64)])
        nm = norm.cpu().numpy().astype(np.float64)
        sd = np.maximum(f.std(1, ddof=1), 1e-6)
        last = 2.0 * np.spacing(np.abs(f).max(1).astype(np.float32)).astype(np.float64)
        last[29] = 0.0
        assert np.all(np.abs(nm[:30] - f.mean(1)) <= last + 1e-6 * np.abs(f.mean(1)))
        got = 1.0 / nm[32:62]
        moved = last if spread > 0 else 0.0
        var_tol = 100 * 1.1e-16 * (f ** 2).mean(1)
        assert np.all(got ** 2 <= (sd * (1 + 1e-6) + moved) ** 2 + var_tol), got / sd
        assert np.all(got ** 2 >= np.maximum(sd * (1 - 1e-6) - moved, 0.0) ** 2 - var_tol), got / sd

    check(T)
    check(T + 1.0e4)  # far above any digester's, still a number
