"""What the tests beside it leave open: the bits of decompressed values, signs of
zero among them; the outlier list of a small batch that overflows; both bounds of
the corrected histograms on grids of few rows."""
import numpy as np
import pytest

import oracle
from paper_2212_10733_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.fixture(scope="module")
def aq():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2212_10733_gb300 import aeqc
    aeqc.load()
    return aeqc


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV)


@pytest.mark.parametrize("grid", [(39, 39), (32, 39), (17, 30)])
@pytest.mark.parametrize("tau", [1e-4, 0.3, 1e-30, 4e-300])
def test_bits_of_decompressed_values(aq, grid, tau):
    """f = fl(fl(fl(xhat + q Delta) a) b) with the sign of every zero and the place
    of every NaN, for decoded values of all signs and sizes; a is read off the
    point whose x' is 1, with lambda_0 alone so that b = 1."""
    P, n = grid[0] * grid[1], 24
    rng = np.random.default_rng(7)
    mu = (rng.standard_normal(P) * 2.0 ** rng.uniform(-60, 20, P)).astype(np.float32)
    mu[:40] *= np.float32(2.0 ** -100)
    mu[40:60] = 0.0
    mu[60:80] = -0.0
    dl = 2.0 ** np.floor(np.log2(tau))
    q = np.rint(rng.standard_normal((n, P)) * 10.0 ** rng.uniform(0, 4.4, (n, 1))).astype(np.int16)
    q[:, 5::50] = oracle.ZERO_CODE
    q[:, 7::30] = 0
    q[:, 40:80:2] = 0
    if 1e-30 <= tau < 1:  # decoded values on the code lattice: exact cancellation
        mu[9::20] = (-q[0, 9::20].astype(np.float64) * dl).astype(np.float32)
    mu[100:106] = [0.0, -0.0, np.inf, np.nan, -np.inf, 1e-45]
    mu[0], q[:, 0] = 1.0, 0
    lam = np.zeros((n, 4))
    lam[1:, 0] = rng.standard_normal(n - 1) * 10.0 ** rng.uniform(-12, 0.5, n - 1)
    m = aq.Model(P, 32, 8)
    z = lambda *s: np.zeros(s)  # noqa: E731
    m.set_group(0, dict(W1=z(P, 32), b1=z(32), W2=z(32, 8), b2=z(8), b3=z(32), b4=z(P),
                        mu=mu.astype(np.float64), sigma=np.ones(P)))
    c = aq.Compressed(n, P, 8, torch.float32, DEV, 16)
    c.latent.zero_()
    c.scale.fill_(1.0)
    c.codes.copy_(dev(q))
    c.lam.copy_(dev(lam))
    c.status.copy_(dev(np.ones(n, np.uint16)))
    g = aq.Grid(*synth.grid_arrays(*grid))
    f = aq.decompress_batch(m, g, c, aq.params_default(tau=tau)).cpu().numpy()
    xhat = aq.ae_decode(m, c.latent, c.scale)[:, :P].cpu().numpy()
    with np.errstate(invalid="ignore", over="ignore"):
        xp = np.where(q == oracle.ZERO_CODE, 0.0,
                      xhat.astype(np.float64) + q.astype(np.float64) * dl)
        want = xp * f[:, :1]
    nan = np.isnan(want)
    assert nan.any() and (want[~nan] == 0).any()
    np.testing.assert_array_equal(np.isnan(f), nan)
    np.testing.assert_array_equal(f.view(np.int64)[~nan], want.view(np.int64)[~nan])


@pytest.mark.parametrize("n,grid,cap", [(90, (37, 33), 50), (40, (39, 39), 2000), (60, (8, 8), 0),
                                        (20, (5, 4), 7)])
def test_outlier_list_of_a_small_batch_overflows(aq, n, grid, cap):
    """The count is that of all escapes; the entries that fit are different points
    of the batch with their values; nothing is written behind them; a histogram has
    the overflow bit if its entries do not all fit, and those that have none do
    not."""
    P, tau = grid[0] * grid[1], 1e-4
    x = synth.histograms(n, 33, grid=grid)
    xh = synth.stand_in_xhat(x, 3)
    for r in range(0, n, 4):
        xh[r, : P // 3] = np.float32(1e9)       # escapes
    for r in range(1, n, 8):
        x[r, 2] = np.nan                        # stored verbatim
    o = aq.Compressed(n, P, 1, torch.float32, DEV, cap + 4096)
    o.index.fill_(-77)
    o.value.fill_(-77.0)
    o.c.outliers.capacity = cap
    aq.quantize_correct(aq.Grid(*synth.grid_arrays(*grid)), dev(x), dev(xh),
                        aq.params_default(tau=tau, kernel=aq.KERNEL_FP64), out=o)
    torch.cuda.synchronize()
    codes, st = o.codes.cpu().numpy(), o.status.cpu().numpy()
    per_row = (codes == oracle.ESCAPE).sum(axis=1)
    total = int(o.count.item())
    assert total == per_row.sum() > cap
    idx, val = o.index.cpu().numpy(), o.value.cpu().numpy()
    assert (idx[cap:] == -77).all() and (val[cap:] == -77.0).all()
    idx, val = idx[:cap], val[:cap]
    # the list is filled in whatever order histograms come, so some of its places
    # belong to one that does not fit as a whole: every place below cap is written
    assert len(np.unique(idx)) == cap and ((idx >= 0) & (idx < n * P)).all()
    assert (codes.reshape(-1)[idx] == oracle.ESCAPE).all()
    np.testing.assert_array_equal(val.view(np.int64), x.reshape(-1)[idx].view(np.int64))
    listed = np.bincount(idx // P, minlength=n)
    over = (st & aq.ST_OUTLIER_OVERFLOW) != 0
    np.testing.assert_array_equal(over, listed < per_row)


@pytest.mark.parametrize("kernel", ["fast", "fp64"])
@pytest.mark.parametrize("grid", [(33, 5), (2, 2), (4, 4), (32, 2), (20, 30)])
def test_bounds_on_grids_of_few_rows(aq, grid, kernel):
    """On grids whose systems are close to singular the multipliers themselves are
    not compared; what they are for is: every point within the bound and every
    moment within qoi_check of its target, with sums in extended precision."""
    P, n, tau = grid[0] * grid[1], 203, 1e-3
    vpar, vperp, vol = synth.grid_arrays(*grid)
    x = synth.histograms(n, 78, grid=grid)
    xh = np.zeros((n, aq.XHAT_LD), np.float32)
    xh[:, :P] = synth.stand_in_xhat(x, 6)[:, :P]
    p = aq.params_default(tau=tau,
                          kernel=aq.KERNEL_FAST if kernel == "fast" else aq.KERNEL_FP64)
    o = aq.quantize_correct(aq.Grid(vpar, vperp, vol), dev(x), dev(xh), p,
                            outlier_capacity=n * P, want_f=True)
    f = o.f.cpu().numpy().astype(np.longdouble)
    st = o.status.cpu().numpy()
    assert np.all(np.abs(f - x) <= tau * x.max(axis=1, keepdims=True) * (1 + 1e-15))
    v = np.tile(vpar, grid[1]).astype(np.longdouble)
    w = np.repeat(np.square(vperp), grid[0]).astype(np.longdouble)
    phi = np.stack([np.ones(P, np.longdouble), v, w, v * v], axis=1)
    g = np.abs((f - x) @ phi) * vol
    s = (np.abs(x).astype(np.longdouble) @ np.abs(phi)) * vol
    assert np.all(g <= 1.0001e-10 * s)
    assert ((st & (oracle.CONVERGED | oracle.ROUND2 | oracle.VERBATIM)) != 0).all()
