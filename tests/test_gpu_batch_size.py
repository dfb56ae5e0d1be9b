"""A histogram's result does not depend on how many others its call has: the
FP64 kernel gives a few histograms to clusters of blocks and many to warps, and
both forms have the same bits (codes, scales, multipliers, step counts,
statuses, corrected values).  Nothing here has a tolerance."""
import numpy as np
import pytest

from paper_2212_10733_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"
FIELDS = ("codes", "scale", "lam", "iters", "status")
MANY = 1000


@pytest.fixture(scope="module")
def aq():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2212_10733_gb300 import aeqc
    aeqc.load()
    return aeqc


def bits(t):
    a = t.cpu().contiguous()
    return {8: lambda: a.view(torch.int64), 4: lambda: a.view(torch.int32),
            2: lambda: a.view(torch.int16), 1: lambda: a}[a.element_size()]().numpy()


def batch(n, grid, tau, seed):
    """Histograms and decoded rows with every course of the correction among
    them: zero and invalid rows, escapes, retries, verbatim rows, -0."""
    P = grid[0] * grid[1]
    x = synth.histograms(n, seed, grid=grid)
    xh = np.zeros((n, 1536), np.float32)
    xh[:, :P] = synth.stand_in_xhat(x, seed)[:, :P]
    rng = np.random.default_rng(seed)
    for r in range(3, n, 9):
        c = rng.integers(0, P)
        k = (r // 9) % 8
        if k == 0:
            x[r] = 0.0
        elif k == 1:
            x[r, c] = np.nan
        elif k == 2:
            x[r, c] = -1e-3
        elif k == 3:
            xh[r, c] = np.inf
        elif k == 4:
            xh[r, :P] += np.float32(3e4 * tau * x[r].max())
        elif k == 5:
            xh[r, : P // 2] = np.float32(1e9)
        elif k == 6:  # every point a little off: the bound fails at both levels
            xh[r, :P] = (x[r] + 0.49 * tau * x[r].max()).astype(np.float32)
        else:
            x[r, c] = -0.0
    return torch.as_tensor(x, device=DEV), torch.as_tensor(xh, device=DEV)


@pytest.mark.parametrize("n", [1, 7, 58, 320, 321])
@pytest.mark.parametrize("grid,tau,options", [
    ((39, 39), 1e-4, {}),
    ((39, 39), 1e-3, {"step_s": 0.9}),
    ((37, 33), 1e-3, {}),
    ((32, 48), 1e-3, {}),      # every point of the largest histogram
    ((64, 24), 1e-2, {}),
    ((20, 20), 1e-3, {"max_iter": 2}),
    ((10, 10), 1e-3, {}),
    ((5, 3), 1e-3, {}),
    ((2, 7), 1e-4, {"tol": 1e-9}),
])
def test_fp64_form_of_a_few_and_of_many(aq, grid, tau, options, n):
    g = aq.Grid(*synth.grid_arrays(*grid))
    P = grid[0] * grid[1]
    x, xh = batch(MANY, grid, tau, 60 + grid[0])
    p = aq.params_default(tau=tau, kernel=aq.KERNEL_FP64, **options)
    many = aq.quantize_correct(g, x, xh, p, outlier_capacity=MANY * P, want_f=True)
    few = aq.quantize_correct(g, x[:n].contiguous(), xh[:n].contiguous(), p,
                              outlier_capacity=n * P, want_f=True)
    torch.cuda.synchronize()
    for name in FIELDS:
        np.testing.assert_array_equal(bits(getattr(few, name)), bits(getattr(many, name)[:n]),
                                      err_msg=name)
    np.testing.assert_array_equal(bits(few.f), bits(many.f[:n]), err_msg="f")


@pytest.mark.parametrize("grid,line", [((7, 9), 63), ((8, 8), 47), ((10, 10), 51),
                                       ((39, 25), 148), ((39, 39), 209)])
def test_fp64_form_on_both_sides_of_the_line(aq, grid, line):
    """The number of histograms that clusters take depends on the points of one."""
    g = aq.Grid(*synth.grid_arrays(*grid))
    P = grid[0] * grid[1]
    x, xh = batch(line + 1, grid, 1e-3, 17)
    p = aq.params_default(tau=1e-3, kernel=aq.KERNEL_FP64)
    a, b = (aq.quantize_correct(g, x[:n].contiguous(), xh[:n].contiguous(), p,
                                outlier_capacity=n * P, want_f=True) for n in (line, line + 1))
    torch.cuda.synchronize()
    for name in FIELDS + ("f",):
        np.testing.assert_array_equal(bits(getattr(a, name)), bits(getattr(b, name)[:line]),
                                      err_msg=name)


@pytest.mark.parametrize("grid", [(39, 39), (20, 20)])
@pytest.mark.parametrize("tau,n,piece", [(1e-4, 5000, 1250), (1e-3, 5000, 1250), (1e-2, 900, 300)])
def test_fast_form_in_pieces(aq, grid, tau, n, piece):
    """The fast kernel's deferred list is above the limit in one call and below
    it in the pieces (at the larger bounds)."""
    g = aq.Grid(*synth.grid_arrays(*grid))
    x, xh = batch(n, grid, tau, 5)
    p = aq.params_default(tau=tau, kernel=aq.KERNEL_FAST)
    whole = aq.quantize_correct(g, x, xh, p, outlier_capacity=4 << 20, want_f=True)
    for at in range(0, n, piece):
        part = aq.quantize_correct(g, x[at:at + piece], xh[at:at + piece], p,
                                   outlier_capacity=4 << 20, want_f=True)
        torch.cuda.synchronize()
        for name in FIELDS + ("f",):
            np.testing.assert_array_equal(bits(getattr(part, name)),
                                          bits(getattr(whole, name)[at:at + piece]),
                                          err_msg="%s from %d" % (name, at))


@pytest.mark.parametrize("kernel,tau,chunk", [("fp64", 1e-4, 4800), ("fast", 1e-3, 1536)])
def test_host_stream_with_a_short_tail(aq, kernel, tau, chunk):
    """compress_batch_host's promise where the chunks lie on both sides of the limit."""
    P, H, L, n = 1521, 64, 16, 5000
    x = torch.as_tensor(synth.histograms(n, synth.config_seed(1) + 56))
    m = aq.Model(P, H, L, dtype=aq.DTYPE_F32)
    m.set_group(0, synth.ae_init(P, H, L, 9))
    m.fit_normalizer(0, x[8:72].to(DEV))
    grid = aq.Grid(*synth.grid_arrays())
    p = aq.params_default(tau=tau, kernel=aq.KERNEL_FAST if kernel == "fast" else aq.KERNEL_FP64)
    ref = aq.compress_batch(m, grid, x.to(DEV), p, outlier_capacity=1 << 20)
    got = aq.compress_batch_host(m, grid, x.pin_memory(), p, chunk=chunk, outlier_capacity=1 << 20)
    torch.cuda.synchronize()
    for name in ("latent",) + FIELDS:
        np.testing.assert_array_equal(bits(getattr(got, name)), bits(getattr(ref, name)),
                                      err_msg=name)
