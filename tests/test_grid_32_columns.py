"""Grids of exactly 32 v_par columns: a lane of the fast correction kernel walks
one column and no columns are left over.  (The host set-up divided by the number
of those left over, which ended the process with SIGFPE on x86.)"""
import ctypes as C
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2212_10733_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


class GridK(C.Structure):
    _fields_ = [("n_par", C.c_int), ("n_perp", C.c_int), ("P", C.c_int), ("has_vol", C.c_int),
                ("vol", C.c_void_p), ("vol_uniform", C.c_double), ("vpar", C.c_double * 64),
                ("vperp2", C.c_double * 64)]


class FastGridK(C.Structure):
    _fields_ = [("ok", C.c_int), ("i_c", C.c_int), ("b", C.c_double), ("c0", C.c_double),
                ("d2", C.c_double), ("vol", C.c_float * 2), ("d2q", C.c_float * 6),
                ("coef", C.c_float * 50), ("bc_f", C.c_float * 2), ("vw_max", C.c_float * 2),
                ("wk", C.c_float * 4), ("seg_nchunk", C.c_int), ("seg_rpc", C.c_int),
                ("seg_mul", C.c_int)]


def segments(n_par, n_perp):
    """ok and the lane segments of make_fast_grid for a uniform grid."""
    from paper_2212_10733_gb300 import aeqc
    vpar, vperp, vol = synth.grid_arrays(n_par, n_perp)
    g, f = GridK(n_par, n_perp, n_par * n_perp, 0, None, vol), FastGridK()
    g.vpar[:n_par] = list(vpar)
    g.vperp2[:n_perp] = list(np.square(vperp))
    make = getattr(aeqc.load(), "_ZN4aeqc14make_fast_gridERKNS_5GridKEPNS_9FastGridKE")
    assert make(C.byref(g), C.byref(f)) == 0
    return f.ok, f.seg_nchunk, f.seg_rpc, f.seg_mul


@pytest.mark.parametrize("grid", [(31, 39), (32, 39), (32, 2), (33, 39), (64, 24), (2, 2)])
def test_lane_segments_of_the_host_set_up(grid):
    """In a process of its own: a signal there is a failure here."""
    from paper_2212_10733_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c",
                        "import sys; sys.path.insert(0, 'tests');"
                        "from test_grid_32_columns import segments;"
                        "print(*segments(%d, %d))" % grid],
                       cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])
    ok, nchunk, rpc, mul = map(int, r.stdout.split())
    assert ok == 1
    rest = grid[0] % 32 if grid[0] < 64 else 32
    if rest == 0:
        assert (nchunk, rpc, mul) == (0, 0, 0)
        return
    assert nchunk == 32 // rest and nchunk * rpc >= grid[1]
    assert [(lane * mul) >> 16 for lane in range(32)] == [lane // rest for lane in range(32)]


@pytest.fixture(scope="module")
def aq():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2212_10733_gb300 import aeqc
    aeqc.load()
    return aeqc


@pytest.mark.gpu
@pytest.mark.parametrize("n_perp", [5, 39, 48])
def test_codes_and_values_on_32_columns(aq, n_perp):
    """Codes, scales and statuses of both kernels against the oracle's quantizer
    on every row, and decompression equal to compression bit for bit."""
    import torch
    P, n, tau = 32 * n_perp, 203, 1e-4
    x = synth.histograms(n, 31, grid=(32, n_perp))
    xh = synth.stand_in_xhat(x, 7)[:, :P].copy()
    x[5], x[7, 3], x[9, 2] = 0.0, np.nan, -1.0
    xh[11] = 0.0
    g = aq.Grid(*synth.grid_arrays(32, n_perp))
    pad = np.zeros((n, aq.XHAT_LD), np.float32)
    pad[:, :P] = xh
    xd, hd = torch.as_tensor(x).cuda(), torch.as_tensor(pad).cuda()
    o = [aq.quantize_correct(g, xd, hd, aq.params_default(tau=tau, kernel=k),
                             outlier_capacity=n * P, want_f=True)
         for k in (aq.KERNEL_FAST, aq.KERNEL_FP64)]
    for name in ("codes", "scale", "status"):
        a, b = (getattr(c, name).cpu().numpy() for c in o)
        np.testing.assert_array_equal(a, b, err_msg=name)
    st = o[0].status.cpu().numpy()
    s = o[0].scale.cpu().numpy()
    codes = o[0].codes.cpu().numpy()
    plain = (st & (oracle.VERBATIM | oracle.ALPHA_RETRY | oracle.ZERO_IMAGE)) == 0
    assert plain.sum() >= n - 12
    q = oracle.quantize(x[plain], xh[plain], tau)[0]
    np.testing.assert_array_equal(codes[plain], q)
    f = o[0].f.cpu().numpy()
    ok = np.isfinite(x).all(axis=1)
    assert np.all(np.abs(f - x)[ok] <= tau * s[ok, None] * (1 + 1e-12))
