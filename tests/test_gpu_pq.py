"""Product quantisation of the latents on the GPU against the oracle
(Sec. III Stage 3, Sec. V-B).

* The start table (no iteration) equals the oracle's bit for bit.
* Given a table, the codes equal the oracle's nearest-centroid decisions bit
  for bit (both in float32, ties to the lowest index), and decoding equals the
  table lookup.
* After Lloyd iterations the tables agree within the fixed-point resolution
  of the sums plus one float32 rounding, per subdomain, with ragged and empty
  subdomains, non-finite latents and bfloat16 latents.
* The whole pipeline with PQ'd latents (encode, quantise the latents, decode
  from the table, quantise the residual, correct) keeps every point within
  the bound and the moments to 1e-10."""
import numpy as np
import pytest

from oracle import pq as opq
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


def latents(n, L, seed):
    rng = np.random.default_rng(seed)
    scale = np.exp(rng.uniform(-3, 3, L))
    z = rng.standard_normal((n, L)) * scale + rng.uniform(-2, 2, L) * scale
    # a few clumps so that K-means has structure
    z[: n // 4] = np.round(z[: n // 4] / scale * 2) * scale / 2
    return z.astype(np.float32)


def table_tol(z, c):
    # fixed-point resolution of the sums (2^-62 of max|z| times the row
    # count) plus one float32 rounding of each centroid
    amax = np.nanmax(np.abs(np.where(np.isfinite(z), z, 0)), axis=0)[:, None]
    return amax * 2.0 ** (-62 + np.ceil(np.log2(max(len(z), 2)))) * 4 + np.spacing(np.abs(c))


@pytest.mark.parametrize("k", [16, 64, 256])
def test_start_table_and_codes_bit_exact(aq, k):
    n, L = 5000, 32
    z = latents(n, L, 1)
    zd = torch.as_tensor(z, device=DEV)
    t0 = aq.pq_train(zd, k=k, iters=0)
    np.testing.assert_array_equal(t0.cpu().numpy()[0], opq.init_centroids(z, k))
    ref = opq.train(z, k, 3)
    tab = torch.as_tensor(ref[None], device=DEV)
    zq = torch.empty_like(zd)
    codes, _ = aq.pq_encode(zd, tab, zq=zq)
    torch.cuda.synchronize()
    oc = opq.assign(z, ref)
    np.testing.assert_array_equal(codes.cpu().numpy(), oc)
    np.testing.assert_array_equal(zq.cpu().numpy(), opq.decode(oc, ref))
    dec = aq.pq_decode(codes, tab, torch.float32)
    np.testing.assert_array_equal(dec.cpu().numpy(), opq.decode(oc, ref))


@pytest.mark.parametrize("iters", [1, 10])
def test_lloyd_tables_match_oracle(aq, iters):
    n, L, k = 20000, 16, 16
    z = latents(n, L, 2)
    t = aq.pq_train(torch.as_tensor(z, device=DEV), k=k, iters=iters).cpu().numpy()[0]
    ref = opq.train(z, k, iters)
    if iters == 1:  # same start, same decisions: only the mean's rounding differs
        assert np.all(np.abs(t - ref) <= table_tol(z, ref))
    else:  # later decisions may flip at exact midpoints; the quantiser is as good
        codes = opq.assign(z, t)
        jg = opq.objective(z, codes, t)
        jo = opq.objective(z, opq.assign(z, ref), ref)
        assert abs(jg - jo) <= 1e-6 * jo
        assert np.mean(np.abs(t - ref) <= table_tol(z, ref)) > 0.99


def test_groups_ragged_empty_nonfinite_and_bf16(aq):
    L, k = 8, 16
    sizes = [3000, 0, 17, 1200]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    z = latents(int(off[-1]), L, 3)
    z[5, 2] = np.nan
    z[3010, 0] = np.inf
    zb = torch.as_tensor(z, device=DEV).to(torch.bfloat16)
    zf = zb.float().cpu().numpy()  # the values the GPU sees
    goff = torch.as_tensor(off, device=DEV)
    G = len(sizes)
    t = aq.pq_train(zb, k=k, iters=1, group_offsets=goff, G=G).cpu().numpy()
    ref = opq.train_grouped(zf, off, k, 1)
    for g in range(G):
        zg = zf[off[g]:off[g + 1]]
        if len(zg) == 0:
            np.testing.assert_array_equal(t[g], 0.0)
            continue
        assert np.all(np.abs(t[g] - ref[g]) <= table_tol(zg, ref[g])), g
    tab = torch.as_tensor(ref, device=DEV)
    zq = torch.empty_like(zb)
    codes, _ = aq.pq_encode(zb, tab, group_offsets=goff, zq=zq)
    torch.cuda.synchronize()
    for g in range(G):
        zg = zf[off[g]:off[g + 1]]
        oc = opq.assign(zg, ref[g])
        np.testing.assert_array_equal(codes.cpu().numpy()[off[g]:off[g + 1]], oc)
        want = torch.as_tensor(opq.decode(oc, ref[g])).to(torch.bfloat16).float().numpy()
        np.testing.assert_array_equal(zq.float().cpu().numpy()[off[g]:off[g + 1]], want)
    assert codes[5, 2].item() == 0 and codes[3010, 0].item() == 0


def test_argument_checks(aq):
    z = torch.zeros((10, 4), device=DEV)
    for bad in (dict(k=1), dict(k=257), dict(iters=-1)):
        with pytest.raises(aq.AeqcError):
            aq.pq_train(z, **{**dict(k=16, iters=1), **bad})
    with pytest.raises(aq.AeqcError):
        aq.pq_train(z, k=16, iters=1, G=2)  # G > 1 without offsets


def test_pipeline_with_pq_latents_keeps_the_bounds(aq):
    P, H, L, n, tau = 1521, 128, 16, 4000, 1e-4
    x = torch.as_tensor(synth.histograms(n, synth.config_seed(1) + 5), device=DEV)
    m = aq.Model(P, H, L, dtype=aq.DTYPE_BF16)
    m.set_group(0, synth.ae_init(P, H, L, 21))
    m.fit_normalizer(0, x[:512])
    ws = None
    for t in range(60):
        ws = m.train_step(x[(t * 64) % 3900:(t * 64) % 3900 + 64], lr=2e-3, ws=ws)
    z, s = aq.ae_encode(m, x)
    tab = aq.pq_train(z, k=16, iters=10)
    codes, _ = aq.pq_encode(z, tab, zq=z)  # z now holds the decoded latents
    xhat = aq.ae_decode(m, z, s)
    grid = aq.Grid(*synth.grid_arrays())
    p = aq.params_default(tau=tau, kernel=aq.KERNEL_FAST)
    out = aq.quantize_correct(grid, x, xhat, p, want_f=True, outlier_capacity=64 * P)
    torch.cuda.synchronize()
    st = out.status.cpu().numpy()
    ok = (st & aq.ST_VERBATIM) == 0
    assert ok.mean() > 0.99
    f, xx = out.f.cpu().numpy()[ok], x.cpu().numpy()[ok]
    e = tau * xx.max(axis=1, keepdims=True)
    assert np.all(np.abs(f - xx) <= e)
    vpar, vperp, vol = synth.grid_arrays()
    V, W = np.meshgrid(vpar, vperp)
    phi = np.stack([np.ones(P), V.ravel(), W.ravel() ** 2, V.ravel() ** 2])
    qf, qx = f @ phi.T * vol, xx @ phi.T * vol
    sk = np.abs(xx) @ np.abs(phi).T * vol
    assert np.max(np.abs(qf - qx) / sk) <= 1e-10


@pytest.mark.parametrize("k", [2, 3, 16, 33, 256])
def test_assignment_any_table(aq, k):
    """The bisection gives the index of the full search (and the oracle's) for
    every table a caller may pass: ascending, with equal or adjacent-float or
    descending neighbours, with infinities and NaN; at centroids, midpoints,
    their neighbouring floats, and values far outside the table."""
    rng = np.random.default_rng(k)
    L = 8
    t = np.sort(rng.standard_normal((L, k)).astype(np.float32), axis=1)
    t[1, k // 2] = t[1, k // 2 - 1]
    t[2, k // 2] = np.nextafter(t[2, k // 2 - 1], np.float32(9))
    t[3] = t[3][::-1]
    t[4] = (1e7 + np.arange(k)).astype(np.float32)
    t[5, -1] = np.inf
    t[6, 0] = np.nan
    t[7] = (t[7] * np.float32(1e-42)).astype(np.float32)
    with np.errstate(invalid="ignore", over="ignore"):
        mid = (t[:, :-1] + t[:, 1:]) / np.float32(2)
        cols = [t, mid, np.nextafter(mid, np.float32(9)), np.nextafter(mid, np.float32(-9)),
                np.nextafter(t, np.float32(9)), rng.standard_normal((L, 64)).astype(np.float32),
                np.tile(np.float32([0, -0.0, 1e30, -1e30, 3e38, np.inf, -np.inf, np.nan, 1e-45,
                                    16777216, 0.4]), (L, 1)),
                t[:, :1] - np.float32(4194304) * (t[:, 1:2] - t[:, :1]) *
                np.float32([[0.25, 0.5, 0.75, 1, 2]])]
        z = np.ascontiguousarray(np.concatenate(cols, axis=1).T.astype(np.float32))
        # the full search starts from centroid 0, whose NaN distance nothing beats
        ref = np.zeros(z.shape, np.uint8)
        best = np.abs(z - t[:, 0])
        for j in range(1, k):
            d = np.abs(z - t[:, j])
            ref[d < best] = j
            best = np.where(d < best, d, best)
        fin = ~np.isnan(t).any(axis=1)
        np.testing.assert_array_equal(ref[:, fin], opq.assign(z, t)[:, fin])
    codes, _ = aq.pq_encode(torch.as_tensor(z, device=DEV), torch.as_tensor(t[None], device=DEV))
    np.testing.assert_array_equal(codes.cpu().numpy(), ref)


@pytest.mark.parametrize("n,L", [(1, 32), (7, 16), (4097, 32), (3001, 5)])
def test_one_iteration_wide_magnitudes(aq, n, L):
    """Means of columns whose values span 40 binades, subnormals among them
    (shifts either side of the fixed point's last place), at row counts around
    the unrolled loads of a block."""
    rng = np.random.default_rng(n)
    z = (rng.standard_normal((n, L)) * 2.0 ** rng.uniform(-30, 10, (n, L))).astype(np.float32)
    z[:, L // 2] *= np.float32(2.0 ** -130)
    t = aq.pq_train(torch.as_tensor(z, device=DEV), k=16, iters=1).cpu().numpy()[0]
    ref = opq.train(z, 16, 1)
    assert np.all(np.abs(t - ref) <= table_tol(z, ref))


@pytest.mark.parametrize("n,L,G,k,kind", [
    (20000, 32, 1, 16, "normal"), (20000, 5, 2, 16, "normal"), (150000, 16, 2, 16, "normal"), (70000, 8, 1, 16, "patterns"), (3000, 16, 5, 16, "normal"),
    (70000, 8, 1, 256, "normal"), (200000, 3, 1, 16, "patterns"), (5000, 8, 1, 2, "offset")])
def test_bf16_counts_equal_values(aq, n, L, G, k, kind):
    """bfloat16 latents (counted by value) and the same values as float32
    (summed one by one) give the same tables bit for bit: few and very many
    distinct values, non-finite patterns, ragged groups, rows that are not
    multiples of eight elements, an unaligned first row."""
    rng = np.random.default_rng(n + L)
    if kind == "patterns":
        z = torch.as_tensor(rng.integers(0, 65536, (n + 1, L)).astype(np.uint16).view(np.int16),
                            device=DEV).view(torch.bfloat16)
    else:
        z = torch.as_tensor(latents(n + 1, L, n), device=DEV).to(torch.bfloat16)
    z = z[1:] if kind == "offset" else z[:n].contiguous()
    off = np.sort(np.concatenate([[0, n], rng.integers(0, n, G - 1)])).astype(np.int64)
    goff = torch.as_tensor(off, device=DEV) if G > 1 else None
    a = aq.pq_train(z, k=k, iters=6, group_offsets=goff, G=G)
    b = aq.pq_train(z.float(), k=k, iters=6, group_offsets=goff, G=G)
    np.testing.assert_array_equal(a.cpu().numpy().view(np.int32), b.cpu().numpy().view(np.int32))


@pytest.mark.parametrize("dtype", ["bfloat16", "float32"])
@pytest.mark.parametrize("n,L,G,k,iters", [(3000, 8, 1, 16, 4), (70000, 32, 2, 64, 2),
                                           (500, 1, 3, 2, 3), (900, 16, 1, 256, 1)])
def test_workspace_of_the_sums_alone(aq, n, L, G, k, iters, dtype):
    """A workspace with room for the iterations' sums only (keys, shifts, sums and
    member counts, each rounded to 256 bytes) is enough, with the same table; one
    byte less is refused, and nothing behind the given bytes is touched."""
    z = torch.as_tensor(latents(n, L, n), device=DEV).to(getattr(torch, dtype))
    off = torch.as_tensor(np.linspace(0, n, G + 1).astype(np.int64), device=DEV)
    goff = off if G > 1 else None
    want = aq.pq_train(z, k=k, iters=iters, group_offsets=goff, G=G)
    need = sum((b * G * L + 255) // 256 * 256 for b in (8, 4, 8 * k, 8 * k))
    ws = torch.full((need + 65536,), 0x5A, dtype=torch.uint8, device=DEV)
    got = torch.empty_like(want)

    def call(nbytes):
        aq._check(aq.load().pq_train(aq._ptr(z), aq._dtype_code(z.dtype), n, L, aq._ptr(goff), G,
                                     k, iters, aq._ptr(got), aq._ptr(ws), nbytes, aq._stream()))

    call(need)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(got.cpu().numpy().view(np.int32),
                                  want.cpu().numpy().view(np.int32))
    assert bool((ws[need:] == 0x5A).all())
    with pytest.raises(aq.AeqcError):
        call(need - 1)


@pytest.mark.parametrize("iters", [0, 1, 2])
@pytest.mark.parametrize("n,L,k", [(1, 32, 16), (1000, 7, 64), (65535, 32, 16), (65536, 32, 16)])
def test_few_iterations_counted_or_not(aq, n, L, k, iters):
    """bfloat16 latents and the same values as float32 give the same table bit for
    bit on both sides of the line from which they are counted."""
    z = torch.as_tensor(latents(n, L, n + iters), device=DEV).to(torch.bfloat16)
    a = aq.pq_train(z, k=k, iters=iters).cpu().numpy()
    b = aq.pq_train(z.float(), k=k, iters=iters).cpu().numpy()
    np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))


@pytest.mark.parametrize("L,k", [(31, 66), (32, 64), (128, 16), (8, 256), (64, 64), (33, 62),
                                 (64, 100)])
def test_codes_with_tables_around_the_staged_sizes(aq, L, k):
    """Tables of 2,046 entries, of 2,048 and of more, even and odd k, up to one that
    has no room for the additional copy: the oracle's codes."""
    z = latents(700, L, k)
    t = np.ascontiguousarray(opq.init_centroids(z, k))
    codes, _ = aq.pq_encode(torch.as_tensor(z, device=DEV), torch.as_tensor(t[None], device=DEV))
    np.testing.assert_array_equal(codes.cpu().numpy(), opq.assign(z, t))
