"""Performance cases: the work that a user of this package has it do, through the public calls of
``paper_2212_10733_gb300.aeqc``, from one small batch to a million histograms.

Kinds: the whole calls (``round_trip``, ``compress``, ``subdomains``, ``decompress``, ``correct``), the
autoencoder's two halves (``encode``, ``decode``), its gradient (``train``), the residual coder (``rice``) and
the latent quantiser (``pq``).  Inputs are ``synth``'s histograms; network weights are the principal directions
of a sample of them (the minimiser of the training loss for the tied linear network), so that residuals, codes
and the Newton iteration are those of a trained model.

The outlier list of a compressed batch is filled in the order its atomics arrive, so its entries are compared
through the decompressed values they become, not as a list.
"""
import math

import numpy as np
import torch

from paper_2212_10733_gb300 import aeqc, synth

GRIDS = {"39x39": (39, 39), "37x33": (37, 33)}


def listed():
    return [
        # one cell's batch with everything at its default (FP32 network, FP64 correction): compress, then
        # decompress; launches and latency
        dict(name="round_trip_64", kind="round_trip", n=64, grid="39x39", H=128, L=16, dtype="f32", layers=2,
             k_max=3, heavy=0.0, tau=1e-3),
        # one time step of one process at a tight bound: the plain-scale workload, the largest call
        dict(name="compress_1m", kind="compress", n=1048576, grid="39x39", H=256, L=32, dtype="bf16", layers=2,
             k_max=3, heavy=0.0, tau=1e-4),
        # the precision workload: wide network, a tenth of the histograms with a heavy tail
        dict(name="compress_precision", kind="compress", n=262144, grid="39x39", H=512, L=32, dtype="bf16",
             layers=2, k_max=4, heavy=0.1, tau=1e-4),
        # subdomains of uneven size, each with its own network, in one call
        dict(name="compress_subdomains", kind="subdomains", G=24, layout=3, grid="39x39", H=256, L=32,
             dtype="bf16", layers=2, k_max=3, heavy=0.0, tau=1e-4),
        # the paper's own network and grid: one tied FP32 layer, latent 4
        dict(name="compress_paper_shape", kind="compress", n=262144, grid="37x33", H=4, L=4, dtype="f32",
             layers=1, k_max=3, heavy=0.0, tau=1e-4),
        # reading a compressed precision batch back
        dict(name="decompress_precision", kind="decompress", n=150001, grid="39x39", H=512, L=32, dtype="bf16",
             layers=2, k_max=4, heavy=0.1, tau=1e-4),
        # stages 4-5 alone, on rows decoded elsewhere (quantised latents, another network)
        dict(name="correct_100k", kind="correct", n=100003, grid="39x39", k_max=3, heavy=0.0, tau=1e-4),
        # latents only
        dict(name="encode_precision", kind="encode", n=262144, grid="39x39", H=512, L=32, dtype="bf16",
             layers=2, k_max=4, heavy=0.1),
        # decoded rows only
        dict(name="decode_precision", kind="decode", n=262144, grid="39x39", H=512, L=32, dtype="bf16",
             layers=2, k_max=4, heavy=0.1),
        # one training batch of the paper's size: loss and gradients, forward and backward
        dict(name="train_128", kind="train", n=128, grid="39x39", H=512, L=32, dtype="bf16", layers=2,
             k_max=4, heavy=0.0),
        # entropy coding of residual codes and back
        dict(name="rice_128k", kind="rice", n=131072, P=1521),
        # product quantisation of a time step's latents: tables trained, then every latent coded
        dict(name="pq_1m", kind="pq", n=1048576, L=32, k=16, iters=10, dtype="bf16"),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["round_trip", "compress", "subdomains", "decompress", "correct", "encode", "decode",
                       "train", "rice", "pq"])
    if kind == "rice":
        return dict(kind=kind, n=_size(rng, 100, 130000), P=rng.choice([1521, 1221]))
    if kind == "pq":
        return dict(kind=kind, n=_size(rng, 1000, 1000000), L=rng.choice([16, 32]), k=rng.choice([16, 64]),
                    iters=rng.randint(4, 10), dtype=rng.choice(["f32", "bf16"]))
    if kind == "correct":
        return dict(kind=kind, n=_size(rng, 50, 100000), grid=rng.choice(["39x39", "37x33"]), k_max=3,
                    heavy=0.0, tau=rng.choice([1e-3, 1e-4]))
    c = dict(kind=kind, grid="39x39", H=rng.choice([128, 256, 512]), L=rng.choice([16, 32]), dtype="bf16",
             layers=2, k_max=rng.choice([3, 4]), heavy=rng.choice([0.0, 0.1]))
    if kind == "train":
        c.update(n=rng.randint(32, 700), dtype=rng.choice(["bf16", "f32"]), heavy=0.0)
        return c
    if kind in ("encode", "decode"):
        c.update(n=_size(rng, 200, 260000))
        return c
    c.update(tau=rng.choice([1e-3, 1e-4]))
    if kind == "round_trip":
        c.update(n=_size(rng, 1, 1000), H=128, L=16, dtype="f32", heavy=0.0)
    elif kind == "subdomains":
        c.update(G=rng.randint(2, 24), layout=rng.randint(0, 1000), H=rng.choice([128, 256]), heavy=0.0)
    else:
        c.update(n=_size(rng, 200, 250000))
        if rng.random() < 0.25:
            c.update(grid="37x33", H=4, L=4, dtype="f32", layers=1, heavy=0.0)
    return c


# --- inputs -----------------------------------------------------------------------------------


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _points(c):
    npar, nperp = GRIDS[c["grid"]]
    return npar * nperp


def _grid(c):
    vpar, vperp, vol = synth.grid_arrays(*GRIDS[c["grid"]])
    return aeqc.Grid(vpar, vperp, vol)


def _group_sizes(c):
    return synth.group_sizes(c["G"], synth.config_seed(c["layout"]))


def _rows(c):
    return int(_group_sizes(c).sum()) if c["kind"] == "subdomains" else c["n"]


def _histograms(c, seed, n):
    return synth.histograms_torch(n, synth.config_seed(seed), _dev(), k_max=c["k_max"], heavy_frac=c["heavy"],
                                  grid=GRIDS[c["grid"]])


def _normaliser(x):
    y = x / x.amax(1, keepdim=True)
    mu = y.mean(0)
    sd = (y - mu).square().mean(0).sqrt().clamp_min(1e-6)
    return (y - mu) / sd, mu, sd


def _network(W1, c, P, mu, sd):
    """Parameters as a user hands them over: float64 arrays of float32 values.  On cells that hold nothing in
    any histogram (the v_perp = 0 row) training has no gradient, so W1 has its initial values there."""
    H, L = c["H"], c["L"]
    init = torch.as_tensor(synth.ae_init(P, H, L, synth.BASE_SEED)["W1"], device=W1.device)
    W1 = torch.where((sd <= 1e-6)[:, None], init, W1[:, :H])
    W2 = torch.zeros((H, L), dtype=torch.float64, device=W1.device)
    W2[:L, :L] = torch.eye(L, dtype=torch.float64, device=W1.device)
    z = lambda k: torch.zeros(k, dtype=torch.float64, device=W1.device)  # noqa: E731
    p = dict(W1=W1, b1=z(H), W2=W2, b2=z(L), b3=z(H), b4=z(P), mu=mu, sigma=sd)
    return {k: v.float().double().contiguous() for k, v in p.items()}


def _principal(u):
    """Principal directions of u, the largest first."""
    _, vec = torch.linalg.eigh(u.T @ u / len(u))
    return vec.flip(1)


def _weights(c, seed):
    """One group's parameters, from a sample of its own of the same kind of histograms."""
    x = _histograms(c, seed + 1000003, 4096)
    u, mu, sd = _normaliser(x)
    return _network(_principal(u), c, _points(c), mu, sd)


def _group_weights(c, seed, x, off):
    """Parameters of every subdomain from its own histograms: the pooled principal directions carried one
    power iteration towards each subdomain's own."""
    pooled = _principal(_normaliser(x[:: max(1, len(x) // 4096)])[0])[:, : c["H"]]
    out = []
    for g in range(c["G"]):
        u, mu, sd = _normaliser(x[off[g]: off[g + 1]][:1024])
        q, _ = torch.linalg.qr(u.T @ (u @ pooled))
        out.append(_network(q, c, _points(c), mu, sd))
    return out


def _model(c, groups):
    m = aeqc.Model(_points(c), c["H"], c["L"], n_groups=len(groups), layers=c["layers"],
                   dtype=aeqc.DTYPE_BF16 if c["dtype"] == "bf16" else aeqc.DTYPE_F32)
    for g, p in enumerate(groups):
        m.set_group(g, {k: v.cpu().numpy() for k, v in p.items()})
    return m


def _params(c):
    kernel = aeqc.KERNEL_FP64 if c["kind"] == "round_trip" else aeqc.KERNEL_FAST
    return aeqc.params_default(tau=c["tau"], kernel=kernel)


def _generator(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(7919 * seed + 17)
    return g


def _decoded_elsewhere(x, seed, rel=1e-2, floor=2e-3):
    """Rows near x, as another decoder leaves them: float32, padded to XHAT_LD columns."""
    g = _generator(seed)
    n, P = x.shape
    e1 = torch.randn((n, P), generator=g, device=x.device)
    e2 = torch.randn((n, P), generator=g, device=x.device)
    out = torch.zeros((n, aeqc.XHAT_LD), dtype=torch.float32, device=x.device)
    out[:, :P] = x * (1.0 + rel * e1) + floor * x.amax(1, keepdim=True) * e2
    return out


def _residual_codes(c, seed):
    """Residual codes as the quantiser leaves them: the zero-level code on the v_perp = 0 row and in the empty
    tail, two-sided geometric levels whose width differs from histogram to histogram, a few escapes."""
    g, n, P = _generator(seed), c["n"], c["P"]
    npar = 39 if P == 1521 else 37
    width = torch.exp(torch.randn((n, 1), generator=g, device=_dev()) * 0.6 + 4.0)
    u = torch.rand((n, P), generator=g, device=_dev()) - 0.5
    q = (-torch.sign(u) * torch.log1p(-2.0 * u.abs().clamp_max(0.499999)) * width).round().clamp(-32000, 32000)
    q[torch.rand((n, P), generator=g, device=_dev()) < 0.05] = aeqc.CODE_ZERO
    q[torch.rand((n, P), generator=g, device=_dev()) < 1e-5] = aeqc.CODE_ESCAPE
    q[:, :npar] = aeqc.CODE_ZERO
    return q.to(torch.int16)


def _latents(c, seed):
    """Latents of a linear encoder: columns of falling spread, off centre."""
    g = _generator(seed)
    spread = 20.0 * torch.arange(1, c["L"] + 1, device=_dev()) ** -0.8
    z = torch.randn((c["n"], c["L"]), generator=g, device=_dev()) * spread + 0.2 * spread
    return z.to(torch.bfloat16 if c["dtype"] == "bf16" else torch.float32)


def _train_weights(c, seed):
    P = _points(c)
    init = synth.ae_init(P, c["H"], c["L"], synth.config_seed(seed))
    _, mu, sd = _normaliser(_histograms(c, seed + 1000003, 2048))
    p = {k: torch.as_tensor(v, device=_dev()) for k, v in init.items()}
    p.update(mu=mu, sigma=sd)
    return {k: v.float().double() for k, v in p.items()}


def _decoder_inputs(c, seed):
    """Latents and scales as the encoder leaves them (bfloat16, or float32 for the FP32 network)."""
    x = _histograms(c, seed, c["n"])
    p = _weights(c, seed)
    s = x.amax(1)
    z = torch.cat([((xc / xc.amax(1, keepdim=True) - p["mu"]) / p["sigma"]) @ (p["W1"] @ p["W2"])
                   for xc in x.split(1 << 15)])
    return z.to(torch.bfloat16 if c["dtype"] == "bf16" else torch.float32), s, p


def prepare(case, seed):
    c = case
    k = c["kind"]
    if k == "rice":  # the streams of several batches go back to back into one store, half the codes' size
        return dict(c=c, codes=_residual_codes(c, seed),
                    store=torch.zeros(max(64, c["n"] * c["P"] // 2), dtype=torch.int32, device=_dev()))
    if k == "pq":
        return dict(c=c, z=_latents(c, seed))
    if k == "train":
        return dict(c=c, m=_model(c, [_train_weights(c, seed)]), x=_histograms(c, seed, c["n"]))
    if k == "decode":
        z, s, p = _decoder_inputs(c, seed)
        return dict(c=c, m=_model(c, [p]), z=z, s=s)
    n, P = _rows(c), _points(c)
    st = dict(c=c, grid=_grid(c), x=_histograms(c, seed, n), goff=None)
    if k == "correct":
        st.update(prm=_params(c), xhat=_decoded_elsewhere(st["x"], seed),
                  out=aeqc.Compressed(n, P, 1, torch.float32, _dev(), max(1024, 4 * n)),
                  ws=torch.empty(int(aeqc.load().quantize_correct_workspace_size(n)), dtype=torch.uint8,
                                 device=_dev()))
        return st
    if k == "subdomains":
        off = np.concatenate([[0], np.cumsum(_group_sizes(c))])
        st.update(m=_model(c, _group_weights(c, seed, st["x"], off)), goff=torch.as_tensor(off, device=_dev()))
    else:
        st.update(m=_model(c, [_weights(c, seed)]))
    if k == "encode":
        return st
    st.update(prm=_params(c))
    if k == "round_trip":
        return st
    st.update(out=aeqc.Compressed(n, P, c["L"], st["m"].latent_dtype(), _dev(), max(1024, 16 * n)),
              ws=aeqc.compress_batch_workspace(st["m"], n, _dev()))
    if k == "decompress":  # what is read back was written by the same library
        aeqc.compress_batch(st["m"], st["grid"], st.pop("x"), st["prm"], out=st["out"], ws=st["ws"])
        st.update(ws=aeqc.decompress_batch_workspace(st["m"], n, _dev()),
                  f=torch.empty((n, P), dtype=torch.float64, device=_dev()))
    return st


# --- one pass ---------------------------------------------------------------------------------


def _compressed(o):
    return dict(latent=o.latent, scale=o.scale, codes=o.codes, lam=o.lam, iters=o.iters, status=o.status,
                count=o.count)


def run(state):
    st = state
    c = st["c"]
    k = c["kind"]
    if k == "round_trip":
        o = aeqc.compress_batch(st["m"], st["grid"], st["x"], st["prm"])
        return dict(_compressed(o), f=aeqc.decompress_batch(st["m"], st["grid"], o, st["prm"]))
    if k in ("compress", "subdomains"):
        return _compressed(aeqc.compress_batch(st["m"], st["grid"], st["x"], st["prm"],
                                               group_offsets=st["goff"], out=st["out"], ws=st["ws"]))
    if k == "decompress":
        return aeqc.decompress_batch(st["m"], st["grid"], st["out"], st["prm"], f=st["f"], ws=st["ws"])
    if k == "correct":
        o = aeqc.quantize_correct(st["grid"], st["x"], st["xhat"], st["prm"], out=st["out"], ws=st["ws"])
        return dict(scale=o.scale, codes=o.codes, lam=o.lam, iters=o.iters, status=o.status, count=o.count)
    if k == "encode":
        z, s = aeqc.ae_encode(st["m"], st["x"])
        return dict(latent=z, scale=s)
    if k == "decode":
        return aeqc.ae_decode(st["m"], st["z"], st["s"])[:, : _points(c)]
    if k == "train":
        loss, grad = st["m"].loss_grad(st["x"])
        return dict(loss=loss, grad=grad)
    if k == "rice":
        r = aeqc.rice_encode(st["codes"])
        st["store"][: len(r.words)].copy_(r.words)
        return dict(kparam=r.kparam, nbits=r.nbits, offsets=r.offsets, words=st["store"],
                    codes=aeqc.rice_decode(r, c["P"]))
    table = aeqc.pq_train(st["z"], k=c["k"], iters=c["iters"])
    codes, zq = aeqc.pq_encode(st["z"], table, zq=torch.empty_like(st["z"]))
    return dict(table=table, codes=codes, zq=zq)


# --- what a pass cannot do without ------------------------------------------------------------


def work(case):
    c = case
    k = c["kind"]
    if k == "rice":  # the codes read, about 8.4 bits a code written and read again, the codes written
        return dict(bytes=c["n"] * c["P"] * (2 + 2 * 8.4 / 8 + 2), flops=0)
    if k == "pq":  # latents read, code and decoded latent written; a distance per centroid and pass
        b = 2 if c["dtype"] == "bf16" else 4
        return dict(bytes=c["n"] * c["L"] * (2 * b + 1), flops=2.0 * c["n"] * c["L"] * c["k"] * (c["iters"] + 1))
    P, n = _points(c), _rows(c)
    if k == "correct":
        return dict(bytes=n * (12 * P + 2 * P + 43), flops=0)
    H, L, b = c["H"], c["L"], 2 if c["dtype"] == "bf16" else 4
    one_way = 2.0 * n * L * P if c["layers"] == 1 else 2.0 * n * H * (P + L)
    weights = (1 if c["kind"] != "subdomains" else c["G"]) * H * (P + L) * b
    if k == "encode":
        return dict(bytes=n * (8 * P + b * L + 8) + weights, flops=one_way)
    if k == "decode":
        return dict(bytes=n * (4 * P + b * L + 8) + weights, flops=one_way)
    if k == "train":  # forward, and the two products of each layer backward
        return dict(bytes=n * 8 * P + 8 * H * (P + L), flops=6 * one_way)
    comp = n * (8 * P + 2 * P + b * L + 43) + weights
    back = n * (8 * P + 2 * P + b * L + 42) + weights
    if k == "decompress":
        return dict(bytes=back, flops=one_way)
    if k == "round_trip":
        return dict(bytes=comp + back, flops=3 * one_way)
    return dict(bytes=comp, flops=2 * one_way)


# --- the same in 64 bits, without the library -------------------------------------------------


def _exact_encode(x, p, rows=1 << 15):
    """(latents, scales) of one group's network; W1 W2 is one matrix, since the activation is the identity."""
    A = p["W1"] @ p["W2"]
    off = p["b1"] @ p["W2"] + p["b2"]
    z = torch.cat([((xc / xc.amax(1, keepdim=True) - p["mu"]) / p["sigma"]) @ A + off for xc in x.split(rows)])
    return z, x.amax(1)


def _exact_train(x, p, tied_order=("W1", "b1", "W2", "b2", "b3", "b4")):
    s = x.amax(1, keepdim=True)
    u = (x / s - p["mu"]) / p["sigma"]
    h1 = u @ p["W1"] + p["b1"]
    z = h1 @ p["W2"] + p["b2"]
    h3 = z @ p["W2"].T + p["b3"]
    d = h3 @ p["W1"].T + p["b4"] - u
    loss = d.square().mean()
    dy = 2.0 * d / d.numel()
    dh3 = dy @ p["W1"]
    dz = dh3 @ p["W2"]
    dh1 = dz @ p["W2"].T
    g = dict(W1=dy.T @ h3 + u.T @ dh1, b1=dh1.sum(0), W2=dh3.T @ z + h1.T @ dz, b2=dz.sum(0), b3=dh3.sum(0),
             b4=dy.sum(0))
    return dict(loss=loss.reshape(1), grad=torch.cat([g[k].reshape(-1) for k in tied_order]))


def _exact_correct(c, x, xhat):
    """Multipliers and scales: quantise, solve the four moment equations by Newton, check the bound, once more
    at a quarter of the bin width where it fails; a histogram that fails again is stored as it is."""
    vpar, vperp, vol = synth.grid_arrays(*GRIDS[c["grid"]])
    v = torch.as_tensor(np.tile(vpar, len(vperp)), device=x.device)
    w = torch.as_tensor(np.repeat(vperp ** 2, len(vpar)), device=x.device)
    phi = torch.stack([torch.ones_like(v), v, w, v * v], 1)
    pairs = (phi[:, :, None] * phi[:, None, :]).reshape(-1, 16)
    n, P = x.shape
    lam = torch.zeros((n, 4), dtype=torch.float64, device=x.device)
    for r0 in range(0, n, 8192):
        xr = x[r0: r0 + 8192]
        hr = xhat[r0: r0 + 8192, :P].double()
        e = c["tau"] * xr.amax(1, keepdim=True)
        todo = torch.arange(len(xr), device=x.device)
        for alpha in (0.5, 0.125):
            xs, hs, es = xr[todo], hr[todo], e[todo]
            dl = torch.exp2(torch.floor(torch.log2(2.0 * alpha * es)))
            g = hs + torch.round((xs - hs) / dl) * dl
            xp = torch.where((g < 0) | (g > 2.0 * xs), torch.zeros_like(g), g)
            Q = vol * (xs @ phi)
            l = torch.zeros((len(xs), 4), dtype=torch.float64, device=x.device)
            for _ in range(6):
                f = xp * torch.exp(-(l @ phi.T))
                M = vol * (f @ pairs).reshape(-1, 4, 4)
                l = l + torch.linalg.solve(M, vol * (f @ phi) - Q)
            f = xp * torch.exp(-(l @ phi.T))
            bad = ((f - xs).abs() > es).any(1)
            lam[r0 + todo[~bad]] = l[~bad]
            todo = todo[bad]
            if not len(todo):
                break
    return dict(scale=x.amax(1), codes=None, lam=lam, iters=None, status=None, count=None)


def _exact_pq(c, z):
    """Lloyd iterations from k evenly spaced centroids: nearest by the float32 distance, means in 64 bits, a
    table of float32 values."""
    zf, k = z.float(), c["k"]
    lo, hi = zf.amin(0).double(), zf.amax(0).double()
    j = torch.arange(k, device=z.device, dtype=torch.float64) + 0.5
    table = (lo[:, None] + j * ((hi - lo) / k)[:, None]).float()
    for _ in range(c["iters"]):
        for d in range(c["L"]):
            a = (zf[:, d, None] - table[d]).abs().argmin(1)
            cnt = torch.bincount(a, minlength=k)
            tot = torch.zeros(k, dtype=torch.float64, device=z.device).index_add_(0, a, zf[:, d].double())
            table[d] = torch.where(cnt > 0, tot / cnt.clamp_min(1), table[d].double()).float()
    zq = torch.stack([table[d][(zf[:, d, None] - table[d]).abs().argmin(1)] for d in range(c["L"])], 1)
    return dict(table=table[None].double(), codes=None, zq=zq.double())


def exact(case, seed):
    c = case
    k = c["kind"]
    if k in ("rice", "decompress"):  # whole numbers; codes that only the library's own decoded rows complete
        return None
    if k == "pq":
        return _exact_pq(c, _latents(c, seed))
    if k == "train":
        return _exact_train(_histograms(c, seed, c["n"]), _train_weights(c, seed))
    if k == "decode":
        z, s, p = _decoder_inputs(c, seed)
        A = p["W2"].T @ p["W1"].T
        off = p["b3"] @ p["W1"].T + p["b4"]
        return torch.cat([sc[:, None] * (p["sigma"] * (zc.double() @ A + off) + p["mu"])
                          for zc, sc in zip(z.split(1 << 15), s.split(1 << 15))])
    n = _rows(c)
    x = _histograms(c, seed, n)
    if k == "correct":
        return _exact_correct(c, x, _decoded_elsewhere(x, seed))
    if k == "subdomains":
        off = np.concatenate([[0], np.cumsum(_group_sizes(c))])
        zs = [_exact_encode(x[off[g]: off[g + 1]], p)
              for g, p in enumerate(_group_weights(c, seed, x, off))]
        z, s = torch.cat([a for a, _ in zs]), torch.cat([b for _, b in zs])
    else:
        z, s = _exact_encode(x, _weights(c, seed))
    if k == "encode":
        return dict(latent=z, scale=s)
    o = dict(latent=z, scale=s, codes=None, lam=None, iters=None, status=None, count=None)
    return dict(o, f=None) if k == "round_trip" else o
