"""Workloads that the reconstruction framework is timed on.

Each case is one call of a public entry point of paper_1704_04511_gb300.recon on synthetic data:
series of damped exponentials inside random ellipses, variable-density sampling, 30 dB of noise.
One context (with the stream it works on) is kept for the whole process, as a reconstruction
service keeps it; every state has inputs and output buffers of its own, as successive scans have.

exact() is the same mathematics in complex128 with plain torch, without the framework's code.
"""

import math

import torch

from paper_1704_04511_gb300 import recon

SIZES = (32, 64, 128, 192, 256)
LAM, GAMMA, EPS0 = 1e-3, 1.4, 0.01
COIL_LAM = 1.0  # many coils at 6x: the data term alone is a noisy fit


def listed():
    return [
        # whole reconstructions (Algorithm 1); the smallest, 200 CG steps of a few microseconds
        dict(name="solve_32x32x8", kind="solve", P=32, Q=32, T=8, N1=5, N2=5, M=2, irls=20, cg=10,
             bf16=False),
        # the benchmark's series and settings
        dict(name="solve_256x256x16", kind="solve", P=256, Q=256, T=16, N1=9, N2=9, M=3, irls=30,
             cg=15, bf16=False),
        # several scans at once, k-space stored as bfloat16 pairs
        dict(name="batch4_256x256x16_bf16", kind="batch", n=4, P=256, Q=256, T=16, N1=9, N2=9, M=3,
             irls=10, cg=15, bf16=True),
        # the volume workload with fewer iterations, the largest working set (streams from HBM)
        dict(name="volume_128x128x64x12", kind="volume", P=128, Q=128, R=64, T=12, N1=7, N2=7, N3=3,
             M=2, irls=2, cg=15),
        # twelve receiver coils, the paper's in-vivo geometry
        dict(name="coils12_128x128x12", kind="coils", nc=12, P=128, Q=128, T=12, N1=9, N2=9, M=3,
             irls=2, cg=10),
        # the comparison with the pixel-wise prior
        dict(name="hlr_voxel_128x128x12", kind="variant", variant=2, P=128, Q=128, T=12, N1=1, N2=1,
             M=3, irls=5, cg=10),
        # least-squares steps alone over the grids of the served mix and the largest grid
        dict(name="cg_64x64x21", kind="cg", P=64, Q=64, T=21, N1=7, N2=7, M=2, cg=15),
        dict(name="cg_192x192x24", kind="cg", P=192, Q=192, T=24, N1=9, N2=9, M=3, cg=15),
        dict(name="cg_512x512x16", kind="cg", P=512, Q=512, T=16, N1=5, N2=5, M=2, cg=10),
        # the other steps of an IRLS iteration, and the T2 map of a recovered series
        dict(name="gram_256x256x16", kind="gram", P=256, Q=256, T=16, N1=9, N2=9, M=3),
        dict(name="weight_256x256_s243", kind="weight", P=256, Q=256, T=16, N1=9, N2=9, M=3),
        dict(name="t2fit_256x256x16", kind="t2fit", P=256, Q=256, T=16),
    ]


def draw(rng):
    def frames(P, Q, lo=4, hi=24, most=1 << 20):
        return rng.randint(lo, max(lo, min(hi, most // (P * Q), 8533 // Q)))

    kind = rng.choice(["solve", "batch", "volume", "coils", "variant", "cg", "cg", "gram", "weight",
                       "t2fit"])
    if kind == "volume":
        P, Q, R = rng.choice((32, 64, 128)), rng.choice((32, 64, 128)), rng.choice((16, 32, 64))
        return dict(kind=kind, P=P, Q=Q, R=R, T=rng.randint(3, 12), N1=rng.randint(2, 7),
                    N2=rng.randint(2, 7), N3=rng.randint(1, 3), M=2, irls=rng.randint(1, 2),
                    cg=rng.randint(5, 15))
    sizes = SIZES + (512,) if kind in ("cg", "t2fit") else SIZES
    P, Q = rng.choice(sizes), rng.choice(sizes)
    if kind == "t2fit":
        return dict(kind=kind, P=P, Q=Q, T=frames(P, Q, most=1 << 22))
    c = dict(kind=kind, P=P, Q=Q, T=frames(P, Q, most=1 << 22 if kind == "cg" else 1 << 20),
             N1=rng.randint(2, 9), N2=rng.randint(2, 9), M=rng.randint(1, 3))
    if kind == "solve":
        c.update(irls=rng.randint(2, 20), cg=rng.randint(5, 15), bf16=rng.random() < 0.3)
    elif kind == "batch":
        c.update(n=rng.randint(2, 4), irls=rng.randint(2, 10), cg=rng.randint(5, 15),
                 bf16=rng.random() < 0.3)
    elif kind == "coils":
        P, Q = rng.choice((32, 64, 128)), rng.choice((32, 64, 128))
        c.update(P=P, Q=Q, T=rng.randint(4, 12), nc=rng.randint(2, 12), irls=rng.randint(1, 2),
                 cg=rng.randint(5, 10))
    elif kind == "variant":
        P, Q = rng.choice((32, 64, 128)), rng.choice((32, 64, 128))
        v = rng.choice((recon.RECON_VARIANT_GIRAF, recon.RECON_VARIANT_HLR_VOXEL))
        c.update(P=P, Q=Q, T=rng.randint(6, 16), variant=v, M=rng.randint(2, 3), irls=rng.randint(2, 5),
                 cg=rng.randint(5, 10))
        if v == recon.RECON_VARIANT_HLR_VOXEL:
            c.update(N1=1, N2=1)
    elif kind == "cg":
        c.update(cg=rng.randint(5, 15))
    return c


# ---- synthetic scans ----

def _grid(case):
    return ((case["R"],) if "R" in case else ()) + (case["P"], case["Q"])


def _filt(case):
    return (case["N1"], case["N2"]) + ((case["N3"],) if "N3" in case else ()) + (case["M"],)


def _dims(x):
    return tuple(range(1, x.dim()))


def _times(T):
    return [1.0 + 59.0 * n / (T - 1) for n in range(T)]


def _freq2(grid):
    """Squared distance from DC per k-space position (natural order), 1 at the edge of an axis."""
    f = torch.zeros(grid, device="cuda")
    for ax, n in enumerate(grid):
        v = torch.fft.fftfreq(n, device="cuda") * 2
        f = f + (v * v).reshape([-1 if i == ax else 1 for i in range(len(grid))])
    return f


def _series(grid, T, gen):
    """Ellipses of random intensity with a smooth map of relaxation times, complex64 (T, *grid)."""
    axes = torch.meshgrid(*[(torch.arange(n, device="cuda") + 0.5) / n - 0.5 for n in grid], indexing="ij")
    rho = torch.zeros(grid, device="cuda")
    for _ in range(8):
        u = torch.rand(2 * len(grid) + 1, generator=gen, device="cuda")
        d = sum(((a - 0.5 * (u[2 * i] - 0.5)) / (0.08 + 0.25 * u[2 * i + 1])) ** 2
                for i, a in enumerate(axes))
        rho = rho + (0.2 + 0.8 * u[-1]) * (d < 1)
    noise = torch.randn(grid, generator=gen, device="cuda")
    low = torch.fft.ifftn(torch.fft.fftn(noise) * torch.exp(-40.0 * _freq2(grid))).real
    low = (low - low.min()) / (low.max() - low.min())
    t2 = 20.0 + 100.0 * low
    t = torch.tensor(_times(T), device="cuda").reshape((T,) + (1,) * len(grid))
    return (rho * torch.exp(-t / t2)).to(torch.complex64)


def _masks(grid, T, gen, undersampling):
    """Variable-density masks, uint8 (T, *grid): exactly n / undersampling samples a frame, drawn
    without replacement, with a full block around DC."""
    n = math.prod(grid)
    f = _freq2(grid)
    logp = -torch.log1p(16.0 * f).reshape(1, n)
    centre = f <= (4.0 / min(grid)) ** 2
    u = torch.rand((T, n), generator=gen, device="cuda").clamp_(1e-7, 1 - 1e-7)
    keys = logp - torch.log(-torch.log(u))
    keys.masked_fill_(centre.reshape(1, n), 1e9)
    at = torch.topk(keys, max(1, round(n / undersampling)), dim=1).indices
    return torch.zeros((T, n), dtype=torch.uint8, device="cuda").scatter_(1, at, 1).reshape((T,) + grid)


def _coil_maps(nc, grid, gen):
    axes = torch.meshgrid(*[(torch.arange(n, device="cuda") + 0.5) / n - 0.5 for n in grid], indexing="ij")
    maps = []
    for c in range(nc):
        u = torch.rand(3, generator=gen, device="cuda")
        ang = 2 * math.pi * c / nc
        d2 = (axes[0] - 0.6 * math.cos(ang)) ** 2 + (axes[1] - 0.6 * math.sin(ang)) ** 2
        phase = 2 * math.pi * (u[0] + (u[1] - 0.5) * axes[0] + (u[2] - 0.5) * axes[1])
        maps.append(torch.polar(torch.exp(-d2 / 0.32), phase))
    maps = torch.stack(maps)
    return (maps / maps.abs().square().sum(0).sqrt()).contiguous()


def _scan(case, seed):
    """x_true, masks, k-space (and coil maps) of one scan, complex64."""
    grid, T = _grid(case), case["T"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
    x = _series(grid, T, gen)
    masks = _masks(grid, T, gen, 6.0)
    coils = _coil_maps(case["nc"], grid, gen) if case["kind"] == "coils" else None
    img = x if coils is None else coils[:, None] * x
    full = torch.fft.fftn(img, dim=tuple(range(img.dim() - len(grid), img.dim())), norm="ortho")
    clean = full * masks
    noise = torch.randn(clean.shape, generator=gen, device="cuda", dtype=torch.complex64) * masks
    b = clean + noise * (torch.linalg.vector_norm(clean) / torch.linalg.vector_norm(noise) * 10.0 ** -1.5)
    if case.get("bf16"):
        b = torch.view_as_real(b).to(torch.bfloat16)
    return dict(x=x, masks=masks, b=b.contiguous(), coils=coils)


# ---- the method in complex128 (plain torch) ----

def _c128(b):
    if b.dtype == torch.bfloat16:
        b = torch.view_as_complex(b.float().contiguous())
    return b.to(torch.complex128)


def _adjoint(b, masks):
    return torch.fft.ifftn(b * masks, dim=_dims(masks), norm="ortho")


def _pairs(M):
    return [(a, b) for a in range(M) for b in range(a, M)]


def _taps(filt):
    """Tap coordinates in column order, grid axes as in _grid (depth first for volumes)."""
    N1, N2, N3 = filt[0], filt[1], filt[2] if len(filt) == 4 else None
    ax = ([N3] if N3 else []) + [N1, N2]
    return torch.cartesian_prod(*[torch.arange(n, device="cuda") for n in ax]).reshape(-1, len(ax)), ax


def _gram(x, filt, circular=False):
    """Lags as the full transforms of the pair products, and G (s, s) complex128."""
    M, grid = filt[-1], x.shape[1:]
    T = x.shape[0]
    if circular:
        x = torch.cat([x, x[:M - 1]]) if M > 1 else x
    k = T if circular else T - M + 1
    taps, _ = _taps(filt)
    diff = taps[:, None] - taps[None]
    at = tuple(diff[..., i] % n for i, n in enumerate(grid))
    n = taps.shape[0]
    G = torch.zeros((M * n, M * n), dtype=torch.complex128, device="cuda")
    full = []
    for a, b in _pairs(M):
        q = (x[M - 1 - a:M - 1 - a + k].conj() * x[M - 1 - b:M - 1 - b + k]).sum(0)
        f = torch.fft.fftn(q)
        full.append(f)
        G[a * n:(a + 1) * n, b * n:(b + 1) * n] = f[at]
        G[b * n:(b + 1) * n, a * n:(a + 1) * n] = f[at].conj().T
    return torch.stack(full), G


def _lags(full, filt):
    """The (2N-1)-sized block of lags around zero of the full transforms."""
    _, ax = _taps(filt)
    for i, n in enumerate(ax):
        idx = torch.arange(-(n - 1), n, device="cuda") % full.shape[i + 1]
        full = full.index_select(i + 1, idx)
    return full


def _weight(G, eps, filt, grid):
    """Summed diagonals of (G + eps)^-1 and S(r), complex128."""
    M = filt[-1]
    taps, ax = _taps(filt)
    n = taps.shape[0]
    H = torch.linalg.inv(G + eps * torch.eye(G.shape[0], dtype=G.dtype, device="cuda"))
    size = [2 * v - 1 for v in ax]
    diff = taps[None] - taps[:, None] + torch.tensor([v - 1 for v in ax], device="cuda")  # l - l' at [l', l]
    at = torch.zeros((n, n), dtype=torch.long, device="cuda")
    for i, v in enumerate(size):
        at = at * v + diff[..., i]
    ds, S = [], []
    for a, b in _pairs(M):
        blk = H[b * n:(b + 1) * n, a * n:(a + 1) * n]
        d = torch.zeros(math.prod(size), dtype=G.dtype, device="cuda").index_add_(0, at.reshape(-1), blk.reshape(-1))
        d = d.reshape(size)
        ds.append(d)
        z = torch.zeros(grid, dtype=G.dtype, device="cuda")
        idx = torch.meshgrid(*[torch.arange(-(v - 1), v, device="cuda") % g for v, g in zip(ax, grid)], indexing="ij")
        S.append(torch.fft.fftn(z.index_put_(idx, d, accumulate=True)))
    return torch.stack(ds), torch.stack(S)


def _voxel_gram(x, M):
    k = x.shape[0] - M + 1
    w = torch.stack([x[M - 1 - m:M - 1 - m + k] for m in range(M)], -1)  # (k, P, Q, M)
    return torch.einsum("jpqa,jpqb->pqab", w.conj(), w)


def _apply_w(S, x, M, circular=False):
    T = x.shape[0]
    y = torch.zeros_like(x)
    pairs = _pairs(M)
    for a in range(M):
        for b in range(M):
            s = S[pairs.index((a, b))] if a <= b else S[pairs.index((b, a))].conj()
            if circular:
                y += s * torch.roll(x, b - a, 0)
            else:
                k = T - M + 1
                y[M - 1 - a:M - 1 - a + k] += s * x[M - 1 - b:M - 1 - b + k]
    return y


def _normal(x, masks, S, lam, M, coils=None, circular=False):
    dim = _dims(x)
    if coils is None:
        y = torch.fft.ifftn(torch.fft.fftn(x, dim=dim) * masks, dim=dim)
    else:
        y = torch.zeros_like(x)
        for c in coils:
            y += c.conj() * torch.fft.ifftn(torch.fft.fftn(c * x, dim=dim) * masks, dim=dim)
    return y + lam * _apply_w(S, x, M, circular)


def _cg(x, r, steps, op):
    p, rr = r.clone(), r.abs().square().sum()
    for _ in range(steps):
        q = op(p)
        alpha = rr / (p.conj() * q).real.sum()
        x = x + alpha * p
        r = r - alpha * q
        new = r.abs().square().sum()
        p = r + (new / rr) * p
        rr = new
    return x, r


def _solve(case, scan):
    filt, grid, M = _filt(case), _grid(case), case["M"]
    b, masks = _c128(scan["b"]), scan["masks"]
    coils = None if scan["coils"] is None else scan["coils"].to(torch.complex128)
    lam = COIL_LAM if coils is not None else LAM
    variant = case.get("variant", recon.RECON_VARIANT_PROPOSED)
    circ = variant == recon.RECON_VARIANT_GIRAF
    if coils is None:
        x0 = _adjoint(b, masks)
    else:
        x0 = sum(c.conj() * _adjoint(bc, masks) for c, bc in zip(coils, b))
    x, eps = x0, None
    for _ in range(case["irls"]):
        if variant == recon.RECON_VARIANT_HLR_VOXEL:
            G = _voxel_gram(x, M)
            if eps is None:
                eps = EPS0 * torch.linalg.eigvalsh(G.cpu()).max().item()
            H = torch.linalg.inv(G + eps * torch.eye(M, dtype=G.dtype, device="cuda"))
            S = torch.stack([H[..., bb, a] for a, bb in _pairs(M)])
        else:
            G = _gram(x, filt, circ)[1]
            if eps is None:
                eps = EPS0 * torch.linalg.eigvalsh(G.cpu()).max().item()
            S = _weight(G, eps, filt, grid)[1]
        op = lambda v: _normal(v, masks, S, lam, M, coils, circ)  # noqa: E731, B023
        x = _cg(x, x0 - op(x), case["cg"], op)[0]
        eps /= GAMMA
    return x


# ---- the calls ----

_kept = {}


def _context():
    """The process's context and the stream that it works on."""
    if not _kept:
        stream = torch.cuda.Stream()
        _kept.update(stream=stream, ctx=recon.Context(0, cuda_stream=stream.cuda_stream))
    return _kept["ctx"].h, _kept["stream"]


def prepare(case, seed):
    kind, grid, T = case["kind"], _grid(case), case["T"]
    h, stream = _context()
    st = dict(case=case, h=h, stream=stream)
    scan = _scan(case, seed)
    if kind in ("solve", "volume", "coils", "variant"):
        st.update(b=scan["b"], masks=scan["masks"], coils=scan["coils"],
                  out=torch.empty((T,) + grid, dtype=torch.complex64, device="cuda"))
    elif kind == "batch":
        scans = [scan] + [_scan(case, int(seed) + 100003 * i) for i in range(1, case["n"])]
        st.update(b=[s["b"] for s in scans], masks=[s["masks"] for s in scans],
                  out=[torch.empty((T,) + grid, dtype=torch.complex64, device="cuda") for _ in scans])
    elif kind == "t2fit":
        st.update(x=_recovered(scan, case, seed), times=_times(T),
                  t2=torch.empty(grid, device="cuda"), amp=torch.empty(grid, device="cuda"))
    else:
        x0, G, S = _step(case, scan)
        npair, s = len(_pairs(case["M"])), G.shape[0]
        lagshape = (npair, 2 * case["N1"] - 1, 2 * case["N2"] - 1)
        if kind == "cg":
            st.update(x0=x0, x=torch.empty_like(x0), r=torch.empty_like(x0), masks=scan["masks"], S=S)
        elif kind == "gram":
            st.update(x=x0, G=torch.empty((s, s), dtype=torch.complex128, device="cuda"),
                      lags=torch.empty(lagshape, dtype=torch.complex128, device="cuda"))
        else:  # weight: the library reads G column-major
            st.update(G=G.T.contiguous(), S=torch.empty((npair,) + grid, dtype=torch.complex64, device="cuda"),
                      dsum=torch.empty(lagshape, dtype=torch.complex128, device="cuda"))
    return st


def _recovered(scan, case, seed):
    """A recovered series: the true one with a residual error of 30 dB."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 18)
    x = scan["x"]
    e = torch.randn(x.shape, generator=gen, device="cuda", dtype=torch.complex64)
    return x + e * (torch.linalg.vector_norm(x) / torch.linalg.vector_norm(e) * 10.0 ** -1.5)


def _step(case, scan):
    """x0 = A^H b, its Gram matrix and (least-squares steps) a weight S(r) with the eps of the
    twentieth IRLS iteration."""
    x0 = _adjoint(_c128(scan["b"]), scan["masks"]).to(torch.complex64)
    filt, grid = _filt(case), _grid(case)
    G = _gram(x0.to(torch.complex128), filt)[1]
    S = None
    if case["kind"] == "cg":
        eps = EPS0 / GAMMA ** 20 * torch.linalg.eigvalsh(G.cpu()).max().item()
        S = _weight(G, eps, filt, grid)[1].to(torch.complex64).contiguous()
    return x0.contiguous(), G, S


def run(st):
    c, h = st["case"], st["h"]
    kind = c["kind"]
    if kind == "solve":
        recon.recon_solve(h, st["b"], st["masks"], _filt(c), LAM, 0.0, c["irls"], c["cg"], st["out"])
        return st["out"]
    if kind == "batch":
        recon.recon_solve_batch(h, st["b"], st["masks"], _filt(c), LAM, 0.0, c["irls"], c["cg"], st["out"])
        return st["out"]
    if kind == "volume":
        recon.recon_solve3(h, st["b"], st["masks"], _filt(c), LAM, 0.0, c["irls"], c["cg"], st["out"])
        return st["out"]
    if kind == "coils":
        recon.recon_solve_coils(h, st["b"], st["masks"], st["coils"], _filt(c), COIL_LAM, 0.0, c["irls"],
                                c["cg"], st["out"])
        return st["out"]
    if kind == "variant":
        recon.recon_solve_variant(h, st["b"], st["masks"], _filt(c), LAM, 0.0, c["irls"], c["cg"],
                                  st["out"], c["variant"])
        return st["out"]
    if kind == "cg":
        # the iterate starts at x0 = A^H b on every pass; the residual that is left is the rounding
        # of the far larger A^H A p, so that the iterate is the result
        with torch.cuda.stream(st["stream"]):
            st["x"].copy_(st["x0"])
        recon.recon_cg(h, st["masks"], _filt(c), None, st["S"], LAM, st["x"], st["r"], c["cg"])
        return st["x"]
    if kind == "gram":
        recon.recon_gram(h, st["x"], _filt(c), st["G"], st["lags"])
        return st["G"], st["lags"]
    if kind == "weight":  # eps = 0.01 lambda_max(G), as in the first iteration
        eps = recon.recon_weight(h, (c["T"], c["P"], c["Q"]), _filt(c), st["G"], -EPS0, 0.0, st["S"], st["dsum"])
        return st["S"], st["dsum"], eps
    recon.recon_t2fit(h, st["x"], st["times"], st["t2"], st["amp"])
    return st["t2"], st["amp"]


def exact(case, seed):
    kind = case["kind"]
    scan = _scan(case, seed)
    if kind in ("solve", "volume", "coils", "variant"):
        return _solve(case, scan)
    if kind == "batch":
        return [_solve(case, scan)] + [_solve(case, _scan(case, int(seed) + 100003 * i))
                                       for i in range(1, case["n"])]
    if kind == "t2fit":
        return _t2_exact(_recovered(scan, case, seed), _times(case["T"]))
    x0, G, S = _step(case, scan)
    filt, grid = _filt(case), _grid(case)
    x = x0.to(torch.complex128)
    if kind == "cg":
        S = S.to(torch.complex128)
        op = lambda v: _normal(v, scan["masks"], S, LAM, case["M"])  # noqa: E731
        return _cg(x, -LAM * _apply_w(S, x, case["M"]), case["cg"], op)[0]
    if kind == "gram":
        full, G = _gram(x, filt)
        return G.T.contiguous(), _lags(full, filt)
    eps = EPS0 * torch.linalg.eigvalsh(G.cpu()).max().item()
    ds, S = _weight(G, eps, filt, grid)
    return S, ds, eps


def _t2_exact(x, times, steps=60):
    """The mono-exponential fit in float64, iterated to its fixed point; the foreground as the
    framework states it (FP32, separately rounded operations)."""
    m0 = torch.sqrt(x[0].real * x[0].real + x[0].imag * x[0].imag)
    fg = m0 > m0.max() * torch.tensor(0.1, device="cuda")
    y = x.to(torch.complex128).abs()
    t = torch.tensor(times, dtype=torch.float32, device="cuda").double().reshape(-1, 1, 1)
    ly = y.clamp_min(1e-30).log()
    dt = t - t.mean()
    R = (-(dt * (ly - ly.mean(0))).sum(0) / (dt * dt).sum()).clamp_min(1e-4)
    A = torch.exp(ly.mean(0) + R * t.mean())
    for _ in range(steps):
        e = torch.exp(-t * R)
        res, jr = A * e - y, -t * A * e
        a11, a12, a22 = (e * e).sum(0), (e * jr).sum(0), (jr * jr).sum(0)
        g1, g2 = (e * res).sum(0), (jr * res).sum(0)
        det = a11 * a22 - a12 * a12
        A = A - (a22 * g1 - a12 * g2) / det
        R = (R - (a11 * g2 - a12 * g1) / det).clamp_min(1e-4)
    nan = torch.full_like(R, float("nan"))
    return torch.where(fg, 1.0 / R, nan), torch.where(fg, A, nan)


def work(case):
    """Inputs and outputs once; the operations of the transforms, products and sums themselves."""
    kind, T, M = case["kind"], case["T"], case.get("M", 1)
    pix = math.prod(_grid(case))
    E, npair = T * pix, M * (M + 1) // 2
    if kind == "t2fit":  # start and 20 Gauss-Newton steps of ~16 operations a sample
        return dict(bytes=8 * E + 8 * pix, flops=20 * 16 * E)
    N = [case["N1"], case["N2"]] + ([case["N3"]] if "N3" in case else [])
    s, nlag = M * math.prod(N), npair * math.prod(2 * n - 1 for n in N)
    step = E * (10 * math.log2(pix) * case.get("nc", 1) + 8 * (2 * M - 1) + 20)  # one CG step
    gram = 8 * npair * E + 10 * npair * pix * math.log2(pix)
    weight = 8 * s ** 3 / 2 + 5 * npair * pix * math.log2(pix)
    if kind == "gram":
        return dict(bytes=8 * E + 16 * (s * s + nlag), flops=gram)
    if kind == "weight":
        return dict(bytes=16 * (s * s + nlag) + 8 * npair * pix, flops=weight)
    if kind == "cg":
        return dict(bytes=8 * E + E + 8 * npair * pix + 16 * E, flops=case["cg"] * step)
    if case.get("variant") == recon.RECON_VARIANT_HLR_VOXEL:
        gram, weight = 8 * npair * E, 8 * M ** 3 * pix
    n, nc = case.get("n", 1), case.get("nc", 1)
    kb = 4 if case.get("bf16") else 8
    return dict(bytes=n * (kb * nc * E + E + 8 * E + (8 * nc * pix if nc > 1 else 0)),
                flops=n * case["irls"] * (case["cg"] * step + gram + weight))
