"""GPU kernels at the sizes where their tiling can go wrong (tile edges, remainders, the smallest
and largest of a range), against plain FP64 references."""

import numpy as np
import pytest

from tests.gpu_util import assert_close, pairs_from_full, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1704_04511_gb300 import recon
    ctx = recon.Context(0)
    yield recon, ctx
    ctx.close()


def _spectrum(kind, s, rng):
    if kind == "random":  # a relative top gap of a fraction of a percent
        X = rng.standard_normal((20 * s, s)) + 1j * rng.standard_normal((20 * s, s))
        return X.conj().T @ X
    U = np.linalg.qr(rng.standard_normal((s, s)) + 1j * rng.standard_normal((s, s)))[0]
    lam = np.where(np.arange(s) < 1, 1.0, 1e-3) if kind == "one" else np.logspace(0, -8, s)
    return {"large": 1e60, "small": 1e-60}.get(kind, 1e6) * (U * lam) @ U.conj().T


@pytest.mark.parametrize("kind", ["random", "decades", "one", "large", "small"])
@pytest.mark.parametrize("filt", [(1, 1, 1), (2, 1, 1), (5, 1, 1), (7, 3, 1), (4, 8, 2), (5, 5, 3),
                                  (9, 9, 3), (7, 15, 3), (9, 9, 6)])
def test_lambda_max(R, filt, kind):
    """lambda_max of s x s matrices from s = 1 (one step) over 128 +- 1 threads, 151 worker CTAs and
    more rows than CTAs to s = 486: eps = lambda_max at eps_in = -1. The iteration ends once the
    value stands to 1e-15 of itself; its sums have s terms of rounding: 4 s 2^-53 + 1e-13."""
    import torch
    recon, ctx = R
    N1, N2, M = filt
    s = N1 * N2 * M
    G = _spectrum(kind, s, np.random.default_rng(s))
    G = 0.5 * (G + G.conj().T)
    S = torch.empty((M * (M + 1) // 2, 32, 32), dtype=torch.complex64, device="cuda")
    Gd = to_dev(np.ascontiguousarray(G.T))
    lam = np.linalg.eigvalsh(G)[-1]
    first = recon.recon_weight(ctx.h, (8, 32, 32), filt, Gd, -1.0, 0.0, S)
    assert abs(first - lam) <= (4 * s * 2.0 ** -53 + 1e-13) * lam
    for _ in range(3):  # the scratch is left ready for the next launch, and the value is the same
        assert recon.recon_weight(ctx.h, (8, 32, 32), filt, Gd, -1.0, 0.0, S) == first


@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 6])
def test_voxel_inverse(R, M):
    """The p = 0 weight alone (the inverse without an eigendecomposition), from T = M (one window)
    over T = 2 M - 1 (no frame that all pairs share) to many frames. FP64 inside at condition numbers
    of about 20, so the result is the rounding of S to FP32: 2 x 2^-24."""
    import torch
    from oracle import variants as V
    recon, ctx = R
    rng = np.random.default_rng(M)
    for T in sorted({M, 2 * M - 1, 2 * M, 13}):
        x = (rng.standard_normal((T, 16, 32)) + 1j * rng.standard_normal((T, 16, 32))).astype(np.complex64)
        x[:, 3, 5] = 0
        G = V.voxel_grams(x.astype(np.complex128), M)
        lmax = np.linalg.eigvalsh(G)[..., -1]
        eps = 0.05 * lmax + 1e-6 * lmax.max()
        ref = pairs_from_full(V.voxel_S(V.voxel_weights(G, eps, 0.0)))
        S = torch.empty(ref.shape, dtype=torch.complex64, device="cuda")
        recon.recon_voxel_weight(ctx.h, to_dev(x), M, to_dev(eps), 0.0, S)
        got = S.cpu().numpy()
        assert np.all(np.abs(got - ref) <= 2.0 ** -23 * np.abs(ref).max(axis=0))


@pytest.mark.parametrize("first", [False, True])
@pytest.mark.parametrize("T,P,Q,M", [(1, 16, 16, 1), (2, 16, 16, 2), (7, 32, 16, 3), (21, 64, 64, 2),
                                     (6, 32, 32, 6), (13, 128, 64, 4), (16, 256, 256, 3),
                                     (24, 192, 192, 1), (24, 16, 256, 5), (11, 512, 512, 2)])
def test_residual_carry(R, T, P, Q, M, first):
    """r + lam W_{S_old - S_new} x (no CG step), runs of 2, 4, 8 and 16 frames with remainders. Each
    element is a sum of M^2 complex products and r: (4 M^2 + 4) roundings of 2^-24."""
    import torch
    recon, ctx = R
    rng = np.random.default_rng(T * P + M)

    def c(*shape):
        return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)

    npair, k, lam = M * (M + 1) // 2, T - M + 1, 0.37
    x, r, So, Sn = c(T, P, Q), c(T, P, Q), c(npair, P, Q), c(npair, P, Q)
    e = 0
    full = np.zeros((M, M, P, Q), dtype=np.complex128)
    for a in range(M):
        for b in range(a, M):
            for S in (So, Sn):
                if a == b:
                    S[e].imag = 0
            d = -Sn[e].astype(np.complex128) + (0 if first else So[e])
            full[a, b], full[b, a] = d, d.conj()
            e += 1
    ref = np.zeros((T, P, Q), dtype=np.complex128) if first else r.astype(np.complex128)
    for a in range(M):
        for b in range(M):
            ref[M - 1 - a:M - 1 - a + k] += lam * full[a, b] * x[M - 1 - b:M - 1 - b + k]
    rd = to_dev(r)
    hist = recon.recon_cg(ctx.h, to_dev(np.ones((T, P, Q), np.uint8)), (3, 3, M),
                          None if first else to_dev(So), to_dev(Sn), lam, to_dev(x), rd, 0)
    got = rd.cpu().numpy()
    assert_close(got, ref, (4 * M * M + 4) * 2.0 ** -24)
    rr = float(np.sum(np.abs(got.astype(np.complex128)) ** 2))
    assert abs(hist[0] - rr) <= 1e-6 * rr


@pytest.mark.parametrize("T", [2, 8, 9, 16, 17, 31, 33, 64])
def test_t2fit_frame_counts(R, T):
    """Frame counts at the edges of the register variants, FP32 against the FP64 fit: the gate of the
    other fit tests."""
    import torch
    from oracle import t2fit
    recon, ctx = R
    rng = np.random.default_rng(T)
    times = [1.0 + 59.0 * n / max(T - 1, 1) for n in range(T)]
    t2 = 20 + 100 * rng.random((32, 32))
    x = np.exp(-np.array(times)[:, None, None] / t2) * (0.2 + rng.random((32, 32)))
    x = (x + 0.005 * (rng.standard_normal(x.shape) + 1j * rng.standard_normal(x.shape))).astype(np.complex64)
    out = torch.empty((32, 32), dtype=torch.float32, device="cuda")
    recon.recon_t2fit(ctx.h, to_dev(x), times, out)
    ref = t2fit.fit_t2(x.astype(np.complex128), times)
    got = out.cpu().numpy().astype(np.float64)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert t2fit.t2_rel_l2(ref, got) < 1e-4


@pytest.mark.parametrize("kind", ["solve", "bf16", "coils", "voxel", "volume"])
def test_graph_serves_other_buffers(R, kind):
    """One context over several scans in buffers of their own, with the masks of one changed in place
    between calls and another shape in between: bitwise the results of a fresh context without
    graphs and of one with a budget (whose graphs point into the caller's buffers)."""
    import torch
    recon, _ = R
    rng = np.random.default_rng(7)

    def scan(T, R_, P, Q):
        shape = (T, R_, P, Q) if R_ else (T, P, Q)
        n = 3 if kind == "coils" else 0
        b = rng.standard_normal(((n,) if n else ()) + shape + (2,)).astype(np.float32)
        b = torch.from_numpy(b).cuda()
        b = b.to(torch.bfloat16) if kind == "bf16" else torch.view_as_complex(b).contiguous()
        m = torch.from_numpy((rng.random(shape) < 0.4).astype(np.uint8)).cuda()
        C = torch.from_numpy((rng.standard_normal((3, P, Q)) + 1j).astype(np.complex64)).cuda() if n else None
        return b, m, C

    def call(ctx, b, m, C):
        out = torch.empty(tuple(m.shape), dtype=torch.complex64, device="cuda")
        if kind == "coils":
            recon.recon_solve_coils(ctx.h, b, m, C, (3, 3, 2), 0.1, 0.0, 2, 4, out)
        elif kind == "voxel":
            recon.recon_solve_variant(ctx.h, b, m, (1, 1, 3), 1e-2, 0.0, 2, 4, out, recon.RECON_VARIANT_HLR_VOXEL)
        elif kind == "volume":
            recon.recon_solve3(ctx.h, b, m, (3, 2, 2, 2), 1e-2, 0.0, 2, 4, out)
        else:
            recon.recon_solve(ctx.h, b, m, (3, 3, 2), 1e-2, 0.0, 3, 4, out)
        return out

    dims = [(5, 16, 32, 16)] * 3 if kind == "volume" else [(6, 0, 32, 64)] * 3
    scans = [scan(*d) for d in dims] + [scan(4, 16 if kind == "volume" else 0, 16, 32)]
    order = [0, 1, 2, 0, 3, 1, 0, 0]
    with recon.Context(0) as kept, recon.Context(0) as plain, recon.Context(0, mem_budget_bytes=1 << 30) as tight:
        recon.recon_set_option(plain.h, recon.RECON_OPT_GRAPHS, 0)
        for step, i in enumerate(order):
            b, m, C = scans[i]
            if step == 6:
                m.copy_(torch.flip(m, dims=(-1,)))
                torch.cuda.synchronize()
            got = call(kept, b, m, C)
            ref = call(plain, b, m, C)
            assert torch.equal(torch.view_as_real(got), torch.view_as_real(ref))
            assert torch.equal(torch.view_as_real(call(tight, b, m, C)), torch.view_as_real(ref))


@pytest.mark.parametrize("T", [10, 11, 12])
@pytest.mark.parametrize("Q", [128, 256])
def test_shared_memory_next_to_the_default_limit(Q, T):
    """Frame counts whose dynamic shared memory alone is just under the 48 KB of a launch without
    opt-in, and over it with the kernel's static arrays (256-point rows, T = 11), in a process state
    where no larger series came before."""
    import subprocess
    import sys
    code = ("import torch\n"
            "from paper_1704_04511_gb300 import recon\n"
            f"T, P, Q = {T}, 16, {Q}\n"
            "c = recon.Context(0)\n"
            "x = torch.randn((T, P, Q), dtype=torch.complex64, device='cuda')\n"
            "m = torch.ones((T, P, Q), dtype=torch.uint8, device='cuda')\n"
            "S = torch.zeros((1, P, Q), dtype=torch.complex64, device='cuda')\n"
            "y = torch.empty_like(x)\n"
            "torch.cuda.synchronize()\n"
            "recon.recon_apply_normal(c.h, m, (3, 3, 1), S, 0.5, x, y)\n"
            "assert (y - x).abs().max() < 1e-5 * x.abs().max()\n")
    subprocess.run([sys.executable, "-c", code], check=True, timeout=120)


def _series(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


def _hermitian_pairs(rng, M, P, Q):
    S = _series(rng, M * (M + 1) // 2, P, Q)
    full = np.zeros((M, M, P, Q), dtype=np.complex128)
    e = 0
    for a in range(M):
        S[e].imag = 0
        for b in range(a, M):
            full[a, b], full[b, a] = S[e], S[e].conj()
            e += 1
    return S, full


def _w(full, x, circ):
    M, T = full.shape[0], x.shape[0]
    y = np.zeros(x.shape, dtype=np.complex128)
    for a in range(M):
        for b in range(M):
            if circ:
                y += full[a, b] * np.roll(x, b - a, 0)
            else:
                k = T - M + 1
                y[M - 1 - a:M - 1 - a + k] += full[a, b] * x[M - 1 - b:M - 1 - b + k]
    return y


@pytest.mark.parametrize("T,P,Q,M", [(1, 16, 16, 1), (300, 16, 16, 2), (8, 32, 32, 2), (150, 16, 32, 3),
                                     (21, 64, 64, 2), (5, 192, 64, 5), (24, 192, 192, 3), (17, 32, 192, 6),
                                     (13, 512, 512, 2), (16, 16, 512, 4), (3, 512, 16, 3),
                                     (13, 256, 128, 3), (12, 128, 256, 2)])
def test_operators_at_run_edges(R, T, P, Q, M):
    """A^H A + lam W over row lengths 16 to 512 with frame counts that leave remainders in the runs of
    frames and in the CTAs' sequences, the time-circular form, three coils and the adjoint, against
    FP64: the gates of the operator parity tests (1e-5; 2e-6 for the adjoint)."""
    import torch
    recon, ctx = R
    rng = np.random.default_rng(T + P + Q)
    x = _series(rng, T, P, Q)
    S, full = _hermitian_pairs(rng, M, P, Q)
    m = (rng.random((T, P, Q)) < 0.4).astype(np.uint8)
    lam, xd = 0.7, to_dev(x)
    y = torch.empty_like(xd)

    def aha(v):
        return np.fft.ifft2(m * np.fft.fft2(v, norm="ortho"), norm="ortho")

    for circ, variant in ((False, recon.RECON_VARIANT_PROPOSED), (True, recon.RECON_VARIANT_GIRAF)):
        recon.recon_apply_normal_variant(ctx.h, to_dev(m), (1, 1, M), variant, to_dev(S), lam, xd, y)
        assert_close(y.cpu().numpy(), aha(x) + lam * _w(full, x, circ), 1e-5)
    recon.recon_adjoint(ctx.h, xd, to_dev(m), y)
    assert_close(y.cpu().numpy(), np.fft.ifft2(m * x, norm="ortho"), 2e-6)
    if 4 * T * Q + Q > 220 * 1024 // 8:
        return
    C = _series(rng, 3, P, Q)
    recon.recon_apply_normal_coils(ctx.h, to_dev(m), to_dev(C), (1, 1, M), to_dev(S), lam, xd, y)
    ref = sum(c.conj() * aha(c * x) for c in C.astype(np.complex128)) + lam * _w(full, x, False)
    assert_close(y.cpu().numpy(), ref, 1e-5)
    b = _series(rng, 3, T, P, Q)
    recon.recon_adjoint_coils(ctx.h, to_dev(b), to_dev(m), to_dev(C), y)
    assert_close(y.cpu().numpy(), sum(c.conj() * np.fft.ifft2(m * v, norm="ortho") for c, v in zip(C, b)), 2e-6)


@pytest.mark.parametrize("T,P,Q,N1,N2,M", [(2, 16, 64, 1, 1, 2), (3, 64, 192, 4, 9, 3), (16, 32, 256, 9, 2, 1),
                                           (5, 512, 64, 3, 40, 2), (13, 16, 512, 2, 5, 5), (16, 16, 512, 3, 3, 6),
                                           (9, 192, 32, 16, 3, 3), (4, 16, 128, 16, 1, 4)])
def test_gram_row_lengths(R, T, P, Q, N1, N2, M):
    """G and its lags over row lengths on both sides of the real-product variant, one to many lags on
    either axis, no shared twiddle rows (40 taps of 64) and the two largest filters: FP32 products of the
    FP32 series with compensated sums, so at most the rounding of a product (2 x 2^-24); G exactly
    Hermitian."""
    import torch
    from oracle import slr
    recon, ctx = R
    rng = np.random.default_rng(T * P + Q)
    x = _series(rng, T, P, Q)
    s, npair = N1 * N2 * M, M * (M + 1) // 2
    G = torch.empty((s, s), dtype=torch.complex128, device="cuda")
    lags = torch.empty((npair, 2 * N1 - 1, 2 * N2 - 1), dtype=torch.complex128, device="cuda")
    recon.recon_gram(ctx.h, to_dev(x), (N1, N2, M), G, lags)
    Gn = G.cpu().numpy().T
    assert_close(Gn, slr.gram_fft(x.astype(np.complex128), N1, N2, M), 2.0 ** -23)
    assert np.array_equal(Gn, Gn.conj().T)
    ln = lags.cpu().numpy()
    for a in range(M):
        e = a * (2 * M - a + 1) // 2
        assert np.array_equal(ln[e], ln[e, ::-1, ::-1].conj())


@pytest.mark.parametrize("T,P,Q,M", [(1, 16, 256, 1), (24, 32, 256, 3), (25, 16, 256, 4), (33, 16, 256, 2),
                                     (9, 256, 256, 5), (31, 16, 256, 6), (3, 16, 128, 2), (33, 16, 128, 3),
                                     (66, 32, 128, 1), (17, 64, 128, 6), (2, 512, 128, 2)])
def test_operator_in_frame_runs(R, T, P, Q, M):
    """A^H A + lam W with rows of 128 and 256 elements: one and several runs of frames, runs that leave
    threads and warps without a frame, valid and time-circular form, against FP64: the gate of the
    operator parity tests (1e-5)."""
    import torch
    recon, ctx = R
    rng = np.random.default_rng(T + P + Q + M)
    x = _series(rng, T, P, Q)
    S, full = _hermitian_pairs(rng, M, P, Q)
    m = (rng.random((T, P, Q)) < 0.4).astype(np.uint8)
    aha = np.fft.ifft2(m * np.fft.fft2(x, norm="ortho"), norm="ortho")
    xd = to_dev(x)
    y = torch.empty_like(xd)
    for circ, variant in ((False, recon.RECON_VARIANT_PROPOSED), (True, recon.RECON_VARIANT_GIRAF)):
        recon.recon_apply_normal_variant(ctx.h, to_dev(m), (1, 1, M), variant, to_dev(S), 0.7, xd, y)
        assert_close(y.cpu().numpy(), aha + 0.7 * _w(full, x, circ), 1e-5)


@pytest.mark.parametrize("T,P,Q", [(7, 64, 64), (16, 128, 128), (15, 128, 128), (64, 64, 64), (7, 256, 192),
                                   (9, 128, 256), (1, 512, 512), (512, 32, 16)])
@pytest.mark.parametrize("steps", [1, 2, 5])
def test_cg_steps_around_the_deferred_update(R, T, P, Q, steps):
    """x and r after CG steps on both sides of 2^18 elements, where x += alpha p moves to the next step's
    first pass and stays with the last one, against FP64 CG on a well-conditioned operator (eigenvalues
    0.5 to about 3): the rounding of the operator, 1e-5."""
    recon, ctx = R
    rng = np.random.default_rng(T + P + Q + steps)
    S = np.abs(rng.standard_normal((1, P, Q))).clip(0.5, 2.0).astype(np.complex64)
    x = _series(rng, T, P, Q)
    m = (rng.random((T, P, Q)) < 0.4).astype(np.uint8)
    xd, rd = to_dev(x), to_dev(np.zeros_like(x))
    recon.recon_cg(ctx.h, to_dev(m), (1, 1, 1), None, to_dev(S), 1.0, xd, rd, steps)

    def op(v):
        return np.fft.ifft2(m * np.fft.fft2(v, norm="ortho"), norm="ortho") + S[0].real * v

    ref = x.astype(np.complex128)
    r = -S[0].real * ref
    p, rr = r.copy(), np.vdot(r, r).real
    for _ in range(steps):
        q = op(p)
        alpha = rr / np.vdot(p, q).real
        ref = ref + alpha * p
        r = r - alpha * q
        new = np.vdot(r, r).real
        p, rr = r + new / rr * p, new
    scale = np.linalg.norm(x)
    assert np.linalg.norm(xd.cpu().numpy() - ref) < 1e-5 * scale
    assert np.linalg.norm(rd.cpu().numpy() - r) < 1e-5 * scale


@pytest.mark.parametrize("T", [15, 16])
def test_coil_and_volume_solves_around_the_deferred_update(R, T):
    """The same for the coil and the volume passes: one IRLS iteration against the oracle, whose
    parity gate (1e-4) it takes."""
    import torch
    from oracle import slr, slr3
    recon, ctx = R
    rng = np.random.default_rng(T)
    m = (rng.random((T, 128, 128)) < 0.4).astype(np.uint8)
    C = _series(rng, 2, 128, 128)
    C /= np.sqrt((np.abs(C) ** 2).sum(0))
    b = _series(rng, 2, T, 128, 128) * m
    out = torch.empty(m.shape, dtype=torch.complex64, device="cuda")
    recon.recon_solve_coils(ctx.h, to_dev(b), to_dev(m), to_dev(C), (2, 2, 2), 0.1, 0.0, 1, 3, out)
    ref = slr.irls(b.astype(np.complex128), m, 2, 2, 2, 0.1, 0.0, 1, 3, coils=C.astype(np.complex128))
    assert_close(out.cpu().numpy(), ref, 1e-4)
    m3 = (rng.random((T, 16, 32, 32)) < 0.4).astype(np.uint8)
    b3 = _series(rng, T, 16, 32, 32) * m3
    out = torch.empty(m3.shape, dtype=torch.complex64, device="cuda")
    recon.recon_solve3(ctx.h, to_dev(b3), to_dev(m3), (2, 2, 2, 2), 0.1, 0.0, 1, 3, out)
    ref = slr3.irls3(b3.astype(np.complex128), m3, 2, 2, 2, 2, 0.1, 0.0, 1, 3)
    assert_close(out.cpu().numpy(), ref, 1e-4)


@pytest.mark.parametrize("T,grid", [(10, (256, 192)), (11, (512, 192)), (21, (256, 192)), (21, (512, 192)),
                                    (21, (16, 16, 192)), (31, (192, 192)), (32, (192, 192)), (32, (16, 32, 192)),
                                    (42, (128, 192)), (42, (32, 16, 192)), (44, (192, 192))])
def test_operator_with_192_point_rows(R, T, grid):
    """A^H A + lam W with rows of 192 elements, whose 24 threads a frame do not divide a CTA, in frame
    counts on both sides of a run's ten frames and with enough image rows that the runs are as long
    as they get: valid and time-circular form and volumes, against FP64: the gate of the operator
    parity tests (1e-5)."""
    import torch
    recon, ctx = R
    rng = np.random.default_rng(T + grid[0])
    x = _series(rng, T, *grid)
    S, full = _hermitian_pairs(rng, 2, int(np.prod(grid[:-1])), grid[-1])
    S, full = S.reshape((3,) + grid), full.reshape((2, 2) + grid)
    m = (rng.random((T,) + grid) < 0.4).astype(np.uint8)
    axes = tuple(range(1, x.ndim))
    aha = np.fft.ifftn(m * np.fft.fftn(x, axes=axes), axes=axes)
    xd = to_dev(x)
    y = torch.empty_like(xd)
    if len(grid) == 3:
        recon.recon_apply_normal3(ctx.h, to_dev(m), (1, 1, 1, 2), to_dev(S), 0.7, xd, y)
        assert_close(y.cpu().numpy(), aha + 0.7 * _w(full, x, False), 1e-5)
        return
    for circ, variant in ((False, recon.RECON_VARIANT_PROPOSED), (True, recon.RECON_VARIANT_GIRAF)):
        recon.recon_apply_normal_variant(ctx.h, to_dev(m), (1, 1, 2), variant, to_dev(S), 0.7, xd, y)
        assert_close(y.cpu().numpy(), aha + 0.7 * _w(full, x, circ), 1e-5)


@pytest.mark.parametrize("filt", [(8, 1, 1), (5, 2, 1), (4, 3, 1), (7, 1, 2), (8, 2, 1), (6, 3, 1), (6, 2, 2),
                                  (8, 8, 1), (8, 4, 3)])
@pytest.mark.parametrize("kind", ["random", "decades", "rank"])
def test_lambda_max_at_the_last_step(R, filt, kind):
    """The same bits from every launch where the iteration can end with the step of a check: s = 8 to
    24 (the end of the Krylov space), 64 and 96 (the limit of the steps) and matrices of rank 8 and 12,
    and the value within 4 s 2^-53 + 1e-13."""
    import torch
    recon, ctx = R
    N1, N2, M = filt
    s = N1 * N2 * M
    rng = np.random.default_rng(s)
    if kind == "rank":
        X = rng.standard_normal((min(8 + s % 8, s), s)) + 1j * rng.standard_normal((min(8 + s % 8, s), s))
        G = X.conj().T @ X
    else:
        G = _spectrum(kind, s, rng)
    G = 0.5 * (G + G.conj().T)
    S = torch.empty((M * (M + 1) // 2, 32, 32), dtype=torch.complex64, device="cuda")
    Gd = to_dev(np.ascontiguousarray(G.T))
    lam = np.linalg.eigvalsh(G)[-1]
    got = {recon.recon_weight(ctx.h, (8, 32, 32), filt, Gd, -1.0, 0.0, S) for _ in range(200)}
    assert len(got) == 1
    assert abs(got.pop() - lam) <= (4 * s * 2.0 ** -53 + 1e-13) * lam


@pytest.mark.parametrize("T,P,Q", [(21, 256, 256), (24, 256, 256), (15, 256, 128), (16, 256, 128), (21, 512, 128),
                                   (24, 256, 192), (5, 512, 512)])
def test_cg_steps_where_pass_a_takes_x_or_not(R, T, P, Q):
    """Series of 2^18 elements and more with x in the first pass and without (second waves of CTAs, 128-point
    rows below 2^19 elements)."""
    test_cg_steps_around_the_deferred_update(R, T, P, Q, 3)


@pytest.mark.parametrize("T,P,Q,M", [(8, 16, 256, 5), (9, 32, 256, 6), (17, 256, 256, 4), (21, 256, 256, 5),
                                     (6, 16, 256, 6), (33, 16, 256, 4), (25, 64, 128, 5), (21, 128, 128, 4),
                                     (33, 16, 128, 6), (17, 16, 128, 3)])
def test_operator_in_frame_runs_of_many_taps(R, T, P, Q, M):
    """Rows of 128 and 256 elements with four to six taps, whose loads follow the transform, and frame
    counts that leave a partial round of W's tasks."""
    test_operator_in_frame_runs(R, T, P, Q, M)


@pytest.mark.parametrize("T,P,Q,M", [(11, 512, 192, 4), (16, 64, 192, 4), (17, 64, 192, 3), (17, 64, 192, 6),
                                     (6, 16, 512, 6), (5, 256, 512, 5), (11, 16, 64, 6), (13, 32, 32, 5),
                                     (20, 64, 16, 6)])
def test_operators_of_many_taps(R, T, P, Q, M):
    """The other row lengths with three to six taps at the edges of their runs of frames."""
    test_operators_at_run_edges(R, T, P, Q, M)


@pytest.mark.parametrize("first", [False, True])
@pytest.mark.parametrize("T,P,Q,M", [(4, 512, 512, 3), (5, 256, 512, 5), (16, 256, 256, 6), (8, 256, 128, 6),
                                     (11, 512, 192, 2), (3, 128, 256, 3), (2, 256, 256, 1)])
def test_residual_carry_run_lengths(R, T, P, Q, M, first):
    """Runs no longer than the series, and of 16 frames for many taps."""
    test_residual_carry(R, T, P, Q, M, first)


@pytest.mark.parametrize("T", [34, 36, 37, 40, 41, 61])
def test_t2fit_long_series(R, T):
    """More than 32 frames, on both sides of the groups of four that are left out beyond the last one."""
    test_t2fit_frame_counts(R, T)
