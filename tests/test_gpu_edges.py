"""GPU kernels at the sizes where their tiling can go wrong (tile edges, remainders, the smallest
and largest of a range), against plain FP64 references."""

import numpy as np
import pytest

from tests.gpu_util import to_dev

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
    lam = np.logspace(0, -8, s) if kind == "decades" else np.where(np.arange(s) < 1, 1.0, 1e-3)
    return 1e6 * (U * lam) @ U.conj().T


@pytest.mark.parametrize("kind", ["random", "decades", "one"])
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
