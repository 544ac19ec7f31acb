"""GPU parity of the device calibration (Table alg:kvrobin steps 1-2; cobra_calibrate_heads)
against the oracle's (oracle/calibrate.py: numpy's symmetric eigen-solver) and the library's
host calibration, on the Llama-3-8B model's heads: K heads with the attention-KL weights
(their group's calibration queries), V heads with the MSE weights.

Both sides work in fp64.  The eigenvalues agree to 1e-10 of the largest, the weights to 1e-9
relative, the directions (after the sign rule) to 1e-7 per component: an eigenvector moves by
about (rounding x |A|) / (gap to its neighbours), and the synthetic spectra keep relative gaps
above ~1e-3 down to the 128th eigenvalue.  The allocator's order of the directions must be the
same permutation."""
import numpy as np
import pytest
import torch

from oracle import calibrate as ocal
from paper_2609_24298_gb300 import cobra, pipeline, synth

from .gpu_util import DEV

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    cobra.lib()


def heads(cfg=2, layers=(0, 17), n_kv=8):
    spec = synth.CONFIGS[cfg]
    G = spec["q_heads"] // spec["kv_heads"]
    srcs, xs, qs = [], [], []
    for side in (0, 1):
        for l in layers:
            for h in range(n_kv):
                s = synth.HeadSource(cfg, l, h, side, spec["alpha"])
                srcs.append(s)
                xs.append(s.calibration(512))
                qs.append(synth.calibration_queries(cfg, l, h, G, 512, spec["alpha"]) if side == 0 else None)
    return srcs, xs, qs


def check(got, want):
    lmax = float(np.max(want["lam"]))
    np.testing.assert_allclose(got["mu"], want["mu"], rtol=0, atol=1e-12 * max(1.0, float(np.max(np.abs(want["mu"])))))
    np.testing.assert_allclose(got["lam"], want["lam"], rtol=0, atol=1e-10 * lmax)
    np.testing.assert_allclose(got["w"], want["w"], rtol=1e-9, atol=1e-12 * float(np.max(want["w"])))
    np.testing.assert_allclose(got["U"], want["U"], rtol=0, atol=1e-7)


def test_device_calibration_matches_oracle_and_host():
    srcs, xs, qs = heads()
    dev = pipeline.calibrate_heads_device(xs, qs, device=DEV)
    host = pipeline.calibrate_heads(xs, qs)
    for d, hcal, x, q in zip(dev, host, xs, qs):
        want = ocal.calibrate_head(np.asarray(x, np.float64), q)
        check(d, want)
        check(d, hcal)


def test_device_calibration_feeds_the_same_allocation():
    srcs, xs, qs = heads(layers=(3,))
    dev = pipeline.calibrate_heads_device(xs, qs, device=DEV)
    host = pipeline.calibrate_heads(xs, qs)
    n = len(xs) // 2
    for part in (slice(0, n), slice(n, 2 * n)):
        a = cobra.cobra_allocate(np.stack([c["w"] for c in dev[part]]), 1.0)
        b = cobra.cobra_allocate(np.stack([c["w"] for c in host[part]]), 1.0)
        assert np.array_equal(a["r"], b["r"]) and np.array_equal(a["b"], b["b"])


@pytest.mark.parametrize("n_tok,n_q,n", [(1, 0, 1), (2, 3, 2), (31, 33, 1), (100, 1, 3), (128, 0, 2), (130, 64, 1), (700, 37, 5)])
def test_device_calibration_of_any_rank(n_tok, n_q, n):
    """Rank-deficient heads (fewer vectors than dimensions, equal vectors): the directions of a
    multiple eigenvalue are not unique, so the check is of what defines a decomposition - orthonormal
    directions that give the covariance back to rounding (512 eps of its norm, four roundings for each of
    128 dimensions), the rank-deficient ones too: the shift of 2^-40 of the largest entry that their
    factor needs is taken off the eigenvalues again."""
    g = np.random.default_rng(n_tok)
    A = g.standard_normal((n, 128, 128)) * (np.arange(1, 129) ** -1.3)[None, None, :]
    x = (g.standard_normal((n, n_tok, 128)) @ A.transpose(0, 2, 1) + 0.5).astype(np.float32)
    x[-1, n_tok // 2:] = x[-1, 0]  # the last head holds the same vector over and over
    q = g.standard_normal((n, n_q, 128)).astype(np.float32) if n_q else None
    xd = torch.tensor(x, device=DEV)
    qd = torch.tensor(q, device=DEV) if n_q else None
    f64 = lambda *s: torch.full(s, float("nan"), dtype=torch.float64, device=DEV)
    mu, lam, U, w = f64(n, 128), f64(n, 128), f64(n, 128 * 128), f64(n, 128)
    cobra.cobra_calibrate_heads(xd, qd, mu, lam, U, w)
    torch.cuda.synchronize()
    mu, lam, U, w = mu.cpu().numpy(), lam.cpu().numpy(), U.cpu().numpy().reshape(n, 128, 128), w.cpu().numpy()
    for h in range(n):
        xh = x[h].astype(np.float64)
        c = xh - xh.mean(axis=0)
        cov = c.T @ c / n_tok
        norm = np.linalg.norm(cov)
        np.testing.assert_allclose(mu[h], xh.mean(axis=0), rtol=0, atol=1e-12 * max(1.0, np.abs(xh).max()))
        assert np.abs(U[h] @ U[h].T - np.eye(128)).max() < 512 * 2.2e-16
        assert np.abs(U[h].T @ (lam[h][:, None] * U[h]) - cov).max() <= 512 * 2.2e-16 * norm + 1e-300
        assert np.all(np.diff(w[h]) <= 0)
        assert all(u[np.argmax(np.abs(u))] > 0 for u in U[h])
        if n_q:
            var = ((q[h].astype(np.float64) @ U[h].T) ** 2).mean(axis=0)
            np.testing.assert_allclose(w[h], var * lam[h], rtol=1e-9, atol=1e-12 * max(np.abs(w[h]).max(), 1e-300))
        else:
            assert np.array_equal(w[h], lam[h])
