"""The fit's products by exact splitting, through opinf_fit: partial tiles, stages, chunks and splits of k, both storage
orders, and operands that use the digits to their limits."""
import numpy as np
import pytest

from paper_2511_20687_gb300 import osam


def snapshots(kind, ns, n, rng):
    """Matrices whose leading singular values are within a factor of 10 of the first."""
    U = rng.standard_normal((ns, n))
    if kind == "full_digits":     # every element the largest mantissa, signs of a random matrix: sums at their bound
        U = np.sign(U) * (1 - 2.0 ** -53)
    elif kind == "constant":      # one direction with all digits of one sign, plus a random part
        U = 0.5 * U + (1 - 2.0 ** -53)
    elif kind == "wide":          # 80 binades along n, so that every chunk has its own exponent
        U = U * 2.0 ** (80 * np.arange(n) / n)
    elif kind == "tiny":
        U = U * 1e-120
    return U


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["random", "full_digits", "constant", "wide", "tiny"])
@pytest.mark.parametrize("ns,n", [(33, 4097), (64, 2048), (65, 70001), (130, 1023), (191, 1025)])
def test_pod_and_projection(kind, ns, n):
    """Singular values against LAPACK's and the projections against numpy.  The Gram matrix is rounded at 2^-52 of
    sigma_0^2 in each of ns^2 entries, so sigma_i is off by at most ns 2^-53 sigma_0^2 / sigma_i^2, where
    sigma_0^2 / sigma_i^2 < 100 (constant: sigma_0 itself only); the basis is re-orthonormalised to rounding."""
    rng = np.random.default_rng(11)
    U = snapshots(kind, ns, n, rng)
    A = rng.standard_normal((ns, n))
    S = rng.standard_normal((ns, 40))
    r = 6
    o = osam.opinf_fit(U, A, S, r, 1e-2, r_s=3, r_s_max=3, quadratic=False)
    s = np.linalg.svd(U, compute_uv=False)
    lead = 1 if kind == "constant" else r
    assert (s[0] / s[lead - 1]) ** 2 < 100
    assert np.abs(o["sigma"][:lead] / s[:lead] - 1).max() < 100 * ns * 2.0 ** -53
    assert np.abs(o["Phi"].T @ o["Phi"] - np.eye(r)).max() < 1e-13
    # the regression's normal equations in numpy on the returned bases: K = O^T's first block
    D = np.concatenate([U @ o["Phi"], S @ o["Phi_S"], np.ones((ns, 1))], 1)
    O = np.linalg.solve(D.T @ D + 1e-2 * np.eye(D.shape[1]), D.T @ (A @ o["Phi"]))
    scale = np.abs(O).max(axis=1)      # a row of O belongs to one feature
    cond = np.linalg.cond(D.T @ D + 1e-2 * np.eye(D.shape[1]))
    if cond < 1e10:
        assert (np.abs(o["K"].T - O[:r]).max(axis=1) <= 1e3 * cond * 2.0 ** -52 * scale.max()).all()

