"""The integer element kernels (linear elastic, Neo-Hookean and Saint Venant-Kirchhoff force, vector-Jacobian products): their arithmetic on
the CPU against extended precision, and the element-level calls against plain torch."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2511_20687_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
H = 0.0123


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    exe = str(tmp_path_factory.mktemp("ie") / "check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-x", "c++", "-I", os.path.join(ROOT, "paper_2511_20687_gb300/csrc"), "-o",
                    exe, os.path.join(ROOT, "tests/integer_elements_check.cpp")], check=True)

    def run(u, x, nu):
        lam, mu = W.lame(1e9, nu)
        text = "\n".join(" ".join(repr(float(v)) for v in [H, lam, mu, *a.reshape(-1), *b.reshape(-1)])
                         for a, b in zip(u, x))
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return np.array([[float(v) for v in line.split()] for line in out.splitlines()])

    return run


def directions(kind, n, rng):
    """Random; a large common value with small differences; magnitudes over many orders; one component only."""
    x = rng.standard_normal((n, 3, 8))
    if kind == "rigid":
        x = rng.standard_normal((n, 3, 1)) + 1e-4 * x
    elif kind == "spread":
        x *= 10.0 ** (-6 * np.abs(rng.standard_normal((n, 3, 8))))
    elif kind == "single":
        x[:, 1:] = 0.0
    return x


@pytest.mark.parametrize("nu", [0.25, 0.45, -0.1])
@pytest.mark.parametrize("amp", [0.0, 1e-9, 1e-3, 0.2])
@pytest.mark.parametrize("kind", ["random", "rigid", "spread", "single"])
@pytest.mark.parametrize("size", [1.0, 1e-80, 1e90])
def test_closer_than_fp64(check, nu, amp, kind, size):
    """Errors in units of the largest exact entry: a corner value sums about 40 terms rounded at 2^-56 of the formats'
    unit, the direction's largest Walsh coefficient is at least 2^-4 of it: 40 x 2^-56 x 2^4 / 10 < 1e-15; and the
    rms over the sample is below that of the same formula in double."""
    rng = np.random.default_rng(4)
    u = H * (0.1 + amp * rng.uniform(-1, 1, (150, 3, 8)) / 2)
    r = check(u, size * directions(kind, 150, rng), nu)
    assert r[:, :2].all()
    assert r[:, [2, 4]].max() < 1e-15
    for k in (2, 4, 6, 8):
        assert np.sqrt(np.mean(r[:, k] ** 2)) <= np.sqrt(np.mean(r[:, k + 1] ** 2))


@pytest.mark.parametrize("nu", [0.25, 0.45, -0.1])
@pytest.mark.parametrize("amp,inside", [(0.0, True), (1e-12, True), (1e-3, True), (0.2, True), (3.0, False)])
def test_saint_venant_kirchhoff_is_closer_than_fp64(check, nu, amp, inside):
    """As above, with the error bound of the linear elastic force; strains of order one leave the range."""
    rng = np.random.default_rng(6)
    u = H * (0.3 + amp * rng.uniform(-1, 1, (150, 3, 8)))
    r = check(u, rng.standard_normal((150, 3, 8)), nu)
    good = r[:, 10] == 1
    assert good.all() if inside else good.mean() < 0.1
    assert (r[good, 11] < 1e-15).all()
    assert not good.any() or np.sqrt(np.mean(r[good, 11] ** 2)) <= np.sqrt(np.mean(r[good, 12] ** 2))


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e-310])
def test_operands_outside_the_formats_are_reported(check, bad):
    x = np.zeros((1, 3, 8))
    x[0, 1, 3] = bad
    assert check(np.zeros((1, 3, 8)), x, 0.25)[0, 0] == 0


def reference(torch, dims, h, material, lam, mu, u):
    """Internal force in plain torch FP64 (2x2x2 Gauss points), per-element lam and mu."""
    nx, ny, nz = dims
    k, j, i = torch.meshgrid(*(torch.arange(n, device=u.device) for n in (nz, ny, nx)), indexing="ij")
    n0 = (i + (nx + 1) * (j + (ny + 1) * k)).reshape(-1)
    corner = [(a & 1, (a >> 1) & 1, a >> 2) for a in range(8)]
    conn = n0[:, None] + torch.tensor([a + (nx + 1) * (b + (ny + 1) * c) for a, b, c in corner], device=u.device)
    q = [(1 - 1 / math.sqrt(3)) / 2, (1 + 1 / math.sqrt(3)) / 2]
    B = torch.zeros(8, 8, 3, dtype=torch.float64)
    for g, p in enumerate(corner):
        for a, s in enumerate(corner):
            l = [q[p[d]] if s[d] else 1 - q[p[d]] for d in range(3)]
            e = [1 if s[d] else -1 for d in range(3)]
            B[g, a] = torch.tensor([e[0] * l[1] * l[2], l[0] * e[1] * l[2], l[0] * l[1] * e[2]], dtype=torch.float64) / h
    B = B.to(u.device)
    G = torch.einsum("eac,gak->egck", u[conn], B)
    lam, mu = lam[:, None, None, None], mu[:, None, None, None]
    eye = torch.eye(3, device=u.device, dtype=torch.float64)
    if material == "le":
        P = lam * G.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] * eye + mu * (G + G.mT)
    elif material == "svk":
        E = 0.5 * (G + G.mT + G.mT @ G)
        P = (G + eye) @ (lam * E.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] * eye + 2 * mu * E)
    else:
        F = G + eye
        J = torch.det(F)[..., None, None]
        C = J * torch.linalg.inv(F).mT
        P = mu * J ** (-2 / 3) * F + (0.5 * (lam + 2 / 3 * mu) * (J * J - 1)
                                      - mu / 3 * J ** (-2 / 3) * (F * F).sum((-2, -1), keepdim=True)) / J * C
    f = torch.zeros_like(u)
    return f.index_add(0, conn.reshape(-1), h ** 3 / 8 * torch.einsum("egck,gak->eac", P, B).reshape(-1, 3))


@pytest.mark.gpu
@pytest.mark.parametrize("material", ["nh", "le"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (3, 1, 2), (4, 4, 1), (5, 7, 9), (17, 16, 15)])
@pytest.mark.parametrize("shift", [0.0, 20.0])   # 20 edges of translation: beyond the fixed-point range
def test_element_calls_match_torch(dims, material, shift):
    """Partial lane groups, warps and blocks.  The reference rounds grad u at 2^-53 of u / h (up to 20) on strains of
    1e-2, so 1e-12 (1 + 100 shift) relative; the gradient is compared through autograd of the reference."""
    import torch

    from paper_2511_20687_gb300.autograd import hex8_force
    g = torch.Generator(device="cuda").manual_seed(7)
    nn = (dims[0] + 1) * (dims[1] + 1) * (dims[2] + 1)
    ne = dims[0] * dims[1] * dims[2]
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    u = (H * (0.02 * (rand(nn, 3) - 0.5) + shift)).requires_grad_(True)
    lam = (4e8 * (1 + 0.2 * rand(ne))).requires_grad_(True)
    mu = (4e8 * (1 + 0.2 * rand(ne))).requires_grad_(True)
    y = rand(nn, 3) - 0.5
    f = hex8_force(u, lam, mu, dims, H, material)
    r = reference(torch, dims, H, material, lam, mu, u)
    got = (f,) + torch.autograd.grad(f, (u, lam, mu), y)
    want = (r,) + torch.autograd.grad(r, (u, lam, mu), y)
    for a, b in zip(got, want):
        assert (a - b).norm() <= 1e-12 * (1 + 100 * shift) * b.norm()


@pytest.mark.gpu
@pytest.mark.parametrize("material", ["nh", "le", "svk"])
@pytest.mark.parametrize("dims", [(16, 32, 32), (17, 31, 33), (64, 32, 32), (33, 65, 31)])   # sides of the size rules
def test_large_meshes_match_torch(dims, material):
    import torch

    from paper_2511_20687_gb300 import osam
    g = torch.Generator(device="cuda").manual_seed(9)
    nn = (dims[0] + 1) * (dims[1] + 1) * (dims[2] + 1)
    ne = dims[0] * dims[1] * dims[2]
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    u = H * 0.02 * (rand(nn, 3) - 0.5)
    u[: nn // 50] += 30 * H          # some elements beyond the fixed-point range, some torn across it
    lam, mu = 4e8 * (1 + 0.2 * rand(ne)), 4e8 * (1 + 0.2 * rand(ne))
    f = torch.empty_like(u)
    osam.hex8_force(dims, H, material, 0.0, 0.0, u, f, lam_e=lam, mu_e=mu)
    r = reference(torch, dims, H, material, lam, mu, u)
    near = torch.isfinite(r).all(1)   # the torn layer may be inverted: the law is undefined there
    near[nn // 50 - 2 * (dims[0] + 1) * (dims[1] + 1): nn // 50 + 2 * (dims[0] + 1) * (dims[1] + 1)] = False
    assert (f - r)[near].norm() <= 1e-12 * (1 + 100 * 30) * r[near].norm()


@pytest.mark.gpu
@pytest.mark.parametrize("material", ["nh", "le", "svk"])
@pytest.mark.parametrize("n,nz", [(16, 64), (17, 57), (24, 30)])   # 16384 elements, the size rule's last, and above it
@pytest.mark.parametrize("per_element", [False, True])
def test_step_on_both_sides_of_the_size_rule(material, n, nz, per_element):
    """Against the FP64 gather kernels (rounding of a step: 1e-12); a tenth of an edge of noise sends many Neo-Hookean
    elements out of the fixed-point range."""
    from paper_2511_20687_gb300 import osam
    p = W.bar_chain("rule", n, [nz, nz], ["fom", "fom"], material, 1e9, 0.25, 1000.0, 1e-3, 1e-6, 4, max_iters=2)
    rng = np.random.default_rng(5)
    for sd in p.subdomains:
        sd.u0 = sd.u0 + W.random_field(sd.n_nodes, 1e-3, 3)
        sd.u0[sd.dirichlet == 7] = 0.0
        if per_element:
            sd.lam_e = sd.lam * (1 + 0.3 * rng.uniform(-1, 1, sd.n_elements))
            sd.mu_e = sd.mu * (1 + 0.3 * rng.uniform(-1, 1, sd.n_elements))
    a, b = osam.Problem(p), osam.Problem(p, scatter=osam.SCATTER_GATHER)
    a.step()
    b.step()
    for i in range(2):
        for f in range(3):
            x, y = a.state(i)[f], b.state(i)[f]
            assert np.linalg.norm(x - y) <= 1e-12 * np.linalg.norm(y)


@pytest.mark.gpu
@pytest.mark.parametrize("material", ["nh", "le", "svk"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_displacement_spreads_to_its_elements(material, bad):
    import torch

    from paper_2511_20687_gb300 import osam
    dims = (5, 4, 6)
    u = torch.zeros(6 * 5 * 7, 3, device="cuda", dtype=torch.float64)
    u[3, 1] = bad
    f = torch.empty_like(u)
    osam.hex8_force(dims, H, material, 1e9, 1e9, u, f)
    assert not torch.isfinite(f[3]).any()
    assert torch.isfinite(f[6 * 5 * 3:]).all()
