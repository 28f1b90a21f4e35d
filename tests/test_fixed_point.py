"""The fixed-point Neo-Hookean force: its arithmetic on the CPU against extended precision, and the explicit
step that uses it against the FP64 kernels and the oracle."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import oracle as O
from paper_2511_20687_gb300 import osam
from paper_2511_20687_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
H = 0.0123


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    exe = str(tmp_path_factory.mktemp("fx") / "check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-x", "c++", "-I", os.path.join(ROOT, "paper_2511_20687_gb300/csrc"), "-o",
                    exe, os.path.join(ROOT, "tests/fixed_point_check.cpp")], check=True)

    def run(elements, nu):
        lam, mu = W.lame(1e9, nu)
        text = "\n".join(" ".join(repr(float(v)) for v in [H, lam, mu, *e.reshape(-1)]) for e in elements)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return np.array([[float(v) for v in line.split()] for line in out.splitlines()])

    return run


CORNERS = np.array([[a & 1, (a >> 1) & 1, a >> 2] for a in range(8)], float)


def elements(amp, n, rotate, shift, seed):
    """n elements [3][8]: random nodal perturbations of amp edges on a rotated, translated cube."""
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(n):
        Q = np.linalg.qr(rng.standard_normal((3, 3)))[0] if rotate else np.eye(3)
        Q *= np.linalg.det(Q)
        x = (CORNERS + 0.5 * amp * rng.uniform(-1, 1, (8, 3))) @ Q.T + shift * rng.uniform(-1, 1, 3)
        out.append(H * (x - CORNERS).T)
    return out


@pytest.mark.parametrize("nu", [0.25, 0.45])
@pytest.mark.parametrize("amp", [0.0, 1e-9, 1e-3, 0.05, 0.25])
def test_element_force_is_closer_than_fp64(check, amp, nu):
    """Every corner force within the error that the formats allow: 2^-54 times the ~40 rounded terms of a
    corner force and the factor 2 of kappa at nu = 0.45 (10 at most), each in units of wq = h^2 / 32 times a
    scale below 2 max(kappa / 2, mu): 2^-54 x 40 x 20 / 32 < 1.4e-15 (the displacement's own rounding through
    1/h adds 2^-53 x 0.1 x 10); and the rms error below that of the same formula in double."""
    r = check(elements(amp, 200, False, 0.1, 1), nu)
    assert r[:, 0].all()
    assert r[:, 1].max() < 1.6e-15
    assert np.sqrt(np.mean(r[:, 1] ** 2)) <= np.sqrt(np.mean(r[:, 2] ** 2))


@pytest.mark.parametrize("amp,rotate,shift,inside", [
    (0.02, True, 0.5, None),      # large rotations: inside unless a component spreads over 2.75 edges
    (1.6, False, 0.0, False),     # strains of order one
    (0.01, False, 30.0, False),   # translations beyond 12 edges
    (0.01, False, 3.0, True),
])
def test_range_check(check, amp, rotate, shift, inside):
    """An element is either reported outside the range or evaluated to the formats' accuracy (a rotated
    element's displacement is rounded at 2^-54 of up to 4 edges: 10 times the bound above)."""
    r = check(elements(amp, 300, rotate, shift, 2), 0.25)
    good = r[:, 0] == 1
    if inside is not None:
        assert good.all() if inside else good.mean() < 0.2
    assert good.sum() > 100 or inside is False
    assert (r[good, 1] < 1.6e-14).all()


def bar(dims, amplitude, per_element, seed=3):
    n, nz = dims
    p = W.bar_chain("fixed", n, [nz, nz], ["fom", "fom"], "nh", 1e9, 0.25, 1000.0, 1e-3, 1e-6, 6, max_iters=3)
    rng = np.random.default_rng(seed)
    for sd in p.subdomains:
        sd.u0 = sd.u0 + W.random_field(sd.n_nodes, amplitude, seed)
        sd.u0[sd.dirichlet == 7] = 0.0
        if per_element:
            sd.lam_e = sd.lam * (1 + 0.3 * rng.uniform(-1, 1, sd.n_elements))
            sd.mu_e = sd.mu * (1 + 0.3 * rng.uniform(-1, 1, sd.n_elements))
    return p


@pytest.mark.gpu
@pytest.mark.parametrize("dims", [(1, 4), (3, 7), (5, 33), (16, 32)])
@pytest.mark.parametrize("per_element", [False, True])
@pytest.mark.parametrize("amplitude", [0.0, 1e-5, 1e-3])
def test_step_matches_fp64_and_oracle(dims, per_element, amplitude):
    """The fixed-point step against the FP64 gather kernels (rounding of a step: 1e-12) and the oracle (1e-9).
    1e-3 is a tenth of an edge of noise at every node: many elements leave the range and take the FP64 path."""
    p = bar(dims, amplitude, per_element)
    a, b = osam.Problem(p), osam.Problem(p, scatter=osam.SCATTER_GATHER)
    ref = O.Problem(p)
    for _ in range(2):
        a.step(); b.step(); ref.step()
    for i in range(2):
        for f in range(3):
            x, y, z = a.state(i)[f], b.state(i)[f], ref.state(i)[f]
            scale = np.linalg.norm(z)
            assert np.linalg.norm(x - y) <= 1e-12 * scale
            assert np.linalg.norm(x - z) <= 1e-9 * scale


@pytest.mark.gpu
@pytest.mark.parametrize("shift", [0.05, 5.0])
def test_far_translation_equals_fp64(shift):
    """A free block moved by 5 and by 500 edges: inside and outside the fixed-point range."""
    p = W.single_bar("moved", 3, 6, "nh", 1e9, 0.25, 1000.0, 1e-3, 1e-6, 8)
    sd = p.subdomains[0]
    sd.dirichlet = None
    sd.u0 = sd.u0 + shift
    a, b = osam.Problem(p), osam.Problem(p, scatter=osam.SCATTER_GATHER)
    a.step(); b.step()
    for f in range(3):
        x, y = a.state(0)[f], b.state(0)[f]
        # u / h is rounded at 2^-53 of |u| / h: strains of 1e-2 carry that relative to |u| / h
        assert np.linalg.norm(x - y) <= 1e-12 * (1 + shift / 1e-2) * np.linalg.norm(y)
