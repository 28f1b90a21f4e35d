"""Which elements the integer Neo-Hookean force may evaluate: the range checks at their limits, on the CPU with the
kernels' own functions and on the GPU against the FP64 kernels."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2511_20687_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
H = 0.0123
CORNERS = np.array([[a & 1, (a >> 1) & 1, a >> 2] for a in range(8)], float)


def build(tmp_path_factory, source):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    exe = str(tmp_path_factory.mktemp("ranges") / "check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-x", "c++", "-I", os.path.join(ROOT, "paper_2511_20687_gb300/csrc"), "-o",
                    exe, os.path.join(ROOT, "tests", source)], check=True)

    def run(lines):
        text = "\n".join(" ".join(repr(float(v)) for v in np.concatenate([np.ravel(a) for a in line])) for line in lines)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return np.array([[float(v) for v in line.split()] for line in out.splitlines()])

    return run


@pytest.fixture(scope="module")
def force(tmp_path_factory):
    return build(tmp_path_factory, "fixed_point_check.cpp")


@pytest.mark.parametrize("stretch", [2.8, 4.0, 8.0, 15.9, 16.1, 16.3, 17.0, 18.0, 20.0, 23.8])
@pytest.mark.parametrize("component", [0, 1, 2])
def test_stretch_across_the_format_is_reported(force, stretch, component):
    """One component of an element spreads over up to 24 edges, half of it on either side of the origin (so that every
    node is inside the format's 12 edges): out of range for every amount, direction and sign."""
    lam, mu = W.lame(1e9, 0.25)
    lines = []
    for axis in range(3):
        for sign in (-1.0, 1.0):
            u = np.zeros((3, 8))
            u[component] = H * sign * stretch * (CORNERS[:, axis] - 0.5)
            lines.append(((H, lam, mu), u))
    assert (force(lines)[:, 0] == 0).all()


@pytest.mark.gpu
@pytest.mark.parametrize("dims", [(6, 5, 4), (41, 41, 41)])   # 8 lanes and one thread per element
@pytest.mark.parametrize("stretch", [2.9, 16.3, 17.0, 23.0])
def test_stretched_layer_matches_torch(dims, stretch):
    """A layer of elements stretched by 2.9 to 23 edges along x (u split evenly about 0); the rest moves rigidly with a
    hundredth of an edge of noise.  The reference rounds grad u at 2^-53 of u / h (up to 12) on strains of 1e-2, so
    1e-12 (1 + 100 stretch / 2) relative to the force of the unstretched part."""
    import torch

    from paper_2511_20687_gb300 import osam
    from tests.test_integer_elements import reference
    g = torch.Generator(device="cuda").manual_seed(3)
    nn = [d + 1 for d in dims]
    ne = dims[0] * dims[1] * dims[2]
    u = H * 0.01 * (torch.rand(nn[2], nn[1], nn[0], 3, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    cut = dims[0] // 2
    u[:, :, :cut + 1, 0] -= 0.5 * stretch * H
    u[:, :, cut + 1:, 0] += 0.5 * stretch * H
    u = u.reshape(-1, 3).contiguous()
    f = torch.empty_like(u)
    osam.hex8_force(dims, H, "nh", 4e8, 4e8, u, f)
    full = lambda v: torch.full((ne,), v, device="cuda", dtype=torch.float64)  # noqa: E731
    r = reference(torch, dims, H, "nh", full(4e8), full(4e8), u)
    assert torch.isfinite(r).all()
    x = torch.arange(nn[0], device="cuda").repeat(nn[1] * nn[2])
    for part in ((x == cut) | (x == cut + 1), (x < cut) | (x > cut + 1)):
        assert (f - r)[part].norm() <= 1e-12 * (1 + 50 * stretch) * r[part].norm()


@pytest.mark.gpu
@pytest.mark.parametrize("n,nz", [(4, 8), (26, 26)])   # 8 lanes and one thread per element
def test_step_with_a_stretched_layer(n, nz):
    """The explicit step across the same kind of layer against the FP64 kernels (rounding of a step: 1e-12; the
    stretched elements carry almost all of the force, so both paths round the same FP64 formula there)."""
    from paper_2511_20687_gb300 import osam
    p = W.single_bar("stretched", n, nz, "nh", 1e9, 0.25, 1000.0, 1e-3, 1e-6, 2)
    sd = p.subdomains[0]
    sd.dirichlet = None
    k = np.arange(nz + 1).repeat((n + 1) ** 2)
    sd.u0 = W.random_field(sd.n_nodes, 1e-5, 3)
    sd.u0[:, 2] += np.where(k <= nz // 2, -0.5, 0.5) * 16.3 * sd.h
    a, b = osam.Problem(p), osam.Problem(p, scatter=osam.SCATTER_GATHER)
    a.step()
    b.step()
    for f in range(3):
        x, y = a.state(0)[f], b.state(0)[f]
        assert np.linalg.norm(x - y) <= 1e-12 * np.linalg.norm(y)


@pytest.fixture(scope="module")
def contrast_force(tmp_path_factory):
    return build(tmp_path_factory, "fixed_point_contrast_check.cpp")


@pytest.mark.parametrize("nu", [0.25, 0.45])
@pytest.mark.parametrize("strain", [1e-9, 1e-4, 1e-3, 0.1])
@pytest.mark.parametrize("contrast", [1.0, 1.5, 2.0, 7.9, 8.1, 16.0, 33.0, 1e2, 1e4, 1e6, 1e12])
def test_soft_element_of_a_stiff_mesh(contrast_force, contrast, strain, nu):
    """The force of an element softer than the mesh's stiffest by any factor: rms error over the sample no larger than
    that of the same formula in double, which rounds relative to the element itself."""
    lam, mu = W.lame(1e9, nu)
    rng = np.random.default_rng(8)
    lines = [((H, lam, mu, contrast), H * 0.5 * strain * rng.uniform(-1, 1, (3, 8))) for _ in range(200)]
    r = contrast_force(lines)
    assert r[:, 0].all()
    assert np.sqrt(np.mean(r[:, 1] ** 2)) <= np.sqrt(np.mean(r[:, 2] ** 2))


@pytest.mark.gpu
@pytest.mark.parametrize("n,nz", [(4, 8), (26, 26)])   # 8 lanes and one thread per element
@pytest.mark.parametrize("contrast", [1.0, 6.0, 20.0, 1e2, 1e4, 1e6])
@pytest.mark.parametrize("precision", ["fp64", "f32x2"])
def test_step_of_a_soft_and_a_stiff_half(n, nz, contrast, precision):
    """Accelerations after a step, compared inside either half alone.  At strains of 1e-3 the FP64 formula itself is off
    by 4e-13 of the force (rms); the two paths' difference stays within five times that."""
    from paper_2511_20687_gb300 import osam
    dt = 2e-7 / np.sqrt(contrast)
    p = W.single_bar("halves", n, nz, "nh", 1e9, 0.25, 1000.0, 1e-3, dt, 2)
    sd = p.subdomains[0]
    sd.dirichlet = None
    k = np.arange(nz).repeat(n * n)
    scale = np.where(k < nz // 2, contrast, 1.0)
    sd.lam_e, sd.mu_e = sd.lam * scale, sd.mu * scale
    sd.u0 = 0.5e-3 * sd.h * np.random.default_rng(5).uniform(-1, 1, (sd.n_nodes, 3))
    mode = {"fp64": osam.FP64, "f32x2": osam.F32X2_FORCE}[precision]
    a, b = osam.Problem(p, precision=mode), osam.Problem(p, scatter=osam.SCATTER_GATHER)
    a.step()
    b.step()
    x, y = a.state(0)[2], b.state(0)[2]
    kn = np.arange(nz + 1).repeat((n + 1) ** 2)
    for half in (kn < nz // 2, kn > nz // 2):
        assert np.linalg.norm((x - y)[half]) <= 2e-12 * np.linalg.norm(y[half])


def test_buffer_entry_holds_either_kind(tmp_path):
    """Integers below 2^60 and FP64 values share an entry: every value comes back, zero and -inf through their codes."""
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    (tmp_path / "held.cpp").write_text("""
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include <limits>
#include "fixed_math.cuh"
using namespace osam::fx;
int main() {
    const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
    int bad = 0;
    for (int e = -766; e < 769; ++e)
        for (double m : {1.0, 1.25, 2.0 - 0x1p-52})
            for (double s : {-1.0, 1.0}) {
                const double v = std::ldexp(s * m, e);
                bad += !held_f64(hold_f64(v)) || f64_held(hold_f64(v)) != v;
            }
    for (double v : {0.0, -0.0, inf, -inf, -0x1p-900, 0x1p1000, -0x1p768})
        bad += !held_f64(hold_f64(v)) || f64_held(hold_f64(v)) != v;
    for (double v : {nan, -nan}) bad += !held_f64(hold_f64(v)) || !std::isnan(f64_held(hold_f64(v)));
    bad += f64_held(hold_f64(0x1p-800)) != 0.0 || f64_held(hold_f64(-0x1p900)) != -inf;
    for (int n = 0; n < 60; ++n)
        for (i64 x : {(i64)1 << n, ((i64)1 << n) - 1, ((i64)2 << n) - 1, (i64)0x123456789abcdefLL >> n})
            bad += held_f64(x) || held_f64(-x) || held_f64(~x);
    std::printf("%d\\n", bad);
}
""")
    exe = str(tmp_path / "held")
    subprocess.run(["g++", "-O2", "-std=c++17", "-x", "c++", "-I", os.path.join(ROOT, "paper_2511_20687_gb300/csrc"), "-o",
                    exe, str(tmp_path / "held.cpp")], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout.strip() == "0"


@pytest.mark.gpu
def test_fixed_point_group_takes_no_more_memory():
    """The default explicit group holds its element forces and predictor in the FP64 group's buffers."""
    import torch

    from paper_2511_20687_gb300 import osam
    p = W.single_bar("memory", 40, 80, "nh", 1e9, 0.25, 1000.0, 1e-3, 1e-7, 2)

    def taken(**kw):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        q = osam.Problem(p, **kw)
        torch.cuda.synchronize()
        used = before - torch.cuda.mem_get_info()[0]
        q.close()
        return used

    taken()                                       # one-time allocations of the library
    gather = taken(scatter=osam.SCATTER_GATHER)
    assert taken() <= gather + (4 << 20)          # the tuner's block lists; a second buffer would be 24 MB


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1e-170, 1.0, 1e160])
def test_units_outside_the_buffers_range(scale):
    """Moduli and density scaled together leave the motion as it is; 1e-170 and 1e160 take the FP64 kernels."""
    from paper_2511_20687_gb300 import osam
    out = []
    for s, mode in ((scale, osam.SCATTER_AUTO), (1.0, osam.SCATTER_GATHER)):
        p = W.single_bar("units", 4, 8, "nh", 1e9, 0.25, 1000.0, 1e-3, 1e-6, 4)
        sd = p.subdomains[0]
        sd.lam, sd.mu, sd.rho = sd.lam * s, sd.mu * s, sd.rho * s
        q = osam.Problem(p, scatter=mode)
        q.step()
        out.append(q.state(0))
    for x, y in zip(*out):
        assert np.linalg.norm(x - y) <= 1e-12 * np.linalg.norm(y)


@pytest.fixture(scope="module")
def lanes(tmp_path_factory):
    return build(tmp_path_factory, "lane_range_check.cpp")


def test_lane_range_check_bounds_every_intermediate(lanes):
    """Whatever passes the lane kernels' check keeps its Walsh coefficients below 11 and its gradients below 3.75, so no
    64-bit value wraps; elements that wrap are refused, among them one corner pulled out by 10.9 edges (coefficients
    of 10.9, a gradient of 7.8 in a format that ends at 4) and components spread over up to 24 edges."""
    rng = np.random.default_rng(12)
    lines = []
    for _ in range(4000):   # corners reached by steps of up to 2.8 edges along random paths: many at the limit
        size = rng.choice([0.5, 2.0, 2.74, 2.8, 6.0, 12.0])
        v = np.zeros(8)
        for a in range(1, 8):
            near = [v[a ^ d] for d in (1, 2, 4) if a & d]
            v[a] = np.mean([max(near), min(near)]) + size * rng.choice([-1, 1]) * rng.choice([1.0, rng.uniform()])
        lines.append((np.clip(v - 0.5 * (v.max() + v.min()), -11.99, 11.99),))
    for corner in range(8):
        for x in (-10.9, 10.9):
            lines.append((np.eye(8)[corner] * x,))
    for axis in range(3):
        for x in (2.8, 8.0, 16.0, 20.0, 23.9):
            lines.append((x * (CORNERS[:, axis] - 0.5),))
    r = lanes(lines)
    ok = r[:, 0] == 1
    assert 500 < ok.sum() < 3900
    assert (r[ok, 1] < 11.001).all() and (r[ok, 2] < 3.751).all() and not r[ok, 3].any()
    assert r[~ok, 3].any() and not ok[4000:].any()


@pytest.fixture(scope="module")
def refit(tmp_path_factory):
    return build(tmp_path_factory, "fixed_point_refit_check.cpp")


@pytest.mark.parametrize("amp", [1e-3, 0.25])
@pytest.mark.parametrize("shift", [0.0, 11.0, 13.0, 15.9, 16.1, 31.0, 33.0, 500.0, 1e5])
def test_translated_element_stays_in_range(refit, shift, amp):
    """An element anywhere within 2^22 edges keeps the format's accuracy (1.6e-15, see test_fixed_point.py) up to the
    rounding of u / h at 2^-62 of it, times the ten units that a corner force amplifies it by; and stays closer than
    the same formula in double."""
    lam, mu = W.lame(1e9, 0.25)
    rng = np.random.default_rng(13)
    lines = [((H, lam, mu), H * (0.5 * amp * rng.uniform(-1, 1, (3, 8)) + shift * rng.choice([-1, 1], (3, 1))))
             for _ in range(200)]
    r = refit(lines)
    assert r[:, 0].all() and r[:, 3].all()
    assert r[:, 1].max() < 1.6e-15 + 10 * shift * 2.0 ** -62
    assert np.sqrt(np.mean(r[:, 1] ** 2)) <= np.sqrt(np.mean(r[:, 2] ** 2))


@pytest.mark.parametrize("stretch", [2.8, 16.3, 29.5, 31.0, 32.0, 33.0, 64.0, 1024.0, 1e6, 5e6, np.inf, np.nan])
def test_torn_element_is_reported_however_far(refit, stretch):
    """Among them spreads that vanish modulo 32 edges."""
    lam, mu = W.lame(1e9, 0.25)
    lines = []
    for axis in range(3):
        for component in range(3):
            u = np.zeros((3, 8))
            u[component] = H * np.where(CORNERS[:, axis] > 0, stretch, 0.0)
            lines.append(((H, lam, mu), u))
    assert (refit(lines)[:, 0] == 0).all()


@pytest.mark.gpu
@pytest.mark.parametrize("dims", [(6, 5, 4), (41, 41, 41)])   # 8 lanes and one thread per element
@pytest.mark.parametrize("edges", [13, 64, 4096])
def test_translated_mesh_gets_the_same_force(dims, edges):
    """u and h on a binary grid, so that a translation changes no digit of the differences: every element's force and
    gradient stay the same bit for bit, and a node's differ by the order of eight FP64 additions (a few 2^-53; the FP64
    kernels' own rounding at strains of 1e-2 is 1e-14)."""
    import torch

    from paper_2511_20687_gb300 import osam
    h = 2.0 ** -6
    g = torch.Generator(device="cuda").manual_seed(17)
    nn = (dims[0] + 1) * (dims[1] + 1) * (dims[2] + 1)
    u = torch.randint(-2 ** 20, 2 ** 20, (nn, 3), generator=g, device="cuda").double() * 2.0 ** -32
    y = torch.rand(nn, 3, generator=g, device="cuda", dtype=torch.float64)
    out = []
    for x in (u, u + edges * h):
        f, ub = torch.empty_like(u), torch.empty_like(u)
        osam.hex8_force(dims, h, "nh", 4e8, 4e8, x, f)
        osam.hex8_force_vjp(dims, h, "nh", 4e8, 4e8, x, y, ub)
        out.append((f, ub))
    for a, b in zip(*out):
        assert (a - b).norm() <= 1e-15 * a.norm()


@pytest.mark.gpu
@pytest.mark.parametrize("n,nz,integrator", [(4, 8, "explicit"), (26, 26, "explicit"), (4, 8, "implicit")])
@pytest.mark.parametrize("shift", [14.0, 40.0])
def test_step_of_a_translated_bar(n, nz, integrator, shift):
    """Against the oracle: u / h is rounded at 2^-53 of the shift on strains of 1e-2."""
    from oracle import oracle as O
    from paper_2511_20687_gb300 import osam
    p = W.single_bar("moved", n, nz, "nh", 1e9, 0.25, 1000.0, 1e-3, 1e-6, 2)
    sd = p.subdomains[0]
    sd.dirichlet = np.zeros(sd.n_nodes, np.uint8)
    sd.integrator = integrator
    sd.u0 = sd.u0 + shift * sd.h
    a, b = osam.Problem(p), O.Problem(p)
    a.step()
    b.step()
    for f in range(3):
        x, y = a.state(0)[f], b.state(0)[f]
        assert np.linalg.norm(x - y) <= 1e-12 * (1 + 100 * shift) * np.linalg.norm(y)


@pytest.mark.gpu
@pytest.mark.parametrize("n,nz", [(4, 8), (26, 26)])   # 8 lanes and one thread per element
def test_step_with_a_layer_torn_by_the_modulus(n, nz):
    """A layer stretched by 32 edges, which vanishes modulo 32, against the FP64 kernels as in
    test_step_with_a_stretched_layer."""
    from paper_2511_20687_gb300 import osam
    p = W.single_bar("torn", n, nz, "nh", 1e9, 0.25, 1000.0, 1e-3, 1e-6, 2)
    sd = p.subdomains[0]
    sd.dirichlet = None
    k = np.arange(nz + 1).repeat((n + 1) ** 2)
    sd.u0 = W.random_field(sd.n_nodes, 1e-5, 3)
    sd.u0[:, 2] += np.where(k <= nz // 2, -0.5, 0.5) * 32.0 * sd.h
    a, b = osam.Problem(p), osam.Problem(p, scatter=osam.SCATTER_GATHER)
    a.step()
    b.step()
    for f in range(3):
        x, y = a.state(0)[f], b.state(0)[f]
        assert np.linalg.norm(x - y) <= 1e-12 * np.linalg.norm(y)


@pytest.fixture(scope="module")
def fixed_u(tmp_path_factory):
    return build(tmp_path_factory, "fixed_u_check.cpp")


NEAR_TWO = [np.nextafter(0.5, 1), 0.5 * (1 + 1e-11), np.nextafter(0.0078125, 1), 2.0 ** -7 * (1 + 2.0 ** -33)]


@pytest.mark.parametrize("h", [H, 0.0125, 1.0, 0.5, np.nextafter(0.5, 0)] + NEAR_TWO)
def test_displacements_of_every_mantissa(fixed_u, h):
    """Mantissas of u and of 1/h up to the largest: half a unit of rounding and 0.75 2^-58 of the value, in units of
    2^-59; only |u| / h >= 12 is marked."""
    rng = np.random.default_rng(31)
    m = np.concatenate([1 + rng.uniform(0, 1, 200), 2 - 2.0 ** -np.arange(1, 53), 1 + 2.0 ** -np.arange(1, 53)])
    u = np.concatenate([s * m * 2.0 ** e for s in (-1, 1) for e in range(-60, 12)])
    r = fixed_u([(h, v) for v in u])
    x = np.abs(r[:, 2])
    bound = 0.51 + 1.5 * x
    assert (np.isnan(r[:, 0]) == (x >= 12)).mean() > 0.999 and not np.isnan(r[x < 11.99, 0]).any()
    assert np.isnan(r[x > 12.01, 0]).all()
    near = ~np.isnan(r[:, 0])
    assert (np.abs(r[near, 0]) <= bound[near]).all()
    assert (np.abs(r[:, 1]) <= bound).all()
    assert (np.abs(r[:, 3] - 256 * r[:, 2]) <= 1.001).all()


@pytest.mark.gpu
@pytest.mark.parametrize("material", ["nh", "le", "svk"])
@pytest.mark.parametrize("h", NEAR_TWO)
@pytest.mark.parametrize("dims", [(5, 4, 3), (41, 41, 41)])   # 8 lanes and one thread per element
def test_edges_just_above_a_power_of_two(material, h, dims):
    """1/h with a mantissa just below 2, against plain torch as in test_integer_elements.py (strains of 1e-2: 1e-12)."""
    import torch

    from paper_2511_20687_gb300 import osam
    from tests.test_integer_elements import reference
    g = torch.Generator(device="cuda").manual_seed(19)
    nn = (dims[0] + 1) * (dims[1] + 1) * (dims[2] + 1)
    ne = dims[0] * dims[1] * dims[2]
    u = h * 0.02 * (torch.rand(nn, 3, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    f = torch.empty_like(u)
    osam.hex8_force(dims, h, material, 4e8, 4e8, u, f)
    full = torch.full((ne,), 4e8, device="cuda", dtype=torch.float64)
    r = reference(torch, dims, h, material, full, full, u.clone().requires_grad_(material != "svk"))
    assert (f - r).norm() <= 1e-12 * r.norm()
    if material != "svk":
        y = torch.rand(nn, 3, generator=g, device="cuda", dtype=torch.float64)
        ub = torch.empty_like(u)
        osam.hex8_force_vjp(dims, h, material, 4e8, 4e8, u, y, ub)
        v = u.clone().requires_grad_(True)
        w, = torch.autograd.grad(reference(torch, dims, h, material, full, full, v), v, y)
        assert (ub - w).norm() <= 1e-12 * w.norm()


@pytest.mark.gpu
@pytest.mark.parametrize("material", ["nh", "le", "svk"])
@pytest.mark.parametrize("integrator", ["explicit", "implicit"])
def test_step_with_edges_just_above_a_power_of_two(material, integrator):
    """The step against the oracle (1e-9 as everywhere)."""
    from oracle import oracle as O
    from paper_2511_20687_gb300 import osam
    p = W.single_bar("near", 4, 8, material, 1e9, 0.25, 1000.0, 1e-3, 1e-6, 2, h=float(np.nextafter(0.0078125, 1)))
    p.subdomains[0].integrator = integrator
    a, b = osam.Problem(p), O.Problem(p)
    a.step()
    b.step()
    for f in range(3):
        x, y = a.state(0)[f], b.state(0)[f]
        assert np.linalg.norm(x - y) <= 1e-9 * np.linalg.norm(y)
