"""The voxel-grid form at the ends of its range: any spacing and any voxel values that a volume
may have.  The energy scales: with every length times a power of two (steps too) the same
image gives the same bits, centres and radii scaled, and so does every voxel times a power
of two (and the step size by its inverse), energies scaled; quotients at the ends of the
range of the kernel's own division are CUDA's."""
import dataclasses
import math
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_quotients_at_the_ends_of_their_range(tmp_path):
    from paper_1804_06304_gb300 import build
    exe = str(tmp_path / "quotient_range")
    subprocess.run([build.NVCC, *build.ARCH, "-O3", "-std=c++17", "-I" + build.INCLUDE, "-o", exe,
                    os.path.join(HERE, "_quotient_range_ref.cu")], check=True, capture_output=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.split() == ["0", "0"]


def _evolve(ndim, dtype, s, v=1.0):
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(ndim)
    dims = (40, 33) if ndim == 2 else (24, 20, 12)
    image = (rng.random(dims[::-1]) * 200).astype(dtype)
    V = ac.ac_create_volume(image * dtype(v), spacing=(s, s, 2.0 * s))
    p = ac.default_params(ndim, 3.0, 100.0, N=1, T=6, path=ac.AC_PATH_GRID)
    p = dataclasses.replace(p, dR=p.dR * s, Rmin=p.Rmin * s, Rmax=p.Rmax * s, max_step=p.max_step * s, eps0=p.eps0 * s * s / v)
    C = ac.ac_seed(V, stride=4.0 * s, R0=3.0 * s)
    ac.ac_evolve(C, p)
    return ac.ac_get_state(C)


# 2D energies are formed with (2R)^-2, 3D with (2R)^-3 and the voxel's volume: as far as those
# stay normal numbers
@pytest.mark.parametrize("ndim,exponent", [(2, -20), (2, -30), (2, -45), (2, -50), (2, 20), (2, 40), (2, 50),
                                           (3, -20), (3, -36), (3, 20), (3, 36)])
@pytest.mark.parametrize("dtype", [np.uint8, np.float32])
def test_lengths_scale(ndim, dtype, exponent):
    want, got = _evolve(ndim, dtype, 1.0), _evolve(ndim, dtype, 2.0**exponent)
    assert np.ptp(want[3]) > 0
    np.testing.assert_array_equal(got[:4] / np.float32(2.0**exponent), want[:4])
    np.testing.assert_array_equal(got[4], want[4])


@pytest.mark.parametrize("ndim", [2, 3])
@pytest.mark.parametrize("exponent", [-95, -80, -60, 60, 80, 100])
def test_voxels_scale(ndim, exponent):
    want, got = _evolve(ndim, np.float32, 1.0), _evolve(ndim, np.float32, 1.0, 2.0**exponent)
    np.testing.assert_array_equal(got[:4], want[:4])
    np.testing.assert_array_equal(got[4] / np.float32(2.0**exponent), want[4])


@pytest.mark.parametrize("dtype", [np.float16, np.float32])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_nonfinite_voxels_are_reported(bad, dtype):
    """Balls with such a voxel stop with a status, those without are not touched by it."""
    from paper_1804_06304_gb300 import ac
    image = np.random.default_rng(1).random((40, 40)).astype(dtype)
    seeds = np.array([[8, 8, 0, 3], [30, 30, 0, 3]], np.float32)
    p = ac.EvolveParams(N=1, T=1, eps0=0.0, Rmin=0.5, Rmax=9.0, path=ac.AC_PATH_GRID)
    C = ac.ac_seed(ac.ac_create_volume(image), explicit=seeds)
    ac.ac_evolve(C, p)
    want = ac.ac_get_state(C)
    image[8, 8] = bad
    C = ac.ac_seed(ac.ac_create_volume(image), explicit=seeds)
    import torch
    trace = torch.zeros((1, 2, 9), device="cuda")
    ac.ac_evolve(C, p, trace=(trace, 0, 2, 1, 2))
    with pytest.raises(ac.ACError):
        ac.ac_get_state(C)
    t = trace.cpu().numpy()[0]
    assert not np.isfinite(t[0, 4]) and np.array_equal(t[1, 4:5], want[4, 1:2])
    assert np.isfinite(t[0, 6:8]).all()   # the centre voxel has no direction


# balls with a voxel within half a unit in the last place of their border: the rows in which it lies
# end with or without it, by whether Ro^2 - dy^2 is rounded once or twice
BORDER = [(1.7738727, 5.1184683, 10.407612), (4.389767, 4.105155, 11.386679), (6.4855967, 2.9813597, 9.075569),
          (7.028953, 5.40722, 11.078195), (0.670507, 4.689889, 11.703898), (0.19110374, 5.8286586, 8.98151),
          (0.95753396, 1.2068299, 8.581024), (0.53011334, 1.3633039, 10.179406), (7.610154, 3.7508016, 11.948878),
          (1.1282305, 2.1320808, 11.602594), (0.6849803, 2.5642705, 11.291962)]


@pytest.mark.parametrize("lanes", [0, 8, 16])
def test_rows_end_where_the_fused_difference_says(lanes):
    """A ball's dE/dR over a constant image, in 64 bits over the voxels of the rows that binary32 gives
    with Ro^2 - dy^2 rounded once; a voxel more or less changes it by 2e-2 and more, rounding by 1e-4."""
    import torch
    from paper_1804_06304_gb300 import ac
    f = np.float32
    sp = np.array([0.5, 0.7], f)
    V = ac.ac_create_volume(np.full((10, 18), 100, np.uint8), spacing=(0.5, 0.7, 1.0))
    seeds = np.array([(x, y, 0.0, r) for x, y, r in BORDER], f)
    C = ac.ac_seed(V, explicit=seeds)
    trace = torch.zeros((1, len(seeds), 9), device="cuda")
    p = ac.EvolveParams(N=64, T=1, eps0=0.0, Rmin=0.5, Rmax=22.0, path=ac.AC_PATH_GRID, lanes_per_contour=lanes)
    ac.ac_evolve(C, p, trace=(trace, 0, len(seeds), 1, 2))
    inv, rho = f(1) / sp, 2.0 ** -0.5
    for t, (x, y, _, R) in zip(trace.cpu().numpy()[0], seeds):
        Ro = f(R + f(0.5))
        sums = np.zeros(2)
        for j in range(int(np.ceil(f(f(y - Ro) * inv[1]))), int(np.floor(f(f(y + Ro) * inv[1]))) + 1):
            dy = f(float(f(j)) * float(sp[1]) - float(y))
            rem = f(float(Ro) ** 2 - float(f(dy * dy)))   # exact in 64 bits, rounded once
            if rem < 0:
                continue
            chord = np.sqrt(rem)
            i = np.arange(int(np.ceil(f(f(x - chord) * inv[0]))), int(np.floor(f(f(x + chord) * inv[0]))) + 1)
            r = np.hypot(i * float(sp[0]) - float(x), float(dy))
            t1, t2 = (r - rho * float(R)) / rho + 0.5, r - float(R) + 0.5
            border = np.abs(t2 - 1.0) < 1e-6    # in the band: a voxel of the ball
            t2 = np.where(border, 1.0, t2)
            sums[0] += (-1.0 + 2.0 * np.clip(t1, 0, 1) - np.clip(t2, 0, 1)).sum()
            sums[1] += (-2.0 * ((t1 >= 0) & (t1 <= 1)) + ((t2 >= 0) & (t2 <= 1))).sum()
        want = (sums[1] - 2.0 * sums[0] / float(R)) * 100.0 * 0.5 * 0.7 / (2.0 * float(R)) ** 2
        assert abs(float(t[5]) - want) < 1e-2, (x, y, R, t[5], want)


@pytest.mark.parametrize("ndim", [2, 3])
@pytest.mark.parametrize("dtype", [np.uint8, np.float32])
def test_voxels_on_and_at_the_centre_inside_a_band(ndim, dtype):
    """Radii of half a band and less, whose centre voxel lies inside the bands: on the centre (no
    direction), off it by less than the Newton steps reach (a direction of length one), and anywhere,
    against sums in 64 bits."""
    import torch
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(ndim)
    dims = (20, 17) if ndim == 2 else (12, 11, 10)
    n, rho = 400, 2.0 ** (-1.0 / ndim)
    c = np.zeros((n, 3))
    c[:, :ndim] = rng.random((n, ndim)) * (np.array(dims) - 1)
    c[:200, :ndim] = np.round(c[:200, :ndim])                         # on a voxel
    c[:100, 0] = rng.choice([0.0, 1e-15, 3e-15, 1e-14, 1e-20], 100)   # near the first of its row
    seeds = np.column_stack([c, rng.uniform(0.2, 0.6, n)]).astype(np.float32)
    image = (rng.random(dims[::-1]) * 200).astype(dtype)
    C = ac.ac_seed(ac.ac_create_volume(image), explicit=seeds)
    trace = torch.zeros((1, n, 9), device="cuda")
    p = ac.EvolveParams(N=1, T=1, eps0=0.0, Rmin=0.1, Rmax=9.0, path=ac.AC_PATH_GRID)
    ac.ac_evolve(C, p, trace=(trace, 0, n, 1, 2))
    off = np.stack(np.meshgrid(*[np.arange(-2, 3)] * ndim, indexing="ij"), -1).reshape(-1, ndim)
    for got, s in zip(trace.cpu().numpy()[0].astype(np.float64), seeds.astype(np.float64)):
        at, R = s[:ndim], s[3]
        v = np.round(at).astype(int) + off
        x = v - at
        r = np.sqrt((x ** 2).sum(1))
        keep = r <= R + 0.5
        v, x, r = v[keep], x[keep], r[keep]
        I = image[tuple(np.clip(v[:, d], 0, dims[d] - 1) for d in reversed(range(ndim)))].astype(np.float64)
        t1, t2 = (r - rho * R) / rho + 0.5, r - R + 0.5
        b1, b2 = (t1 >= 0) & (t1 <= 1), (t2 >= 0) & (t2 <= 1)
        J = ((-1.0 + 2.0 * np.clip(t1, 0, 1) - np.clip(t2, 0, 1)) * I).sum()
        slope = np.where(r > 0, (b1 * (-2.0 / rho) + b2) * I / np.maximum(r, 1e-300), 0.0)
        inv = (2.0 * R) ** -ndim
        want = np.array([J, ((b1 * -2.0 + b2) * I).sum() - ndim * J / R] + [(slope * x[:, d]).sum() for d in range(ndim)]) * inv
        np.testing.assert_allclose(got[4:6 + ndim], want, rtol=1e-4, atol=2e-3, err_msg=str(s))
