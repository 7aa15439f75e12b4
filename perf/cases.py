"""The work that users of the snakuscule library have it do, as timed cases.

A pass is the call sequence of a program that holds its image on the GPU and keeps
its volume, contour and plan handles: load the voxels, write the seeding lattice (or
restore a checkpoint), evolve every contour for a window of iterations, and hand back
the whole contour state (cx, cy, cz, R, E of every contour); or the localization of an
evolved state.  Windows are the 10 iterations by which the request loop advances its
tiles (20 with the energy rule): descent is sensitive to its input where a contour sits
between touching nuclei, so longer runs of the same arithmetic drift apart from any
rounding difference and say less about a kernel than these windows do.  Images follow
the library's synthetic workloads: bright round nuclei on a darker background with
noise, made on the GPU from the seed.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_1804_06304_gb300 import ac

VOXEL = {"u8": torch.uint8, "u16": torch.uint16, "f16": torch.float16, "f32": torch.float32}
BYTES = {"u8": 1, "u16": 2, "f16": 2, "f32": 4}
CONTRAST = {"u8": 170.0, "u16": 1700.0, "f16": 1700.0, "f32": 0.7}


def listed():
    return [
        # The smallest volume the library is used on (a test crop around a few cells): launches and latency.
        dict(name="small-3d", kind="evolve", ndim=3, nx=64, ny=64, nz=32, dtype="u8", sz=1.0, stride=4.0, N=256,
             first=1, T=10),
        # One tile of the request loop for one round: the smallest tile of the serving workload.
        dict(name="tile-3d", kind="evolve", ndim=3, nx=128, ny=128, nz=128, dtype="u16", sz=1.0, stride=6.0, N=512,
             first=1, T=10),
        # The headline volume, a whole brain-like confocal stack: throughput.
        dict(name="brain-3d", kind="evolve", ndim=3, nx=1024, ny=1024, nz=256, dtype="u16", sz=2.0, stride=6.0, N=512,
             first=1, T=10),
        # A ragged stack stored as binary16, resumed from a checkpoint late in its evolution: contours of many
        # radii, away from the lattice.
        dict(name="resume-3d-f16", kind="evolve", ndim=3, nx=431, ny=389, nz=117, dtype="f16", sz=2.0, stride=6.0,
             N=512, first=41, T=10),
        # The batching form: uneven volumes, one plan with autotuned bricks replayed as a graph.  The lanes per contour
        # are fixed (to what the tuner takes on this workload), as a program that wants the same bits on every run does.
        dict(name="batch-3d", kind="batch", count=12, dtype="u8", stride=4.0, N=256, first=1, T=10),
        # A crop of a slide image: the smallest 2D call.
        dict(name="crop-2d", kind="evolve", ndim=2, nx=512, ny=512, nz=1, dtype="u8", sz=1.0, stride=6.0, N=128,
             first=1, T=10),
        # A slide image: the 2D workload of the benchmark.
        dict(name="large-2d", kind="evolve", ndim=2, nx=4096, ny=4096, nz=1, dtype="u8", sz=1.0, stride=6.0, N=128,
             first=1, T=10),
        # A ragged image in single precision with energy culling: the contours that the rule leaves running go on
        # compacted.
        dict(name="cull-2d-f32", kind="cull", ndim=2, nx=1531, ny=1117, nz=1, dtype="f32", sz=1.0, stride=6.0, N=128,
             first=1, T=20, cull=10),
        # The voxel-grid form of the energy (the paper's integration before sampling), in 2D and 3D.
        dict(name="grid-2d", kind="grid", ndim=2, nx=1024, ny=1024, nz=1, dtype="u8", sz=1.0, stride=6.0, N=1,
             first=1, T=10),
        dict(name="grid-3d", kind="grid", ndim=3, nx=256, ny=250, nz=64, dtype="u16", sz=2.0, stride=6.0, N=1,
             first=1, T=10),
        # Localization of an evolved state: a small crop, and a large stack.
        dict(name="localize-small", kind="localize", ndim=3, nx=64, ny=64, nz=32, dtype="u8", sz=1.0, stride=4.0),
        dict(name="localize-large", kind="localize", ndim=3, nx=768, ny=1024, nz=200, dtype="u8", sz=2.0, stride=6.0),
    ]


def draw(rng):
    def spread(lo, hi):   # log-uniform whole number
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    dtype = rng.choice(["u8", "u16", "u16", "f16", "f32"])
    stride = rng.choice([4.0, 5.0, 6.0, 6.0, 6.5])
    kind = rng.choice(["evolve", "evolve", "evolve", "evolve", "batch", "cull", "grid", "localize"])
    ndim = rng.choice([2, 3, 3]) if kind != "cull" else 2
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 16), dtype=dtype, stride=max(4.0, stride),
                    N=rng.choice([128, 200, 256, 384]), first=1, T=10)
    if ndim == 2:
        n = spread(200, 4096)
        dims = dict(nx=n, ny=max(64, int(n * rng.uniform(0.5, 1.0))), nz=1, sz=1.0)
        N = rng.choice([64, 100, 128, 128, 256, spread(24, 400)])
    else:
        n = spread(64, 640)
        dims = dict(nx=n, ny=max(40, int(n * rng.uniform(0.6, 1.0))), nz=spread(24, max(32, n // 3)),
                    sz=rng.choice([1.0, 2.0]))
        N = rng.choice([256, 512, 512, spread(32, 1100)])
    case = dict(kind=kind, ndim=ndim, dtype=dtype, stride=stride, **dims)
    if kind == "localize":
        return case
    if kind == "grid":
        return dict(case, N=1, first=1, T=10)
    if kind == "cull":
        return dict(case, N=N, first=1, T=20, cull=rng.randint(5, 15))
    return dict(case, N=N, first=rng.choice([1, 1, 41]), T=10)


# ------------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _image(g, shape_xyz, spacing, dtype, ndim):
    """An image [z, y, x] (or [y, x]): balls on a background, with noise, as `dtype`."""
    nx, ny, nz = shape_xyz
    vox = torch.zeros(nz * ny * nx, device="cuda")
    per, rmin, rmax = (1400, 5.0, 10.0) if ndim == 2 else (2700 / spacing[2], 3.0, 8.0)
    count = max(4, int(nx * ny * nz / per))
    ext = torch.tensor([(n - 1) * s for n, s in zip(shape_xyz, spacing)], device="cuda", dtype=torch.float64)
    c = _uniform(g, 0.0, 1.0, count, 3) * ext
    r = _uniform(g, rmin, rmax, count)
    bright = torch.ones(count, device="cuda")
    if dtype in ("u16", "f16"):   # log-normal brightness
        bright = torch.exp(0.4 * torch.randn(count, generator=g, device="cuda"))
    reach = [int(rmax / s) + 1 if d < ndim else 0 for d, s in enumerate(spacing)]
    axes = [torch.arange(-h, h + 1, device="cuda") for h in reach]
    off = torch.cartesian_prod(*axes)                                     # (o, 3): x, y, z
    sp = torch.tensor(spacing, device="cuda", dtype=torch.float64)
    n = torch.tensor(shape_xyz, device="cuda")
    step = max(1, (1 << 25) // len(off))
    for i in range(0, count, step):
        idx = torch.round(c[i:i + step] / sp).long()[:, None, :] + off
        d2 = ((idx * sp - c[i:i + step, None, :]) ** 2)[..., :ndim].sum(-1)
        inside = (d2 < (r[i:i + step] ** 2)[:, None]) & (idx >= 0).all(-1) & (idx < n).all(-1)
        flat = (idx[..., 2] * ny + idx[..., 1]) * nx + idx[..., 0]
        val = bright[i:i + step, None].expand(flat.shape)
        vox.scatter_reduce_(0, flat[inside], val[inside], "amax")
    back, fore, noise = {"u8": (30.0, 200.0, 15.0), "f32": (0.1, 0.8, 0.06)}.get(dtype, (300.0, 2000.0, 50.0))
    level = torch.full_like(vox, back)
    if dtype in ("u16", "f16"):   # an uneven background
        level = level.view(nz * ny, nx).add_(torch.linspace(0.0, 600.0, nx, device="cuda")).view(-1)
    vox = torch.where(vox > 0, vox * fore, level)
    vox += noise * torch.randn(vox.shape, generator=g, device="cuda")
    if dtype == "u8":
        vox = vox.round_().clamp_(0, 255).to(torch.uint8)
    elif dtype in ("u16", "f16"):
        vox = vox.round_().clamp_(0, 65535 if dtype == "u16" else 60000).to(torch.int32 if dtype == "u16" else torch.float16)
        vox = vox.to(VOXEL[dtype])
    return vox.view(nz, ny, nx) if ndim == 3 else vox.view(ny, nx)


def _lattice(shape_xyz, spacing, stride, ndim):
    """Seed positions as the library lays them out: (C, 3) float64 holding float32 values, x fastest."""
    axes, s32 = [], float(np.float32(stride))
    for d in range(3):
        if d >= ndim:
            axes.append(torch.zeros(1, dtype=torch.float64, device="cuda"))
            continue
        ext = shape_xyz[d] * spacing[d]
        L = max(1, int(math.floor(ext / stride)))
        first = float(np.float32(-0.5 * spacing[d] + 0.5 * (ext - L * stride) + 0.5 * stride))
        axes.append((torch.arange(L, device="cuda", dtype=torch.float64) * s32 + first).float().double())
    z, y, x = torch.meshgrid(axes[2], axes[1], axes[0], indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)


def _dims(case):
    return (case["nx"], case["ny"], case["nz"]), (1.0, 1.0, case["sz"])


def _params(case, ndim, seed):
    R0 = case["stride"] / math.sqrt(1.5)
    kw = {}
    if case["kind"] == "grid":
        kw["path"] = ac.AC_PATH_GRID
    if case["kind"] == "cull":   # a fifth of the detection threshold, tested at iteration `cull`
        kw.update(cull_iter=case["cull"], cull_E=0.2 * ac.default_E0(ndim, CONTRAST[case["dtype"]]))
    if case["first"] > 1:
        kw["first_iter"] = case["first"]
    return ac.default_params(ndim, R0, CONTRAST[case["dtype"]], N=case["N"], T=case["T"], seed=int(seed), **kw)


def _checkpoint(g, case, shape, spacing):
    """A state late in an evolution: centres moved off the lattice, radii of many sizes."""
    ndim, R0 = case["ndim"], case["stride"] / math.sqrt(1.5)
    c = _lattice(shape, spacing, case["stride"], ndim)
    state = torch.zeros(5, len(c), device="cuda")
    for d in range(ndim):
        x = c[:, d] + _uniform(g, -0.6, 0.6, len(c)) * case["stride"]
        state[d] = x.clamp(0.0, (shape[d] - 1) * spacing[d]).float()
    state[3] = _uniform(g, 0.6 * R0, 1.8 * R0, len(c)).float()
    return state


def _evolved(g, case, shape, spacing):
    """A converged state: contours gathered on cells with low energies, the others above the threshold."""
    ndim, R0 = case["ndim"], case["stride"] / math.sqrt(1.5)
    C = len(_lattice(shape, spacing, case["stride"], ndim))
    ext = torch.tensor([(n - 1) * s for n, s in zip(shape, spacing)], device="cuda", dtype=torch.float64)
    cells = _uniform(g, 0.0, 1.0, max(2, C // 24), 3) * ext
    home = torch.randint(len(cells), (C,), generator=g, device="cuda")
    on = _uniform(g, 0.0, 1.0, C) < 0.4
    near = cells[home] + 0.7 * torch.randn(C, 3, generator=g, device="cuda", dtype=torch.float64)
    c = torch.where(on[:, None], near, _uniform(g, 0.0, 1.0, C, 3) * ext)
    c = torch.minimum(c.clamp(min=0.0), ext)
    E0 = ac.default_E0(ndim, CONTRAST[case["dtype"]])
    E = torch.where(on, E0 * _uniform(g, 0.8, 4.0, C), E0 * _uniform(g, -1.0, 0.98, C))
    R = R0 * (1.1 + 0.15 * torch.randn(C, generator=g, device="cuda", dtype=torch.float64)).clamp(0.6, 2.0)
    state = torch.cat([c.T, R[None], E[None]]).float()
    if ndim == 2:
        state[2] = 0.0
    return state.contiguous()


def _batch_shapes(case):
    """Uneven volumes from 64^3 to 512x512x128, voxel counts spread over their logarithm."""
    t = (np.arange(case["count"]) * 0.618034 + 0.3) % 1.0
    return [(int(round(64 * 8 ** v)), int(round(64 * 8 ** v)), int(round(64 * 2 ** v))) for v in t]


class _Device:
    """The state of a contour handle as an array that torch can view; a view keeps the handle (and its memory) alive."""

    def __init__(self, contours):
        self.contours = contours
        self.__cuda_array_interface__ = {"data": (ac.ac_state_device_ptr(contours), False), "shape": (5, contours.count),
                                         "typestr": "<f4", "version": 3}


def _state_view(contours):
    return torch.as_tensor(_Device(contours), device="cuda")


# ------------------------------------------------------------------------ the calls
def prepare(case, seed):
    g = _generator(seed)
    if case["kind"] == "batch":
        s = dict(case=case, images=[], volumes=[], sets=[], states=[])
        for shape in _batch_shapes(case):
            s["images"].append(_image(g, shape, (1.0, 1.0, 1.0), case["dtype"], 3))
            s["volumes"].append(ac.ac_create_volume(s["images"][-1]))
            s["sets"].append(ac.ac_seed(s["volumes"][-1], stride=case["stride"]))
            s["states"].append(_state_view(s["sets"][-1]))
        p = ac.ac_autotune(s["sets"], dataclasses.replace(_params(case, 3, seed), lanes_per_contour=8))
        s["plan"] = ac.ac_plan_create(s["sets"], p, [(i, case["first"], case["T"], 0) for i in range(case["count"])])
        return s
    shape, spacing = _dims(case)
    s = dict(case=case, image=_image(g, shape, spacing, case["dtype"], case["ndim"]))
    s["volume"] = ac.ac_create_volume(s["image"], spacing=spacing)
    s["contours"] = ac.ac_seed(s["volume"], stride=case["stride"])
    s["state"] = _state_view(s["contours"])
    if case["kind"] == "localize":
        s["E0"], s["cap"] = ac.default_E0(case["ndim"], CONTRAST[case["dtype"]]), _cap(case)
        s["state"].copy_(_evolved(g, case, shape, spacing))
    else:
        s["params"] = _params(case, case["ndim"], seed)
        if case["first"] > 1:
            s["checkpoint"] = _checkpoint(g, case, shape, spacing)
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind == "localize":
        cells = ac.ac_localize(s["contours"], s["E0"], s["cap"])
        return {k: cells[k] for k in ("c", "r", "E", "id")}
    if kind == "batch":
        for image, volume, contours in zip(s["images"], s["volumes"], s["sets"]):
            ac.ac_load_volume(volume, image)
            ac.ac_reseed(contours)
        ac.ac_plan_launch(s["plan"], use_graph=True)
        return s["states"]
    ac.ac_load_volume(s["volume"], s["image"])
    if "checkpoint" in s:
        s["state"].copy_(s["checkpoint"])
    else:
        ac.ac_reseed(s["contours"])
    ac.ac_evolve(s["contours"], s["params"])
    return s["state"]


# ------------------------------------------------------------------------ what a pass cannot do without
def _cap(case):
    """The best cells that a program asks for: fewer than the state holds, so that every seed gives as many."""
    return max(4, _count(*_dims(case), case["stride"], case["ndim"]) // 64)


def _count(shape, spacing, stride, ndim):
    return math.prod(max(1, math.floor(shape[d] * spacing[d] / stride)) for d in range(ndim))


def work(case):
    b = BYTES[case["dtype"]]
    if case["kind"] == "batch":
        parts = [((x, y, z), (1.0, 1.0, 1.0), 3) for x, y, z in _batch_shapes(case)]
    else:
        parts = [(*_dims(case), case["ndim"])]
    C = sum(_count(sh, sp, case["stride"], nd) for sh, sp, nd in parts)
    voxels = sum(math.prod(sh) for sh, _, _ in parts)
    if case["kind"] == "localize":   # the state in, the cells out; a distance per pair of a cell's contours
        return {"bytes": 20.0 * C + 24.0 * _cap(case), "flops": 10.0 * 10 * 0.4 * C}
    ndim = parts[0][2]
    if case["kind"] == "grid":       # the voxels of a ball, about 30 operations each
        Ro = case["stride"] / math.sqrt(1.5) + 0.5
        points = math.pi * Ro * Ro if ndim == 2 else 4.0 / 3.0 * math.pi * Ro ** 3 / case["sz"]
        ops = 30.0
    else:                            # integer and floating operations of one sample
        points, ops = case["N"], 65.5 if ndim == 2 else 117.75
    iters = case["T"] if case["kind"] != "cull" else case["cull"] + 0.2 * (case["T"] - case["cull"])
    return {"bytes": float(voxels * b + 36.0 * C), "flops": ops * points * iters * C}


# ------------------------------------------------------------------------ the same in 64 bits
_M0, _M1, _LOW = 0xD2511F53, 0xCD9E8D57, 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    k0, k1 = key & _LOW, (key >> 32) & _LOW
    for _ in range(10):
        p0, p1 = c0 * _M0, c2 * _M1                   # modulo 2^64
        h0, h1 = (p0 >> 32) & _LOW, (p1 >> 32) & _LOW
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, p1 & _LOW, h0 ^ c3 ^ k1, p0 & _LOW
        k0, k1 = (k0 + 0x9E3779B9) & _LOW, (k1 + 0xBB67AE85) & _LOW
    return c0, c1, c2, c3


def _interpolate(img, idx, ndim):
    """Clamp-to-edge multilinear interpolation of img [z, y, x] at index positions (list x, y, z)."""
    n = img.shape[::-1]
    base, frac = [], []
    for d in range(ndim):
        x = idx[d].clamp(0.0, n[d] - 1.0)
        b = torch.floor(x).clamp(max=n[d] - 2.0)
        base.append(b.long())
        frac.append(x - b)
    flat, pitch, at = img.reshape(-1), (1, n[0], n[0] * n[1]), 0
    for d in range(ndim):
        at = at + base[d] * pitch[d]

    def along(d, at):
        if d < 0:
            return flat[at].double()
        lo, hi = along(d - 1, at), along(d - 1, at + pitch[d])
        return lo + frac[d] * (hi - lo)

    return along(ndim - 1, at)


def _sums(img, spacing, ndim, p, c, R, n, k, stream, grid):
    """J, dJ/dR and dJ/dc of Eqs. 5-10 for contours at c (C, 3) with radii R."""
    rho = 2.0 ** (-1.0 / ndim)
    dR = float(np.float32(p.dR))
    dr = rho * dR
    Ro = R + 0.5 * dR
    if grid:
        reach = [int(float(Ro.max()) / spacing[d]) + 1 if d < ndim else 0 for d in range(3)]
        off = torch.cartesian_prod(*[torch.arange(-h, h + 1, device="cuda") for h in reach])
        vox = [torch.round(c[:, d:d + 1] / spacing[d]).long() + off[None, :, d] for d in range(3)]
        x = [vox[d] * spacing[d] - c[:, d:d + 1] for d in range(ndim)]
        r = torch.sqrt(sum(v * v for v in x))
        at = [vox[d].clamp(0, img.shape[2 - d] - 1) for d in range(3)]
        I = torch.where(r <= Ro[:, None], img[at[2], at[1], at[0]].double(), 0.0)
        unit = [torch.where(r > 0, v / r.clamp(min=1e-300), 0.0) for v in x]
        measure = math.prod(spacing[:ndim])
    else:
        m = torch.arange((p.N + 1) // 2, device="cuda")[None, :]
        kk = k[:, None]
        nn, ss = torch.full_like(kk, n), torch.full_like(kk, stream)
        w = _philox(m.expand(len(k), -1), nn.expand(-1, m.shape[1]), kk.expand(-1, m.shape[1]),
                    ss.expand(-1, m.shape[1]), int(p.seed))
        w0 = torch.stack([w[0], w[2]], -1).reshape(len(k), -1)[:, :p.N]
        w1 = torch.stack([w[1], w[3]], -1).reshape(len(k), -1)[:, :p.N]
        if ndim == 3:
            rad = ((w0 >> 11).double() * 2.0 ** -21) ** (1.0 / 3.0)
            t = (w1 & 0x1FFFFF).double() * 2.0 ** -21
            a = (((w0 & 0x7FF) << 10) | (w1 >> 22)).double() * (2.0 * math.pi * 2.0 ** -21)
            s = 2.0 * torch.sqrt(t * (1.0 - t))
            unit = [s * torch.cos(a), s * torch.sin(a), 1.0 - 2.0 * t]
        else:
            rad = torch.sqrt((w0 >> 8).double() * 2.0 ** -24)
            a = (w1 >> 8).double() * (2.0 * math.pi * 2.0 ** -24)
            unit = [torch.cos(a), torch.sin(a)]
        r = rad * Ro[:, None]
        I = _interpolate(img, [(c[:, d:d + 1] + r * unit[d]) / spacing[d] for d in range(ndim)], ndim)
        measure = ((4.0 / 3.0 * math.pi * Ro ** 3 if ndim == 3 else math.pi * Ro ** 2) / p.N)
    t1 = (r - rho * R[:, None]) / dr + 0.5
    t2 = (r - R[:, None]) / dR + 0.5
    b1 = ((t1 >= 0) & (t1 < 1)).double()
    b2 = ((t2 >= 0) & (t2 < 1)).double()
    S = -1.0 + 2.0 * t1.clamp(0, 1) - t2.clamp(0, 1)
    J = (S * I).sum(1) * measure
    JR = ((b1 * (-2.0 * rho / dr) + b2 / dR) * I).sum(1) * measure
    slope = (b1 * (-2.0 / dr) + b2 / dR) * I            # -S'(r) I
    Jc = [(slope * u).sum(1) * measure for u in unit]
    return J, JR, Jc


def _evolve64(img, spacing, ndim, p, state, stream, chunk):
    """Free-running evolution of `state` (5, C) float64 over the window of p."""
    img = img.reshape(-1, *img.shape[-2:]).to(torch.int32) if img.dtype == torch.uint16 else img.reshape(-1, *img.shape[-2:])
    first = p.first_iter or 1
    f = lambda v: float(np.float32(v))   # the parameters as the library takes them  # noqa: E731
    top = [(img.shape[2 - d] - 1) * spacing[d] for d in range(3)]
    for lo in range(0, state.shape[1], chunk):
        st = state[:, lo:lo + chunk]
        c, R = st[:3].T.clone(), st[3].clone()
        E = torch.zeros_like(R)
        k = torch.arange(lo, lo + len(R), device="cuda")
        live = torch.ones_like(R, dtype=torch.bool)
        for n in range(first, first + p.T):
            J, JR, Jc = _sums(img, spacing, ndim, p, c, R, n, k, stream, p.path == ac.AC_PATH_GRID)
            inv = (2.0 * R) ** -ndim
            E = torch.where(live, J * inv, E)
            if p.cull_iter and n == p.cull_iter:
                live = live & ~(E > f(p.cull_E))
            if n == first + p.T - 1:
                break
            eta = 0.5 * f(p.eps0) / math.sqrt(n)
            d = torch.stack([-eta * j * inv for j in Jc], 1)
            norm = d.norm(dim=1, keepdim=True)
            d = torch.where(norm > f(p.max_step), d * (f(p.max_step) / norm.clamp(min=1e-300)), d)
            dRr = (-eta * (JR - ndim * J / R) * inv).clamp(-f(p.max_step), f(p.max_step))
            R = torch.where(live, (R + dRr).clamp(f(p.Rmin), f(p.Rmax)), R)
            for a in range(ndim):
                c[:, a] = torch.where(live, (c[:, a] + d[:, a]).clamp(0.0, top[a]), c[:, a])
        state[:, lo:lo + chunk] = torch.cat([c.T, R[None], E[None]])
    return state


def _localize64(state, E0, ndim, cap):
    """Greedy overlap competition in order of (E, k): the first `cap` kept contours, in that order."""
    rho = 2.0 ** (-1.0 / ndim)
    s = state.double().cpu().numpy()
    keep = np.flatnonzero(s[4] <= float(np.float32(E0)))
    order = keep[np.argsort(s[4][keep], kind="stable")]
    c, R = s[:3, order].T, s[3, order]
    h = rho * R.max()
    box = {}
    kept = []
    for i, cell in enumerate(map(tuple, np.floor(c / h).astype(int))):
        x, r = c[i], R[i]
        free = True
        for dx in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dz in (-1, 0, 1) if ndim == 3 else (0,):
                    for j in box.get((cell[0] + dx, cell[1] + dy, cell[2] + dz), ()):
                        if math.dist(x, c[j]) < rho * max(r, R[j]):
                            free = False
                            break
                    if not free:
                        break
                if not free:
                    break
            if not free:
                break
        if free:
            box.setdefault(cell, []).append(i)
            kept.append(i)
    kept = np.array(kept, dtype=int)
    kept = kept[:cap]
    return {"c": c[kept], "r": rho * R[kept], "E": s[4, order[kept]], "id": order[kept].astype(np.int32)}


def exact(case, seed):
    if work(case)["flops"] > 4e11:   # more than some seconds of double precision
        return None
    g = _generator(seed)
    if case["kind"] == "batch":
        out = []
        for i, shape in enumerate(_batch_shapes(case)):
            img = _image(g, shape, (1.0, 1.0, 1.0), case["dtype"], 3)
            out.append(_start(case, shape, (1.0, 1.0, 1.0), 3))
            _evolve64(img, (1.0, 1.0, 1.0), 3, _params(case, 3, seed), out[-1], i, (1 << 25) // case["N"])
        return out
    shape, spacing = _dims(case)
    ndim = case["ndim"]
    img = _image(g, shape, spacing, case["dtype"], ndim)
    if case["kind"] == "localize":
        if _count(shape, spacing, case["stride"], ndim) > 200_000:
            return None
        return _localize64(_evolved(g, case, shape, spacing), ac.default_E0(ndim, CONTRAST[case["dtype"]]), ndim,
                           _cap(case))
    state = _start(case, shape, spacing, ndim)
    if case["first"] > 1:
        state = _checkpoint(g, case, shape, spacing).double()
    points = case["N"] if case["kind"] != "grid" else 40 ** ndim
    return _evolve64(img, spacing, ndim, _params(case, ndim, seed), state, 0, max(1, (1 << 25) // points))


def _start(case, shape, spacing, ndim):
    c = _lattice(shape, spacing, case["stride"], ndim)
    state = torch.zeros(5, len(c), dtype=torch.float64, device="cuda")
    state[:3] = c.T
    state[3] = float(np.float32(case["stride"] / math.sqrt(1.5)))
    return state
