"""The workloads whose speed this repository follows, over the range a user runs.

A case is one call (or one short chain of calls) through the package's Python
binding: rsx.Context.run, the single image rsx.Context.scatter_angle, and the
chain of single steps.  The sizes are those of the benchmark's and the tests'
grids (the paper's 1024 x 1024 x 128 and 2048 x 2048 x 64 studies, the
2048 x 2048 film, the 128 x 128 x 16 sample) and generic ones between them.

Inputs are drawn on the GPU from the seed: a partition of the box into c
materials (smooth fractions, or one material per voxel), alignment s in
[0, 1], Euler angles over their whole range, and resonant optical constants
near the carbon K edge.  exact() evaluates the same images in 64 bits with
plain torch, from five Fourier transforms of the per-voxel tensor.
"""
from __future__ import annotations

import math

import torch

from paper_2209_13121_gb300 import rsx

HC_EV_NM = 1239.84198
TWO_PI = 2.0 * math.pi


def _case(name, kind, nx, ny, nz, c, **more):
    d = dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, c=c, voxel_nm=5.0, precision=32,
             algorithm=1, lab=False, binary=False, energies=1, increment=2.0, end=180.0,
             host_out=False)
    d.update(more)
    return d


def listed():
    return [
        # One detector image of a small model: what an interactive check or a
        # fitting loop on a toy model asks for.  Launches and host calls count.
        _case("image_64x64x16", "image", 64, 64, 16, 2),
        # A preview of a model at low resolution, all angles, images read on
        # the host: the small sample the CPU baseline also runs.
        _case("run_128x128x16", "run", 128, 128, 16, 4, energies=2, host_out=True),
        # A model whose box was cut from a measurement or another simulation:
        # no side is a power of two; the frame-consistent reading of U^T p.
        _case("run_300x180x45", "run", 300, 180, 45, 3, lab=True, energies=2, increment=5.0,
              end=175.0),
        # A film one voxel thick (the paper's 2-D studies), two materials.
        _case("film_2048x2048x1", "run", 2048, 2048, 1, 2, binary=True, energies=2),
        # A thin stack at the usual lateral size.
        _case("run_1024x1024x16", "run", 1024, 1024, 16, 3, energies=2),
        # The smaller grid of the paper's multi-GPU study.
        _case("run_512x512x64", "run", 512, 512, 64, 4, energies=2),
        # The paper's largest grid at four materials: the benchmark's workload.
        _case("run_1024x1024x128", "run", 1024, 1024, 128, 4),
        # The paper's material-scaling grid, the largest call listed here.
        _case("run_2048x2048x64", "run", 2048, 2048, 64, 4),
        # Double precision, as used to check an FP32 study.
        _case("fp64_256x256x32", "run", 256, 256, 32, 4, precision=64, increment=10.0),
        # Algorithm 2 (N_t once per energy), which saves memory at many materials.
        _case("alg2_1024x1024x32", "run", 1024, 1024, 32, 4, algorithm=2, energies=2,
              increment=5.0),
        # Algorithm 3, the linearity restatement: a spectrum at full size.
        _case("alg3_1024x1024x128", "run", 1024, 1024, 128, 4, algorithm=3, energies=2),
        # The chain of single steps, for work on one stage at a time.
        _case("steps_256x256x32", "steps", 256, 256, 32, 3),
    ]


def _angles(case):
    return 1 + int(math.floor(case["end"] / case["increment"] + 1e-6))


def _largest_prime(n):
    p, f = 1, 2
    while n > 1:
        while n % f == 0:
            n, p = n // f, f
        f += 1
    return p


def _cost(case):
    """Voxel-angles, weighted by how dear the path is, to bound what draw() gives."""
    n = case["nx"] * case["ny"] * case["nz"] * case["energies"]
    k = 4.0 if case["algorithm"] == 3 else float(_angles(case)) if case["kind"] == "run" else 4.0
    if case["precision"] == 64:
        k *= 30.0
    if any(v & (v - 1) for v in (case["nx"], case["ny"])):
        k *= 6.0 * (1.0 + max(_largest_prime(case["nx"]), _largest_prime(case["ny"])) / 16.0)
    return n * k * (2.0 if case["algorithm"] == 2 else 1.0)


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def side():
        return 1 << rng.randint(5, 11) if rng.random() < 0.5 else log_int(24, 1500)

    nx = side()
    ny = nx if rng.random() < 0.6 else side()
    nz = 1 << rng.randint(0, 7) if rng.random() < 0.5 else log_int(1, 128)
    u = rng.random()
    kind = "run" if u < 0.75 else "image" if u < 0.9 else "steps"
    case = _case("", kind, nx, ny, nz, rng.randint(1, 8))
    del case["name"]
    case["voxel_nm"] = rng.choice([5.0, 5.0, 5.0, 2.0, 10.0])
    case["precision"] = 64 if rng.random() < 0.15 else 32
    case["algorithm"] = rng.choice([1, 1, 1, 1, 1, 2, 3]) if kind == "run" else 1
    case["lab"] = rng.random() < 0.25
    case["binary"] = rng.random() < 0.5
    case["host_out"] = kind == "run" and rng.random() < 0.25
    if kind == "run":
        case["energies"] = rng.randint(1, 3)
        case["increment"] = rng.choice([1.0, 2.0, 3.0, 5.0, 7.5, 15.0, 30.0])
        case["end"] = rng.choice([90.0, 170.0, 180.0, 360.0 - case["increment"]])
    # within the largest listed case: fewer angles, energies and slices until it is
    while _cost(case) > 2.0e10 or case["c"] * case["nx"] * case["ny"] * case["nz"] > 2 ** 29:
        if kind == "run" and case["increment"] < 45.0:
            case["increment"], case["end"] = case["increment"] * 2.0, 180.0
        elif case["energies"] > 1:
            case["energies"] -= 1
        else:
            case["nz"] = max(1, case["nz"] // 2)
            case["c"] = max(1, case["c"] - 1)
    return case


# ------------------------------------------------------------------ inputs
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _generator(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed))
    return g


def _morphology(case, seed):
    """[c][nz][ny][nx][4] (v, s, phi, theta) in the case's precision."""
    dev, g = _dev(), _generator(seed)
    c, grid = case["c"], (case["nz"], case["ny"], case["nx"])
    dt = torch.float32 if case["precision"] == 32 else torch.float64
    M = torch.empty((c,) + grid + (4,), device=dev, dtype=dt)
    # domains a few voxels wide: white noise on a coarser grid, interpolated
    total, best, win = None, None, None
    coarse = [max(1, -(-n // 4)) for n in grid]
    for j in range(c):
        f = torch.rand([1, 1] + coarse, generator=g, device=dev)
        f = torch.nn.functional.interpolate(f, size=grid, mode="trilinear", align_corners=False)
        f = f[0, 0]
        if case["binary"]:
            if best is None:
                best, win = f, torch.zeros(grid, dtype=torch.uint8, device=dev)
            else:
                win[f > best] = j
                best = torch.maximum(best, f)
        else:
            f = f.pow_(4).add_(1e-6)
            M[j, ..., 0] = f
            total = f.clone() if total is None else total.add_(f)
        del f
    for j in range(c):
        if case["binary"]:
            M[j, ..., 0] = win == j
        else:
            M[j, ..., 0] /= total
        for k, top in ((1, 1.0), (2, TWO_PI), (3, math.pi)):
            M[j, ..., k] = torch.rand(grid, generator=g, device=dev, dtype=dt) * top
    return M


def _constants(case, seed):
    """Energies (eV) and [n_E][c][4] (delta_par, beta_par, delta_perp, beta_perp)
    near the carbon K edge; the last of several materials is vacuum."""
    g = torch.Generator()
    g.manual_seed(int(seed) + 77)

    def u(lo, hi):
        return lo + (hi - lo) * float(torch.rand((), generator=g, dtype=torch.float64))

    n, c = case["energies"], case["c"]
    e0 = u(270.0, 310.0)
    E = [e0 + 2.5 * i for i in range(n)]
    K = [[[0.0] * 4 for _ in range(c)] for _ in range(n)]
    for j in range(c):
        d0, b0, res, half = u(1e-4, 1e-3), u(1e-5, 1e-4), u(282.0, 288.0), u(0.5, 2.0)
        ab, ad, par, perp = u(1e-3, 5e-3), u(5e-4, 2e-3), u(0.5, 1.5), u(0.5, 1.5)
        if c > 1 and j == c - 1:
            continue
        for i in range(n):
            x = (E[i] - res) / half
            D, L = x / (x * x + 1.0), 1.0 / (x * x + 1.0)
            K[i][j] = [d0 + par * ad * D, b0 + par * ab * L, d0 + perp * ad * D, b0 + perp * ab * L]
    return E, K


def _alpha(seed):
    g = torch.Generator()
    g.manual_seed(int(seed) + 5)
    return math.pi * float(torch.rand((), generator=g, dtype=torch.float64))


# --------------------------------------------------------------- the calls
def prepare(case, seed):
    nx, ny, nz, c = case["nx"], case["ny"], case["nz"], case["c"]
    M = _morphology(case, seed)
    E, K = _constants(case, seed)
    ctx = rsx.Context(nx, ny, nz, c, case["voxel_nm"], precision=case["precision"],
                      algorithm=case["algorithm"],
                      frame=rsx.RSX_FRAME_LAB if case["lab"] else rsx.RSX_FRAME_LITERAL)
    ctx.set_morphology(M)
    ctx.set_optical_constants(E, K)
    st = {"kind": case["kind"], "ctx": ctx, "alpha": _alpha(seed),
          "angles": (0.0, case["increment"], case["end"]), "out": None}
    if case["kind"] == "run" and not case["host_out"]:
        st["out"] = torch.empty((case["energies"], ny, nx), device="cuda", dtype=M.dtype)
    if case["kind"] in ("image", "steps"):
        st["out"] = torch.empty((ny, nx), device="cuda", dtype=M.dtype)
    if case["kind"] == "steps":
        st["p"] = torch.empty((3, nz, ny, nx, 2), device="cuda", dtype=M.dtype)
        st["acc"] = torch.empty((ny, nx), device="cuda", dtype=M.dtype)
    return st


def run(state):
    ctx, alpha = state["ctx"], state["alpha"]
    if state["kind"] == "run":
        return ctx.run(state["angles"], out=state["out"])
    if state["kind"] == "image":
        return ctx.scatter_angle(0, alpha, state["out"])
    state["acc"].zero_()
    ctx.polarization(0, alpha, state["p"])
    ctx.fft3d(state["p"])
    ctx.ewald(0, state["p"], state["out"])
    ctx.rotate_accumulate(state["out"], alpha, state["acc"])
    return state["p"], state["out"], state["acc"]


def work(case):
    """Bytes: the morphology once per energy, the images (the steps: p~ too).
    Operations: the tensor of each voxel and material once per energy; then
    per angle p of each voxel, its z transform, and the lateral transforms of
    the q_z planes the Ewald sphere meets (5 n log2 n real operations each);
    Algorithm 3: five transforms per energy and a sum per pixel and angle."""
    nx, ny, nz, c, ne = (case[k] for k in ("nx", "ny", "nz", "c", "energies"))
    n, npix, r = nx * ny * nz, nx * ny, case["precision"] // 8
    k = TWO_PI * 270.0 / HC_EV_NM
    q2 = min(k * k, 2.0 * (math.pi / case["voxel_nm"]) ** 2)
    planes = nz
    if case["kind"] != "steps":
        depth = (k - math.sqrt(k * k - q2)) * nz * case["voxel_nm"] / TWO_PI
        planes = min(nz, 2 + int(depth))
    fft = 5.0 * (n * math.log2(nz) + planes * npix * math.log2(npix))
    per = 45.0 * npix
    ang = _angles(case) if case["kind"] == "run" else 1
    if case["algorithm"] == 3:
        flops = ne * (40.0 * c * n + 5.0 * fft + ang * (40.0 + per / npix) * npix)
    else:
        flops = ne * (40.0 * c * n + ang * (30.0 * n + 3.0 * fft + per))
    data = ne * (4 * r * c * n + r * npix)
    if case["kind"] == "steps":
        data += 6 * r * n + r * npix
    return {"bytes": float(data), "flops": float(flops)}


# ---------------------------------------------------------- in 64 bits
def _tensor(case, M, K):
    """The entries xx, xy, yy, xz, yz of sum_j (N_rot N_rot - I) / (4 pi),
    [5][nz][ny][nx] complex128.  With a uniaxial N_eff = a I + b d d^T its
    square is a^2 I + (2 a b + b^2) d d^T."""
    grid = tuple(M.shape[1:4])
    nt = torch.zeros((5,) + grid, dtype=torch.complex128, device=M.device)
    step = max(1, (1 << 24) // (grid[1] * grid[2]))
    for z in range(0, grid[0], step):
        o = nt[:, z:z + step]
        for j in range(case["c"]):
            v, s, phi, th = (M[j, z:z + step, ..., k].double() for k in range(4))
            n_par, n_perp = complex(1.0 - K[j][0], K[j][1]), complex(1.0 - K[j][2], K[j][3])
            iso = (n_par + 2.0 * n_perp) / 3.0
            a = v * (s * n_perp + (1.0 - s) * iso)
            b = v * s * (n_par - n_perp)
            f = 2.0 * a * b + b * b
            a = a * a - 1.0
            st = torch.sin(th)
            d = (torch.cos(phi) * st, torch.sin(phi) * st, torch.cos(th))
            for e, (p, q) in enumerate(((0, 0), (0, 1), (1, 1), (0, 2), (1, 2))):
                o[e] += f * (d[p] * d[q])
                if p == q:
                    o[e] += a
    return nt.div_(4.0 * math.pi)


def _p_of(x, y, alpha, lab):
    """Uᵀ (x cos a + y sin a) of the three components (lab: without Uᵀ)."""
    ca, sa = math.cos(alpha), math.sin(alpha)
    p = [ca * u + sa * w for u, w in zip(x, y)]
    return p if lab else [ca * p[0] + sa * p[1], ca * p[1] - sa * p[0], p[2]]


def _sphere(case, E, dev):
    nx, ny, nz, d = case["nx"], case["ny"], case["nz"], case["voxel_nm"]
    k = TWO_PI / (HC_EV_NM / E)
    qx = TWO_PI * torch.fft.fftfreq(nx, d, dtype=torch.float64, device=dev)[None, :]
    qy = TWO_PI * torch.fft.fftfreq(ny, d, dtype=torch.float64, device=dev)[:, None]
    rad = k * k - qx * qx - qy * qy
    on = rad >= 0.0
    qz = torch.where(on, torch.sqrt(rad.clamp(min=0.0)) - k, torch.zeros_like(rad))
    t = qz / (TWO_PI / (nz * d))
    b = torch.floor(t)
    bins = [torch.remainder(b + i, nz).long() for i in (0, 1)]
    r = [(qx + 0.0 * rad) / k, (qy + 0.0 * rad) / k, (k + qz) / k]
    return k, on, bins, t - b, r


def _image(sphere, bins):
    """fftshifted image from p~ at the two bins, bins[i] = its three components."""
    k, on, _, w, r = sphere
    X = torch.zeros_like(w)
    for v, wt in zip(bins, (1.0 - w, w)):
        rv = sum(ri * vi for ri, vi in zip(r, v))
        X += wt * sum((k * k * (vi - ri * rv)).abs().square() for ri, vi in zip(r, v))
    return torch.fft.fftshift(torch.where(on, X, torch.zeros_like(X)))


def _rotate(img, alpha):
    ny, nx = img.shape
    ca, sa = math.cos(alpha), math.sin(alpha)
    x = torch.arange(nx, dtype=torch.float64, device=img.device)[None, :] - nx // 2
    y = torch.arange(ny, dtype=torch.float64, device=img.device)[:, None] - ny // 2
    fx = nx // 2 + ca * x - sa * (nx / ny) * y
    fy = ny // 2 + sa * (ny / nx) * x + ca * y
    x0, y0 = torch.floor(fx), torch.floor(fy)
    tx, ty = fx - x0, fy - y0
    out = torch.zeros_like(img)
    for dy, wy in ((0, 1.0 - ty), (1, ty)):
        for dx, wx in ((0, 1.0 - tx), (1, tx)):
            xx, yy = (x0 + dx).long(), (y0 + dy).long()
            ok = (xx >= 0) & (xx < nx) & (yy >= 0) & (yy < ny)
            out += torch.where(ok, img[yy.clamp(0, ny - 1), xx.clamp(0, nx - 1)] * wx * wy, 0.0)
    return out


def exact(case, seed):
    if not torch.cuda.is_available() and case["nx"] * case["ny"] * case["nz"] > 1 << 20:
        return None
    M = _morphology(case, seed)
    E, K = _constants(case, seed)
    alpha, dev = _alpha(seed), M.device
    images = []
    for i in range(case["energies"]):
        nt = _tensor(case, M, K[i])
        sphere = _sphere(case, E[i], dev)
        if case["kind"] == "steps":
            p = _p_of((nt[0], nt[1], nt[3]), (nt[1], nt[2], nt[4]), alpha, case["lab"])
            p = [torch.fft.fftn(f) for f in p]
            iy = torch.arange(case["ny"], device=dev)[:, None]
            ix = torch.arange(case["nx"], device=dev)[None, :]
            img = _image(sphere, [[f[b, iy, ix] for f in p] for b in sphere[2]])
            return torch.view_as_real(torch.stack(p)), img, _rotate(img, alpha)
        # the five entries' transforms at each pixel's two bins: [bin][entry]
        at = [[], []]
        for e in range(5):
            f = torch.fft.fft2(torch.fft.fft(nt[e], dim=0))
            for k in (0, 1):
                at[k].append(torch.gather(f, 0, sphere[2][k][None])[0])
            del f
        del nt

        def image(a):
            return _image(sphere, [_p_of((t[0], t[1], t[3]), (t[1], t[2], t[4]), a, case["lab"])
                                   for t in at])

        if case["kind"] == "image":
            return image(alpha)
        n = _angles(case)
        acc = torch.zeros((case["ny"], case["nx"]), dtype=torch.float64, device=dev)
        for j in range(n):
            a = math.radians(case["increment"] * j)
            acc += _rotate(image(a), a)
        images.append(acc / n)
    return torch.stack(images)
