"""The work that a user of the library has it do, as measured cases.

A case is one FFM product v = G W u through the Python binding:

* op "product": plan + apply + destroy on points the library has not seen (the paper's use: everything is
  recomputed for each product);
* op "apply":   one product with a plan that the program keeps (iterative solves, served scenes).

Point clouds, wavenumbers, weights and densities have the shapes of `paper_1909_05600_gb300.workloads`, drawn
here on the GPU.  Densities are single precision, as in the served requests (the library computes its fields in
FP32 whatever the density's type).  Plans take the library's defaults.
"""
import math

import numpy as np
import torch

from paper_1909_05600_gb300 import ffm, workloads

KERNEL = {"laplace": ffm.LAPLACE, "helmholtz": ffm.HELMHOLTZ, "double_layer": ffm.LAPLACE_DL,
          "gradient": ffm.LAPLACE_GRAD}
SURFACES = ("sphere", "cube_surface")


def case(op, kernel, geometry, nx, ny, eps, nrhs=1, points="f64", density="f32", **more):
    return dict(op=op, kernel=kernel, geometry=geometry, nx=nx, ny=ny, eps=eps, nrhs=nrhs, points=points,
                density=density, **more)


def listed():
    return [
        # the smallest product of an iterative solve: launches and latency
        case("apply", "laplace", "sphere", 9_973, 10_007, 1e-3, name="apply_laplace_sphere_10k"),
        # the plain Laplace configuration (points and weights in double precision), all of it per call
        case("product", "laplace", "sphere", 20_000, 20_000, 1e-3, name="product_laplace_sphere_20k"),
        # a served request of middling size: uniform volume, the tighter accuracy
        case("product", "laplace", "cube_volume", 250_000, 249_989, 1e-4, name="product_laplace_volume_250k"),
        # requests of one scene merged into one product of several densities
        case("apply", "laplace", "sphere", 100_000, 100_000, 1e-3, nrhs=8, name="apply_laplace_sphere_100k_8rhs"),
        # clustered volume in single precision, a plan that many products use
        case("apply", "laplace", "clustered", 10_000_000, 10_000_000, 1e-3, points="f32",
             name="apply_laplace_clustered_10M"),
        # the largest: the clustered volume of 1e8 + 1e8 points, all of it per call
        case("product", "laplace", "clustered", 100_000_000, 100_000_000, 1e-3, points="f32",
             name="product_laplace_clustered_1e8"),
        # the Helmholtz configuration at ten points per wavelength (k = 177), all of it per call
        case("product", "helmholtz", "sphere", 1_000_000, 1_000_000, 1e-3, density="c64",
             name="product_helmholtz_sphere_1M"),
        # a served Helmholtz request: uniform volume, low wavenumber per box, the tighter accuracy
        case("product", "helmholtz", "cube_volume", 120_011, 120_000, 1e-4, density="c64",
             name="product_helmholtz_volume_120k"),
        # many right-hand sides (scattering from many directions) on the cube's surface, X = Y
        case("apply", "helmholtz", "cube_surface", 200_000, 200_000, 1e-4, nrhs=64, density="c64",
             name="apply_helmholtz_cube_200k_64rhs"),
        # the double layer of a boundary integral equation
        case("apply", "double_layer", "sphere", 200_000, 200_000, 1e-3, name="apply_double_layer_sphere_200k"),
        # the gradient of the single layer (fields, MFIE): three outputs per target
        case("apply", "gradient", "sphere", 300_000, 299_993, 1e-3, name="apply_gradient_sphere_300k"),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["apply_laplace", "product_laplace", "multi_laplace", "clustered", "product_helmholtz",
                         "multi_helmholtz", "double_layer", "gradient"])
    eps = rng.choice([1e-3, 1e-4])
    geometry = rng.choice(["sphere", "cube_surface", "cube_volume"])
    if family == "clustered":
        n = _size(rng, 1_000_000, 100_000_000)
        return case(rng.choice(["product", "apply"]) if n < 20_000_000 else "product", "laplace", "clustered", n,
                    int(n * rng.uniform(0.9, 1.0)), 1e-3, points="f32")
    if family == "multi_helmholtz":
        n = _size(rng, 20_000, 200_000)
        return case("apply", "helmholtz", "cube_surface", n, n, 1e-4, nrhs=_size(rng, 2, 64), density="c64")
    if family == "product_helmholtz":
        n = _size(rng, 10_000, 1_000_000 if geometry in SURFACES else 300_000)
        return case("product", "helmholtz", geometry, n, int(n * rng.uniform(0.7, 1.0)), eps, density="c64")
    if family == "double_layer":
        n = _size(rng, 10_000, 1_000_000)
        return case("apply", "double_layer", "sphere", n, int(n * rng.uniform(0.7, 1.0)), eps)
    if family == "gradient":
        n = _size(rng, 10_000, 1_000_000)
        return case("apply", "gradient", rng.choice(["sphere", "cube_volume"]), n, int(n * rng.uniform(0.7, 1.0)), eps)
    if family == "multi_laplace":
        n = _size(rng, 10_000, 500_000)
        return case("apply", "laplace", geometry, n, int(n * rng.uniform(0.7, 1.0)), eps, nrhs=_size(rng, 2, 16))
    n = _size(rng, 10_000, 2_000_000)
    return case("apply" if family == "apply_laplace" else "product", "laplace", geometry, n,
                int(n * rng.uniform(0.7, 1.0)), eps)


# ---------------------------------------------------------------- inputs


def _points(geometry, n, dtype, g):
    dev = "cuda"
    if geometry == "sphere":
        p = torch.randn((n, 3), dtype=torch.float64, device=dev, generator=g)
        p = p / p.norm(dim=1, keepdim=True)
    elif geometry == "cube_surface":
        p = torch.rand((n, 3), dtype=torch.float64, device=dev, generator=g)
        face = torch.randint(0, 6, (n, 1), device=dev, generator=g)
        p.scatter_(1, face % 3, (face // 3).double())
    elif geometry == "cube_volume":
        p = torch.rand((n, 3), dtype=torch.float64, device=dev, generator=g)
    else:  # the 8-Gaussian mixture with the shared centres of workloads.gaussian_mixture
        c = torch.as_tensor(np.random.default_rng(7).random((8, 3)), dtype=dtype, device=dev)
        p = torch.randn((n, 3), dtype=dtype, device=dev, generator=g).mul_(0.05)
        p += c[torch.randint(0, 8, (n,), device=dev, generator=g)]
    return p.to(dtype).contiguous()


def _wavenumber(c):
    return workloads.wavenumber_ppw(max(c["nx"], c["ny"]), c["geometry"]) if c["kernel"] == "helmholtz" else 0.0


def _inputs(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dtype = torch.float32 if c["points"] == "f32" else torch.float64
    ny, nrhs, k = c["ny"], c["nrhs"], _wavenumber(c)
    X = _points(c["geometry"], c["nx"], dtype, g)
    shape = (ny,) if nrhs == 1 else (nrhs, ny)
    if c["kernel"] == "helmholtz" and nrhs > 1:
        Y = X.clone()  # one surface, plane-wave densities e^{i k d.y} from directions uniform on the sphere
        d = _points("sphere", nrhs, torch.float64, g)
        u = torch.polar(torch.ones(shape, dtype=torch.float64, device="cuda"), k * (d @ Y.double().T)).to(torch.complex64)
    else:
        Y = _points(c["geometry"], ny, dtype, g)
        if c["geometry"] == "clustered":
            u = torch.rand(shape, dtype=torch.float32, device="cuda", generator=g).mul_(2.0).sub_(1.0)
        elif c["kernel"] == "helmholtz":
            u = torch.randn(shape + (2,), dtype=torch.float32, device="cuda", generator=g)
            u = torch.view_as_complex(u)
        else:
            u = torch.randn(shape, dtype=torch.float32, device="cuda", generator=g)
    area = 1.0 if c["geometry"] == "clustered" else workloads.AREA[c["geometry"]]
    w = torch.full((ny,), area / ny, dtype=dtype, device="cuda")
    normals = Y.clone() if c["kernel"] == "double_layer" else None  # the unit sphere's own normals
    return X, Y, u.contiguous(), w, normals, k


def _plan(c, X, Y, w, normals, k):
    return ffm.Plan(X, Y, KERNEL[c["kernel"]], k, c["eps"], weights=w, normals=normals)


def prepare(case, seed):
    X, Y, u, w, normals, k = _inputs(case, seed)
    if case["op"] == "apply":
        return {"plan": _plan(case, X, Y, w, normals, k), "u": u}
    return {"case": case, "points": (X, Y, w, normals, k), "u": u}


def run(state):
    if "plan" in state:
        return state["plan"].apply(state["u"])
    with _plan(state["case"], *state["points"]) as plan:
        return plan.apply(state["u"])


# ---------------------------------------------------------------- what a pass cannot do without


def work(case):
    nx, ny, nrhs = case["nx"], case["ny"], case["nrhs"]
    real = 4 if case["points"] == "f32" else 8
    outs = 3 if case["kernel"] == "gradient" else 1
    value = 8 if case["density"] == "c64" else 4
    # the points and weights are read once in a product; with a kept plan a pass still reads a position (FP32)
    # per point and a weight per source
    per_point = 3 * real if case["op"] == "product" else 12
    nbytes = per_point * (nx + ny) + real * ny + value * nrhs * (ny + outs * nx)
    # each target meets the points of its own and the touching leaves (about 24 points in a leaf; 9 leaves on a
    # surface, 27 in a volume), about ten operations a pair (twenty for a complex exponential)
    near = nx * 24 * (9 if case["geometry"] in SURFACES else 27) * (20 if case["kernel"] == "helmholtz" else 10)
    return {"bytes": float(nbytes), "flops": float(near * outs * (1 if nrhs == 1 else 1 + 0.2 * nrhs))}


# ---------------------------------------------------------------- the same products as direct sums in 64 bits


def exact(case, seed):
    nx, ny, nrhs = case["nx"], case["ny"], case["nrhs"]
    helm = case["kernel"] == "helmholtz"
    if float(nx) * ny * ((4.0 + 2.0 * nrhs) if helm else (1.0 + 0.2 * nrhs)) > 2.0e11:
        return None
    X, Y, u, w, normals, k = _inputs(case, seed)
    X, Y = X.double(), Y.double()
    q = (u.reshape(nrhs, ny).to(torch.complex128 if helm else torch.float64) * w.double()).T.contiguous()
    out = [torch.empty((nrhs, nx), dtype=q.dtype, device="cuda") for _ in range(3 if case["kernel"] == "gradient" else 1)]
    step = max(1, (1 << 25) // ny)
    for a in range(0, nx, step):
        x = X[a:a + step]
        d = [x[:, j, None] - Y[None, :, j] for j in range(3)]
        r2 = (d[0] * d[0]).addcmul_(d[1], d[1]).addcmul_(d[2], d[2])
        zero = r2 == 0
        if helm:
            r = r2.sqrt_()
            G = torch.polar((4.0 * math.pi * r).reciprocal_().masked_fill_(zero, 0.0), r.mul_(k))
            out[0][:, a:a + step] = (G @ q).T
            continue
        inv = r2.rsqrt_().masked_fill_(zero, 0.0)
        if case["kernel"] == "laplace":
            out[0][:, a:a + step] = (inv @ q).T
            continue
        inv = inv * inv * inv
        if case["kernel"] == "double_layer":
            n = normals.double()
            dot = (d[0] * n[:, 0]).addcmul_(d[1], n[None, :, 1]).addcmul_(d[2], n[None, :, 2])
            out[0][:, a:a + step] = (inv.mul_(dot) @ q).T
        else:
            for j in range(3):
                out[j][:, a:a + step] = -((d[j] * inv) @ q).T
    if not helm:
        out = [o / (4.0 * math.pi) for o in out]
    if case["kernel"] == "gradient":
        v = torch.stack(out, dim=1)  # (nrhs, 3, nx)
        return v[0] if nrhs == 1 else v
    return out[0][0] if nrhs == 1 else out[0]
