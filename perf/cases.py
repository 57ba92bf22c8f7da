"""Work that a user of this package has it do, as cases that can be timed and compared.

A case is one call, or one short sequence of calls, through the public entry
points: the projector pair (`sipo_project`, `sipo_backproject` and their
autograd forms), with attenuation and a point spread function where the case
says so, and solves of the projection LP (`sipo_solve`, `sipo_solve_batched`).

`listed()` names the cases, `draw(rng)` makes further ones of the same ranges,
`prepare(case, seed)` makes what a program holds before the call, `run(state)`
is one pass, `work(case)` the bytes and operations that no implementation can
do without, and `exact(case, seed)` the outputs in 64-bit arithmetic from the
definitions, in plain torch.

Layouts: volume [ny][nx][nz], sinogram [views][bins][nz], z fastest.  Voxel
centres at i - (n - 1)/2, detector coordinate u = x cos + y sin + (bins - 1)/2,
linear interpolation between the bins floor(u) and floor(u) + 1.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2604_08997_gb300 as sipo
from paper_2604_08997_gb300 import _abi, autograd

KASE = {"general": sipo.SIPO_GENERAL, "case1": sipo.SIPO_CASE1, "case2": sipo.SIPO_CASE2}
STORAGE = {"f32": sipo.SIPO_F32, "f64": sipo.SIPO_F64, "bf16": sipo.SIPO_BF16}
BATCH_VIEWS = (180, 250, 391, 333)  # view counts of a sweep's members, in this order
MASK64 = (1 << 63) - 1


def _case(name, kind, nx, ny, nz, views, bins, dtype="f32", full_turn=False, vial=0.0, mu=0.0,
          sigma=(0.0, 0.0, 0.0), trunc=4.0, lp="general", iters=0, members=0):
    """vial: radius as a share of the smaller side (0: none); mu: attenuation per voxel."""
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "views": views, "bins": bins,
            "dtype": dtype, "full_turn": full_turn, "vial": vial, "mu": mu, "sx": sigma[0], "sy": sigma[1],
            "sz": sigma[2], "trunc": trunc, "lp": lp, "iters": iters, "members": members}


def listed():
    blur = dict(vial=0.46875, mu=0.005, sigma=(1.5, 1.5, 2.5))
    return [
        # the smallest operator calls: both directions on one 64 x 64 slice in double
        # precision, as a check or an outer loop around the operators makes them
        _case("slice64-pair-f64", "pair", 64, 64, 1, 96, 91, "f64"),
        # a 2-D design of the published size over a full turn, differentiated: the
        # projector forward and backward inside a gradient-based program
        _case("slice512-project-grad", "project_grad", 512, 512, 1, 360, 512, full_turn=True),
        # a printed part of the published 3-D size (z not a multiple of 4) with the
        # 5-tap blur: its dose forward and backward
        _case("part130-dose-grad", "dose_grad", 128, 128, 130, 360, 128, sigma=(1.0, 1.0, 1.0), trunc=2.0),
        # one member of a sweep over part sizes, whose z extents and views are uneven
        _case("part96-pair", "pair", 96, 90, 96, 391, 101, vial=0.47),
        # the headline size: one application of the projector, and one of its adjoint
        # with attenuation, as own solvers and evaluations call them
        _case("part256-project", "project", 256, 256, 256, 360, 256, vial=0.46875),
        _case("part256-dose", "dose", 256, 256, 256, 360, 256, vial=0.46875, mu=0.005),
        # the headline size with attenuation and blur, differentiated in the input and
        # in the blur widths (calibration of the point spread function)
        _case("part256-blur-grad", "project_grad", 256, 256, 256, 360, 256, **blur),
        # solves, by one check period of 64 iterations and the returned point: the 2-D
        # workload in double precision, where launches and scalar steps count
        _case("slice64-solve-f64", "solve", 64, 64, 1, 96, 91, "f64", lp="case1", iters=64),
        # a 2-D design of the published size over a full turn
        _case("slice512-solve", "solve", 512, 512, 1, 360, 512, full_turn=True, lp="general", iters=64),
        # a tolerance and inhibition sweep over parts of several sizes, solved as one batch
        _case("sweep-solve", "batch", 64, 64, 64, 180, 64, vial=0.47, lp="case1", iters=64, members=4),
        # the headline solve, and the attenuated and blurred one in bf16 storage
        _case("part256-solve", "solve", 256, 256, 256, 360, 256, vial=0.46875, lp="case2", iters=64),
        _case("part384-blur-solve-bf16", "solve", 384, 384, 384, 540, 384, "bf16", vial=0.46875, mu=0.0033,
              sigma=(2.0, 2.0, 3.0), lp="case2", iters=32),
    ]


def _size(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "project", "dose", "project_grad", "dose_grad", "solve", "solve", "batch"])
    flat = rng.random() < 0.35 and kind != "batch"
    dtype = rng.choice(["f32", "f32", "f32", "f64"]) if kind != "batch" else "f32"
    if kind == "solve" and not flat and rng.random() < 0.35:
        dtype = "bf16"
    top = 512 if flat else (256 if dtype != "f64" else 96)
    nx = _size(rng, 48, top)
    ny = max(40, nx + rng.choice([0, 0, 0, -1, 3, -6]))
    nz = 1
    if not flat:
        nz = rng.choice([nx, nx, 16 * max(1, nx // 16), _size(rng, 16, max(20, nx)), 2 * max(8, nx // 2 - 3)])
    views = _size(rng, 60, 400)
    bins = max(nx, ny) if rng.random() < 0.6 else int(math.ceil(1.42 * max(nx, ny)))
    vial = rng.choice([0.0, 0.46875, 0.47]) if flat else rng.choice([0.46875, 0.47])
    mu = 1.28 / nx if vial > 0 and rng.random() < 0.35 else 0.0
    sigma, trunc = (0.0, 0.0, 0.0), 4.0
    if rng.random() < 0.4 or kind == "dose_grad":
        s = rng.choice([1.0, 1.25, 1.5, 2.0])
        sigma, trunc = (s, s, 0.0 if flat else rng.choice([s, 2.5])), rng.choice([2.0, 4.0, 4.0])
    lp = rng.choice(["general", "case1", "case2"])
    c = _case("", kind, nx, ny, nz, views, bins, dtype, flat and rng.random() < 0.5, vial, mu, sigma, trunc, lp,
              64 if kind in ("solve", "batch") else 0, rng.choice([3, 4, 6]) if kind == "batch" else 0)
    if kind == "batch":
        c.update(nx=64, ny=64, nz=64, bins=64, vial=0.47, mu=0.0, sx=0.0, sy=0.0, sz=0.0,
                 views=rng.choice([180, 211]), lp=rng.choice(["case1", "case2"]))
    del c["name"]
    return c


# ------------------------------------------------------------------- inputs
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _real(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _sigma(case):
    return (case["sx"], case["sy"], case["sz"])


def _vial(case):
    return case["vial"] * min(case["nx"], case["ny"])


def _angles(case):
    span = 2.0 * math.pi if case["full_turn"] else math.pi
    return np.arange(case["views"], dtype=np.float64) * (span / case["views"])


def _generator(seed, salt):
    g = torch.Generator(device=_device())
    g.manual_seed((seed * 1000003 + salt * 7919 + 12345) & MASK64)
    return g


def target(case, seed):
    """A binary part, float32 [ny][nx][nz]: balls (discs in 2-D) and rings of
    feature sizes between a twenty-fifth and a quarter of the side, inside the
    vial with room for the band."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    dev, side = _device(), min(nx, ny)
    rng = np.random.default_rng([seed, nx, ny, nz])
    x = (torch.arange(nx, device=dev) - (nx - 1) / 2)[None, :, None]
    y = (torch.arange(ny, device=dev) - (ny - 1) / 2)[:, None, None]
    z = (torch.arange(nz, device=dev) - (nz - 1) / 2)[None, None, :]
    inner = 0.43 * side - max(2.0, 10 * side / 256)
    f = torch.zeros((ny, nx, nz), dtype=torch.bool, device=dev)
    for i in range(6):
        r = rng.uniform(0.04, 0.13) * side
        rho, phi = max(0.0, inner - 1.6 * r) * math.sqrt(rng.uniform()), rng.uniform(0, 2 * math.pi)
        dx, dy = x - rho * math.cos(phi), y - rho * math.sin(phi)
        dz = z - rng.uniform(-0.3, 0.3) * (nz - 1)
        if i % 3 == 2:  # a ring about the z direction
            f |= ((dx * dx + dy * dy).sqrt() - r) ** 2 + dz * dz <= (0.45 * r) ** 2
        else:
            f |= dx * dx + dy * dy + dz * dz <= r * r
    f &= x * x + y * y <= inner * inner
    if not bool(f.any()):
        f |= x * x + y * y + z * z <= (0.1 * side) ** 2
    return f.to(torch.float32).contiguous()


def _volume(case, seed):
    """Signed volume, as the duals that a solver projects."""
    shape = (case["ny"], case["nx"], case["nz"])
    return torch.randn(shape, generator=_generator(seed, 1), device=_device(), dtype=_real(case))


def _sinogram(case, seed, salt=2):
    """Non-negative projections, about half of them dark."""
    shape = (case["views"], case["bins"], case["nz"])
    return torch.randn(shape, generator=_generator(seed, salt), device=_device(), dtype=_real(case)).relu_()


def _band_width(case):
    return max(2, int(round(10 * min(case["nx"], case["ny"]) / 256)))


def _geometry(case):
    return dict(nx=case["nx"], ny=case["ny"], nz=case["nz"], angles=_angles(case), n_det=case["bins"],
                vial_radius=_vial(case), mu=case["mu"], psf_sigma=_sigma(case), psf_trunc=case["trunc"])


def _lp(case, member=0):
    return dict(kase=KASE[case["lp"]], w1=1.0, w2=1.0, tol_lo=0.05 + 0.02 * member, tol_hi=0.05 + 0.02 * member,
                inhibit_ratio=0.8 + 0.02 * member, band_width=_band_width(case))


def _context(case, seed, member=0):
    tol = dict(kkt_tol=0.0, max_iter=max(1, case["iters"]), check_every=min(64, max(1, case["iters"])),
               storage=STORAGE[case["dtype"]])
    return sipo.sipo_create(_geometry(case), target(case, seed), _lp(case, member), tol)


def _members(case):
    """The LPs of a batch: parts of growing size, 64, 96, 112, 80, ... voxels a side."""
    out = []
    for i in range(case["members"]):
        n = (64, 96, 112, 80)[i % 4]
        out.append(dict(case, kind="solve", nx=n, ny=n, nz=n, bins=n,
                        views=case["views"] if i % 4 == 0 else BATCH_VIEWS[i % 4]))
    return out


def _point(ctx, real):
    """Buffers for the point that a solve returns: projections and duals."""
    return {"y": torch.empty(ctx.sino_shape, dtype=real, device="cuda"),
            "lam_up": torch.empty(ctx.vol_shape, dtype=real, device="cuda"),
            "lam_lo": torch.empty(ctx.vol_shape, dtype=real, device="cuda")}


def prepare(case, seed):
    state = {"case": case}
    if case["kind"] == "batch":
        parts = _members(case)
        state["ctxs"] = [_context(c, seed + i, i) for i, c in enumerate(parts)]
        state["points"] = [_point(c, torch.float32) for c in state["ctxs"]]
        return state
    ctx = state["ctx"] = _context(case, seed)
    if case["kind"] == "solve":
        state["point"] = _point(ctx, _real(case))
        state["dose"] = torch.empty(ctx.vol_shape, dtype=_real(case), device="cuda")
        return state
    if case["kind"] in ("pair", "project", "project_grad"):
        state["vol"] = _volume(case, seed)
    if case["kind"] in ("pair", "dose", "dose_grad", "project_grad"):
        state["sino"] = _sinogram(case, seed)
    if case["kind"] == "dose_grad":
        state["vol"] = _volume(case, seed)
    state["out_sino"] = torch.empty(ctx.sino_shape, dtype=_real(case), device="cuda")
    state["out_vol"] = torch.empty(ctx.vol_shape, dtype=_real(case), device="cuda")
    if max(_sigma(case)) > 0:
        state["sigma"] = torch.tensor(_sigma(case), dtype=torch.float64, requires_grad=True)
    return state


# --------------------------------------------------------------------- pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        sipo.sipo_solve_batched(state["ctxs"])
        for ctx, p in zip(state["ctxs"], state["points"]):
            sipo.sipo_get_state(ctx, p["y"], p["lam_up"], p["lam_lo"])
        return state["points"]
    ctx = state["ctx"]
    if kind == "solve":
        p = state["point"]
        sipo.sipo_solve(ctx)
        sipo.sipo_get_state(ctx, p["y"], p["lam_up"], p["lam_lo"])
        if case["dtype"] == "bf16":  # the point in its storage type
            return {k: v.to(torch.bfloat16) for k, v in p.items()}
        sipo.sipo_get_array(ctx, _abi.ARRAY_DOSE, state["dose"])
        return dict(p, dose=state["dose"])
    if kind == "pair":
        sipo.sipo_project(ctx, state["vol"], state["out_sino"])
        sipo.sipo_backproject(ctx, state["sino"], state["out_vol"])
        return {"sino": state["out_sino"], "vol": state["out_vol"]}
    if kind == "project":
        return {"sino": sipo.sipo_project(ctx, state["vol"], state["out_sino"])}
    if kind == "dose":
        return {"vol": sipo.sipo_backproject(ctx, state["sino"], state["out_vol"])}
    fwd = autograd.project if kind == "project_grad" else autograd.backproject
    src, seed_grad = (state["vol"], state["sino"]) if kind == "project_grad" else (state["sino"], state["vol"])
    leaf = src.detach().requires_grad_(True)
    sigma = state.get("sigma")
    out = fwd(ctx, leaf, sigma)
    wrt = [leaf] if sigma is None else [leaf, sigma]
    grads = torch.autograd.grad(out, wrt, seed_grad)
    res = {"out": out.detach(), "grad": grads[0]}
    if sigma is not None:
        res["grad_sigma"] = grads[1].to(torch.float32)
    return res


# --------------------------------------------------------------------- work
def _inside(case, dev):
    nx, ny = case["nx"], case["ny"]
    a = 2 * torch.arange(nx, device=dev) - (nx - 1)
    b = 2 * torch.arange(ny, device=dev) - (ny - 1)
    r = _vial(case)
    if r <= 0:
        return torch.ones((ny, nx), dtype=torch.bool, device=dev)
    return (a * a)[None, :] + (b * b)[:, None] <= math.floor(4.0 * r * r)


def _radii(case):
    return [int(math.ceil(case["trunc"] * s)) if s > 0 else 0 for s in _sigma(case)]


def _labels(case, seed):
    """0 exterior, 1 band, 2 gel: the band is every other voxel in the vial
    within the band width of the gel or in the blur's support of it."""
    gel = target(case, seed) != 0
    w = _band_width(case)
    x = gel.to(torch.float32)[None, None]
    near = torch.zeros_like(gel)
    reach = min(w, case["nz"] - 1)
    for dz in range(-reach, reach + 1):  # one 2-D dilation by a disc per z offset, then a shift along z
        rr = w * w - dz * dz
        h = int(math.isqrt(rr))
        layer = torch.zeros_like(gel)
        for dy in range(-h, h + 1):
            hx = int(math.isqrt(rr - dy * dy))
            p = torch.nn.functional.max_pool3d(x, (1, 2 * hx + 1, 1), 1, (0, hx, 0))[0, 0] > 0
            lo, hi = max(0, dy), min(case["ny"], case["ny"] + dy)
            layer[lo:hi] |= p[lo - dy:hi - dy]
        lo, hi = max(0, dz), min(case["nz"], case["nz"] + dz)
        near[:, :, lo:hi] |= layer[:, :, lo - dz:hi - dz]
    rad = _radii(case)
    if max(rad) > 0:
        near |= torch.nn.functional.max_pool3d(x, (2 * rad[1] + 1, 2 * rad[0] + 1, 2 * rad[2] + 1), 1,
                                               (rad[1], rad[0], rad[2]))[0, 0] > 0
    inside = _inside(case, gel.device)[:, :, None]
    return torch.where(gel & inside, 2, torch.where(near & inside & ~gel, 1, 0)).to(torch.uint8)


def _needed(case, lab):
    """Columns whose dose the LP's rows read."""
    need = (lab != 0).any(dim=2)
    rad = _radii(case)
    if max(rad) > 0:
        need = torch.nn.functional.max_pool2d(need.float()[None, None], (2 * rad[1] + 1, 2 * rad[0] + 1), 1,
                                              (rad[1], rad[0]))[0, 0] > 0
        need &= _inside(case, lab.device)
    return need


def work(case):
    """Per operator application: two taps (a multiply and an add each) per voxel,
    view and z; its input read once and its output written once.  Per iteration
    of a solve: one application each way over the columns that the rows read,
    and the iterates read and written once.  The blur: its taps per voxel."""
    if case["kind"] == "batch":
        parts = [work(c) for c in _members(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    vol, sino = case["nx"] * case["ny"] * case["nz"], case["views"] * case["bins"] * case["nz"]
    size = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
    taps = sum(2 * r + 1 for r in _radii(case) if r > 0)
    if case["kind"] == "solve":
        cols = int(_needed(case, _labels(case, 0)).sum().item())
        flops = 2 * (2 * 2 * cols * case["nz"] * case["views"] + 2 * taps * cols * case["nz"])
        # y, its anchor and the column sums read, y and y-bar written and read; the
        # duals, their anchors, the dose and its anchor, the row sums and the labels
        # read, the duals, the dose and their difference written and read
        byte = sino * (5 * size + 4) + cols * case["nz"] * (8 * size + 17)
        return {"bytes": case["iters"] * byte, "flops": case["iters"] * flops}
    inside = int(_inside(case, "cpu").sum().item())
    op = {"bytes": size * (vol + sino), "flops": 4 * inside * case["nz"] * case["views"] + 2 * taps * vol}
    times = {"pair": 2, "project": 1, "dose": 1, "project_grad": 2, "dose_grad": 2}[case["kind"]]
    out = {k: times * v for k, v in op.items()}
    if taps and case["kind"].endswith("_grad"):  # the three derivatives of the blur and their inner products
        out["flops"] += 3 * (2 * taps + 2) * vol + 4 * inside * case["nz"] * case["views"] * (case["kind"] == "project_grad")
    return out


# -------------------------------------------------------------------- exact
class _Exact:
    """The operators from their definitions, 64-bit, one view at a time."""

    def __init__(self, case):
        self.case = case
        dev = _device()
        nx, ny = case["nx"], case["ny"]
        self.x = (torch.arange(nx, dtype=torch.float64, device=dev) - (nx - 1) / 2)[None, :]
        self.y = (torch.arange(ny, dtype=torch.float64, device=dev) - (ny - 1) / 2)[:, None]
        self.inside = _inside(case, dev)
        self.ang = _angles(case)

    def _view(self, k):
        """Bins and weights [2][ny*nx] of view k; off the detector the weight is 0."""
        case = self.case
        c, s = math.cos(self.ang[k]), math.sin(self.ang[k])
        u = self.x * c + self.y * s + (case["bins"] - 1) / 2
        i0 = torch.floor(u)
        w1 = u - i0
        idx = torch.stack((i0, i0 + 1)).to(torch.int64).reshape(2, -1)
        wt = torch.stack((1 - w1, w1)) * self.inside
        ok = (idx >= 0) & (idx < case["bins"])
        wt = wt.reshape(2, -1) * ok
        r = _vial(case)
        if r > 0:
            sj = idx.to(torch.float64) - (case["bins"] - 1) / 2
            on = sj.abs() <= r
            chord = (r * r - sj * sj).clamp_min(0).sqrt()
            path = (-self.x * s + self.y * c).reshape(1, -1) + chord
            wt = wt * on * (torch.exp(-case["mu"] * path) if case["mu"] else 1.0)
        return idx.clamp(0, case["bins"] - 1), wt

    def adjoint_p(self, sino):
        case = self.case
        out = torch.zeros((case["ny"] * case["nx"], case["nz"]), dtype=torch.float64, device=sino.device)
        for k in range(case["views"]):
            idx, wt = self._view(k)
            for t in range(2):
                out += wt[t][:, None] * sino[k].index_select(0, idx[t])
        return out.reshape(case["ny"], case["nx"], case["nz"])

    def p(self, vol):
        case = self.case
        flat = vol.reshape(-1, case["nz"])
        out = torch.zeros((case["views"], case["bins"], case["nz"]), dtype=torch.float64, device=vol.device)
        for k in range(case["views"]):
            idx, wt = self._view(k)
            for t in range(2):
                out[k].index_add_(0, idx[t], wt[t][:, None] * flat)
        return out

    def blur(self, vol, deriv=-1):
        rad, sig = _radii(self.case), _sigma(self.case)
        for a, dim in ((0, 1), (1, 0), (2, 2)):  # x, y, z
            if rad[a] == 0:
                continue
            i = np.arange(-rad[a], rad[a] + 1, dtype=np.float64)
            e = np.exp(-i * i / (2 * sig[a] ** 2))
            taps = e / e.sum()
            if a == deriv:
                de = e * i * i / sig[a] ** 3
                taps = (de * e.sum() - e * de.sum()) / e.sum() ** 2
            out, n = torch.zeros_like(vol), vol.shape[dim]
            for t, o in zip(taps, range(-rad[a], rad[a] + 1)):
                lo, hi = max(0, -o), min(n, n - o)
                if lo < hi:
                    out.narrow(dim, lo, hi - lo).add_(vol.narrow(dim, lo + o, hi - lo), alpha=float(t))
            vol = out
        return vol

    def project(self, vol):
        return self.p(self.blur(vol))

    def dose(self, sino):
        return self.blur(self.adjoint_p(sino))


def _exact_solve(case, seed):
    """One check period of the reflected Halpern PDHG from zero, and the point of
    the check that ends it (no restart can come before that check)."""
    op = _Exact(case)
    lab = _labels(case, seed)
    band, gel = lab == 1, lab == 2
    has_u, has_v = case["lp"] != "case2", case["lp"] != "case1"
    lp = _lp(case)
    f = {"general": 1.0, "case1": 1.0, "case2": 1.0 / lp["inhibit_ratio"]}[case["lp"]]
    f_up = (1 + lp["tol_hi"]) / (1 - lp["tol_lo"])
    act = op.p(target(case, seed).double()) > 0
    need = _needed(case, lab)[:, :, None]
    row = op.dose(act.double())
    col = op.project(band.double() + 2 * gel.double()) * act
    rup = row + band * float(has_u) + gel * (f if has_v else 0.0)
    up_rows = band | gel
    c_u, c_v = float(has_u), float(has_v)
    col_u, col_v = band.sum().item() * has_u, gel.sum().item() * f * has_v
    rhs = (0.0 if has_u else 1.0) * band + (0.0 if has_v else f_up) * gel  # fixed part of the upper rows
    h2 = (rhs * rhs / rup)[up_rows & (rup > 0)].sum().item() + (f * f / row)[gel & (row > 0)].sum().item()
    c2 = (c_u ** 2 / col_u if col_u else 0.0) + (c_v ** 2 / col_v if col_v else 0.0)
    om = math.sqrt(c2 / h2)
    eta = 0.99
    tau = torch.where(col > 0, eta / (om * col), 0.0)
    sig_up = torch.where(up_rows & (rup > 0), eta * om / rup, 0.0)
    sig_lo = torch.where(gel & (row > 0), eta * om / row, 0.0)
    y, lu, ll, u, v = torch.zeros_like(col), torch.zeros_like(row), torch.zeros_like(row), 0.0, 1.0
    for k in range(case["iters"] + 1):
        up = max(0.0, u - eta / (om * col_u) * (c_u - lu[band].sum().item())) if col_u else u
        vp = max(1.0, v - eta / (om * col_v) * (c_v - f * lu[gel].sum().item())) if col_v else v
        yp = (y - tau * op.project(lu - ll)).clamp_min(0)
        dbar = op.dose(2 * yp - y)
        bound = rhs + (2 * up - u if has_u else 0.0) * band + (f * (2 * vp - v) if has_v else 0.0) * gel
        lup = (lu + sig_up * (dbar - bound)).clamp_min(0) * up_rows
        llp = (ll + sig_lo * (f - dbar)).clamp_min(0) * gel
        if k == case["iters"]:
            break
        w = (k + 1.0) / (k + 2.0)
        y, lu, ll = w * (2 * yp - y), w * (2 * lup - lu), w * (2 * llp - ll)
        u, v = w * (2 * up - u), w * (2 * vp - v) + (1 - w) * 1.0
    return {"y": yp, "lam_up": lup, "lam_lo": llp, "dose": op.blur(op.adjoint_p(yp) * need)}


def exact(case, seed):
    kind, vol = case["kind"], case["nx"] * case["ny"] * case["nz"]
    if kind == "batch" or case["dtype"] == "bf16":
        return None
    if kind == "solve":
        # two applications of about 0.1 ms a view an iteration and more with the volume
        if case["iters"] * case["views"] * (1.0 + vol / 5e5) > 5e4:
            return None
        return _exact_solve(case, seed)
    if vol * case["views"] > 2e10:
        return None
    op = _Exact(case)
    if kind in ("pair", "project", "project_grad", "dose_grad"):
        x = _volume(case, seed).double()
    if kind in ("pair", "dose", "dose_grad", "project_grad"):
        s = _sinogram(case, seed).double()
    if kind == "pair":
        return {"sino": op.project(x), "vol": op.dose(s)}
    if kind == "project":
        return {"sino": op.project(x)}
    if kind == "dose":
        return {"vol": op.dose(s)}
    if kind == "project_grad":
        raw = op.adjoint_p(s)
        res = {"out": op.project(x), "grad": op.blur(raw)}
    else:
        raw = op.adjoint_p(s)
        res = {"out": op.blur(raw), "grad": op.project(x)}
    if max(_sigma(case)) > 0:
        rad = _radii(case)
        res["grad_sigma"] = torch.stack([(raw * op.blur(x, a)).sum() if rad[a] else raw.new_zeros(()) for a in range(3)])
    return res
