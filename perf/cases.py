"""The work that a user of this library has it do, as cases for timing.

A suspension is a staggered lattice of prolate vesicles (or two vesicles in
free space) moved over one time step, the library's own synthetic workloads
made quickly for any size.  The kinds of case:

  step       one time step of a running simulation: upsample X0 and X1, find
             the contacts, their volumes V and dV/dX1 (Stiv.step), and, when
             "adjoint" is set, the gradient rows scattered onto the vertices
             and taken back to the SH coefficients, as an optimiser or the
             contact solver uses them
  autograd   forward and backward of the summed volume (autograd.stiv_sum)
  transform  the synthesis and its adjoint alone (stiv_upsample,
             stiv_grad_to_coef), as surface post-processing calls them
  lcp        the contact LCP of a step: matrix assembly and Newton solve
  fidelity   the mesh-fidelity estimate of Sec. 3.1.2 on the upsampled meshes
  sort       the check-point sort of Alg. 1 (stiv_sort_pairs)

Engines are taken in mid-simulation: they have run one step, so that their
scratch has the size the suspension needs.  Their output buffers have room to
spare, as a program gives them whose contacts come and go; a pass returns
them whole (the tail past the counts stays zero).
"""
import dataclasses
import math

import numpy as np
import torch

from paper_1812_04719_gb300 import autograd as A
from paper_1812_04719_gb300 import scenegen as G
from paper_1812_04719_gb300 import stiv as S

# minimum separation used with the degree-six test: 0.009 at R0 = 1.136,
# scaled to this R0 and inflated by 1 + 2 alpha, alpha = 0.05
D_M = 1.1 * 0.009 / 1.136 * G.R0_PAPER


def _step(name, **kw):
    """A step case with the defaults of a periodic FP64 suspension."""
    c = dict(kind="step", name=name, nx=0, ny=0, nz=0, phi=0.5, aspect=2.0, p="16", tilt=3.0, trans=0.2, flow=0.0,
             rot=1.0, periodic=True, precision="fp64", d_m=False, ee=True, absolute=False, graph=False, grad=True,
             adjoint=False)
    c.update(kw)
    return c


def listed():
    return [
        # a two-body encounter, p = 8 -> 16 in free space: the smallest call,
        # launches and latency
        _step("pair_p8", p="8"),
        # a dilute periodic suspension of 64 vesicles at 30%, default options
        _step("dilute64_p16", nx=4, ny=4, nz=2, phi=0.30, tilt=30.0, trans=0.4, rot=6.0),
        # gradients through the step at 256 vesicles, 50%, p = 12 -> 24:
        # forward and backward of the summed volume by torch.autograd
        _step("lattice256_p12_autograd", kind="autograd", nx=8, ny=4, nz=4, aspect=1.98, p="12", trans=0.4),
        # the dense suspension of the paper's throughput runs, 1440 vesicles at
        # 58%: a graph-replayed step and the adjoint, in FP64 and with the
        # tensor-core synthesis on FP32 vertices
        _step("lattice1440_p16_fp64", nx=12, ny=12, nz=5, phi=0.58, aspect=2.4, graph=True, adjoint=True),
        _step("lattice1440_p16_mixed", nx=12, ny=12, nz=5, phi=0.58, aspect=2.4, graph=True, adjoint=True,
              precision="mixed"),
        # uneven orders with a vortex displacement long against the mesh
        # spacing: 4096 vesicles at 40%, the largest suspension
        _step("uneven4096", nx=16, ny=16, nz=8, phi=0.40, p="8,12,16", tilt=10.0, trans=0.30, flow=2.0, rot=2.0,
              graph=True),
        # the step with a minimum separation d_m > 0 (degree-six test), with
        # an order that is no power of two, launched eagerly
        _step("separation360_p15", nx=6, ny=6, nz=5, phi=0.58, aspect=2.4, p="15", d_m=True),
        # synthesis and adjoint alone at an odd order, FP64
        dict(kind="transform", name="transform999_p21_fp64", n=999, p="21", precision="fp64"),
        # and in the tensor-core form on uneven orders
        dict(kind="transform", name="transform4096_mixed", n=4096, p="8,12,16", precision="mixed"),
        # contact resolution after a dense step: assemble B = J M J^T, solve
        _step("lcp1440_p16", kind="lcp", nx=12, ny=12, nz=5, phi=0.58, aspect=2.4),
        # resolution check of 256 vesicles against the 4x finer grid
        dict(kind="fidelity", name="fidelity256_p12", n=256, p="12", precision="fp64", factor=4),
        # a million check points by 48-bit keys
        dict(kind="sort", name="sort_1m", n=1_000_003, bits=48),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_orders(rng):
    if rng.random() < 0.25:
        return ",".join(str(q) for q in sorted(rng.sample(range(5, 18), rng.randint(2, 3))))
    return str(rng.choice([5, 7, 8, 9, 11, 12, 13, 15, 16, 16, 17, 20, 24]))


def draw(rng):
    kind = rng.choices(["step", "autograd", "transform", "lcp", "fidelity", "sort"], [10, 2, 3, 2, 1.5, 1.5])[0]
    if kind == "sort":
        return dict(kind=kind, n=_log_int(rng, 1000, 1 << 20), bits=rng.randint(20, 60))
    if kind in ("transform", "fidelity"):
        ps = rng.choice([_draw_orders(rng), str(rng.randint(2, 32))])
        work = max(int(q) for q in ps.split(",")) ** (2 if kind == "transform" else 3)
        top = min(4096, (1_000_000 if kind == "transform" else 2_000_000) // work)
        c = dict(kind=kind, n=_log_int(rng, 2, max(3, top)), p=ps, precision=rng.choice(["fp64", "fp64", "mixed"]))
        if kind == "fidelity":
            c["factor"] = rng.randint(2, 4)
        return c
    if kind == "step" and rng.random() < 0.15:   # two vesicles in free space
        c = _step("", p=str(rng.randint(4, 24)), precision=rng.choice(["fp64", "mixed"]), d_m=rng.random() < 0.3,
                  ee=rng.random() < 0.8, graph=rng.random() < 0.4)
        del c["name"]
        return c
    ps = _draw_orders(rng)
    pm = max(int(q) for q in ps.split(","))
    top = min(2048, 360_000 // (pm * pm))
    while True:
        periodic = rng.random() < 0.75
        lo = (4, 4, 2) if periodic else (1, 1, 1)   # a periodic box must exceed twice a vesicle's extent
        nx, ny, nz = _log_int(rng, lo[0], 14), _log_int(rng, lo[1], 14), _log_int(rng, lo[2], 7)
        if 2 * nx * ny * nz <= top:
            break
    phi = rng.uniform(0.35, 0.58)
    c = _step("", kind=kind, nx=nx, ny=ny, nz=nz, phi=round(phi, 3), aspect=round(rng.uniform(2.0, 2.3), 3), p=ps,
              tilt=round(rng.uniform(0.0, 6.0), 2), trans=round(rng.uniform(0.1, 0.4), 3),
              flow=round(rng.choice([0.0, 0.0, 0.0, 0.5, 1.5]) * rng.random(), 3), rot=round(rng.uniform(0.5, 3.0), 2),
              periodic=periodic, precision=rng.choice(["fp64", "fp64", "mixed"]), d_m=rng.random() < 0.2,
              ee=rng.random() < 0.85, absolute=rng.random() < 0.1, graph=rng.random() < 0.5,
              grad=rng.random() < 0.85, adjoint=rng.random() < 0.5)
    if kind != "step":
        c.update(grad=True, ee=True, absolute=False)
    if kind == "lcp":             # a step that leaves contacts to resolve
        c.update(trans=round(rng.uniform(0.25, 0.4), 3), phi=round(rng.uniform(0.45, 0.58), 3), nx=max(nx, 2),
                 ny=max(ny, 2))
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rotations(rng, n, max_deg):
    """n rotations about random axes by angles uniform in [0, max_deg]."""
    ax = rng.normal(size=(n, 3))
    ax /= np.linalg.norm(ax, axis=1, keepdims=True)
    th = np.radians(rng.uniform(0.0, max_deg, n))
    K = np.zeros((n, 3, 3))
    K[:, 0, 1], K[:, 0, 2], K[:, 1, 2] = -ax[:, 2], ax[:, 1], -ax[:, 0]
    K -= K.transpose(0, 2, 1)
    return np.eye(3) + np.sin(th)[:, None, None] * K + (1.0 - np.cos(th))[:, None, None] * (K @ K)


def _perturb(rng, n, p, amp):
    """Random coefficients of degrees 2 .. p, falling off like 1 / (n+1)^2."""
    deg = np.floor(np.sqrt(np.arange((p + 1) ** 2) + 0.5))
    fall = np.where(deg >= 2, amp * G.R0_PAPER / (deg + 1.0) ** 2, 0.0)
    return rng.uniform(-1.0, 1.0, size=(n, 3, (p + 1) ** 2)) * fall


def _suspension(rng, ps, centers, tilt, shift, rot):
    """Coefficients per vesicle of prolate vesicles at the centres, long axes
    within tilt degrees of z, moved by shift and a rotation of up to rot
    degrees, both surfaces with shape noise.  Returns (flat, offsets)."""
    n = len(ps)
    a_ax, b_ax = G.prolate_axes()
    M = _rotations(rng, n, tilt) @ np.diag([b_ax, b_ax, a_ax])
    R = _rotations(rng, n, rot)
    sizes = 6 * (np.asarray(ps, np.int64) + 1) ** 2
    off = np.concatenate([[0], np.cumsum(sizes)[:-1]]).astype(np.int64)
    flat = np.empty(int(sizes.sum()))
    for p in sorted(set(int(q) for q in ps)):
        idx = np.nonzero(np.asarray(ps) == p)[0]
        c0 = _perturb(rng, len(idx), p, 0.01)
        for k, col in ((0, 3), (1, 1), (2, 2)):     # u_x at m = 1, u_y at m = -1, u_z at m = 0
            c0[:, :, col] += math.sqrt(4 * math.pi / 3) * M[idx][:, :, k]
        c1 = R[idx] @ c0 + _perturb(rng, len(idx), p, 0.02)
        c0[:, :, 0] = math.sqrt(4 * math.pi) * centers[idx]
        c1[:, :, 0] = math.sqrt(4 * math.pi) * (centers[idx] + shift[idx])
        nc = (p + 1) ** 2
        flat[off[idx][:, None] + np.arange(6 * nc)] = np.stack([c0, c1], axis=1).reshape(len(idx), 6 * nc)
    return flat, off


def _orders(text, n):
    """Orders per vesicle, mixed in a fixed way (the same for every seed)."""
    return np.random.default_rng(n).choice(np.array([int(q) for q in text.split(",")], dtype=np.int32), size=n)


def _unit(rng, n):
    v = rng.normal(size=(n, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def _scene(case, seed):
    d_m = D_M if case.get("d_m") else 0.0
    rng = np.random.default_rng(seed)
    if "nx" not in case:          # isolated vesicles for transforms and fidelity
        n = int(case["n"])
        ps = _orders(case["p"], n)
        centers = rng.uniform(0.0, 30.0, size=(n, 3))
        flat, off = _suspension(rng, ps, centers, 180.0, 0.2 * G.R0_PAPER * _unit(rng, n), 1.0)
        L = np.zeros(3)
    elif case["nx"] == 0:         # two vesicles closing in free space
        sc = G.two_vesicles(p=int(case["p"]), seed=seed)
        return dataclasses.replace(sc, d_m=d_m)
    else:
        a_ax, b_ax = G.prolate_axes()
        a = (2.0 * (4.0 / 3.0 * math.pi * a_ax * b_ax * b_ax) / case["phi"] / case["aspect"]) ** (1.0 / 3.0)
        c = case["aspect"] * a
        centers, L = G.bcc_lattice(case["nx"], case["ny"], case["nz"], a, c)
        n = len(centers)
        centers = (centers + rng.uniform(0, 1, 3) * np.array([a, a, c])) % L
        ps = _orders(case["p"], n)
        shift = case["trans"] * G.R0_PAPER * _unit(rng, n)
        if case["flow"] > 0:      # Taylor vortex at the centres
            x, y, z = (2 * math.pi * centers / L).T
            shift = shift + case["flow"] * np.stack([np.sin(x) * np.cos(y) * np.sin(z),
                                                     np.cos(x) * np.sin(y) * np.sin(z), 0 * x], axis=1)
        flat, off = _suspension(rng, ps, centers, case["tilt"], shift, case["rot"])
        if not case["periodic"]:
            L = np.zeros(3)
    return G.Scene(name="", p=ps, coef=flat, coef_off=off, L=np.asarray(L, np.float64), centers=centers, d_m=d_m)


def _precision(case):
    return S.STIV_MIXED if case.get("precision") == "mixed" else S.STIV_FP64


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sort":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = int(case["n"])
        keys = torch.randint(0, 1 << int(case["bits"]), (n,), generator=g, device="cuda", dtype=torch.int64)
        nb = S.stiv_sort_scratch_bytes(n)
        return dict(kind=kind, n=n, bits=int(case["bits"]), keys=keys,
                    vals=torch.arange(n, dtype=torch.int32, device="cuda"), ko=torch.empty_like(keys),
                    vo=torch.empty(n, dtype=torch.int32, device="cuda"), nb=nb,
                    scratch=torch.empty(nb, dtype=torch.uint8, device="cuda"))
    sc = _scene(case, seed)
    prec = _precision(case)
    st = dict(kind=kind, ds=S.DeviceScene.from_scene(sc, precision=prec))
    ds = st["ds"]
    if kind in ("transform", "fidelity"):
        st["eng"] = S.Stiv.for_scene(sc, precision=prec)
        st["eng"].upsample(ds)
        if kind == "fidelity":
            st["factor"] = int(case["factor"])
        else:
            g = torch.Generator(device="cuda").manual_seed(seed)
            st["gX"] = torch.randn(ds.verts.numel(), generator=g, dtype=torch.float64, device="cuda")
            st["gcoef"] = torch.zeros_like(ds.coef)
        return st
    cap = int((6 + 5 * case["flow"]) * (sc.p.astype(np.int64) ** 2).sum()) + 4096
    eng = S.Stiv.for_scene(sc, precision=prec, pair_cap=16 * sc.n + 64, contact_cap=cap, include_ee=case["ee"],
                           velocity=S.STIV_VEL_ABSOLUTE if case["absolute"] else S.STIV_VEL_RELATIVE)
    st.update(eng=eng, graph=case["graph"], grad=case["grad"] or case["adjoint"], adjoint=case["adjoint"],
              stream=torch.cuda.Stream() if case["graph"] else torch.cuda.current_stream())
    torch.cuda.synchronize()
    eng.step(ds, grad=st["grad"], use_graph=st["graph"], stream=st["stream"])
    if case["adjoint"]:
        st["gX"] = torch.zeros(ds.verts.numel(), dtype=torch.float64, device="cuda")
        st["gcoef"] = torch.zeros_like(ds.coef)
    if kind == "autograd":
        st["coef"] = ds.coef.clone().requires_grad_(True)
    if kind == "lcp":
        rng = np.random.default_rng(seed + 1)
        st["lcp"] = S.ContactLCP(row_cap=6 * sc.n + 64, nnz_cap=100 * sc.n + 1024)
        st["m"] = torch.as_tensor(rng.uniform(0.5, 2.0, sc.n), device="cuda")
        st["t"] = torch.as_tensor(rng.uniform(0.5, 2.0, sc.n) / (8.0 * sc.p.astype(np.float64) ** 2), device="cuda")
        st["lcp"].assemble(eng, ds, st["m"], st["t"])
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _adjoint(st, stream):
    """Gradient rows of the engine's last step to the SH coefficients."""
    eng, ds = st["eng"], st["ds"]
    b, q = eng.buf, stream.cuda_stream
    with torch.cuda.stream(stream):
        st["gX"].zero_()
    S.stiv_grad_scatter(eng.h, q, ds.p.data_ptr(), b.contacts_struct(), b.counts.data_ptr(), 0, b.grad.data_ptr(),
                        b.gves.data_ptr(), b.gvid.data_ptr(), ds.vert_off.data_ptr(), st["gX"].data_ptr())
    S.stiv_grad_to_coef(eng.h, q, ds.n, ds.p_max, ds.p.data_ptr(), ds.coef_off.data_ptr(), ds.vert_off.data_ptr(),
                        st["gX"].data_ptr(), st["gcoef"].data_ptr())


def run(st):
    kind = st["kind"]
    if kind == "sort":
        S.stiv_sort_pairs(torch.cuda.current_stream().cuda_stream, st["n"], st["bits"], st["keys"].data_ptr(),
                          st["vals"].data_ptr(), st["ko"].data_ptr(), st["vo"].data_ptr(), st["scratch"].data_ptr(),
                          st["nb"])
        return dict(keys=st["ko"], vals=st["vo"])
    eng, ds = st["eng"], st["ds"]
    if kind == "transform":
        eng.upsample(ds)
        S.stiv_grad_to_coef(eng.h, torch.cuda.current_stream().cuda_stream, ds.n, ds.p_max, ds.p.data_ptr(),
                            ds.coef_off.data_ptr(), ds.vert_off.data_ptr(), st["gX"].data_ptr(),
                            st["gcoef"].data_ptr())
        return dict(verts=ds.verts, gcoef=st["gcoef"])
    if kind == "fidelity":
        return dict(err=eng.mesh_fidelity(ds, factor=st["factor"]))
    if kind == "lcp":
        lcp = st["lcp"]
        lcp.assemble(eng, ds, st["m"], st["t"])
        lcp.solve(eng)
        return dict(rows=lcp.dims[:2], row_pair=lcp.row_pair, q=lcp.q, row_ptr=lcp.row_ptr, col=lcp.col, val=lcp.val,
                    lam=lcp.lam)
    if kind == "autograd":
        st["coef"].grad = None
        total = A.stiv_sum(st["coef"], eng, ds)
        total.backward()
        return dict(total=total.detach(), grad=st["coef"].grad)
    r = eng.step(ds, grad=st["grad"], use_graph=st["graph"], stream=st["stream"])
    b = eng.buf
    r = dict(counts=r["counts"][:S.C_STATUS + 1], verts=ds.verts, i=b.ci, j=b.cj, shift=b.cs, pair=b.pair, type=b.type,
             a=b.a, b=b.b, tau=b.tau, w=b.w, V=b.Vc, V_pair=b.Vp)
    if st["grad"]:
        r.update(grad=b.grad, gves=b.gves, gvid=b.gvid)
    if st["adjoint"]:
        _adjoint(st, st["stream"])
        r["gcoef"] = st["gcoef"]
    return r


# ---------------------------------------------------------------------------
# work that a pass cannot do without
# ---------------------------------------------------------------------------
def _mean_over_orders(case, f):
    ps = [int(q) for q in case["p"].split(",")]
    return sum(f(p) for p in ps) / len(ps)


def _synthesis_flops(p):
    """Separable synthesis of one field on the order-2p grid: ring sums with
    the parity of the Legendre functions, then a real FFT per ring."""
    P = 2 * p
    return 2.0 * (p + 1) ** 2 * (P // 2 + 1) + (P + 1) * 2.5 * (2 * P) * math.log2(2 * P)


def work(case):
    kind = case["kind"]
    if kind == "sort":
        return {"bytes": 24.0 * case["n"], "flops": 0.0}
    n = case["n"] if "n" in case else max(2, 2 * case["nx"] * case["ny"] * case["nz"])
    vb = 4.0 if case.get("precision") == "mixed" else 8.0
    coef = n * _mean_over_orders(case, lambda p: 6.0 * (p + 1) ** 2)
    verts = n * _mean_over_orders(case, lambda p: 6.0 * G.nverts(2 * p))
    fields = n * 6 * _mean_over_orders(case, _synthesis_flops)
    if kind == "transform":     # coefficients to vertices, and the X1 half back
        return {"bytes": 8 * coef + vb * verts + 4 * verts + 8 * coef, "flops": 1.5 * fields}
    if kind == "fidelity":
        return {"bytes": 8 * coef + vb * verts + 16 * n,
                "flops": n * 6 * _mean_over_orders(case, lambda p: _synthesis_flops(p) * case["factor"] ** 2)}
    # contacts follow from the density and the step; about 1.5 p^2 per vesicle
    # with edge-edge pairs, a quarter of it without, in a dense suspension
    contacts = n * _mean_over_orders(case, lambda p: 1.5 * p * p) * (1.0 if case["ee"] else 0.25) * \
        (0.05 if case["nx"] == 0 else 1.0)
    rows = contacts * (44.0 + (128.0 if case["grad"] else 0.0))
    if kind == "lcp":
        return {"bytes": contacts * 132.0, "flops": contacts * 48.0}
    out = {"bytes": 8 * coef + vb * verts + rows, "flops": fields + contacts * 800.0}
    if kind == "autograd":      # a step without and one with gradient rows, and the adjoint
        return {"bytes": 2 * out["bytes"] + 8 * coef, "flops": 2 * out["flops"] + 0.5 * fields}
    if case["adjoint"]:
        return {"bytes": out["bytes"] + 8 * coef, "flops": out["flops"] + 0.5 * fields}
    return out


# ---------------------------------------------------------------------------
# the same outputs in 64 bits by plain torch and numpy
# ---------------------------------------------------------------------------
def _basis(p, x, phi):
    """Y [len(x) * len(phi), (p+1)^2]: real orthonormal spherical harmonics at
    cos(theta) = x (rows) and longitudes phi, entry n^2 + n + m."""
    x = np.asarray(x, dtype=np.float64)
    s = np.sqrt((1.0 - x) * (1.0 + x))
    leg = np.zeros((p + 1, p + 1, len(x)))
    leg[0, 0] = math.sqrt(1.0 / (4.0 * math.pi))
    for m in range(p + 1):
        if m:
            leg[m, m] = math.sqrt((2.0 * m + 1.0) / (2.0 * m)) * s * leg[m - 1, m - 1]
        if m < p:
            leg[m + 1, m] = math.sqrt(2.0 * m + 3.0) * x * leg[m, m]
        for n in range(m + 2, p + 1):
            a = math.sqrt((4.0 * n * n - 1.0) / (n * n - m * m))
            b = math.sqrt(((n - 1.0) ** 2 - m * m) / (4.0 * (n - 1.0) ** 2 - 1.0))
            leg[n, m] = a * (x * leg[n - 1, m] - b * leg[n - 2, m])
    Y = np.zeros((len(x), len(phi), (p + 1) ** 2))
    for m in range(p + 1):
        c = np.cos(m * phi) * (math.sqrt(2.0) if m else 1.0)
        d = np.sin(m * phi) * math.sqrt(2.0)
        for n in range(m, p + 1):
            Y[:, :, n * n + n + m] = leg[n, m][:, None] * c[None, :]
            if m:
                Y[:, :, n * n + n - m] = leg[n, m][:, None] * d[None, :]
    return torch.as_tensor(Y.reshape(-1, (p + 1) ** 2), device="cuda")


def _mesh_basis(p):
    """Synthesis matrix of the order-2p mesh: its rings, then the two poles."""
    P = 2 * p
    x = -np.polynomial.legendre.leggauss(P + 1)[0]
    grid = _basis(p, np.sort(x)[::-1], np.pi * np.arange(2 * P) / P)
    return torch.cat([grid, _basis(p, [1.0, -1.0], np.zeros(1))])


def _by_order(sc):
    """(p, vesicles of that order, index of their coefficients, of their vertices)."""
    vo = sc.vert_off()
    for p in sorted(set(sc.p.tolist())):
        idx = np.nonzero(sc.p == p)[0]
        nc, nv = (p + 1) ** 2, G.nverts(2 * p)
        ci = torch.as_tensor(sc.coef_off[idx][:, None] + np.arange(6 * nc), device="cuda").reshape(-1, 6, nc)
        vi = torch.as_tensor(vo[idx][:, None] + np.arange(6 * nv), device="cuda").reshape(-1, 6, nv)
        yield p, idx, ci, vi


def _exact_verts(sc):
    coef = torch.as_tensor(sc.coef, device="cuda")
    X = torch.zeros(sc.n_vert_values(), dtype=torch.float64, device="cuda")
    for p, _, ci, vi in _by_order(sc):
        X[vi] = coef[ci] @ _mesh_basis(p).T
    return X


def _exact_fidelity(sc, factor):
    """Largest distance between the mesh as a map of parameter space and the
    series, over the rings and longitudes of the finer grid."""
    coef, X = torch.as_tensor(sc.coef, device="cuda"), _exact_verts(sc)
    err = torch.zeros(sc.n, 2, dtype=torch.float64, device="cuda")
    for p, idx, ci, vi in _by_order(sc):
        P, W, Pf = 2 * p, 4 * p, 2 * p * factor
        mesh = np.arccos(np.sort(np.polynomial.legendre.leggauss(P + 1)[0])[::-1])
        fine = np.arccos(np.sort(np.polynomial.legendre.leggauss(Pf + 1)[0])[::-1])
        V = X[vi]
        C = coef[ci]
        k = torch.arange(2 * Pf, device="cuda")
        j, j1, b = k // factor, (k // factor + 1) % W, (k % factor).double() / factor
        ring = V[:, :, :-2].reshape(len(idx), 6, P + 1, W)
        worst = torch.zeros(len(idx), 2, dtype=torch.float64, device="cuda")
        for th in fine:
            series = C @ _basis(p, [math.cos(th)], np.pi * np.arange(2 * Pf) / Pf).T
            if th < mesh[0] or th > mesh[-1]:
                north = th < mesh[0]
                tp = th / mesh[0] if north else (math.pi - th) / (math.pi - mesh[-1])
                pole, r = V[:, :, -2 if north else -1][:, :, None], ring[:, :, 0 if north else P]
                on = pole + tp * (r[:, :, j] + b * (r[:, :, j1] - r[:, :, j]) - pole)
            else:
                i = min(int(np.searchsorted(mesh, th, side="right")) - 1, P - 1)
                a = (th - mesh[i]) / (mesh[i + 1] - mesh[i])
                q, r, s, u = ring[:, :, i][:, :, j], ring[:, :, i + 1][:, :, j], ring[:, :, i + 1][:, :, j1], \
                    ring[:, :, i][:, :, j1]
                on = torch.where(a >= b, q + a * (r - q) + b * (s - r), q + b * (u - q) + a * (s - u))
            d = (on - series).reshape(len(idx), 2, 3, -1).square().sum(dim=2).sqrt().amax(dim=-1)
            worst = torch.maximum(worst, d)
        err[torch.as_tensor(idx, device="cuda")] = worst
    return err


def _exact_lcp(case, seed):
    """B = J M J^T and the solution of 0 <= -V + B lam, lam >= 0 from the step's
    gradient rows: dense in torch."""
    st = prepare(case, seed)
    b, n = st["eng"].buf, st["ds"].n
    counts = b.counts.cpu().numpy()
    nc, npair = int(counts[S.C_VF] + counts[S.C_EE]), int(counts[S.C_PAIRS])
    pair = b.pair[:nc].long()
    rows = torch.unique(pair)
    row = torch.searchsorted(rows, pair)
    nr = len(rows)
    lcp = st["lcp"]
    out = {k: torch.zeros_like(getattr(lcp, k)) for k in ("row_pair", "q", "row_ptr", "col", "val", "lam")}
    if nr == 0:
        return dict(out, rows=torch.zeros(2, dtype=torch.int64))
    ves, vid, g = b.gves[:nc].long(), b.gvid[:nc].long(), b.grad[:nc]
    stride = int(vid.max()) + 1
    B = torch.zeros(nr, nr, dtype=torch.float64, device="cuda")
    T = torch.zeros(3, nr, n, dtype=torch.float64, device="cuda")
    r4 = row[:, None].expand(-1, 4).reshape(-1)
    for c in range(3):
        J = torch.sparse_coo_tensor(torch.stack([r4, (ves * stride + vid).reshape(-1)]),
                                    (g[:, :, c] * st["m"][ves].sqrt()).reshape(-1), (nr, n * stride)).coalesce()
        B += torch.sparse.mm(J, J.t().coalesce()).to_dense()
        T[c].index_put_((r4, ves.reshape(-1)), g[:, :, c].reshape(-1), accumulate=True)
        B += (T[c] * st["t"]) @ T[c].T
    vi, vj = b.ci[:npair][rows], b.cj[:npair][rows]
    share = (vi[:, None] == vi) | (vi[:, None] == vj) | (vj[:, None] == vi) | (vj[:, None] == vj)
    at = share.nonzero()
    q = -b.Vp[:npair][rows]
    lam = torch.zeros(nr, dtype=torch.float64, device="cuda")
    for _ in range(100):
        y = q + B @ lam
        act = y < lam
        if torch.minimum(lam, y).abs().max() < 1e-14:
            break
        new = torch.zeros_like(lam)
        new[act] = torch.linalg.solve(B[act][:, act], -q[act])
        lam = new
    out["row_pair"][:nr], out["q"][:nr], out["lam"][:nr] = rows.int(), q, lam
    out["row_ptr"][1:nr + 1] = share.sum(dim=1).cumsum(0)
    out["col"][:len(at)], out["val"][:len(at)] = at[:, 1].int(), B[at[:, 0], at[:, 1]]
    return dict(out, rows=torch.tensor([nr, len(at)]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "sort":
        st = prepare(case, seed)
        keys, order = torch.sort(st["keys"], stable=True)
        return dict(keys=keys, vals=order.int())
    if kind == "lcp":
        return _exact_lcp(case, seed)
    if kind == "autograd":
        return None
    sc = _scene(case, seed)
    if kind == "fidelity":
        return dict(err=_exact_fidelity(sc, int(case["factor"])))
    X = _exact_verts(sc)
    if kind == "step":            # contacts need the library; their vertices do not
        return dict(verts=X)
    g = torch.Generator(device="cuda").manual_seed(seed)
    gX = torch.randn(X.numel(), generator=g, dtype=torch.float64, device="cuda")
    gcoef = torch.zeros(len(sc.coef), dtype=torch.float64, device="cuda")
    for p, _, ci, vi in _by_order(sc):
        gcoef[ci[:, 3:]] = gX[vi[:, 3:]] @ _mesh_basis(p)
    return dict(verts=X, gcoef=gcoef)
