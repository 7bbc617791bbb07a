"""Measured cases: the products and solves a user of the library runs on the GPU.

listed()  the cases by name; draw(rng) one more of the same ranges
prepare() what a program has in hand before the call: a set-up context (mesh, grid, frequency),
          matrices or weights, and the vectors, made from the seed
run()     one pass through the public entry points, its outputs whole
work()    bytes and flops no implementation can do without (inputs read once, outputs written once)
exact()   the same outputs in 64 bits by plain torch, where that needs no boundary integrals

Structures are the repository's own workloads: copper bars (1-100 GHz, FP32 and FP64), gold
split-ring arrays at about 1 THz (where the internal operator is sparse), the AIM grids of both,
and random block-diagonal matrices of the same block sizes.
"""
import math
import random

import numpy as np
import torch

from paper_2108_03991_gb300 import api, synth

DEV = "cuda"


def listed():
    return [
        # one short bar (120 edges): the smallest system product, launches and latency only
        {"name": "matvec_small_bar", "op": "matvec", "mesh": "bars", "nx": 1, "ny": 1, "lmin": 2.0,
         "lmax": 2.0, "mseed": 0, "cross": 1.0, "freq": 10e9, "prec": "c32", "nrhs": 1},
        # the plain method: the copper bar at 10 GHz in FP64 (one block of 2,016)
        {"name": "matvec_copper_bar_c64", "op": "matvec", "mesh": "bars", "nx": 1, "ny": 1,
         "lmin": 20.0, "lmax": 20.0, "mseed": 0, "cross": 2.0, "freq": 10e9, "prec": "c64", "nrhs": 1},
        # the 4 x 4 bar array: what every FGMRES iteration of that workload applies
        {"name": "matvec_bar_array", "op": "matvec", "mesh": "bars", "nx": 4, "ny": 4, "lmin": 5.0,
         "lmax": 40.0, "mseed": 0, "cross": 1.0, "freq": 10e9, "prec": "c32", "nrhs": 1},
        # 4 x 4 gold rings at 1 THz: the same product with the sparse internal operator
        {"name": "matvec_rings", "op": "matvec", "mesh": "rings", "n": 4, "mseed": 2, "freq": 1e12,
         "prec": "c32", "nrhs": 1},
        # four excitations at once on 3 x 3 rings (odd grid): the product of the batched solve
        {"name": "batch_rings", "op": "matvec", "mesh": "rings", "n": 3, "mseed": 2, "freq": 1e12,
         "prec": "c32", "nrhs": 4},
        # many ports: internal products of 64 right-hand sides on the tensor cores, six bars
        {"name": "ports_tensor_core", "op": "ports", "mesh": "bars", "nx": 3, "ny": 2, "lmin": 5.0,
         "lmax": 40.0, "mseed": 1, "cross": 1.0, "freq": 10e9, "nrhs": 64, "tc": True},
        # 16 right-hand sides through the FP32 block products
        {"name": "ports_fp32", "op": "ports", "mesh": "bars", "nx": 3, "ny": 2, "lmin": 5.0,
         "lmax": 40.0, "mseed": 1, "cross": 1.0, "freq": 10e9, "nrhs": 16, "tc": False},
        # the grid step of the full 32 x 32 ring array (three vector-potential components)
        {"name": "conv_ring_grid", "op": "conv", "nx": 512, "ny": 512, "nz": 8, "ncomp": 3, "prec": "c32"},
        # a grid whose padded lengths are not powers of two
        {"name": "conv_ragged_grid", "op": "conv", "nx": 150, "ny": 90, "nz": 21, "ncomp": 3, "prec": "c32"},
        # the 32 x 32 ring array's block-diagonal product (6.8 GB): the bandwidth-bound extreme
        {"name": "gemv_ring_blocks", "op": "gemv", "blocks": 1024, "nmin": 912, "nmax": 912, "mseed": 0,
         "nrhs": 1, "prec": "c32"},
        # the learned correction's network on the bar array's grid, forward and backward
        {"name": "net_grad_bar_grid", "op": "net", "nx": 35, "ny": 35, "nz": 78},
        # a whole preconditioned FP32-bulk solve: plane wave on 2 x 2 rings to 1e-6
        {"name": "solve_rings", "op": "solve", "mesh": "rings", "n": 2, "mseed": 2, "freq": 1e12},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(["matvec", "matvec", "matvec", "ports", "ports", "conv", "conv", "gemv", "gemv",
                     "net", "solve"])
    if op in ("matvec", "ports", "solve"):
        prec = rng.choice(["c32", "c32", "c64"])
        if rng.random() < 0.5 and op != "ports":
            case = {"op": op, "mesh": "rings", "n": rng.randint(1, 3), "mseed": rng.randrange(1000),
                    "freq": round(rng.uniform(0.9, 1.2), 3) * 1e12}
        else:
            nx, ny = rng.randint(1, 4), rng.randint(1, 2)
            case = {"op": op, "mesh": "bars", "nx": nx, "ny": ny, "lmin": 2.0,
                    "lmax": rng.choice([4.0, 8.0, 16.0, 30.0]), "mseed": rng.randrange(1000),
                    "cross": 1.0, "freq": float("%.3g" % _log(rng, 1e9, 1e11))}
        if op == "matvec":
            case.update(prec=prec, nrhs=rng.choice([1, 1, 1, 2, 3, 4]))
        elif op == "ports":
            case.update(tc=rng.random() < 0.6, nrhs=int(round(_log(rng, 1, 128))))
        elif case["mesh"] == "bars":  # a solve: rings only (bars leave the currents ill-determined)
            case = {"op": op, "mesh": "rings", "n": rng.randint(1, 2), "mseed": case["mseed"],
                    "freq": round(rng.uniform(0.9, 1.2), 3) * 1e12}
        return case
    if op == "conv":
        prec = rng.choice(["c32", "c32", "c32", "c64"])
        cap = 2_000_000 if prec == "c32" else 200_000
        nx, ny = int(round(_log(rng, 10, 600))), int(round(_log(rng, 10, 600)))
        nz = rng.choice([8, 8, int(round(_log(rng, 8, 90)))])
        while nx * ny * nz > cap:
            nx, ny = max(10, nx * 3 // 4), max(10, ny * 3 // 4)
        return {"op": "conv", "nx": nx, "ny": ny, "nz": nz, "ncomp": rng.randint(1, 4), "prec": prec}
    if op == "gemv":
        blocks, nmax = int(round(_log(rng, 1, 300))), int(round(_log(rng, 8, 2053)))
        return {"op": "gemv", "blocks": blocks, "nmin": rng.choice([1, nmax]), "nmax": nmax,
                "mseed": rng.randrange(1000), "nrhs": rng.choice([1, 1, 2, 3, 4, 6]),
                "prec": rng.choice(["c32", "c32", "c64"])}
    return {"op": "net", "nx": int(round(_log(rng, 7, 130))), "ny": int(round(_log(rng, 7, 130))),
            "nz": int(round(_log(rng, 7, 80)))}


# ---- structures ----------------------------------------------------------------------------
def _structure(case):
    if case["mesh"] == "rings":
        return synth.srr_array_config(case["mseed"], case["n"], case["freq"])
    rng = np.random.default_rng(case["mseed"])
    a, c = 0.5, case["cross"]
    lengths = np.round(rng.uniform(case["lmin"], case["lmax"], case["nx"] * case["ny"]) / a) * a
    parts = []
    for i in range(case["nx"]):
        for j in range(case["ny"]):
            length = float(lengths[i * case["ny"] + j])
            parts.append(synth.box((5.0 * i, 5.0 * j, 0.0), (c, c, length),
                                   (round(c / a), round(c / a), round(length / a))))
    mesh = synth.merge(parts, [synth.SIGMA_CU] * len(parts))
    return mesh, synth.grid_box(mesh, a), case["freq"]


def _sizes(case):
    rng = random.Random(case["mseed"])
    return [rng.randint(case["nmin"], case["nmax"]) for _ in range(case["blocks"])]


def _prec(case):
    return api.BEM_C64 if case.get("prec") == "c64" else api.BEM_C32


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _cvec(n, seed, prec=api.BEM_C32):
    return torch.randn(n, dtype=api.cdtype(prec), device=DEV, generator=_gen(seed))


# ---- the interface -------------------------------------------------------------------------
def prepare(case, seed):
    op = case["op"]
    if op in ("matvec", "ports", "solve"):
        ctx = api.Context(*_structure(case))
        if op == "matvec":
            return {"op": op, "ctx": ctx, "prec": _prec(case), "nrhs": case["nrhs"],
                    "x": _cvec(case["nrhs"] * ctx.n, seed, _prec(case))}
        if op == "ports":
            return {"op": op, "ctx": ctx, "tc": case["tc"], "nrhs": case["nrhs"],
                    "h": _cvec(case["nrhs"] * ctx.ne, seed)}
        ctx.precond_setup()
        ang = random.Random(seed).uniform(0.0, 2.0 * math.pi)  # polarisation in the rings' plane
        return {"op": op, "ctx": ctx,
                "b": ctx.rhs_plane_wave((math.cos(ang), math.sin(ang), 0.0), (0.0, 0.0, 1.0))}
    if op == "conv":
        # the context of a structure on this grid; the grid step does not depend on the mesh
        grid = synth.Grid(np.array([-1.1, -1.1, -1.1]), np.array([0.5, 0.5, 0.5]),
                          np.array([case["nx"], case["ny"], case["nz"]], dtype=np.int64))
        ctx = api.Context(synth.bar_mesh(1.0, 1.0, 1.0, 0.5), grid, 10e9)
        return {"op": op, "ctx": ctx, "prec": _prec(case), "ncomp": case["ncomp"],
                "sigma": _cvec(case["ncomp"] * ctx.ng, seed, _prec(case))}
    if op == "gemv":
        sizes = _sizes(case)
        n = sum(sizes)
        total = sum(s * ((s + 3) // 4 * 4) for s in sizes)
        A = _cvec(total, seed, _prec(case))
        o = 0
        for s in sizes:
            ld = (s + 3) // 4 * 4
            if ld != s:
                A[o:o + s * ld].view(s, ld)[:, s:] = 0
            o += s * ld
        return {"op": op, "sizes": sizes, "A": A, "x": _cvec(n * case["nrhs"], seed + 1, _prec(case)),
                "y": torch.empty(n * case["nrhs"], dtype=api.cdtype(_prec(case)), device=DEV),
                "nrhs": case["nrhs"], "prec": _prec(case)}
    rng = np.random.default_rng(seed)
    sd = [math.sqrt(2.0 / (27.0 * ci)) for ci, _ in NET]
    w = np.concatenate([s * rng.standard_normal(ci * co * 27) for s, (ci, co) in zip(sd, NET)])
    shape = (8, case["nz"], case["ny"], case["nx"])
    return {"op": op, "w": w.astype(np.float32),
            "x": torch.randn(shape, device=DEV, generator=_gen(seed + 1)),
            "gout": torch.randn(shape, device=DEV, generator=_gen(seed + 2))}


def run(state):
    op = state["op"]
    if op == "matvec":
        if state["nrhs"] == 1:
            return state["ctx"].matvec(state["x"], prec=state["prec"])
        return state["ctx"].matvec_batch(state["x"], prec=state["prec"])
    if op == "ports":
        f = state["ctx"].internal_tc if state["tc"] else state["ctx"].internal
        return f(state["h"], nrhs=state["nrhs"])
    if op == "solve":
        x, _ = state["ctx"].solve(state["b"], tol=1e-6, prec_mode=api.BEM_C32, precond=1)
        return x.to(torch.complex64)  # what a 1e-6 residual determines
    if op == "conv":
        return state["ctx"].conv(state["sigma"], ncomp=state["ncomp"], prec=state["prec"])
    if op == "gemv":
        return api.blockdiag_gemv(state["sizes"], state["A"], state["x"], state["y"], state["nrhs"],
                                  state["prec"])
    return api.convnet_run(state["w"], state["x"], state["gout"])


NET = [(8, 16), (16, 16), (16, 16), (16, 8)]  # channels of the four 3x3x3 layers


def _near_pairs(grid, centres_a, centres_b):
    """Pairs whose anchor nodes lie within two cells of each other on every axis."""
    n = grid.n
    cnt = []
    for c in (centres_a, centres_b):
        idx = np.floor((c - grid.origin) / grid.h + 0.5).astype(np.int64)
        m = np.zeros(tuple(n))
        np.add.at(m, tuple(idx.T), 1.0)
        cnt.append(m)
    s = np.pad(cnt[1], 2)
    for ax in range(3):
        s = sum(np.roll(s, k, axis=ax) for k in range(-2, 3))
    return float((cnt[0] * s[2:-2, 2:-2, 2:-2]).sum())


def _edge_counts(mesh):
    nt = np.bincount(mesh.obj, minlength=mesh.nobj)
    return [int(t) * 3 // 2 for t in nt]  # closed surfaces


def _fft_flops(n):
    p = 8.0 * n[0] * n[1] * n[2]
    return 10.0 * p * math.log2(p) * 0.5  # half the padded points are known zeros or dropped


def work(case):
    op = case["op"]
    cb = 16 if case.get("prec") == "c64" else 8  # bytes of a complex number
    if op in ("matvec", "ports", "solve"):
        mesh, grid, _ = _structure(case)
        ne = _edge_counts(mesh)
        block = float(sum(n * n for n in ne))
        # e = Z h on the rings keeps about 0.39 of the dense block (pairs within 23 skin depths)
        zshare = 0.39 if case["mesh"] == "rings" else 1.0
        if op == "ports":
            r = case["nrhs"]
            z = zshare if not case["tc"] else 1.0
            return {"bytes": 8 * ((1 + z) * block + 3.0 * r * sum(ne)), "flops": 8.0 * (1 + z) * block * r}
        r = case.get("nrhs", 1)
        cen = mesh.verts[mesh.tris].mean(axis=1)
        tri_pairs = _near_pairs(grid, cen, cen)
        near = tri_pairs * (1.0 + 2.25)  # pulses, and 1.5 times as many edges on both sides
        E, T, ng = float(sum(ne)), float(mesh.nt), float(grid.npts)
        once = cb * ((1 + zshare) * block + near) + cb / 2 * (81 * E + 27 * T)
        per = cb * 2 * (E + T)
        flops = 8 * ((1 + zshare) * block + near) + 16 * (81 * E + 27 * T) + 4 * _fft_flops(grid.n)
        if op == "solve":  # the operators and the preconditioner's blocks, read once
            return {"bytes": once + 8.0 * sum((n + n * 2 / 3) ** 2 for n in ne) + 2 * 16 * (E + T),
                    "flops": flops}
        return {"bytes": once + r * per, "flops": r * flops}
    if op == "conv":
        n = (case["nx"], case["ny"], case["nz"])
        return {"bytes": cb * case["ncomp"] * 2.0 * n[0] * n[1] * n[2],
                "flops": case["ncomp"] * _fft_flops(n)}
    if op == "gemv":
        sizes = _sizes(case)
        block = float(sum(s * s for s in sizes))
        return {"bytes": cb * (block + 2.0 * case["nrhs"] * sum(sizes)), "flops": 8.0 * block * case["nrhs"]}
    p = float(case["nx"] * case["ny"] * case["nz"])
    wn = sum(ci * co * 27 for ci, co in NET)
    return {"bytes": 4 * (p * 8 * 4 + 2 * wn), "flops": 3 * 2.0 * wn * p}


def exact(case, seed):
    """In 64 bits by plain torch. The system and internal products and the solve are None: their
    values rest on the singular boundary integrals of the set-up."""
    op = case["op"]
    if op == "conv":
        sigma = prepare_sigma(case, seed).to(torch.complex128)
        n = (case["nz"], case["ny"], case["nx"])
        P = [2 * v for v in n]
        k0 = 2.0 * math.pi * 10e9 / 299792458.0 * 1e-6  # per micrometre
        ax = [torch.arange(p, device=DEV, dtype=torch.float64) for p in P]
        ax = [torch.minimum(a, p - a) * 0.5 for a, p in zip(ax, P)]
        R = torch.sqrt(ax[0][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[2][None, None, :] ** 2)
        G = torch.polar(1.0 / (4.0 * math.pi * R.clamp_min(1e-300)), -k0 * R)
        G[0, 0, 0] = 0  # the self term belongs to the near region
        G = torch.fft.fftn(G)
        out = []
        for s in sigma.view(case["ncomp"], *n):
            f = torch.fft.ifftn(torch.fft.fftn(s, s=P) * G)
            out.append(f[:n[0], :n[1], :n[2]].reshape(-1))
        return torch.cat(out)
    if op == "gemv":
        st = prepare(case, seed)
        n, r = sum(st["sizes"]), case["nrhs"]
        x = st["x"].view(r, n).to(torch.complex128)
        y = torch.empty_like(x)
        o = i = 0
        for s in st["sizes"]:
            ld = (s + 3) // 4 * 4
            B = st["A"][o:o + s * ld].view(s, ld)[:, :s].to(torch.complex128)
            y[:, i:i + s] = x[:, i:i + s] @ B.T
            o, i = o + s * ld, i + s
        return y.reshape(-1)
    if op == "net":
        st = prepare(case, seed)
        bf = lambda t: t.to(torch.bfloat16).to(torch.float64)  # noqa: E731  the net's inputs are BF16
        ws, o = [], 0
        w = bf(torch.from_numpy(st["w"]).to(DEV))
        for ci, co in NET:
            ws.append(w[o:o + ci * co * 27].view(co, ci, 3, 3, 3).clone().requires_grad_())
            o += ci * co * 27
        x = bf(st["x"]).requires_grad_()
        h = x[None]
        for i, k in enumerate(ws):
            h = torch.nn.functional.conv3d(h, k, padding=1)
            if i + 1 < len(ws):
                h = torch.relu(h)
        out = h[0]
        grads = torch.autograd.grad(out, ws + [x], st["gout"].to(torch.float64))
        gw = torch.cat([g.reshape(-1) for g in grads[:-1]]).cpu().numpy()
        return out.detach(), gw, grads[-1]
    return None


def prepare_sigma(case, seed):
    return _cvec(case["ncomp"] * case["nx"] * case["ny"] * case["nz"], seed, _prec(case))
