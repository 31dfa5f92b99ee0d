"""Workloads on which the convolution is timed: the calls that a program built on this library makes.

A case names one layer (irreps, harmonics, radial width), one graph size and one call:

    fwd    inference of one layer                                   conv_fwd
    bwd    adjoints of all four arguments                           conv_bwd
    train  a training step of a model without forces                conv_fwd, conv_bwd
    dbwd   second order, as a loss on forces needs it               conv_dbwd
    step   one training step on energies and forces                 conv_fwd, conv_bwd, conv_dbwd
    force  one step of molecular dynamics: positions in, forces out edge_vectors, conv_geo_fwd, conv_geo_bwd, position_gradient

Graphs are radius graphs of uniform random positions at the density of a liquid (0.1 atoms per cubic Angstrom), with the
cutoff that gives the wanted mean degree; `batch` disjoint ones side by side stand for a batch of molecules.
"""
import math

import numpy as np
import torch

import paper_2607_18074_b200 as sobek

DENSITY = 0.1
ENVELOPE = 6
# radial basis of a case -> the library's constant
BASES = {"bessel": sobek.BASIS_BESSEL, "gaussian": sobek.BASIS_GAUSSIAN}


def _case(name, irreps_in, irreps_out, l_max, K, nodes, degree, call, batch=1, mode="uvw", layout="ir_mul", basis="bessel"):
    c = dict(irreps_in=irreps_in, irreps_out=irreps_out, l_max=l_max, K=K, nodes=nodes, degree=degree, call=call,
             batch=batch, mode=mode, layout=layout, basis=basis)
    return dict(name=name, **c) if name else c


def listed():
    tiny, nequip = "8x0e+8x1o", "32x0e+32x1o+32x2e"
    mid, wide = "64x0e+64x1o+64x2e", "64x0e+64x1o+64x2e+64x3o+64x4e"
    mixed, uvu = "128x0e+64x1o+64x2e", "128x0e+128x1o+128x2e"
    return [
        # a small molecule through a small model: an interactive call, bound by latency
        _case("tiny_fwd", tiny, tiny, 2, 8, 64, 17, "fwd", basis="gaussian"),
        # the same model in a training step on energies and forces: all three orders, one after another
        _case("tiny_step", tiny, tiny, 2, 8, 64, 17, "step", basis="gaussian"),
        # a NequIP-like layer on a liquid of some thousand atoms: inference
        _case("nequip_fwd", nequip, nequip, 2, 8, 5000, 30, "fwd"),
        # the same layer trained on energies, the number of atoms as it comes
        _case("nequip_train", nequip, nequip, 2, 8, 4999, 30, "train"),
        # molecular dynamics with it: positions in, forces out, nothing stored per edge but its vector
        _case("md_force", nequip, nequip, 2, 8, 2003, 36, "force"),
        # a batch of 31 molecules of 101 atoms in the layout that e3nn programs use (mul_ir), trained on energies
        _case("molecules_train", mid, mid, 2, 16, 101, 32, "train", batch=31, layout="mul_ir"),
        # a large periodic-box-like system through a 64-channel layer: inference at a million edges
        _case("million_fwd", mid, mid, 2, 16, 31250, 32, "fwd"),
        # long neighbourhoods (a large cutoff) and unequal multiplicities: backward
        _case("dense_bwd", mixed, mixed, 2, 16, 2048, 255, "bwd"),
        # a MACE-like layer from two orders to four: the second-order call of force training
        _case("mace_dbwd", "128x0e+128x1o", "128x0e+128x1o+128x2e+128x3o", 3, 8, 20000, 30, "dbwd"),
        # the channelwise mode on a batch of small molecules: training
        _case("channelwise_train", uvu, uvu, 2, 16, 128, 32, "train", batch=127, mode="uvu"),
        # multiplicities and a radial width that no tile fits: training of a small hand-made model
        _case("odd_train", "20x0e+7x1o+5x2e", "12x0e+9x1o+5x2e", 2, 10, 701, 25, "train"),
        # the widest layer of all, l up to 4 at 64 channels and two million edges: a whole force-training step
        _case("wide_step", wide, wide, 4, 16, 50000, 40, "step"),
    ]


# layers that drawn cases pick from: (orders of the input, orders of the output, l_max, mode)
_LAYERS = [((0, 1), (0, 1), 2, "uvw"), ((0, 1, 2), (0, 1, 2), 2, "uvw"), ((0, 1, 2), (0, 1, 2), 2, "uvw"),
           ((0, 1), (0, 1, 2, 3), 3, "uvw"), ((0, 1, 2, 3), (0, 1), 3, "uvw"), ((0, 1, 2, 3), (0, 1, 2, 3), 3, "uvw"),
           ((0, 1, 2, 3, 4), (0, 1, 2, 3, 4), 4, "uvw"), ((0, 1, 2), (0, 1, 2), 2, "uvu")]
_MULTS = (8, 16, 24, 32, 32, 48, 64, 64, 64, 96, 128, 128)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    ceiling = 0.5 * _cost(listed()[-1])
    while True:
        l_in, l_out, l_max, mode = rng.choice(_LAYERS)
        m = rng.choice(_MULTS)
        text = lambda ls, mult: "+".join("%dx%d%s" % (mult(l), l, "eo"[l % 2]) for l in ls)
        if mode == "uvu" or rng.random() < 0.6:
            mi = mo = lambda l: m                                            # one multiplicity for all orders
        elif rng.random() < 0.7:
            mi = mo = lambda l: m if l == 0 else max(8, m // 2)              # wider scalars
        else:
            odd = [rng.randint(3, 40) for _ in range(5)]                     # as they come
            mi = mo = lambda l: odd[l]
        call = rng.choice(("fwd", "fwd", "bwd", "train", "train", "dbwd", "step", "force"))
        if call == "force" and (mode == "uvu" or max(l_in + l_out) > 2 or any(mi(l) % 16 or mi(l) > 64 for l in l_in + l_out)):
            call = "train"                 # the geometry front end does not take every layer
        K = rng.choice((8, 8, 10, 16, 16))
        batch = rng.choice((1, 1, 1, _log_int(rng, 2, 200)))
        nodes = _log_int(rng, 32, 40000) if batch == 1 else _log_int(rng, 16, 300)
        degree = min(_log_int(rng, 4, 120), nodes // 2)
        layout = "mul_ir" if call != "force" and rng.random() < 0.2 else "ir_mul"
        c = _case(None, text(l_in, mi), text(l_out, mo), l_max, K, nodes, degree, call, batch, mode, layout,
                  rng.choice(("bessel", "bessel", "gaussian")))
        # multiplicities that no tile fits run on the FP32 pipes, about ten times as long
        slow = 10 if any(mi(l) % 8 for l in l_in + l_out) else 1
        if slow * _cost(c) <= ceiling and nodes * batch * degree <= 2_000_000:
            return c


# ---- inputs ---------------------------------------------------------------------------------------------------


def _irreps(text):
    out = []
    for block in text.split("+"):
        mul, ir = block.split("x")
        out.append((int(mul), int(ir[:-1]), 1 if ir[-1] == "e" else -1))
    return out


def _dim(irreps):
    return sum(mul * (2 * l + 1) for mul, l, _ in irreps)


def _cutoff(nodes, degree, side):
    """Cutoff at which `nodes` uniform points of a cube have `degree` neighbours each on average."""
    lo, hi = 0.0, 1.0
    for _ in range(60):
        t = 0.5 * (lo + hi)
        p = 4 / 3 * math.pi * t ** 3 - 1.5 * math.pi * t ** 4 + 1.6 * t ** 5 - t ** 6 / 6       # of a pair in the unit cube
        lo, hi = (t, hi) if (nodes - 1) * p < degree else (lo, t)
    return lo * side


def _radius_graph(nodes, batch, degree, gen):
    """Positions [batch * nodes, 3], receiver-sorted CSR (row_ptr, senders, receivers) and cutoff of `batch` disjoint
    radius graphs.  The cutoff is taken from the positions, so that there are nodes * batch * degree edges whatever the seed."""
    side = (nodes / DENSITY) ** (1 / 3)
    reach = 2 * side if nodes <= 600 else 1.15 * _cutoff(nodes, degree, side)
    pos = torch.rand(batch, nodes, 3, generator=gen, device="cuda") * side
    recv, send, dist2 = [], [], []
    rows = max(1, 40_000_000 // nodes)
    for b in range(batch):
        p = pos[b]
        for i in range(0, nodes, rows):
            d2 = sum((p[i:i + rows, k, None] - p[None, :, k]) ** 2 for k in range(3))
            i_, j_ = ((d2 < reach * reach) & (d2 > 0)).nonzero(as_tuple=True)
            recv.append(i_ + (b * nodes + i))
            send.append(j_ + b * nodes)
            dist2.append(d2[i_, j_])
    recv, send, dist2 = torch.cat(recv), torch.cat(send), torch.cat(dist2)
    order = torch.sort(dist2, stable=True).indices[:nodes * batch * degree // 2 * 2]
    r_c = float(dist2[order[-1]]) ** 0.5 * (1 + 1e-6)
    keep = order.sort().values
    recv, send = recv[keep], send[keep]
    row_ptr = torch.zeros(batch * nodes + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.bincount(recv, minlength=batch * nodes).cumsum(0)
    return pos.reshape(-1, 3), row_ptr, send.to(torch.int32), recv, r_c


def _harmonics(l_max, v):
    """Real spherical harmonics of unit vectors, [E, (l_max+1)^2], component normalisation, sine branch at m < 0."""
    x, y, z = v.double().unbind(1)
    out = [None] * (l_max + 1) ** 2
    a, b = torch.ones_like(x), torch.zeros_like(x)          # Re, Im of (x + iy)^m
    for m in range(l_max + 1):
        q = {m: torch.full_like(z, float(math.prod(range(1, 2 * m, 2))))}       # P_l^m / sin^m
        for l in range(m + 1, l_max + 1):
            q[l] = ((2 * l - 1) * z * q[l - 1] - ((l + m - 1) * q[l - 2] if l - 2 >= m else 0)) / (l - m)
        for l in range(m, l_max + 1):
            c = math.sqrt((2 * l + 1) * math.factorial(l - m) / math.factorial(l + m) * (2 if m else 1))
            out[l * l + l + m] = c * q[l] * a
            if m:
                out[l * l + l - m] = c * q[l] * b
        a, b = x * a - y * b, y * a + x * b
    return torch.stack(out, 1).float()


def _radial(basis, K, r_c, r):
    """Radial embedding [E, K] of the distances r."""
    r = r.double()[:, None]
    if basis == "gaussian":
        step = r_c / (K - 1)
        return torch.exp(-0.5 * ((r - step * torch.arange(K, device=r.device)) / step) ** 2).float()
    n, d, p = torch.arange(1, K + 1, device=r.device), r / r_c, ENVELOPE
    u = 1 - (p + 1) * (p + 2) / 2 * d ** p + p * (p + 2) * d ** (p + 1) - p * (p + 1) / 2 * d ** (p + 2)
    return (math.sqrt(2 / r_c) * torch.sin(n * math.pi * d) / r * u).float()


def _weight_scale(plan):
    """1 / sqrt(fan-in) per column of R."""
    paths = [plan.path(k) for k in range(plan.info.n_paths)]
    uvu = plan.mode == "uvu"
    fan = {}
    for p in paths:
        fan[p.i_out] = fan.get(p.i_out, 0) + (1 if uvu else p.c_in)
    std = np.zeros(plan.info.N_w, dtype=np.float32)
    for p in paths:
        std[p.w_off:p.w_off + (p.c_in if uvu else p.c_in * p.c_out)] = (plan.info.K * fan[p.i_out]) ** -0.5
    return torch.from_numpy(std).cuda()


class State:
    """What a program keeps from call to call: plan, graph with its sender view, workspace, inputs and output buffers."""


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = State()
    s.call = case["call"]
    s.plan = sobek.Plan(_irreps(case["irreps_in"]), _irreps(case["irreps_out"]), case["l_max"], case["K"], mode=case["mode"],
                        layout=case["layout"])
    i = s.plan.info
    pos, row_ptr, col, recv, s.r_c = _radius_graph(case["nodes"], case["batch"], case["degree"], gen)
    src_ptr, src_perm = sobek.graph_prepare(row_ptr, col)
    s.graph = sobek.make_graph(row_ptr, col, src_ptr, src_perm, sobek.graph_receivers(row_ptr, src_perm))
    N, E = row_ptr.numel() - 1, col.numel()
    new = lambda *shape: torch.empty(shape, device="cuda")
    normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda")
    scale = _weight_scale(s.plan)
    s.x, s.R, s.gy = normal(N, i.C_x), normal(i.K, i.N_w) * scale, normal(N, i.C_y)
    s.y, s.gx, s.gR = new(N, i.C_y), new(N, i.C_x), new(i.K, i.N_w)
    order = {"fwd": 0, "dbwd": 2, "step": 2}.get(s.call, 1)
    s.ws = torch.empty(sobek.workspace_bytes(s.plan, N, E, order), dtype=torch.uint8, device="cuda")
    if s.call == "force":
        s.basis = BASES[case["basis"]]
        s.pos, s.rvec, s.g_rvec, s.gpos = pos, new(E, 3), new(E, 3), new(N, 3)
        return s
    rij = pos[col.long()] - pos[recv]
    r = rij.norm(dim=1)
    s.Y, s.phi = _harmonics(case["l_max"], rij / r[:, None]), _radial(case["basis"], case["K"], s.r_c, r)
    s.gY, s.gphi = new(E, i.dim_sh), new(E, i.K)
    if order == 2:
        s.vx, s.vY, s.vphi, s.vR = normal(N, i.C_x), normal(E, i.dim_sh), normal(E, i.K), normal(i.K, i.N_w) * scale
        s.ggy, s.hx, s.hY, s.hphi, s.hR = new(N, i.C_y), new(N, i.C_x), new(E, i.dim_sh), new(E, i.K), new(i.K, i.N_w)
    return s


def run(s):
    if s.call == "force":
        sobek.edge_vectors(s.graph, s.pos, s.rvec)
        sobek.conv_geo_fwd(s.plan, s.graph, s.rvec, s.basis, s.r_c, ENVELOPE, s.x, s.R, s.y, s.ws)
        sobek.conv_geo_bwd(s.plan, s.graph, s.rvec, s.basis, s.r_c, ENVELOPE, s.x, s.R, s.gy, s.gx, s.g_rvec, None, s.ws)
        sobek.position_gradient(s.graph, s.g_rvec, s.gpos)
        return {"y": s.y, "gx": s.gx, "g_rvec": s.g_rvec, "gpos": s.gpos}
    out = {}
    if s.call in ("fwd", "train", "step"):
        sobek.conv_fwd(s.plan, s.graph, s.x, s.Y, s.phi, s.R, s.y, s.ws)
        out.update(y=s.y)
    if s.call in ("bwd", "train", "step"):
        sobek.conv_bwd(s.plan, s.graph, s.x, s.Y, s.phi, s.R, s.gy, s.gx, s.gY, s.gphi, s.gR, s.ws)
        out.update(gx=s.gx, gY=s.gY, gphi=s.gphi, gR=s.gR)
    if s.call in ("dbwd", "step"):
        sobek.conv_dbwd(s.plan, s.graph, s.x, s.Y, s.phi, s.R, s.gy, s.vx, s.vY, s.vphi, s.vR, s.ggy, s.hx, s.hY, s.hphi,
                        s.hR, s.ws)
        out.update(ggy=s.ggy, hx=s.hx, hY=s.hY, hphi=s.hphi, hR=s.hR)
    return out


# ---- what a pass cannot do without ----------------------------------------------------------------------------


def work(case):
    """Each input read once and each output written once; multiply-adds of the receiver-factorised form (edge state of
    K x components per edge, one contraction with R per node; second order and adjoints as sums of the same maps)."""
    ii, io = _irreps(case["irreps_in"]), _irreps(case["irreps_out"])
    K, dsh, uvu = case["K"], (case["l_max"] + 1) ** 2, case["mode"] == "uvu"
    N = case["nodes"] * case["batch"]
    E = N * case["degree"]
    Cx, Cy = _dim(ii), _dim(io)
    F = Ft = Gf = Gt = Nw = 0
    for ci, li, pi in ii:
        for ls in range(case["l_max"] + 1):
            for co, lo, po in io:
                if abs(li - ls) <= lo <= li + ls and po == pi * (-1) ** ls:
                    w = ci if uvu else ci * co
                    Nw += w
                    F += ci * (2 * lo + 1)
                    Ft += co * (2 * li + 1)
                    Gf += w * (2 * lo + 1)
                    Gt += w * (2 * li + 1)
    R, graph, edge = K * Nw, 8 * N + 4 * E, dsh + K
    # (multiply-adds per edge over K, multiply-adds per node over K, floats in, floats out)
    parts = {
        "fwd": (F, Gf, N * Cx + E * edge + R, N * Cy),
        "bwd": (3 * F + Ft, 2 * Gf + Gt, N * (Cx + Cy) + E * edge + R, N * Cx + E * edge + R),
        "dbwd": (8 * F + 3 * Ft, 5 * Gf + 2 * Gt, N * (2 * Cx + Cy) + 2 * E * edge + 2 * R, N * (Cx + Cy) + E * edge + R),
        # forward and backward from positions, without the adjoint of R
        "force": (3 * F + Ft, 2 * Gf + Gt, N * (Cx + Cy + 3) + R, N * (Cx + Cy + 3) + 3 * E),
    }
    which = {"train": ("fwd", "bwd"), "step": ("fwd", "bwd", "dbwd")}.get(case["call"], (case["call"],))
    floats = sum(parts[k][2] + parts[k][3] for k in which)
    return {"bytes": 4 * floats + graph * len(which), "flops": 2 * K * sum(E * parts[k][0] + N * parts[k][1] for k in which)}


def _cost(case):
    """Time-like figure by which drawn cases are kept below the largest listed one."""
    w = work(case)
    return w["flops"] / 30e12 + w["bytes"] / 3e12


def tolerance(case):
    """Every product is taken as three bf16 products with 32-bit sums, which leaves some 2^-17 of each factor."""
    return {"rel": 4e-5}
