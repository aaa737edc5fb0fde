"""Performance cases of the compressed Deep Potential path on one GPU.

Each case is one pass that an MD program makes over a frame of atoms, through the package's public
calls.  Its fields:
  system  "shell"  random neighbour shells (no coordinates), "copper" fcc with one type, "alloy" fcc with
          three types 90/6/4 %, "water" molecules of two types;
  n0..n2  cells per axis (fcc: 4 atoms each; water: one molecule each; shell: n0 n1 n2 atoms);
  m1, m2  channels of the embedding net (m1/4, m1/2, m1 wide) and of the descriptor's second factor;
  scale   share of the usual neighbour rows and cut-off volume (1: sel 512 / 500 / 138);
  fill    fcc: share of the rows that hold a real neighbour (the lattice constant follows);
  switch  the weighting function: 0 cosine, 1 quintic;
  pass    "step"   the compressed embedding: T and D forward, ds and dR~ backward;
          "chain"  coordinates -> T, D -> dE/dT of a given dE/dD -> forces and virial;
          "model"  the whole energy model: coordinates -> D -> fitting net -> energies, forces, virial;
          "vector" the whole vector model: the fitting net's m1 outputs weight T's x, y, z rows;
          "fitting" the fitting net alone: energies and dE/dD;
  arith   "tc" f64 with the contractions on the tensor cores (the default path), "rows" f32 row by row,
          "moments" f32 by interval moments, "df64" f64 arrays in double-float arithmetic.

The geometries are jittered lattices at the densities of the copper, water and Al-Cu-Mg systems that the
tests and the benchmark use; net weights are random.  Everything is made on the device from the seed.
"""
import math

import numpy as np
import torch

import paper_2107_02103_gb300 as dpc

F64 = torch.float64
DENSITY = 0.0334  # water molecules per cubic angstrom
HIDDEN = (240, 240, 240)  # the fitting net of the paper
STRIDE0, STRIDE1, EXT = 0.01, 0.1, 5.0  # the table's fine and coarse step and its extension
RUN_ROWS = {"shell": 1.5, "copper": 10.0, "alloy": 6.2, "water": 2.7}  # consecutive rows in one table interval


def _case(name, system, cells, kind, arith="tc", m1=100, m2=16, scale=1.0, fill=0.83, switch=0):
    c = dict(system=system, n0=cells[0], n1=cells[1], n2=cells[2], arith=arith, m1=m1, m2=m2, scale=scale, fill=fill,
             switch=switch)
    c["pass"] = kind
    return {"name": name, **c} if name else c


def listed():
    return [
        # a handful of atoms with a small net, as a unit cell or a test run: launches and latency
        _case("shell_step_f64", "shell", (4, 4, 4), "step", m1=32, m2=4),
        # the headline: one step of the descriptor over 4096 copper atoms, 512 rows each
        _case("copper_step_f64", "copper", (8, 8, 16), "step"),
        # the water box of the network-size study: short runs of neighbours, four pair tables
        _case("water_step_f64", "water", (16, 16, 16), "step"),
        # a large three-component frame, nine pair tables, a third of the rows padding
        _case("alloy_step_f64", "alloy", (16, 16, 32), "step", fill=0.7),
        # odd sizes throughout: rows per type, channels, atoms per tile
        _case("ragged_step_f64", "alloy", (6, 7, 9), "step", m1=60, m2=7, scale=0.371, fill=0.77),
        # MD of a small water box from coordinates to forces, environment and forces fused
        _case("water_chain_f64", "water", (8, 8, 8), "chain"),
        # one MD step of the whole energy model on copper, the paper's switch
        _case("copper_model_f64", "copper", (8, 8, 16), "model", switch=1),
        # the same path in single precision, where f32 accuracy is enough
        _case("water_step_f32", "water", (16, 16, 16), "step", arith="rows"),
        _case("copper_step_f32", "copper", (8, 8, 16), "step", arith="moments"),
        # coordinates to forces in double-float arithmetic on the FP32 pipes
        _case("water_chain_df64", "water", (16, 16, 16), "chain", arith="df64"),
        # the fitting net alone, two centre types, forward and backward
        _case("water_fitting_f64", "water", (16, 16, 16), "fitting"),
        # a vector model (dipoles) on the smallest periodic water box: many small launches
        _case("water_vector_f64", "water", (4, 4, 4), "vector"),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "chain", "model", "vector", "fitting"])
    arith = rng.choice(["tc", "tc", "tc", "rows", "moments", "df64"]) if kind in ("step", "chain") else "tc"
    system = rng.choice(["copper", "water", "alloy"] + (["shell"] if kind == "step" else []))
    low, high = {"shell": (11, 3000), "copper": (216, 4096), "alloy": (216, 8192), "water": (64, 4096)}[system]
    if kind != "step":
        high = min(high, 2048)
    cells_wanted = math.exp(rng.uniform(math.log(low), math.log(high)))
    least = {"shell": 1, "copper": 6, "alloy": 6, "water": 4}[system]  # the box spans two cut-offs
    n0 = max(least, round(cells_wanted ** (1 / 3) * rng.uniform(0.75, 1.0)))
    n1 = max(least, round((cells_wanted / n0) ** 0.5))
    n2 = max(least, int(cells_wanted / (n0 * n1)))
    m1 = rng.choice([100, 100, 4 * rng.randint(6, 32)])
    m2 = rng.choice([16, 16, rng.randint(1, 24)])
    scale = rng.choice([1.0, round(rng.uniform(0.3, 1.0), 3)])
    fill = round(rng.uniform(0.35, 0.9), 3)
    return _case(None, system, (n0, n1, n2), kind, arith, m1, m2, scale, fill, rng.randint(0, 1))


# ------------------------------------------------------------------ geometry
def _sizes(case):
    """Rows per type, cut-offs, atoms, expected real rows per atom."""
    cells, sc = case["n0"] * case["n1"] * case["n2"], case["scale"]
    if case["system"] == "shell":
        sel, rc, rcs, nloc = [32], 4.0, 0.5, cells
    elif case["system"] == "copper":
        sel, rc, rcs, nloc = [max(8, round(512 * sc))], 8.0 * sc ** (1 / 3), 2.0, 4 * cells
    elif case["system"] == "alloy":
        sel, rc, rcs, nloc = [max(8, round(x * sc)) for x in (400, 60, 40)], 8.0 * sc ** (1 / 3), 2.0, 4 * cells
    else:
        sel, rc, rcs, nloc = [max(6, round(x * sc)) for x in (46, 92)], 6.0 * sc ** (1 / 3), 0.5, 3 * cells
    share = {"shell": 0.75, "copper": case["fill"], "alloy": case["fill"], "water": 0.65}[case["system"]]
    return sel, rc, rcs, nloc, share * sum(sel)


def _gen(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + tag)
    return g


def _normal(seed, tag, *shape):
    return torch.randn(shape, dtype=F64, device="cuda", generator=_gen(seed, tag))


def _uniform(seed, tag, *shape):
    return torch.rand(shape, dtype=F64, device="cuda", generator=_gen(seed, tag))


def _lattice(case):
    ax = [torch.arange(case[k], device="cuda", dtype=F64) for k in ("n0", "n1", "n2")]
    return torch.stack(torch.meshgrid(*ax, indexing="ij"), dim=-1).reshape(-1, 3)


def _atoms(case, seed):
    """Positions (sorted by type), types and box."""
    cell, shape = _lattice(case), [case["n0"], case["n1"], case["n2"]]
    if case["system"] == "water":
        a = DENSITY ** (-1 / 3)
        o = (cell + 0.5) * a + 0.3 * (2.0 * _uniform(seed, 1, len(cell), 3) - 1.0)
        u = torch.nn.functional.normalize(_normal(seed, 2, len(cell), 3), dim=1)
        w = torch.nn.functional.normalize(torch.linalg.cross(u, _normal(seed, 3, len(cell), 3)), dim=1)
        half = math.radians(104.5) / 2
        h = [o + 0.96 * (math.cos(half) * u + sgn * math.sin(half) * w) for sgn in (1.0, -1.0)]
        pos = torch.cat([o, torch.stack(h, dim=1).reshape(-1, 3)])
        types = torch.cat([torch.zeros(len(cell)), torch.ones(2 * len(cell))]).to("cuda", torch.int32)
    else:
        sel, rc, _, _, real = _sizes(case)
        a = (4.0 * (4.0 / 3.0) * math.pi * rc ** 3 / real) ** (1.0 / 3.0)
        basis = torch.tensor([[0, 0, 0], [0.5, 0.5, 0], [0.5, 0, 0.5], [0, 0.5, 0.5]], dtype=F64, device="cuda")
        pos = ((cell[:, None, :] + basis).reshape(-1, 3) + 0.25) * a
        pos = pos + 0.1 * _normal(seed, 1, len(pos), 3)
        if case["system"] == "alloy":
            x = _uniform(seed, 2, len(pos))
            types = (x > 0.90).to(torch.int32) + (x > 0.96).to(torch.int32)
            order = torch.argsort(types, stable=True)
            pos, types = pos[order], types[order].contiguous()
        else:
            types = torch.zeros(len(pos), dtype=torch.int32, device="cuda")
    box = torch.tensor([n * a for n in shape], dtype=F64, device="cuda")
    return pos, types, box


def _neighbours(pos, types, box, rc, sel):
    """Neighbour list over local atoms and periodic images: per type segment the nearest first, -1 padding."""
    n, b32, p32 = len(pos), box.float(), pos.float()
    segs = [torch.nonzero(types == b).flatten() for b in range(len(sel))]
    step = max(1, (1 << 26) // n)
    out = []
    for lo in range(0, n, step):
        parts = []
        for b, idx in enumerate(segs):
            d2 = torch.zeros((min(step, n - lo), len(idx)), device="cuda")
            for c in range(3):
                d = p32[idx, c][None, :] - p32[lo:lo + step, c][:, None]
                d -= b32[c] * torch.round(d / b32[c])
                d2 += d * d
            d2[d2 < 1e-8] = float("inf")  # the atom itself
            k = min(sel[b], len(idx))
            v, at = torch.topk(d2, k, dim=1, largest=False, sorted=True)
            j = torch.where(v < rc * rc, idx[at], -1)
            parts.append(torch.nn.functional.pad(j, (0, sel[b] - k), value=-1))
        out.append(torch.cat(parts, dim=1))
    j = torch.cat(out)
    hit = j >= 0
    # every (atom, box shift) pair other than the atom itself becomes one image after the local atoms
    jj = j.clamp(min=0)
    shift = -torch.round((pos[jj] - pos[:, None, :]) / box).to(torch.int64)
    code = ((shift[..., 0] + 1) * 3 + shift[..., 1] + 1) * 3 + shift[..., 2] + 1
    image = hit & (code != 13)
    uniq, inv = torch.unique((jj * 27 + code)[image], return_inverse=True)
    c = uniq % 27
    sv = torch.stack([c // 9 - 1, (c // 3) % 3 - 1, c % 3 - 1], dim=1).to(F64)
    # the rows that an MD program sets aside for images: the shell's share of the volume and a margin, the rest far away
    room = math.ceil(1.2 * n * (float(torch.prod(1.0 + 2.0 * rc / box)) - 1.0)) + 64
    far = torch.full((room - len(uniq), 3), 1e3, dtype=F64, device="cuda")
    coord = torch.cat([pos, pos[uniq // 27] + sv * box, far])
    j = torch.where(hit, j, -1)
    j[image] = n + inv
    return coord.contiguous(), j.to(torch.int32).contiguous()


def _switch(r, rcs, rc, kind):
    """The weighting function s(r) (Sec. II of the paper; kind 0: its cosine form)."""
    u = ((r - rcs) / (rc - rcs)).clamp(0.0, 1.0)
    w = u ** 3 * (-6.0 * u * u + 15.0 * u - 10.0) + 1.0 if kind == 1 else 0.5 * torch.cos(math.pi * u) + 0.5
    return w / r


def _rows(d, rcs, rc, kind):
    """(s, R~) of displacement vectors."""
    r = torch.sqrt((d * d).sum(-1))
    s = _switch(r, rcs, rc, kind)
    return s, torch.cat([s[..., None], (s / r)[..., None] * d], dim=-1)


def _inputs(case, seed):
    """The frame in f64: sel, s, R~, valid rows per type, types, and coordinates with their list."""
    sel, rc, rcs, nloc, _ = _sizes(case)
    x = {"sel": sel, "rc": rc, "rcs": rcs}
    nnei = sum(sel)
    if case["system"] == "shell":
        real = 3 * nnei // 4
        r = torch.sort(0.9 + (rc - 0.9) * _uniform(seed, 1, nloc, real), dim=1).values
        d = r[..., None] * torch.nn.functional.normalize(_normal(seed, 2, nloc, real, 3), dim=2)
        d = torch.nn.functional.pad(d, (0, 0, 0, nnei - real))
        hit = (torch.arange(nnei, device="cuda") < real).expand(nloc, nnei)
        x["types"] = torch.zeros(nloc, dtype=torch.int32, device="cuda")
    else:
        pos, x["types"], box = _atoms(case, seed)
        x["coord"], x["nlist"] = _neighbours(pos, x["types"], box, rc, sel)
        hit = x["nlist"] >= 0
        d = x["coord"][x["nlist"].clamp(min=0).long()] - x["coord"][:nloc, None, :]
    s, R = _rows(torch.where(hit[..., None], d, 1.0), rcs, rc, case["switch"])
    x["hit"], x["d"] = hit, d
    x["s"] = torch.where(hit, s, 0.0).contiguous()
    x["Rt"] = torch.where(hit[..., None], R, 0.0).contiguous()
    x["nvalid"] = torch.stack([h.sum(1) for h in hit.split(sel, dim=1)], dim=1).to(torch.int32).contiguous()
    x["range"] = (0.0, float(x["s"].max()))
    return x


# ------------------------------------------------------------------- weights
def _net(seed, tag, widths, count):
    """Per net and layer: W [in][out] ~ N(0, 1/in), then b [out] ~ N(0, 1)."""
    rows = []
    for l in range(len(widths) - 1):
        w = _normal(seed, tag + 2 * l, count, widths[l] * widths[l + 1]) / math.sqrt(widths[l])
        rows += [w, _normal(seed, tag + 2 * l + 1, count, widths[l + 1])]
    return torch.cat(rows, dim=1).contiguous()


def _layers(params, widths):
    at = 0
    for l in range(len(widths) - 1):
        i, o = widths[l], widths[l + 1]
        yield params[:, at:at + i * o].reshape(-1, i, o), params[:, at + i * o:at + i * o + o]
        at += i * o + o


def _table(case, seed, x):
    """The table a compressed model holds, f64 [pairs][intervals][3][m1][2]: the quintics through the net's
    value and first two derivatives at the nodes."""
    m1, nt = case["m1"], len(x["sel"])
    widths = [1, m1 // 4, m1 // 2, m1]
    info = dpc.dp_table_info_make(*x["range"], STRIDE0, STRIDE1, EXT)
    n0, n1 = (round((info.upper - info.lower) / info.stride0), round((info.upper_ext - info.upper) / info.stride1))
    nodes = torch.cat([info.lower + info.stride0 * torch.arange(n0, dtype=F64), info.upper + info.stride1
                       * torch.arange(n1 + 1, dtype=F64)]).cuda()
    h = nodes[None, :, None].expand(nt * nt, -1, 1)
    dh, d2h = torch.ones_like(h), torch.zeros_like(h)
    for w, b in _layers(_net(seed, 100, widths, nt * nt), widths):
        v = torch.tanh(h @ w + b[:, None, :])
        g, g2 = dh @ w, d2h @ w
        dv = (1.0 - v * v) * g
        d2v = (1.0 - v * v) * g2 - 2.0 * v * g * dv
        fold = {1: lambda z: z, 2: lambda z: torch.cat([z, z], dim=2)}.get(w.shape[2] // w.shape[1]) \
            if w.shape[2] in (w.shape[1], 2 * w.shape[1]) else None
        h, dh, d2h = (v + fold(h), dv + fold(dh), d2v + fold(d2h)) if fold else (v, dv, d2v)
    t = torch.diff(nodes)[None, :, None]
    y, y1, dy, dy1, c, c1 = h[:, :-1], h[:, 1:], dh[:, :-1], dh[:, 1:], d2h[:, :-1], d2h[:, 1:]
    k = y1 - y - dy * t - 0.5 * c * t * t
    m = (dy1 - dy - c * t) * t
    q = (c1 - c) * t * t
    co = [(6.0 * k - 3.0 * m + 0.5 * q) / t ** 5, (-15.0 * k + 7.0 * m - q) / t ** 4, (10.0 * k - 4.0 * m + 0.5 * q)
          / t ** 3, 0.5 * c, dy, y]  # of t^5 .. t^0
    tab = torch.stack([torch.stack(co[2 * i:2 * i + 2], dim=-1) for i in range(3)], dim=2)
    return info, nodes, n0, tab.contiguous()


def _fitting(case, seed, x):
    nout = case["m1"] if case["pass"] == "vector" else 1
    widths = [case["m1"] * case["m2"], *HIDDEN, nout]
    counts = torch.bincount(x["types"].long(), minlength=len(x["sel"])).tolist()
    return widths, _net(seed, 200, widths, len(x["sel"])), [0, *np.cumsum(counts).tolist()]


def _given(case, seed, x):
    """Upstream gradients and stand-alone descriptors."""
    n, m1, m2 = len(x["types"]), case["m1"], case["m2"]
    return {"dT": _normal(seed, 10, n, 4, m1), "dD": _normal(seed, 11, n, m1, m2), "dv": _normal(seed, 12, n, 3),
            "D": 0.1 * _normal(seed, 13, n, m1 * m2)}


# ------------------------------------------------------------------ the pass
def prepare(case, seed):
    x = _inputs(case, seed)
    kind, arith = case["pass"], case["arith"]
    f32 = arith in ("rows", "moments")
    dt = torch.float32 if f32 else F64
    given = _given(case, seed, x)
    st = {"case": dict(case), "sel": x["sel"], "types": x["types"], "kind": kind, "arith": arith, "m2": case["m2"]}
    if kind != "fitting":
        info, _, _, tab = _table(case, seed, x)
        st["info"] = info
        if arith == "tc":
            st["plan"] = dpc.dp_tabulate_tc_plan_f64(tab, info, sum(x["sel"]))
            need = dpc.dp_tabulate_tc_work_bytes(info, len(x["types"]), sum(x["sel"]), len(x["sel"]), case["m1"])
            st["work"] = torch.empty(need, dtype=torch.uint8, device="cuda")
        elif arith == "df64":
            hi = tab.float()
            st["table"] = torch.stack([hi, (tab - hi.double()).float()], dim=-1).flatten(-2).contiguous()
        else:
            st["table"] = tab.to(dt)
    if kind == "step":
        st.update(s=x["s"].to(dt), Rt=x["Rt"].to(dt), nvalid=x["nvalid"], dT=given["dT"].to(dt))
    elif kind != "fitting":
        st.update(coord=x["coord"].to(dt), nlist=x["nlist"], env=dpc.env_info(x["rcs"], x["rc"], case["switch"]))
        st.update(dD=given["dD"].to(dt), dv=given["dv"])
    else:
        st["D"] = given["D"]
    if kind in ("model", "vector", "fitting"):
        st["widths"], st["params"], st["start"] = _fitting(case, seed, x)
        st["fwork"] = torch.empty(dpc.dp_fitting_tc_work_bytes(st["widths"], len(x["types"])), dtype=torch.uint8,
                                  device="cuda")
    return st


def run(st):
    kind, arith, sel = st["kind"], st["arith"], st["sel"]
    reuse = dpc.DP_TC_REUSE_RUNS
    if kind == "fitting":
        E, act = dpc.dp_fitting_fwd_tc_f64(st["params"], st["widths"], st["start"], st["D"], work=st["fwork"])
        return {"E": E, "act": act,
                "dD": dpc.dp_fitting_grad_tc_f64(st["params"], st["widths"], st["start"], act, work=st["fwork"])}
    if arith == "tc":
        plan, info, work = st["plan"], st["info"], st["work"]
        if kind == "step":
            args = (plan, info, st["s"], st["Rt"], st["nvalid"], st["types"], sel)
            T, D = dpc.dp_tabulate_fusion_fwd_tc_f64(*args, work=work, M2=st["m2"])
            ds, dRt = dpc.dp_tabulate_fusion_grad_tc_f64(*args, st["dT"], work=work, flags=reuse)
            return {"T": T, "D": D, "ds": ds, "dRt": dRt}
        coord, nlist, env = st["coord"], st["nlist"], st["env"]
        T, D, nvalid = dpc.dp_tabulate_fusion_env_fwd_tc_f64(plan, info, coord, nlist, sel, env, st["types"],
                                                             work=work, M2=st["m2"])
        out = {"D": D, "nvalid": nvalid}
        if kind == "chain":
            dT = dpc.dp_descriptor_contract_grad(T, st["dD"])
        else:
            net = (st["params"], st["widths"], st["start"])
            E, act = dpc.dp_fitting_fwd_tc_f64(*net, D, work=st["fwork"])
            g = None
            if kind == "vector":
                out["v"] = dpc.dp_vector_head(T, E)
                g = dpc.dp_vector_head_grad(T, E, st["dv"], want=("da",))[1]
            dD = dpc.dp_fitting_grad_tc_f64(*net, act, g=g, work=st["fwork"])
            dT = dpc.dp_descriptor_contract_grad(T, dD.view(D.shape))
            if kind == "vector":
                dpc.dp_vector_head_grad(T, E, st["dv"], dT=dT, accumulate=True, want=("dT",))
            out["E"] = E
        F, W = dpc.dp_tabulate_fusion_env_grad_tc_f64(plan, info, coord, nlist, sel, env, st["types"], dT, work=work,
                                                      flags=reuse)
        return {**out, "dT": dT, "F": F, "virial": W}
    df = dpc.DF64 if arith == "df64" else None
    fwd, grad = (dpc.dp_tabulate_fusion_fwd, dpc.dp_tabulate_fusion_grad) if arith == "rows" else \
        (dpc.dp_tabulate_fusion_fwd_moments, dpc.dp_tabulate_fusion_grad_moments)
    if kind == "step":
        s, Rt, nvalid = st["s"], st["Rt"], st["nvalid"]
    else:
        s, Rt, nvalid = dpc.dp_env_mat(st["coord"], st["nlist"], sel, st["env"], arith=df)
    args = (st["table"], st["info"], s, Rt, nvalid, st["types"], sel)
    T = fwd(*args)
    D = dpc.dp_descriptor_contract(T, st["m2"], arith=df)
    if kind == "step":
        ds, dRt = grad(*args, st["dT"])
        return {"T": T, "D": D, "ds": ds, "dRt": dRt}
    dT = dpc.dp_descriptor_contract_grad(T, st["dD"], arith=df)
    ds, dRt = grad(*args, dT)
    F, W = dpc.dp_force_virial(st["coord"], st["nlist"], st["env"], ds, dRt, arith=df)
    return {"D": D, "nvalid": nvalid, "dT": dT, "F": F, "virial": W}


def work(case):
    """Inputs read and outputs written once; the moments (24 FMA a row), the derivatives (40), the contraction
    with the coefficients (24 m1 FMA per run of rows and direction), D (4 m1 m2) and its backward, the net."""
    sel, _, _, n, real = _sizes(case)
    kind, m1, m2, nnei = case["pass"], case["m1"], case["m2"], sum(sel)
    e = 4 if case["arith"] in ("rows", "moments") else 8
    hidden = sum(HIDDEN)
    widths = [m1 * m2, *HIDDEN, m1 if kind == "vector" else 1]
    weights = sum((widths[l] + 1) * widths[l + 1] for l in range(len(widths) - 1))
    net = 2.0 * n * 2 * weights
    if kind == "fitting":
        return {"bytes": 8.0 * (n * (2 * m1 * m2 + 1 + hidden) + len(sel) * weights), "flops": net}
    runs = real / RUN_ROWS[case["system"]]
    flops = 2.0 * n * (64 * real + 48 * m1 * runs + 4 * m1 * m2)
    table = len(sel) ** 2 * 200 * 6 * m1 * e
    if kind == "step":
        rows = n * nnei * 5 * e
        return {"bytes": float(n * real * 5 * e + rows + n * e * (8 * m1 + m1 * m2) + table), "flops": flops}
    moved = n * nnei * 4 + 2 * 3 * n * e + n * e * (m1 * m2 + 4 * m1) + table
    if kind == "chain":
        moved += n * e * m1 * m2
    else:
        moved += len(sel) * weights * e
        flops += net
    return {"bytes": float(moved), "flops": flops + 2.0 * n * 8 * m1 * m2}


# ------------------------------------------------------- the same in 64 bits
def _exact_net(params, widths, start, D):
    E, acts = [], []
    for t in range(len(start) - 1):
        v, keep = D[start[t]:start[t + 1]], []
        layers = list(_layers(params[t:t + 1], widths))
        for w, b in layers[:-1]:
            z = torch.tanh(v @ w[0] + b[0])
            keep.append(z)
            v = z + v if w.shape[1] == w.shape[2] else z
        E.append(v @ layers[-1][0][0] + layers[-1][1][0])
        acts.append(torch.cat(keep, dim=1))
    E = torch.cat(E)
    return (E[:, 0] if E.shape[1] == 1 else E), torch.cat(acts)


def exact(case, seed):
    x, kind = _inputs(case, seed), case["pass"]
    given = _given(case, seed, x)
    if kind == "fitting":
        widths, params, start = _fitting(case, seed, x)
        D = given["D"].requires_grad_(True)
        E, act = _exact_net(params, widths, start, D)
        return {"E": E.detach(), "act": act.detach(), "dD": torch.autograd.grad(E.sum(), D)[0]}
    if case["arith"] in ("rows", "moments"):  # in 64 bits on the values that the 32-bit arrays hold
        if kind == "step":
            for k in ("s", "Rt"):
                x[k] = x[k].float().double()
        else:
            x["coord"] = x["coord"].float().double()
            x["d"] = x["coord"][x["nlist"].clamp(min=0).long()] - x["coord"][:len(x["types"]), None, :]
        given = {k: v.float().double() for k, v in given.items()}
    info, nodes, n0, tab = _table(case, seed, x)
    if case["arith"] in ("rows", "moments"):
        tab = tab.float().double()
    n, m1, m2, nnei, nt = len(x["types"]), case["m1"], case["m2"], sum(x["sel"]), len(x["sel"])
    tab = tab.permute(0, 1, 3, 2, 4).reshape(nt * nt * (len(nodes) - 1), m1, 6)
    seg = torch.repeat_interleave(torch.arange(nt, device="cuda"), torch.tensor(x["sel"], device="cuda"))
    hit, step = x["hit"], max(1, 250_000 // nnei)

    def rows_of(a):  # (s, R~) of atoms a: the input arrays, or from coordinates with their graph
        if kind == "step":
            return None, x["s"][a], x["Rt"][a]
        d = torch.where(hit[a][..., None], x["d"][a], 1.0).requires_grad_(True)
        s, R = _rows(d, x["rcs"], x["rc"], case["switch"])
        return d, torch.where(hit[a], s, 0.0), torch.where(hit[a][..., None], R, 0.0)

    def table_at(s, a):  # g and g' of every row
        sd = s.detach()
        l0 = ((sd - info.lower) / info.stride0).floor().clamp(0, n0 - 1)
        l1 = n0 + ((sd - info.upper) / info.stride1).floor().clamp(min=0)
        l = torch.where(sd < info.upper, l0, l1).long().clamp(max=len(nodes) - 2)
        t = (sd - nodes[l])[..., None]
        pair = x["types"][a].long()[:, None] * nt + seg[None, :]
        c = tab[pair * (len(nodes) - 1) + l]
        g, dg = c[..., 0], torch.zeros_like(c[..., 0])
        for q in range(1, 6):
            dg = dg * t + g
            g = g * t + c[..., q]
        return g * hit[a][..., None], dg * hit[a][..., None]

    T = torch.empty((n, 4, m1), dtype=F64, device="cuda")
    for lo in range(0, n, step):
        a = slice(lo, min(n, lo + step))
        _, s, R = rows_of(a)
        T[a] = R.detach().transpose(1, 2) @ table_at(s, a)[0] / nnei
    out = {}
    if kind == "step":
        dT, D = given["dT"], T.transpose(1, 2) @ T[:, :, :m2]
        out["T"] = T
    else:
        Tg = T.clone().requires_grad_(True)
        D = Tg.transpose(1, 2) @ Tg[:, :, :m2]
        if kind == "chain":
            loss = (D * given["dD"]).sum()
        else:
            widths, params, start = _fitting(case, seed, x)
            E, _ = _exact_net(params, widths, start, D.reshape(n, m1 * m2))
            out["E"] = E.detach()
            if kind == "vector":
                v = (Tg[:, 1:] @ E[:, :, None])[..., 0]
                out["v"] = v.detach()
                loss = (v * given["dv"]).sum()
            else:
                loss = E.sum()
        dT = torch.autograd.grad(loss, Tg)[0]
        D = D.detach()
        F = torch.zeros_like(x["coord"])
        W = torch.zeros((3, 3), dtype=F64, device="cuda")
    ds, dRt = torch.empty((n, nnei), dtype=F64, device="cuda"), torch.empty((n, nnei, 4), dtype=F64, device="cuda")
    for lo in range(0, n, step):
        a = slice(lo, min(n, lo + step))
        d, s, R = rows_of(a)
        g, dg = table_at(s, a)
        dRa = g @ dT[a].transpose(1, 2) / nnei
        dsa = (R.detach() * (dg @ dT[a].transpose(1, 2))).sum(-1) / nnei
        if kind == "step":
            ds[a], dRt[a] = dsa, dRa
            continue
        gd = torch.autograd.grad((s * dsa).sum() + (R * dRa).sum(), d)[0]
        F[:n][a] += gd.sum(1)
        F.index_add_(0, x["nlist"][a].clamp(min=0).long().flatten(), -gd.reshape(-1, 3))
        W -= torch.einsum("bni,bnj->ij", d.detach() * hit[a][..., None], gd)
    out["D"] = D
    if kind == "step":
        return {**out, "ds": ds, "dRt": dRt}
    return {**out, "nvalid": None, "dT": dT, "F": F, "virial": W}
