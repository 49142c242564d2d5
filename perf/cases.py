"""The work that performance is measured on: what programs have this library do.

Evaluations of one cell (host and device buffers), batches of uneven cells as a
server packs them, molecular dynamics (NVE, and the NVT protocol of the paper's
benchmarks) and one convolution with its gradients through autograd; from one
16-atom cell to 112,000 atoms, FP32 and BF16, the SevenNet-0 model and the
smaller models of the paper's benchmarks (degree 2 and 3, 4 to 64 channels).

Structures are disordered cells of the repository's densities: a lattice with
vacancies whose atoms are displaced at random, so that every pair keeps a
physical distance and a large cell takes milliseconds to make.
"""

import math

import numpy as np
import torch
import torch.utils.checkpoint

import paper_2402_03789_gb300 as sn

MASSES = np.array([14.0067, 15.999, 28.0855])       # N, O, Si
SHIFT = (-0.05, -0.03, -0.08)                        # eV per atom of a species: total energies do not cancel to nothing
AMU_G = 1.66053906660e-24
ACC = 9.64853321e-3                                  # eV/A/amu -> A/fs^2
KB = 8.617333262e-5

# name -> (multiplicities, layers, r_cut, radial MLP width, avg. neighbours, readout width)
MODELS = {
    "sevennet0": ((128, 64, 32), 5, 5.0, 64, 34.0, 64),
    "small": ((32, 32), 3, 5.0, 32, 34.0, 16),
}


def model_spec(case):
    """Hyper-parameters of the case's model: a named one, or "bench" (every irrep
    has `channels` channels, r_c 4 A) with the case's layers, channels and lmax."""
    if case["model"] == "bench":
        mul, layers = (case["channels"],) * (case["lmax"] + 1), case["layers"]
        rc, hid, avg, ro = 4.0, 64, 21.4, 64
    else:
        mul, layers, rc, hid, avg, ro = MODELS[case["model"]]
    return dict(n_species=3, n_layers=layers, mul=mul, r_cut=rc, n_basis=8, poly_p=6, mlp_hidden=hid,
                avg_num_neigh=avg, readout_hidden=ro, scale=1.0, shift=SHIFT)


def listed():
    s0 = dict(model="sevennet0")
    return [
        # the smallest request a server or a script sends: latency and launches
        dict(name="eval_16_fp32", kind="host", prec="fp32", atoms=16, rho=2.2, **s0),
        # one call on a parity-sized cell from host buffers
        dict(name="eval_192_bf16", kind="host", prec="bf16", atoms=192, rho=2.2, **s0),
        # a serving batch: cells of 16 to 2,000 atoms, log-uniform, packed together
        dict(name="batch_24_bf16", kind="batch", prec="bf16", structs=24, atoms=2000, rho=2.6, **s0),
        # an ordinary cell in full precision, on device buffers
        dict(name="eval_3000_fp32", kind="dev", prec="fp32", atoms=3000, rho=2.2, **s0),
        # the benchmark's workload: 24,000-atom SiO2, BF16
        dict(name="eval_24000_bf16", kind="dev", prec="bf16", atoms=24000, rho=2.2, **s0),
        # the largest cell: 112,000-atom Si3N4
        dict(name="eval_112000_bf16", kind="dev", prec="bf16", atoms=112000, rho=3.1, **s0),
        # NVE dynamics in full precision, three steps a call and the state read back
        dict(name="md_nve_1000_fp32", kind="md", prec="fp32", atoms=1000, rho=2.2, steps=3, temp=300.0, tau=0.0,
             skin=0.0, **s0),
        # the paper's benchmark protocol: degree-3 model, NVT, here with a Verlet skin
        dict(name="md_nvt_4608_lmax3_bf16", kind="md", prec="bf16", atoms=4608, rho=2.65, steps=4, temp=300.0,
             tau=100.0, skin=0.5, model="bench", layers=3, channels=32, lmax=3),
        # a degree-3 benchmark model with channels that need padding, full precision
        dict(name="eval_1500_lmax3_fp32", kind="dev", prec="fp32", atoms=1500, rho=2.65, model="bench", layers=4,
             channels=16, lmax=3),
        # a degree-2 benchmark model on the paper's 12,960-atom cell
        dict(name="eval_12960_lmax2_bf16", kind="dev", prec="bf16", atoms=12960, rho=2.65, model="bench", layers=5,
             channels=64, lmax=2),
        # one middle block and its gradients through autograd, as a training program calls it
        dict(name="conv_2777_bf16", kind="conv", prec="bf16", atoms=2777, rho=2.2, layer=2, **s0),
        dict(name="conv_803_fp32", kind="conv", prec="fp32", atoms=803, rho=2.2, layer=1, **s0),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["host", "dev", "dev", "batch", "md", "conv"])
    prec = rng.choice(["bf16", "bf16", "fp32"])
    name = rng.choice(["sevennet0", "sevennet0", "bench", "bench", "small"])
    c = dict(kind=kind, prec=prec, model=name, rho=round(rng.uniform(2.2, 3.1), 3))
    if name == "bench":
        c.update(layers=rng.randint(2, 5), channels=rng.choice([4, 8, 16, 24, 32, 48, 64]), lmax=rng.choice([2, 3]))
    top = 6000 if prec == "fp32" else 30000
    if kind == "host":
        c["atoms"] = _log_uniform(rng, 16, 3000)
    elif kind == "dev":
        c["atoms"] = _log_uniform(rng, 16, top)
    elif kind == "batch":
        c.update(structs=rng.randint(2, 48), atoms=_log_uniform(rng, 64, 2000 if prec == "bf16" else 500))
    elif kind == "md":
        c.update(atoms=_log_uniform(rng, 64, top // 4), steps=rng.randint(1, 4), temp=300.0,
                 tau=rng.choice([0.0, 100.0]), skin=rng.choice([0.0, 0.5]))
    else:
        layers = model_spec(c)["n_layers"]
        c.update(atoms=_log_uniform(rng, 16, top // 4), layer=rng.randrange(layers))
    return c


# ------------------------------------------------------------------ inputs
def _structure(n, rho, rng):
    """(pos [n,3], species [n], cell [3,3]): a slightly sheared periodic cell of
    about the density rho (g/cm3), species at random over N, O and Si."""
    species = rng.integers(0, 3, n).astype(np.int32)
    length = (MASSES[species].sum() * AMU_G / rho * 1e24) ** (1.0 / 3.0)
    cell = np.eye(3) * length
    cell[1, 0] = 0.04 * length
    cell[2, 1] = -0.03 * length
    k = max(1, math.ceil(n ** (1.0 / 3.0) - 1e-9))
    site = np.sort(rng.permutation(k ** 3)[:n])
    grid = np.stack([site // (k * k), site // k % k, site % k], 1)
    frac = (grid + 0.5 + rng.uniform(-0.16, 0.16, (n, 3))) / k
    order = rng.permutation(n)                       # the caller's order is not the lattice's
    return (frac @ cell)[order], species, cell


def _sizes(case):
    rng = np.random.default_rng(case["structs"])     # the sizes belong to the case, what fills them to the seed
    lo = 16 if case["atoms"] > 16 else 1
    s = np.exp(rng.uniform(math.log(lo), math.log(case["atoms"] + 1), case["structs"]))
    return np.clip(s.astype(int), lo, case["atoms"])


def _velocities(species, temp, rng):
    m = MASSES[species]
    v = rng.standard_normal((m.size, 3)) * np.sqrt(KB * temp / m * ACC)[:, None]
    return v - (m[:, None] * v).sum(0) / m.sum()


def _inputs(case, seed):
    """Everything drawn for a case, from the seed alone, as numpy arrays."""
    rng = np.random.default_rng(seed)
    spec = model_spec(case)
    d = dict(spec=spec, weights=rng.standard_normal(sum(a * b for _, (a, b) in _layout(spec))))
    if case["kind"] == "batch":
        parts = [_structure(int(n), case["rho"], rng) for n in _sizes(case)]
        d["offsets"] = np.concatenate([[0], np.cumsum([p[0].shape[0] for p in parts])]).astype(np.int64)
        d["pos"], d["species"] = np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts])
        d["cells"] = np.stack([p[2] for p in parts])
        return d
    conv = case["kind"] == "conv"                    # a block's graph belongs to the case, too
    pos, species, cell = _structure(case["atoms"], case["rho"], np.random.default_rng(case["atoms"]) if conv else rng)
    d.update(pos=pos, species=species, cells=cell[None], offsets=np.array([0, pos.shape[0]], np.int64))
    if case["kind"] == "md":
        d["vel"] = _velocities(species, case["temp"], rng)
    if conv:
        dst, src, vec = (t.cpu().numpy() for t in _graph(torch.as_tensor(pos, device="cuda"),
                                                         torch.as_tensor(cell, device="cuda"), spec["r_cut"]))
        order = np.argsort(dst, kind="stable")
        turn, _ = np.linalg.qr(rng.standard_normal((3, 3)))
        vec = vec @ turn * rng.uniform(0.97, 1.0)
        d.update(row_ptr=np.searchsorted(dst[order], np.arange(pos.shape[0] + 1)).astype(np.int32),
                 src=src[order].astype(np.int32), vec=vec[order].astype(np.float32))
        blk = _block(spec, case["layer"])
        xd = sum((2 * l + 1) * m for l, m in blk["inp"].items())
        md = sum((2 * l + 1) * m for l, m in blk["msg"].items())
        d["x"] = rng.standard_normal((pos.shape[0], xd)).astype(np.float32)
        d["gm"] = rng.standard_normal((pos.shape[0], md)).astype(np.float32)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    st = dict(case=case, model=sn.SevenNet(d["spec"], d["weights"], device=0))
    dev = torch.device("cuda", 0)
    kind = case["kind"]
    if kind == "host":
        st.update(pos=d["pos"], species=d["species"], cell=d["cells"][0])
    elif kind in ("dev", "batch"):
        n, s = d["pos"].shape[0], len(d["cells"])
        ew = torch.empty(10 * s, dtype=torch.float64, device=dev)      # energies, then virials
        st.update(offsets=d["offsets"], cells=d["cells"], species=torch.as_tensor(d["species"], device=dev),
                  pos=torch.as_tensor(d["pos"], device=dev), ew=ew,
                  out=(ew[:s], torch.empty((n, 3), dtype=torch.float64, device=dev), ew[s:].view(s, 3, 3)))
    elif kind == "md":
        md = sn.MD(st["model"], d["pos"], d["vel"], d["species"], MASSES, d["cells"][0], case["prec"])
        if case["skin"] > 0:
            md.set_skin(case["skin"])
        if case["tau"] > 0:
            md.set_nose_hoover(case["temp"], case["tau"])
        st["md"] = md
    else:
        from paper_2402_03789_gb300.autograd import conv
        st.update({k: torch.as_tensor(d[k], device=dev) for k in ("row_ptr", "src", "gm")}, conv=conv,
                  x=torch.as_tensor(d["x"], device=dev).requires_grad_(True),
                  vec=torch.as_tensor(d["vec"], device=dev).requires_grad_(True))
    return st


def run(st):
    case, model = st["case"], st["model"]
    kind = case["kind"]
    if kind == "host":
        e, f, w = model.evaluate(st["pos"], st["cell"], st["species"], precision=case["prec"])
        return dict(energy_virial=np.concatenate([[e], w.reshape(-1)]), forces=f)
    if kind in ("dev", "batch"):
        _, f, _ = model.evaluate_batch_dev(st["offsets"], st["cells"], st["species"], st["pos"],
                                           precision=case["prec"], out=st["out"])
        return dict(energy_virial=st["ew"], forces=f)
    if kind == "md":
        ep, ek = st["md"].step(case["steps"], 1.0)
        pos, vel, f = st["md"].state()
        return dict(energies=np.stack([ep, ek]), pos=pos, vel=vel, forces=f)
    m = st["conv"](model, case["layer"], st["x"], st["vec"], st["row_ptr"], st["src"], case["prec"])
    gx, gd = torch.autograd.grad(m, [st["x"], st["vec"]], st["gm"])
    return dict(m=m.detach(), gx=gx, gd=gd)


# ------------------------------------------------------------------ work and tolerance
def _couplings(inp, lmax, last):
    return [(a, b, c, inp[a]) for a in sorted(inp) for b in range(lmax + 1)
            for c in range(abs(a - b), min(a + b, lmax) + 1) if not last or c == 0]


def _block(spec, t):
    mul, lmax = spec["mul"], len(spec["mul"]) - 1
    last = t == spec["n_layers"] - 1
    inp = {0: mul[0]} if t == 0 else dict(enumerate(mul))
    paths = _couplings(inp, lmax, last)
    msg = {}
    for _, _, c, m in paths:
        msg[c] = msg.get(c, 0) + m
    gate = {0: mul[0]} if last else {0: sum(mul), **{l: mul[l] for l in range(1, lmax + 1)}}
    return dict(inp=inp, paths=paths, msg=dict(sorted(msg.items())), gate=gate, last=last, width=sum(p[3] for p in paths))


def _layout(spec):
    """(name, (rows, columns)) of the canonical weight vector, in order."""
    out, h = [("embed", (spec["n_species"], spec["mul"][0]))], spec["mlp_hidden"]
    for t in range(spec["n_layers"]):
        b = _block(spec, t)
        out += [(f"{t}.sc{l}", (b["inp"][l], m)) for l, m in sorted(b["gate"].items()) if l in b["inp"]]
        out += [(f"{t}.lin1{l}", (m, m)) for l, m in sorted(b["inp"].items())]
        out += [(f"{t}.mlp0", (spec["n_basis"], h)), (f"{t}.mlp1", (h, h)), (f"{t}.mlp2", (h, b["width"]))]
        out += [(f"{t}.lin2{l}", (b["msg"][l], m)) for l, m in sorted(b["gate"].items()) if l in b["msg"]]
    return out + [("readout0", (spec["mul"][0], spec["readout_hidden"])), ("readout1", (spec["readout_hidden"], 1))]


def _mean_neighbours(case, spec):
    density = case["rho"] / (MASSES.mean() * AMU_G * 1e24)
    return 4.0 / 3.0 * math.pi * spec["r_cut"] ** 3 * density


def work(case):
    """Multiply-adds counted as two: the tensor product, the radial MLP and the
    node linears of every block, forward and adjoint (the radial MLP depends on
    the distance only, so once per pair of directed edges, and its output twice)."""
    spec = model_spec(case)
    nn = _mean_neighbours(case, spec)
    atoms = case["atoms"]
    if case["kind"] == "batch":                      # mean of a log-uniform size
        lo = min(16, atoms)
        atoms = case["structs"] * ((atoms - lo) / math.log(atoms / lo) if atoms > lo else atoms)
    h, flops = spec["mlp_hidden"], 0.0
    blocks = range(spec["n_layers"]) if case["kind"] != "conv" else [case["layer"]]
    for t in blocks:
        b = _block(spec, t)
        tp = sum(m * ((2 * a + 1) * (2 * c + 1) + 2 * c + 1) for a, _, c, m in b["paths"])
        mlp = spec["n_basis"] * h + h * h + h * b["width"]
        flops += 2.0 * nn * (3 * tp + 1.5 * mlp)
        if case["kind"] != "conv":
            lin = sum((2 * l + 1) * b["inp"][l] * (b["inp"][l] + b["gate"].get(l, 0)) for l in b["inp"])
            lin += sum((2 * l + 1) * b["msg"].get(l, 0) * m for l, m in b["gate"].items())
            flops += 4.0 * lin
    flops *= atoms
    if case["kind"] == "conv":
        b = _block(spec, case["layer"])
        xd = sum((2 * l + 1) * m for l, m in b["inp"].items())
        md = sum((2 * l + 1) * m for l, m in b["msg"].items())
        return dict(bytes=atoms * (4 + 8 * xd + 8 * md) + atoms * nn * (4 + 24) + 4 * h * b["width"], flops=flops)
    steps = case.get("steps", 1)
    params = 4 * sum(a * c for _, (a, c) in _layout(spec))
    return dict(bytes=steps * (atoms * (24 + 24 + 4) + params), flops=steps * flops)


def tolerance(case):
    # about four times the distance from the 64-bit result: FP32 up to 1.4e-6 (forces),
    # BF16 up to 2.3e-3 (forces; the messages of one convolution 4.3e-3)
    return {"rel": 1e-5} if case["prec"] == "fp32" else {"rel": 1e-2}


# ------------------------------------------------------------------ the same in 64 bits, plain torch
def _coupling(a, b, c):
    """Real-basis coupling tensor [2a+1, 2b+1, 2c+1]: Clebsch-Gordan coefficients
    (Racah's formula) carried to the real harmonics, squares summing to 2c + 1,
    the first entry positive."""
    f = math.factorial
    cg = np.zeros((2 * a + 1, 2 * b + 1, 2 * c + 1))
    for m in range(-a, a + 1):
        for n in range(-b, b + 1):
            k = m + n
            if abs(k) > c:
                continue
            pre = (2 * c + 1) * f(c + a - b) * f(c - a + b) * f(a + b - c) / f(a + b + c + 1)
            pre *= f(c + k) * f(c - k) * f(a - m) * f(a + m) * f(b - n) * f(b + n)
            s = 0.0
            for q in range(a + b - c + 1):
                den = [a + b - c - q, a - m - q, b + n - q, c - b + m + q, c - a - n + q]
                if min(den) >= 0:
                    s += (-1) ** q / (f(q) * math.prod(f(v) for v in den))
            cg[m + a, n + b, k + c] = math.sqrt(pre) * s

    def basis(l):
        u = np.zeros((2 * l + 1, 2 * l + 1), complex)
        u[l, l] = 1.0
        for m in range(1, l + 1):
            u[l + m, l + m], u[l + m, l - m] = (-1) ** m / math.sqrt(2), 1 / math.sqrt(2)
            u[l - m, l - m], u[l - m, l + m] = 1j / math.sqrt(2), -1j * (-1) ** m / math.sqrt(2)
        return u

    t = np.einsum("cz,xyz,ax,by->abc", basis(c), cg, basis(a).conj(), basis(b).conj())
    t = t.real if np.abs(t.real).max() >= np.abs(t.imag).max() else t.imag
    t = t * math.sqrt((2 * c + 1) / (t * t).sum())
    t[np.abs(t) < 1e-14] = 0.0
    return t * np.sign(t.reshape(-1)[np.nonzero(np.abs(t.reshape(-1)) > 1e-9)[0][0]])


_TENSORS = {}


def _coupling_t(a, b, c):
    if (a, b, c) not in _TENSORS:
        _TENSORS[a, b, c] = torch.as_tensor(_coupling(a, b, c), device="cuda")
    return _TENSORS[a, b, c]


def _harmonics(d, r, lmax):
    x, y, z = (d / r[:, None]).unbind(1)
    s3, s5, s15 = math.sqrt(3), math.sqrt(5), math.sqrt(15)
    out = [torch.ones_like(x)[:, None], torch.stack([s3 * y, s3 * z, s3 * x], 1)]
    if lmax >= 2:
        out.append(torch.stack([s15 * x * y, s15 * y * z, s5 / 2 * (3 * z * z - 1), s15 * x * z,
                                s15 / 2 * (x * x - y * y)], 1))
    if lmax >= 3:
        a, b, c, e = math.sqrt(70) / 4, math.sqrt(105), math.sqrt(42) / 4, math.sqrt(7) / 2
        out.append(torch.stack([a * y * (3 * x * x - y * y), b * x * y * z, c * y * (5 * z * z - 1),
                                e * z * (5 * z * z - 3), c * x * (5 * z * z - 1), b / 2 * z * (x * x - y * y),
                                a * x * (x * x - 3 * y * y)], 1))
    return out


def _graph(pos, cell, rc):
    """Directed edges (dst, src, d) of one periodic cell, d = r_src - r_dst + image, 0 < |d| < rc."""
    inv = torch.linalg.inv(cell)
    frac = pos @ inv
    frac = frac - torch.floor(frac)
    p = frac @ cell
    n = p.shape[0]
    widths = [1.0 / float(torch.linalg.norm(inv[:, i])) for i in range(3)]
    ks = [range(-math.ceil(rc / w), math.ceil(rc / w) + 1) for w in widths]
    shifts = torch.tensor([(i, j, k) for i in ks[0] for j in ks[1] for k in ks[2]], dtype=p.dtype, device=p.device) @ cell
    # receivers and senders in cubes of the cell, so that a large cell compares near atoms only
    parts = []
    nb = max(1, min(int(min(widths) // (rc * 1.05)), 24)) if n > 20000 else 1
    bins = torch.clamp((frac * nb).long(), max=nb - 1)
    key = (bins[:, 0] * nb + bins[:, 1]) * nb + bins[:, 2]
    members = [torch.nonzero(key == b)[:, 0] for b in range(nb ** 3)]
    for b in range(nb ** 3):
        v = members[b]
        if nb >= 4:                                  # 27 neighbouring cubes hold every sender
            x, y, z = b // (nb * nb), b // nb % nb, b % nb
            w = torch.cat([members[((x + i) % nb * nb + (y + j) % nb) * nb + (z + k) % nb]
                           for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)])
        else:
            w = torch.arange(n, device=p.device)
        step = max(1, (1 << 24) // max(1, w.numel()))
        for v0 in range(0, v.numel(), step):
            vv = v[v0:v0 + step]
            if nb >= 4:                              # wide cells: the nearest image is the only one
                d = p[w][None] - p[vv][:, None]
                d = d - torch.round(d @ inv) @ cell
                hit = torch.nonzero((d.square().sum(-1) < rc * rc) & (w[None] != vv[:, None]))
                parts.append((vv[hit[:, 0]], w[hit[:, 1]], d[hit[:, 0], hit[:, 1]]))
                continue
            for s in shifts:
                d = p[w][None] - p[vv][:, None] + s
                r2 = d.square().sum(-1)
                hit = torch.nonzero((r2 < rc * rc) & (r2 > 0))
                parts.append((vv[hit[:, 0]], w[hit[:, 1]], d[hit[:, 0], hit[:, 1]]))
    return tuple(torch.cat(v) for v in zip(*parts))


def _messages(spec, b, wd, t, x, d, dst, src, n):
    """{l: [n, 2l+1, channels]} of one convolution, by slices of edges that the backward pass computes again."""
    lmax = len(spec["mul"]) - 1

    def part(d, dst, src, *xs):
        x = dict(zip(sorted(b["inp"]), xs))
        r = torch.linalg.norm(d, dim=1)
        q = r / spec["r_cut"]
        p = spec["poly_p"]
        env = 1 - (p + 1) * (p + 2) / 2 * q ** p + p * (p + 2) * q ** (p + 1) - p * (p + 1) / 2 * q ** (p + 2)
        k = torch.arange(1, spec["n_basis"] + 1, dtype=d.dtype, device=d.device)
        basis = 2 / spec["r_cut"] * torch.sin(k * math.pi * q[:, None]) / r[:, None]
        basis = basis * torch.where(q < 1, env, torch.zeros_like(env))[:, None]
        h = basis
        for name in ("mlp0", "mlp1"):
            h = torch.nn.functional.silu(h @ wd[f"{t}.{name}"] / math.sqrt(h.shape[1]))
        w = h @ wd[f"{t}.mlp2"] / math.sqrt(h.shape[1])
        ys = _harmonics(d, r, lmax)
        out, col = {}, 0
        for l1, l2, l3, m in b["paths"]:
            g = torch.einsum("abc,eb->eca", _coupling_t(l1, l2, l3), ys[l2])
            v = torch.matmul(g, x[l1][src]) * w[:, None, col:col + m]
            col += m
            out.setdefault(l3, []).append(torch.zeros((n, 2 * l3 + 1, m), dtype=d.dtype, device=d.device)
                                          .index_add(0, dst, v))
        return tuple(torch.cat(out[l], 2) / spec["avg_num_neigh"] for l in sorted(out))

    xs = [x[l] for l in sorted(b["inp"])]
    total = None
    step = 1 << 18
    for e in range(0, max(1, d.shape[0]), step):
        got = torch.utils.checkpoint.checkpoint(part, d[e:e + step], dst[e:e + step], src[e:e + step], *xs,
                                                use_reentrant=False)
        total = got if total is None else tuple(u + v for u, v in zip(total, got))
    return dict(zip(sorted(b["msg"]), total))


def _weights64(spec, flat):
    flat, off, wd = torch.as_tensor(flat, device="cuda"), 0, {}
    for name, (a, b) in _layout(spec):
        wd[name] = flat[off:off + a * b].view(a, b)
        off += a * b
    return wd


def _energy(spec, wd, species, d, dst, src):
    lin = lambda v, w: v @ w / math.sqrt(w.shape[0])  # noqa: E731
    n, mul = species.shape[0], spec["mul"]
    h = {0: wd["embed"][species][:, None, :]}
    for t in range(spec["n_layers"]):
        b = _block(spec, t)
        m = _messages(spec, b, wd, t, {l: lin(h[l], wd[f"{t}.lin1{l}"]) for l in h}, d, dst, src, n)
        y = {}
        for l in b["gate"]:
            y[l] = lin(m[l], wd[f"{t}.lin2{l}"]) + (lin(h[l], wd[f"{t}.sc{l}"]) if l in h else 0)
        silu = torch.nn.functional.silu
        if b["last"]:
            h = {0: silu(y[0])}
            break
        gates, h, off = silu(y[0][..., mul[0]:]), {0: silu(y[0][..., :mul[0]])}, 0
        for l in range(1, len(mul)):
            h[l] = y[l] * gates[..., off:off + mul[l]]
            off += mul[l]
    e = lin(lin(h[0][:, 0, :], wd["readout0"]), wd["readout1"])[:, 0]
    return e * spec["scale"] + torch.tensor(spec["shift"], dtype=e.dtype, device=e.device)[species]


def _evaluate64(spec, wd, species, pos, cell):
    """(E, F, W) of one cell as torch FP64 values on the GPU."""
    dst, src, d0 = _graph(pos, cell, spec["r_cut"])
    d = d0.detach().requires_grad_(True)
    e = _energy(spec, wd, torch.as_tensor(species, dtype=torch.long, device="cuda"), d, dst, src).sum()
    (g,) = torch.autograd.grad(e, d) if d.numel() else (torch.zeros_like(d),)
    f = torch.zeros_like(pos).index_add(0, dst, g).index_add(0, src, -g)
    return e.detach(), f, -(g.T @ d0)


def exact(case, seed):
    d = _inputs(case, seed)
    spec, wd = d["spec"], None
    wd = _weights64(spec, d["weights"])
    pos = torch.as_tensor(d["pos"], device="cuda")
    if case["kind"] == "conv":
        b = _block(spec, case["layer"])
        rows = torch.as_tensor(d["row_ptr"], device="cuda").long()
        n = rows.numel() - 1
        dst = torch.repeat_interleave(torch.arange(n, device="cuda"), rows[1:] - rows[:-1])
        x64 = torch.as_tensor(d["x"], device="cuda").double().requires_grad_(True)
        vec = torch.as_tensor(d["vec"], device="cuda").double().requires_grad_(True)
        x, off = {}, 0
        for l, m in b["inp"].items():
            x[l] = x64[:, off:off + (2 * l + 1) * m].reshape(n, 2 * l + 1, m)
            off += (2 * l + 1) * m
        got = _messages(spec, b, wd, case["layer"], x, vec, dst, torch.as_tensor(d["src"], device="cuda").long(), n)
        m = torch.cat([got[l].reshape(n, -1) for l in sorted(got)], 1)
        gx, gd = torch.autograd.grad(m, [x64, vec], torch.as_tensor(d["gm"], device="cuda").double())
        return dict(m=m.detach(), gx=gx, gd=gd)
    if case["kind"] != "md":
        off = d["offsets"]
        got = [_evaluate64(spec, wd, d["species"][a:b], pos[a:b], torch.as_tensor(c, device="cuda"))
               for a, b, c in zip(off[:-1], off[1:], d["cells"])]
        return dict(energy_virial=torch.cat([torch.stack([g[0] for g in got]), torch.stack([g[2] for g in got]).view(-1)]),
                    forces=torch.cat([g[1] for g in got]))
    # velocity Verlet, and a Nose-Hoover thermostat around each step where tau > 0
    cell, species = torch.as_tensor(d["cells"][0], device="cuda"), d["species"]
    m = torch.as_tensor(MASSES[species], device="cuda")[:, None]
    vel, xi, kt = torch.as_tensor(d["vel"], device="cuda"), 0.0, KB * case["temp"]
    nf = 3 * pos.shape[0] - 3
    kinetic = lambda v: float(0.5 * (m * v * v).sum() / ACC)  # noqa: E731

    def thermostat(v, xi):
        q = nf * kt * case["tau"] ** 2
        xi += 0.25 * (2 * kinetic(v) - nf * kt) / q
        v = v * math.exp(-0.5 * xi)
        return v, xi + 0.25 * (2 * kinetic(v) - nf * kt) / q

    _, f, _ = _evaluate64(spec, wd, species, pos, cell)
    logs = []
    for _ in range(case["steps"]):
        if case["tau"] > 0:
            vel, xi = thermostat(vel, xi)
        vel = vel + 0.5 * ACC * f / m
        pos = pos + vel
        e, f, _ = _evaluate64(spec, wd, species, pos, cell)
        vel = vel + 0.5 * ACC * f / m
        if case["tau"] > 0:
            vel, xi = thermostat(vel, xi)
        logs.append((float(e), kinetic(vel)))
    return dict(energies=torch.tensor(logs, dtype=torch.float64).T.contiguous(), pos=pos, vel=vel, forces=f)
