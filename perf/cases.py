"""The work that users of this library have it do, as measurable cases.

A case names a field of elements and one pass over it through the package's
public entry points:

    step    build the radiation tree and take J of every gas element: one
            radiation step of a simulation
    build   build the tree, read back its order and take J of a short rung: one
            step of an individual-timestep run, most of it the rebuild
    J       J of a set of receivers in a tree that exists already (a rung of
            an individual-timestep run, or a second pass over all the gas)
    grad    J as a differentiable function of opacity and luminosity, forward
            and backward
    batch   one run of a batch plan: many receiver subsets of several trees

Fields (all in the unit box): a jittered lattice of n^3 gas elements with
lognormal density (P(k) ~ k^-3) and sources in dense gas, or gas clumped
around a few centres as particles of a galaxy are (deep, uneven trees).
"""

import math

import numpy as np
import torch

import paper_2310_15235_gb300 as t2

FLAGS = {"SOFT": t2.SOFT, "THICK": t2.THICK, "LINEAR": t2.LINEAR, "BUCKET": t2.BUCKET,
         "PP": t2.PP, "CSM": t2.CSM}
KAPPA = (10.0, 3.0, 0.5, 1.5)


def _case(name, kind, n, sources, bands=1, nside=2, theta=0.75, **more):
    case = {"kind": kind, "field": "lattice", "n": n, "sources": sources, "bands": bands,
            "nside": nside, "theta": theta, "sigma": 1.5, "bucket": 12, "flags": "",
            "receivers": 0, "refine": 0.0, "subsets": 0, "trees": 1}
    if name:
        case["name"] = name
    case.update(more)
    return case


def listed():
    return [
        # one source in a small uniform box: the smallest whole step, where
        # launches and synchronisations are most of the time
        _case("step_point_16", "step", 16, 1, sigma=0.0),
        # a uniform medium with some tens of sources, one band, default beams
        _case("step_stromgren_32", "step", 32, 64, sigma=0.0),
        # the benchmark: the clumpy multi-band field at full size
        _case("step_clumpy_128", "step", 128, 10_000, 3, 4, 0.5),
        # a step that rebuilds the tree at full size for a short rung of receivers
        _case("build_clumpy_128", "build", 128, 10_000, 3, 4, 0.5, receivers=1000),
        # the shortest rung of an individual-timestep run: a handful of receivers
        _case("rung_clumpy_128_100", "J", 128, 10_000, 3, 4, 0.5, receivers=100),
        # a rung in the middle
        _case("rung_clumpy_128_33333", "J", 128, 10_000, 3, 4, 0.5, receivers=33_333),
        # the paper's per-bucket beams over all the gas
        _case("bucket_clumpy_128", "J", 128, 10_000, 3, 4, 0.5, flags="BUCKET"),
        # the paper's whole scheme at its default beams: per-bucket walks, p-p
        # absorption, the complex source model, optically thick elements
        _case("paper_scheme_64", "J", 64, 1024, 2, 2, 0.75, sigma=1.0,
              flags="BUCKET|PP|CSM|THICK"),
        # unevenly clumped particles (deep tree) with absorption refinement
        _case("clumped_refined_200k", "J", 58, 2_000, 2, 2, 0.75, field="clumps",
              flags="SOFT", refine=0.1, receivers=50_001),
        # fine beams, the comparison scheme of linear averages, finite elements
        _case("fine_beams_40", "J", 40, 700, 2, 8, 0.6, sigma=1.0, flags="LINEAR|SOFT|THICK"),
        # gradients of a loss on J for every opacity and luminosity
        _case("grad_clumpy_64", "grad", 64, 1024, 2, 2, 0.75, sigma=1.0),
        # many receiver subsets of several snapshots in one run of a plan
        _case("batch_clumpy_64", "batch", 64, 1_500, 3, 4, 0.5, trees=4, subsets=64),
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    largest = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["step", "step", "build", "J", "J", "J", "grad", "batch"])
        n = _log_int(rng, 9, 120 if kind in ("step", "build", "J") else 61)
        sources = _log_int(rng, 1, max(2, min(10_000, n ** 3 // 100)))
        nside = rng.choice([1, 2, 2, 2, 4, 4, 8]) if n < 64 else rng.choice([2, 4])
        flags = []
        if kind in ("step", "J", "batch"):
            if rng.random() < 0.45:
                flags.append("BUCKET")
                if rng.random() < 0.4 and nside <= 4:
                    flags.append("PP")
                if rng.random() < 0.4 and n <= 80:
                    flags.append("CSM")
        for f in ("SOFT", "THICK", "LINEAR"):
            if rng.random() < 0.25:
                flags.append(f)
        field = "clumps" if rng.random() < 0.25 and "PP" not in flags else "lattice"
        case = _case("", kind, n, sources, rng.choice([1, 2, 3, 3, 4]), nside,
                     round(rng.uniform(0.45, 0.95), 3), field=field,
                     sigma=round(rng.uniform(0.0, 1.5), 2), bucket=rng.choice([7, 12, 12, 16]),
                     flags="|".join(flags))
        if kind == "build" or (kind == "J" and rng.random() < 0.7):
            case["receivers"] = _log_int(rng, 1, min(n ** 3, 2000 if kind == "build" else n ** 3))
        if kind == "J" and rng.random() < 0.2:
            case["refine"] = round(rng.uniform(0.05, 0.5), 3)
        if kind == "batch":
            case["trees"], case["subsets"] = rng.randint(1, 5), rng.randint(2, 40)
        if _cost(case) <= largest:
            return case


# ---------------------------------------------------------------------------
# Inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _lattice_field(case, gen, dev):
    n, sigma = case["n"], case["sigma"]
    axis = torch.arange(n, dtype=torch.float64, device=dev)
    grid = torch.stack(torch.meshgrid(axis, axis, axis, indexing="ij"), -1).reshape(-1, 3)
    jitter = torch.rand((n ** 3, 3), generator=gen, dtype=torch.float64, device=dev) - 0.5
    gas = (grid + 0.5 + 0.5 * jitter) / n
    rho = torch.ones(n ** 3, dtype=torch.float64, device=dev)
    if sigma > 0:
        white = torch.randn((n, n, n), generator=gen, dtype=torch.float64, device=dev)
        k = torch.fft.fftfreq(n, device=dev, dtype=torch.float64) * n
        k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2
        amp = torch.where(k2 > 0, k2.clamp_min(1e-300) ** -0.75, torch.zeros_like(k2))
        g = torch.fft.ifftn(torch.fft.fftn(white) * amp).real
        g = ((g - g.mean()) / g.std()).reshape(-1)
        rho = torch.exp(sigma * g - 0.5 * sigma * sigma)
    if case["sources"] == 1:  # off the root's split planes
        src = torch.tensor([[0.53, 0.51, 0.52]], dtype=torch.float64, device=dev)
    else:
        cum = torch.cumsum(rho, 0)
        u = torch.rand(case["sources"], generator=gen, dtype=torch.float64, device=dev)
        cell = torch.searchsorted(cum, u * cum[-1]).clamp_max(n ** 3 - 1)
        src = (grid[cell] + torch.rand((case["sources"], 3), generator=gen, dtype=torch.float64,
                                       device=dev)) / n
    return gas, rho / n ** 3, torch.full((n ** 3,), 1.0 / n, dtype=torch.float64, device=dev), src


def _clump_field(case, gen, dev):
    n = case["n"] ** 3

    def rand(*shape):
        return torch.rand(shape, generator=gen, dtype=torch.float64, device=dev)

    def normal(*shape):
        return torch.randn(shape, generator=gen, dtype=torch.float64, device=dev)

    centres, width = 0.2 + 0.6 * rand(6, 3), 0.01 * 12.0 ** rand(6)

    def place(m):
        which = (rand(m) * 6).long().clamp_max(5)
        return (centres[which] + width[which, None] * normal(m, 3)).clamp(0.0, 1.0), which

    gas, which = place(n)
    mass = (0.5 + rand(n)) / n
    # element sizes from the clumps' mean densities
    h = (width[which] ** 3 * 15.75 * 6.0 / n) ** (1.0 / 3.0)
    return gas, mass, h, place(case["sources"])[0]


def _field(case, seed):
    """Positions, masses, opacities, luminosities and sizes of one field."""
    dev = _device()
    gen = torch.Generator(device=dev)
    gen.manual_seed(1_000_003 * seed + 17)
    make = _clump_field if case["field"] == "clumps" else _lattice_field
    gas, mass, h, src = make(case, gen, dev)
    ng, ns, nb = gas.shape[0], src.shape[0], case["bands"]
    kappa = torch.zeros((ng + ns, nb), dtype=torch.float32, device=dev)
    kappa[:ng] = torch.tensor(KAPPA[:nb], dtype=torch.float32, device=dev)
    lum = torch.zeros((ng + ns, nb), dtype=torch.float32, device=dev)
    u = torch.rand(ns, generator=gen, dtype=torch.float64, device=dev)
    lum[ng:] = (1.0 / (1000.0 - 999.0 * u)).float()[:, None]
    return {"pos": torch.cat([gas, src]).contiguous(),
            "mass": torch.cat([mass, torch.zeros(ns, dtype=mass.dtype, device=dev)]).float(),
            "kappa": kappa, "lum": lum,
            "h": torch.cat([h, h.mean().expand(ns)]).float(), "gas": ng, "gen": gen}


def _flags(case):
    return sum(FLAGS[f] for f in case["flags"].split("|") if f)


def _build(case, f):
    return t2.build(f["pos"], f["mass"], f["kappa"], f["lum"], f["h"], box_lo=(0.0, 0.0, 0.0),
                    box_size=1.0, bucket=case["bucket"])


def _active(case, f):
    if case["receivers"] <= 0 or case["receivers"] >= f["gas"]:
        return torch.arange(f["gas"], device=f["pos"].device)
    return torch.randperm(f["gas"], generator=f["gen"],
                          device=f["pos"].device)[:case["receivers"]].sort().values


def _subsets(case, fields):
    """Receiver subsets of 10^U(1.5, 5) elements: row offsets, trees, receivers."""
    sizes = 10.0 ** np.random.RandomState(case["subsets"]).uniform(1.5, 5.0, case["subsets"])
    sizes = np.minimum(sizes.astype(np.int64), fields[0]["gas"])
    tree_of = np.arange(case["subsets"]) % len(fields)
    rows = []
    for size, t in zip(sizes, tree_of):
        f = fields[t]
        rows.append(torch.randperm(f["gas"], generator=f["gen"],
                                   device=f["pos"].device)[:int(size)].sort().values)
    return np.concatenate([[0], np.cumsum(sizes)]), tree_of, torch.cat(rows)


def _seeds(case, seed):
    return [seed + 7919 * t for t in range(case["trees"])]


def prepare(case, seed):
    fields = [_field(case, s) for s in _seeds(case, seed)]
    f = fields[0]
    state = {"case": case, "field": f}
    if case["kind"] != "batch":
        state["active"] = _active(case, f)
    if case["kind"] == "grad":
        state["kappa"] = f["kappa"].clone().requires_grad_()
        state["lum"] = f["lum"].clone().requires_grad_()
        state["weight"] = torch.rand((state["active"].numel(), case["bands"]),
                                     generator=f["gen"], device=f["pos"].device)
    if case["kind"] == "J":
        state["tree"] = _build(case, f)
        state["tree"].prepare(case["nside"])
        if case["refine"] > 0:
            state["tree"].set_tau_refine(case["refine"])
    if case["kind"] == "batch":
        offsets, tree_of, state["active"] = _subsets(case, fields)
        trees = [_build(case, g) for g in fields]
        state["plan"] = t2.Batch(trees, offsets, tree_of, nside=case["nside"],
                                 theta=case["theta"], flags=_flags(case))
    return state


def run(state):
    case, f = state["case"], state["field"]
    if case["kind"] == "batch":
        return state["plan"].run(state["active"])
    if case["kind"] == "grad":
        J = t2.J_fn(f["pos"], f["mass"], state["kappa"], state["lum"], state["active"],
                    nside=case["nside"], theta=case["theta"], h=f["h"], flags=_flags(case),
                    box_lo=(0.0, 0.0, 0.0), box_size=1.0, bucket=case["bucket"])
        gk, gl = torch.autograd.grad((J * state["weight"]).sum(), (state["kappa"], state["lum"]))
        return {"J": J.detach(), "kappa": gk, "lum": gl}
    tree = state["tree"] if case["kind"] == "J" else _build(case, f)
    J = tree.J(state["active"], nside=case["nside"], theta=case["theta"], flags=_flags(case))
    if case["kind"] == "build":
        return {"J": J, "keys": tree.export("keys"), "perm": tree.export("perm")}
    return J


# ---------------------------------------------------------------------------
# What a pass cannot do without


def work(case):
    """Bytes: the arrays that go in and come out, once.  Operations: per walk,
    the cells of the cut that B/d > theta gives (they grow as theta^-3 and
    with the tree's depth), one crossing per beam and cell met, one term of J
    per source, receiver and band; in the gradient twice that again."""
    gas = case["n"] ** 3
    elements = gas + case["sources"]
    nb, npix = case["bands"], 12 * case["nside"] ** 2
    arrays = elements * (24 + 8 + 8 * nb)
    depth = max(1.0, math.log2(max(2.0, elements / case["bucket"])))
    leaves = 2.0 * elements / case["bucket"]
    cells = min(leaves, 7.3 / case["theta"] ** 3 * depth)
    found = min(cells, case["sources"])
    per_walk = 2 * cells * 12 + npix * 15 * (15 + 2 * nb) + found * 30
    per_receiver = found * (12 + 4 * nb)
    if case["kind"] == "batch":
        rows = case["subsets"] * min(gas, 12_300)
        walks = min(rows, case["trees"] * gas)
    else:
        rows = walks = min(gas, case["receivers"]) or gas
    receivers = walks
    if "BUCKET" in case["flags"]:
        walks = min(walks, leaves)
    if "PP" in case["flags"]:
        sphere = min(gas, 4.2 * (npix / 12.566) ** 1.5)
        per_receiver += found * 0.15 * sphere * 20
    flops = walks * per_walk + receivers * per_receiver
    if case["kind"] in ("step", "build"):  # the transmission average of every cell and pair
        flops += leaves * npix / 2 * nb * 15
    if case["kind"] == "grad":
        flops *= 3
    io = 12 * rows if case["kind"] != "grad" else rows * (8 + 8 * nb) + elements * 8 * nb
    io += 12 * elements if case["kind"] == "build" else 0
    inputs = arrays if case["kind"] in ("step", "build", "grad") else min(arrays, walks * cells * 48)
    return {"bytes": inputs + io + 4 * nb * rows, "flops": flops}


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


# ---------------------------------------------------------------------------
# The method in 64 bits with plain tensors: the radiation tree, the cut seen
# from every origin, and every source's optical depth as the sum over all
# cells of the cut that its beam crosses before it.

_SPLIT_BITS = 21


def _spread(v):
    for shift, mask in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F),
                        (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
        v = (v | (v << shift)) & mask
    return v


def _plain_tree(f, bucket):
    """Cyclic x, y, z bisection of the unit cube, nodes breadth first."""
    pos = f["pos"]
    dev, N = pos.device, pos.shape[0]
    cell = torch.floor(pos * 2.0 ** _SPLIT_BITS).clamp(0, 2 ** _SPLIT_BITS - 1).long()
    keys = (_spread(cell[:, 0]) << 2) | (_spread(cell[:, 1]) << 1) | _spread(cell[:, 2])
    keys, perm = torch.sort(keys, stable=True)
    one = torch.zeros(1, dtype=torch.long, device=dev)
    prefix, first, count = one, one, one + N
    out = {"prefix": [], "first": [], "count": [], "child": [], "parent": [], "depth": []}
    begin, parent = [0], one - 1
    for depth in range(64):
        split = (count > bucket) & (depth < 63)
        bit = 1 << max(62 - depth, 0)
        mid = torch.searchsorted(keys, prefix | bit)
        mid = torch.minimum(torch.maximum(mid, first), first + count)
        base = begin[-1] + prefix.numel()
        child = torch.where(split, base + 2 * (torch.cumsum(split.long(), 0) - 1), -one - 1)
        for k, v in (("prefix", prefix), ("first", first), ("count", count), ("child", child),
                     ("parent", parent), ("depth", torch.full_like(prefix, depth))):
            out[k].append(v)
        own = torch.arange(prefix.numel(), device=dev)[split] + begin[-1]
        begin.append(base)
        if own.numel() == 0:
            break
        p, s, c, m = prefix[split], first[split], count[split], mid[split]
        prefix = torch.stack([p, p | bit], 1).reshape(-1)
        first = torch.stack([s, m], 1).reshape(-1)
        count = torch.stack([m - s, s + c - m], 1).reshape(-1)
        parent = own.repeat_interleave(2)
    t = {k: torch.cat(v) for k, v in out.items()}
    t.update(keys=keys, perm=perm, begin=begin)
    axes = []
    for a in range(3):
        k = torch.zeros_like(t["prefix"])
        for l in range(_SPLIT_BITS):
            k = (k << 1) | ((t["prefix"] >> (3 * (_SPLIT_BITS - 1 - l) + 2 - a)) & 1)
        axes.append(k.double() / 2.0 ** _SPLIT_BITS)
    t["lo"] = torch.stack(axes, 1)
    t["ext"] = torch.stack([2.0 ** -((t["depth"] + 2 - a) // 3).double() for a in range(3)], 1)
    t["leaf"] = t["child"] < 0
    leaf_ids = torch.nonzero(t["leaf"]).reshape(-1)
    order = torch.argsort(t["first"][leaf_ids], stable=True)
    leaf_ids = leaf_ids[order]
    leaf_ids = leaf_ids[t["count"][leaf_ids] > 0]
    t["leaf_of"] = torch.repeat_interleave(leaf_ids, t["count"][leaf_ids])
    return t


def _up(t, leaf_values, combine):
    """Values of every node from its leaves' values."""
    levels = {}
    begin = t["begin"]
    for d in range(len(begin) - 2, -1, -1):
        a, b = begin[d], begin[d + 1]
        v = leaf_values[a:b]
        child = t["child"][a:b]
        inner = child >= 0
        if bool(inner.any()):
            c = child[inner] - begin[d + 1]
            below = levels[d + 1]
            v = v.index_put((torch.nonzero(inner).reshape(-1),),
                            combine(below[c], below[c + 1]))
        levels[d] = v
    return torch.cat([levels[d] for d in range(len(begin) - 1)])


def _aggregate(t, f, kappa, lum):
    n = t["prefix"].numel()
    perm, leaf_of = t["perm"], t["leaf_of"]
    L, km = lum[perm], kappa[perm] * f["mass"].double()[perm, None]
    pos = f["pos"][perm]
    Lt = L.sum(1)
    leaf = torch.cat([L, Lt[:, None] * pos, Lt[:, None]], 1)
    zero = torch.zeros((n, leaf.shape[1]), dtype=torch.float64, device=pos.device)
    s = _up(t, zero.index_add(0, leaf_of, leaf), torch.add)
    nb = L.shape[1]
    t["L"], total = s[:, :nb], s[:, -1:]
    middle = t["lo"] + 0.5 * t["ext"]
    t["c"] = torch.where(total > 0, s[:, nb:nb + 3] / total.clamp_min(1e-300), middle)
    corner = torch.maximum(t["c"] - t["lo"], t["lo"] + t["ext"] - t["c"])
    t["B"] = corner.detach().square().sum(1).sqrt()
    volume = t["ext"].prod(1, keepdim=True)
    t["alpha"] = torch.zeros((n, nb), dtype=torch.float64,
                             device=pos.device).index_add(0, leaf_of, km) / volume
    t["Le"], t["pe"] = L, pos
    return t


def _variation(t):
    a = t["alpha"].detach()
    hi, lo = _up(t, a, torch.maximum), _up(t, a, torch.minimum)
    return (hi - lo).amax(1) * t["ext"][:, 2]


def _ring_vectors(nside, dev):
    """HEALPix pixel centres, RING order (Gorski et al. 2005)."""
    z, phi = [], []
    for ring in range(1, 4 * nside):
        north = min(ring, 4 * nside - ring)
        if north < nside:
            size, shift = 4 * north, 0.5
            height = math.copysign(1.0 - north ** 2 / (3.0 * nside ** 2), 2 * nside - ring)
        else:
            size, shift = 4 * nside, 0.5 if (ring - nside) % 2 == 0 else 0.0
            height = 4.0 / 3.0 - 2.0 * ring / (3.0 * nside)
        j = np.arange(size)
        z.append(np.full(size, height))
        phi.append(2.0 * np.pi / size * (j + shift))
    z, phi = np.concatenate(z), np.concatenate(phi)
    s = np.sqrt((1.0 - z) * (1.0 + z))
    v = np.stack([s * np.cos(phi), s * np.sin(phi), z], 1)
    v[np.abs(v) < 1e-15] = 0.0
    return torch.from_numpy(v).to(dev)


def _ring_pixel(nside, v):
    """HEALPix RING pixel of direction vectors (Gorski et al. 2005)."""
    n = nside
    z = v[:, 2] / v.square().sum(1).sqrt()
    t = torch.remainder(torch.atan2(v[:, 1], v[:, 0]), 2.0 * math.pi) / (0.5 * math.pi)
    up, down = n * (0.5 + t) - 0.75 * n * z, n * (0.5 + t) + 0.75 * n * z
    jp, jm = torch.floor(up).long(), torch.floor(down).long()
    ring = n + 1 + jp - jm
    ip = torch.div(jp + jm - n + (1 - ring % 2) + 1, 2, rounding_mode="floor") % (4 * n)
    belt = 2 * n * (n - 1) + (ring - 1) * 4 * n + ip
    frac = t - torch.floor(t)
    width = n * torch.sqrt(3.0 * (1.0 - z.abs()).clamp_min(0.0))
    ring = torch.floor(frac * width).long() + torch.floor((1.0 - frac) * width).long() + 1
    ip = torch.floor(t * ring).long() % (4 * ring)
    cap = torch.where(z > 0, 2 * ring * (ring - 1) + ip, 12 * n * n - 2 * ring * (ring + 1) + ip)
    return torch.where(z.abs() <= 2.0 / 3.0, belt, cap)


def _plain_table(t, nside, linear, dirs):
    """Absorption of every node for every antipodal pair of beams [n, P, nb]."""
    P = dirs.shape[0] // 2
    n = dirs[:P]
    begin, levels = t["begin"], {}
    for d in range(len(begin) - 2, -1, -1):
        a, b = begin[d], begin[d + 1]
        own = t["alpha"][a:b, None, :].expand(b - a, P, t["alpha"].shape[1])
        inner = torch.nonzero(t["child"][a:b] >= 0).reshape(-1)
        if inner.numel():
            c = t["child"][a:b][inner] - begin[d + 1]
            a1, a2 = levels[d + 1][c], levels[d + 1][c + 1]
            if linear:
                value = 0.5 * (a1 + a2)
            else:
                E = t["ext"][a]
                x = d % 3
                y, z = (x + 1) % 3, (x + 2) % 3
                ny = (n[:, y] / n[:, x]).abs().nan_to_num(posinf=1e300)
                nz = (n[:, z] / n[:, x]).abs().nan_to_num(posinf=1e300)
                u = torch.minimum(0.5 * E[x], torch.minimum(E[y] / ny.clamp_min(1e-300),
                                                            E[z] / nz.clamp_min(1e-300)))
                both = 2.0 * (E[y] * E[z] * u - 0.5 * (E[y] * nz + E[z] * ny) * u * u
                              + ny * nz * u ** 3 / 3.0) / E.prod()
                both = torch.where(n[:, x] == 0, torch.zeros_like(both), both)[:, None]
                one = 0.5 - 0.5 * both
                chord = (E / n.abs().clamp_min(1e-300)).amin(1)[:, None]
                x1, x2 = chord * a1, chord * a2
                m = torch.minimum(x1, x2)
                rest = (one * (torch.expm1(m - x1) + torch.expm1(m - x2))
                        + both * torch.expm1(m - 0.5 * (x1 + x2)))
                value = (m - torch.log1p(rest)) / chord
            own = own.index_put((inner,), value)
        levels[d] = own
    return torch.cat([levels[d] for d in range(len(begin) - 1)])


def _cut(t, origin, theta, forced):
    """(origin, node) pairs of the cut and which of them are opened leaves."""
    dev = origin.device
    i = torch.arange(origin.shape[0], device=dev)
    q = torch.zeros_like(i)
    gi, gq, go = [], [], []
    while i.numel():
        x, lo = origin[i], t["lo"][q]
        gap = torch.maximum(lo - x, x - lo - t["ext"][q]).clamp_min(0.0)
        d = gap.square().sum(1).sqrt()
        opens = (d == 0) | (t["B"][q] > theta * d)
        if forced is not None:
            opens |= forced[q]
        down = opens & ~t["leaf"][q]
        keep = ~down
        gi.append(i[keep])
        gq.append(q[keep])
        go.append(opens[keep])
        c = t["child"][q[down]]
        i, q = i[down].repeat_interleave(2), torch.stack([c, c + 1], 1).reshape(-1)
    return torch.cat(gi), torch.cat(gq), torch.cat(go)


def _join(a_key, b_key, n):
    """Index pairs (a, b) with equal keys in [0, n)."""
    a_order, b_order = torch.argsort(a_key, stable=True), torch.argsort(b_key, stable=True)
    nb = torch.bincount(b_key, minlength=n)
    b_start = torch.cumsum(nb, 0) - nb
    reps = nb[a_key[a_order]]
    total = int(reps.sum())
    a = torch.repeat_interleave(a_order, reps, output_size=total)
    start = torch.cumsum(reps, 0) - reps
    within = torch.arange(total, device=a_key.device) - torch.repeat_interleave(
        start, reps, output_size=total)
    return a, b_order[b_start[a_key[a]] + within]


def _tau(t, table, dirs, pair_of, origin, ci, cq, si, sv, beam):
    """Optical depth along each source's beam to its projected distance."""
    n = dirs[beam]
    s = (sv * n).sum(1)
    a, b = _join(si, ci, origin.shape[0])
    x, q, na = origin[ci[b]], cq[b], n[a]
    lo = t["lo"][q] - x
    hi = lo + t["ext"][q]
    flat = na == 0
    safe = torch.where(flat, torch.ones_like(na), na)
    ta, tb = lo / safe, hi / safe
    inside = (lo <= 0) & (hi > 0)
    big = torch.full_like(ta, 1e300)
    near = torch.where(flat, torch.where(inside, -big, big), torch.minimum(ta, tb))
    far = torch.where(flat, big, torch.maximum(ta, tb))
    t0, t1 = near.amax(1).clamp_min(0.0), far.amin(1)
    hit = torch.nonzero((t0 < t1) & (t0 < s.detach()[a])).reshape(-1)
    a, q, t0, t1 = a[hit], q[hit], t0[hit], t1[hit]
    length = torch.minimum(t1, s[a]) - t0
    alpha = table[q, pair_of[beam[a]]]
    tau = torch.zeros((si.numel(), alpha.shape[1]), dtype=torch.float64, device=origin.device)
    return s, tau.index_add(0, a, alpha * length[:, None])


def _kernel(r, h, soft):
    if not soft:
        return 1.0 / (4.0 * math.pi * r * r)
    x = r / (0.48860251190292 * h)
    near = x.clamp_max(30.0)
    g = 0.5 * (1.0 + (near * near - 1.0) / (4.0 * near) * torch.log(
        ((near - 1.0) / (near + 1.0)).square().clamp_min(1e-300)))
    y = 1.0 / x.clamp_min(1.0).square()
    series = sum(y ** m / (4 * m * m - 1) for m in range(1, 12))
    return torch.where(x > 20.0, series, g) / (h * h)


def _plain_J(t, f, case, table, dirs, active):
    """J of the elements `active` (caller order) [A, nb]."""
    flags = case["flags"].split("|")
    dev, theta = f["pos"].device, float(np.float32(case["theta"]))
    pair_of = _ring_pixel(case["nside"], -dirs)
    half = dirs.shape[0] // 2
    index = torch.arange(dirs.shape[0], device=dev)
    pair_of = torch.where(index < half, index, pair_of)
    forced = _variation(t) > case["refine"] if case["refine"] > 0 else None
    inverse = torch.empty_like(t["perm"])
    inverse[t["perm"]] = torch.arange(t["perm"].numel(), device=dev)
    where = inverse[active]
    bucket = "BUCKET" in flags
    if bucket:
        leaves, own = torch.unique(t["leaf_of"][where], return_inverse=True)
        origins = t["lo"][leaves] + 0.5 * t["ext"][leaves]
    else:
        origins, own = t["pe"][where], torch.arange(where.numel(), device=dev)
    chunk, at, rows = 2, 0, []
    while at < origins.shape[0]:
        origin = origins[at:at + chunk]
        ci, cq, opened = _cut(t, origin, theta, forced)
        # sources: luminous cells of the cut, luminous elements of its opened leaves
        cell = (~opened) & (t["L"][cq].detach().sum(1) > 0)
        n_el = torch.where(opened, t["count"][cq], torch.zeros_like(cq))
        total = int(n_el.sum())
        ei = torch.repeat_interleave(ci, n_el, output_size=total)
        start = torch.cumsum(n_el, 0) - n_el
        ej = (torch.repeat_interleave(t["first"][cq], n_el, output_size=total)
              + torch.arange(total, device=dev)
              - torch.repeat_interleave(start, n_el, output_size=total))
        keep = t["Le"][ej].detach().sum(1) > 0
        if not bucket:
            keep &= ej != where[at + ei]
        ei, ej = ei[keep], ej[keep]
        si = torch.cat([ci[cell], ei])
        sp = torch.cat([t["c"][cq[cell]], t["pe"][ej]])
        sl = torch.cat([t["L"][cq[cell]], t["Le"][ej]])
        sv = sp - origin[si]
        good = sv.detach().square().sum(1) > 0
        si, sp, sl, sv = si[good], sp[good], sl[good], sv[good]
        beam = _ring_pixel(case["nside"], sv.detach())
        absorbs = t["absorbs"][cq]
        s, tau = _tau(t, table, dirs, pair_of, origin, ci[absorbs], cq[absorbs], si, sv, beam)
        mine = torch.nonzero((own >= at) & (own < at + origin.shape[0])).reshape(-1)
        a, b = _join(own[mine] - at, si, origin.shape[0])
        who = where[mine][a]
        v = sp[b] - t["pe"][who]
        r2 = v.square().sum(1)
        ok = r2.detach() > 0
        b, a, who, r = b[ok], a[ok], who[ok], r2[ok].sqrt()
        w = _kernel(r, f["h"].double()[t["perm"]][who], "SOFT" in flags)
        term = sl[b] * (w[:, None] * torch.exp(-tau[b] * (r / s[b])[:, None]))
        part = torch.zeros((mine.numel(), sl.shape[1]), dtype=torch.float64, device=dev)
        rows.append((mine, part.index_add(0, a, term)))
        at += chunk
        work_done = max(1, ci.numel() * si.numel() // max(1, origin.shape[0]))
        chunk = int(max(1, min(4096, 1.5e7 * origin.shape[0] // work_done,
                               4e7 / max(1, a.numel()) * origin.shape[0])))
        yield rows.pop()


def _thick(f, kappa, active, flags):
    if "THICK" not in flags.split("|"):
        return 1.0
    tau = (kappa * f["mass"].double()[:, None])[active] / f["h"].double()[active, None] ** 2
    small = tau < 1e-12
    safe = torch.where(small, torch.ones_like(tau), tau)
    return torch.where(small, torch.ones_like(tau), -torch.expm1(-safe) / safe)


def _plain(case, f, active, weight=None):
    """J and, with weights of the rows, the gradients of sum(weight J)."""
    grad = weight is not None
    kappa, lum = f["kappa"].double(), f["lum"].double()
    dirs = _ring_vectors(case["nside"], f["pos"].device)
    with torch.set_grad_enabled(grad):
        kappa.requires_grad_(grad)
        lum.requires_grad_(grad)
        t = _aggregate(_plain_tree(f, case["bucket"]), f, kappa, lum)
        table = _plain_table(t, case["nside"], "LINEAR" in case["flags"], dirs)
        t["absorbs"] = table.detach()[:, 0].sum(1) > 0
        factor = _thick(f, kappa, active, case["flags"])
        roots = [table, t["L"], t["c"], t["Le"]]
        cut = [r.detach().requires_grad_(grad) for r in roots]
        table, t["L"], t["c"], t["Le"] = cut
        J = torch.zeros((active.numel(), case["bands"]), dtype=torch.float64,
                        device=f["pos"].device)
        for mine, part in _plain_J(t, f, case, table, dirs, active):
            J[mine] = part.detach()
            if grad:
                f_rows = factor if isinstance(factor, float) else factor.detach()[mine]
                (part * f_rows * weight[mine].double()).sum().backward()
        if not grad:
            return J * factor
        back = [(r, c.grad) for r, c in zip(roots, cut) if c.grad is not None and r.requires_grad]
        if not isinstance(factor, float):
            back.append((factor, J * weight.double()))
        torch.autograd.backward([r for r, _ in back], [g for _, g in back])
        J = J * (factor if isinstance(factor, float) else factor.detach())
    return {"J": J, "kappa": kappa.grad, "lum": lum.grad}


def exact(case, seed):
    flags = case["flags"].split("|")
    if "PP" in flags or "CSM" in flags:
        return None  # the near field particle by particle takes far longer than 20 seconds
    dev = _device()
    if work(case)["flops"] > 1.6e10 or (case["refine"] > 0 and case["receivers"] > 2000):
        return None  # more origins, or more cells each, than 64 bits can do in 20 seconds
    fields = [_field(case, s) for s in _seeds(case, seed)]
    f = fields[0]
    if case["kind"] == "batch":
        offsets, tree_of, active = _subsets(case, fields)
        rows = torch.repeat_interleave(torch.as_tensor(tree_of, device=dev),
                                       torch.as_tensor(np.diff(offsets), device=dev))
        out = torch.zeros((active.numel(), case["bands"]), dtype=torch.float64, device=dev)
        for k, g in enumerate(fields):
            if bool((rows == k).any()):
                out[rows == k] = _plain(case, g, active[rows == k])
        return out
    active = _active(case, f)
    if case["kind"] == "grad":
        weight = torch.rand((active.numel(), case["bands"]), generator=f["gen"], device=dev)
        return _plain(case, f, active, weight)
    J = _plain(case, f, active)
    return {"J": J, "keys": None, "perm": None} if case["kind"] == "build" else J
