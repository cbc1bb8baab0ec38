"""The work that programs have this library do, as measurable cases.

Structures are the two kinds that the tests and the benchmark use, generated here on the GPU so that inputs of any
size are quick to make: water clusters (0.0334 molecules per cubic Angstrom, O-O at least 2.5 Angstrom, rigid
molecules in random orientations, no spatial order) and periodic boxes of C, H, N, O in the ratio 3:5:1:1 (0.1 atoms
per cubic Angstrom, pairs at least 0.9 Angstrom apart).  A program keeps one `Soap` object per basis for all its
structures, so `prepare` takes it from a small cache; the structure itself, and the output buffers where the call
takes them, are made anew.
"""
from __future__ import annotations

import functools
import math

import torch

import paper_2609_05709_b200 as soap

WATER_DENSITY = 0.0334          # molecules per A^3
WATER_SPACING = WATER_DENSITY ** (-1.0 / 3.0)
OO_MIN, R_OH, HOH_DEG = 2.5, 0.9572, 104.52
BOX_DENSITY, BOX_MIN_DIST = 0.1, 0.9
WATER_SPECIES, BOX_SPECIES = (1, 8), (1, 6, 7, 8)

# A case: call (entry point), structure, size (molecules of a cluster, atoms of a box, structures of a batch), basis
# (rbf, n_max, l_max, r_cut, sigma), centers (0: every atom), crossover, weighted.
DEFAULTS = {"structure": "water", "rbf": "gto", "sigma": 0.5, "centers": 0, "crossover": True, "weighted": False}


def _case(name, call, size, n_max, l_max, r_cut, **more):
    case = dict(DEFAULTS, call=call, size=size, n_max=n_max, l_max=l_max, r_cut=r_cut, **more)
    return dict(case, name=name) if name else case


def listed():
    return [
        # one small molecule cluster after another, sized and allocated by the library: latency and launches only
        _case("tiny_cluster", "derivatives", 8, 4, 3, 5.0),
        # descriptor of one frame of a small periodic simulation cell
        _case("small_box_descriptor", "descriptor", 431, 6, 4, 5.0, structure="box"),
        # the benchmark's step: descriptor and Jacobian of a 3000-atom cluster into buffers that are kept
        _case("cluster_step", "derivatives_into", 1000, 8, 6, 6.0),
        # the published parameters: wide cutoff, small basis
        _case("wide_cutoff", "derivatives", 1000, 7, 3, 10.0),
        # the far end of the hyperparameter map
        _case("large_basis", "derivatives", 400, 12, 10, 6.0),
        # a structure too large for one Jacobian, in batches of centres; a basis between the usual sizes
        _case("centre_batch", "derivatives", 10007, 5, 5, 6.0, centers=1021),
        # four species under periodic boundary conditions, polynomial basis
        _case("box_step", "derivatives_into", 2000, 8, 8, 5.0, structure="box", rbf="polynomial", sigma=0.4),
        # the same kind of box with a radial weighting, rows without the structural zeros
        _case("box_compact_weighted", "derivatives_compact", 1111, 6, 6, 5.0, structure="box", weighted=True),
        # a data set of small molecules in one call
        _case("molecule_batch", "derivatives_batch", 1500, 4, 3, 5.0),
        # descriptors of a large cluster, and of a million atoms
        _case("cluster_descriptor", "descriptor", 9999, 8, 6, 5.0),
        _case("million_atoms", "descriptor", 333334, 8, 6, 5.0),
        # a global descriptor with its derivative by every atom
        _case("averaged", "derivatives_outer", 1000, 8, 6, 6.0),
    ]


def _log_int(rng, low, high):
    return min(high, max(low, round(math.exp(rng.uniform(math.log(low), math.log(high))))))


MAX_JACOBIAN_BYTES = 6.0e9       # the largest listed Jacobian
MAX_DESCRIPTOR_FLOPS = 8.0e10    # about the largest listed descriptor call


def draw(rng):
    while True:
        kind = rng.choice(["cluster", "cluster", "cluster", "box", "box", "descriptor", "descriptor", "descriptor", "batch", "average"])
        n_max, l_max = rng.randint(2, 12), rng.randint(2, 10)
        if kind == "cluster":
            r_cut = 10.0 if rng.random() < 0.3 else round(rng.uniform(4.0, 7.0), 2)
            case = _case("", rng.choice(["derivatives", "derivatives_into"]), _log_int(rng, 5, 2000), n_max, l_max, r_cut)
            case["crossover"] = rng.random() < 0.85
            if case["size"] > 300 and rng.random() < 0.3:
                case["centers"] = rng.randint(64, 2 * case["size"])
        elif kind == "box":
            case = _case("", rng.choice(["derivatives", "derivatives_into", "derivatives_compact"]), _log_int(rng, 50, 2500),
                         rng.randint(2, 8), rng.randint(2, 8), round(rng.uniform(4.0, 5.5), 2), structure="box",
                         rbf=rng.choice(["gto", "polynomial"]), sigma=rng.choice([0.4, 0.5]), weighted=rng.random() < 0.25)
        elif kind == "descriptor":
            box = rng.random() < 0.4
            case = _case("", "descriptor", _log_int(rng, 50 if box else 5, 400000 if box else 333334),
                         rng.randint(2, 8) if box else n_max, rng.randint(2, 8), round(rng.uniform(4.0, 6.0), 2),
                         structure="box" if box else "water")
        elif kind == "batch":
            case = _case("", "derivatives_batch", _log_int(rng, 16, 3000), rng.randint(2, 8), rng.randint(2, 6), round(rng.uniform(4.0, 6.0), 2))
        else:
            case = _case("", rng.choice(["derivatives_outer", "derivatives_inner"]), _log_int(rng, 20, 1200), rng.randint(2, 9),
                         rng.randint(2, 7), round(rng.uniform(4.0, 6.0), 2))
        w = work(case)
        if w["bytes"] <= MAX_JACOBIAN_BYTES and (case["call"] != "descriptor" or w["flops"] <= MAX_DESCRIPTOR_FLOPS):
            return case


# ---------------------------------------------------------------------------------------------- structures
def _rotations(n, gen):
    q = torch.randn((n, 4), generator=gen, device="cuda", dtype=torch.float64)
    a, b, c, d = (q / q.norm(dim=1, keepdim=True)).T
    rows = [a * a + b * b - c * c - d * d, 2 * (b * c - a * d), 2 * (b * d + a * c),
            2 * (b * c + a * d), a * a - b * b + c * c - d * d, 2 * (c * d - a * b),
            2 * (b * d - a * c), 2 * (c * d + a * b), a * a - b * b - c * c + d * d]
    return torch.stack(rows, 1).reshape(n, 3, 3)


def _sphere_sites(n):
    """The n sites of a cubic lattice of water's density that lie nearest its centre."""
    half = int(math.ceil((3.0 * n / (4.0 * math.pi)) ** (1.0 / 3.0))) + 2
    ax = torch.arange(-half, half + 1, device="cuda", dtype=torch.float64)
    sites = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3) + torch.tensor([0.13, 0.29, 0.41], device="cuda", dtype=torch.float64)
    return WATER_SPACING * sites[torch.argsort(sites.square().sum(1))[:n]]


def _molecules(oxygen, gen):
    n = oxygen.shape[0]
    jitter = (WATER_SPACING - OO_MIN) / 2
    oxygen = oxygen + jitter * (2 * torch.rand((n, 3), generator=gen, device="cuda", dtype=torch.float64) - 1)
    half = math.radians(HOH_DEG) / 2
    arms = R_OH * torch.tensor([[math.sin(half), 0, math.cos(half)], [-math.sin(half), 0, math.cos(half)]], device="cuda", dtype=torch.float64)
    rot = _rotations(n, gen)
    pos = torch.stack([oxygen] + [oxygen + rot @ arm for arm in arms], 1)
    return pos.reshape(-1, 3), torch.tensor([8, 1, 1], device="cuda", dtype=torch.int32).repeat(n)


def _water(n, gen):
    return _molecules(_sphere_sites(n)[torch.randperm(n, generator=gen, device="cuda")], gen)


def _box(n, gen):
    edge, m = (n / BOX_DENSITY) ** (1.0 / 3.0), int(math.ceil(n ** (1.0 / 3.0) - 1e-9))
    spacing = edge / m
    site = torch.randperm(m ** 3, generator=gen, device="cuda")[:n]
    xyz = torch.stack([site // (m * m), site // m % m, site % m], 1).double()
    xyz = spacing * (xyz + 0.5) + (spacing - BOX_MIN_DIST) / 2 * (2 * torch.rand((n, 3), generator=gen, device="cuda", dtype=torch.float64) - 1)
    unit = n // 10
    numbers = torch.full((n,), 8, device="cuda", dtype=torch.int32)
    numbers[:9 * unit] = torch.tensor([6] * 3 + [1] * 5 + [7], device="cuda", dtype=torch.int32).repeat(unit)
    numbers = numbers[torch.randperm(n, generator=gen, device="cuda")]
    cell = [[edge if i == k else 0.0 for k in range(3)] for i in range(3)]
    return xyz, numbers.contiguous(), cell


MOST_MOLECULES = 15               # molecules of a structure of a batch: 1 to 15, 3 to 45 atoms


def _batch(n, gen):
    sizes = (torch.arange(n, device="cuda") % MOST_MOLECULES + 1)[torch.randperm(n, generator=gen, device="cuda")]
    ends = sizes.cumsum(0)
    local = torch.arange(int(ends[-1]), device="cuda") - torch.repeat_interleave(ends - sizes, sizes)
    pos, numbers = _molecules(_sphere_sites(MOST_MOLECULES)[local], gen)
    ptr = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), 3 * ends])
    return pos, numbers, ptr


def _structure(case, seed):
    """(positions in fp64, numbers, cell, centres, offsets of a batch) of a case, from the seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    cell = centers = ptr = None
    if case["structure"] == "box":
        pos, numbers, cell = _box(case["size"], gen)
    elif case["call"] == "derivatives_batch":
        pos, numbers, ptr = _batch(case["size"], gen)
    else:
        pos, numbers = _water(case["size"], gen)
    if case["centers"]:
        centers = torch.randperm(pos.shape[0], generator=gen, device="cuda")[:case["centers"]].to(torch.int32).contiguous()
    return pos, numbers, cell, centers, ptr


def _scaled(structure, factor):
    """The structure on the library's terms (fp32 positions), uniformly scaled."""
    pos, numbers, cell, centers, ptr = structure
    return (factor * pos).float().contiguous(), numbers, None if cell is None else [[factor * x for x in row] for row in cell], centers, ptr


def _rows(case, structure):
    """Jacobian rows of the structure."""
    pos, numbers, cell, centers, ptr = structure
    if ptr is None:
        return _handle_of(case).neighbors(pos, numbers, cell, centers)[1]
    sizes = ptr[1:] - ptr[:-1]
    at = torch.arange(3 * MOST_MOLECULES, device="cuda")
    atom = torch.minimum(ptr[:-1, None] + at, ptr[1:, None] - 1)
    xyz = pos.double()[atom]
    d = xyz[:, :, None, :] - xyz[:, None, :, :]
    inside = (d * d).sum(-1) < case["r_cut"] ** 2                 # an atom counts itself: its own row
    there = at < sizes[:, None]
    return int((inside & there[:, :, None] & there[:, None, :]).sum())


_TARGET = {}


def _fitted(case, seed):
    """A structure from the seed with as many Jacobian rows as the case's structure of seed 0, so that the outputs of
    all seeds have one shape: random structures of a kind differ in their row count by a few parts in a thousand,
    which a uniform scaling by even less takes up."""
    first = _structure(case, seed)
    if "derivatives" not in case["call"] or case["call"] in ("derivatives_outer", "derivatives_inner"):
        return _scaled(first, 1.0)
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _TARGET:
        _TARGET[key] = _rows(case, _scaled(_structure(case, 0), 1.0))
    target = _TARGET[key]
    low, high = 0.5, 2.0                                            # few rows at `high`, many at `low`
    factor, step = 1.0, 0.002
    for trial in range(400):
        s = _scaled(first, factor)
        rows = _rows(case, s)
        if rows == target:
            return s
        if rows > target:
            low = max(low, factor)
        else:
            high = min(high, factor)
        if high - low < 1e-8:                                       # several pairs cross the cutoff at once: another structure
            first = _structure(case, seed + 1000003 * (trial + 1))
            low, high, factor, step = 0.5, 2.0, 1.0, 0.002
        elif low == 0.5 or high == 2.0:
            factor, step = factor + (step if rows > target else -step), 2 * step
        else:
            factor = (low + high) / 2
    raise RuntimeError("no structure with the wanted number of rows")


# ---------------------------------------------------------------------------------------------- the cases
@functools.lru_cache(maxsize=3)
def _handle(species, r_cut, n_max, l_max, sigma, rbf, periodic, crossover, weighted):
    weighting = {"function": "poly", "r0": r_cut, "c": 1.0, "m": 2.0, "w0": 1.0} if weighted else None
    return soap.Soap(list(species), r_cut, n_max, l_max, sigma, soap.GTO if rbf == "gto" else soap.POLYNOMIAL, (periodic,) * 3,
                     crossover=crossover, weighting=weighting)


def _handle_of(case):
    box = case["structure"] == "box"
    return _handle(BOX_SPECIES if box else WATER_SPECIES, case["r_cut"], case["n_max"], case["l_max"], case["sigma"], case["rbf"],
                   box, case["crossover"], case["weighted"])


def prepare(case, seed):
    h = _handle_of(case)
    pos, numbers, cell, centers, ptr = _fitted(case, seed)
    state = {"call": case["call"], "soap": h, "pos": pos, "num": numbers, "cell": cell, "centers": centers, "ptr": ptr}
    if case["call"] == "derivatives_into":
        # a time-stepping program sizes its buffers once
        c = pos.shape[0] if centers is None else centers.shape[0]
        _, rows = h.neighbors(pos, numbers, cell, centers)
        state["out"] = (torch.empty((c, h.n_features), device="cuda"), torch.empty((rows, 3, h.n_features), device="cuda"),
                        torch.empty(c + 1, dtype=torch.int64, device="cuda"), torch.empty(rows, dtype=torch.int32, device="cuda"))
    return state


def run(state):
    h, pos, num, cell, centers = state["soap"], state["pos"], state["num"], state["cell"], state["centers"]
    call = state["call"]
    if call == "derivatives_into":
        h.derivatives_into(pos, num, cell, centers, *state["out"])
        return state["out"]
    if call == "descriptor":
        return h.descriptor(pos, num, cell, centers)
    if call == "derivatives_outer":
        return h.derivatives_average("outer", pos, num, cell, centers)
    if call == "derivatives_inner":
        return h.derivatives_average("inner", pos, num, cell, centers)
    if call == "derivatives_compact":
        d = h.derivatives_compact(pos, num, cell, centers)
        return d.descriptor, d.center_rows, d.jacobian, d.row_ptr, d.row_atom
    d = h.derivatives_batch(pos, num, state["ptr"]) if call == "derivatives_batch" else h.derivatives(pos, num, cell, centers)
    return d.descriptor, d.jacobian, d.row_ptr, d.row_atom


def _pairs(case):
    """(atoms, centres, expected ordered pairs inside the cutoff)."""
    rc = case["r_cut"]
    if case["structure"] == "box":
        n = case["size"]
        return n, n, n * BOX_DENSITY * 4.0 / 3.0 * math.pi * rc ** 3
    if case["call"] == "derivatives_batch":
        n = case["size"] * 3 * (MOST_MOLECULES + 1) / 2
        return n, n, n * 0.75 * 3 * (MOST_MOLECULES + 1) / 2      # most of a small molecule lies inside the cutoff
    n = 3 * case["size"]
    radius = (3.0 * case["size"] / (4.0 * math.pi * WATER_DENSITY)) ** (1.0 / 3.0)
    s = min(rc / radius, 2.0)
    pairs = n * (n - 1) * s ** 3 * (1 - 9.0 / 16.0 * s + s ** 3 / 32.0)   # two uniform points of a ball
    c = case["centers"] or n
    return n, c, pairs * c / n


def work(case):
    n_atoms, c, pairs = _pairs(case)
    s, n, l1 = len(BOX_SPECIES if case["structure"] == "box" else WATER_SPECIES), case["n_max"], case["l_max"] + 1
    lm = l1 * l1
    tri, square = n * (n + 1) // 2 * l1, n * n * l1
    features = s * tri + (s * (s - 1) // 2 * square if case["crossover"] else 0)
    touched = tri + ((s - 1) * square if case["crossover"] else 0)            # features that a neighbour's row depends on
    inputs = 16 * n_atoms + 4 * case["centers"]
    # multiply-adds: radial polynomials, harmonics, accumulation, Eq. 4
    fma = pairs * (5 * n * l1 + 3 * lm + n * lm) + c * lm * s * n * (s * n + 1) / 2
    if case["call"] == "descriptor":
        return {"bytes": inputs + 4 * c * features, "flops": 2 * fma}
    # gradients of the coefficients, their contraction with the coefficients, the product rule
    fma += pairs * (5 * n * l1 + 9 * lm + 6 * n * lm + 4 * s * n * lm + 7 * touched)
    if case["call"] in ("derivatives_outer", "derivatives_inner"):
        return {"bytes": inputs + 4 * features + 12 * n_atoms * features, "flops": 2 * fma}
    rows = pairs + c
    width = (touched + 7) // 8 * 8 if case["call"] == "derivatives_compact" else features
    out = 4 * c * features + 12 * rows * width + 4 * rows + 8 * (c + 1)
    if case["call"] == "derivatives_compact":
        out += 12 * c * features
    return {"bytes": inputs + out, "flops": 2 * fma}


def tolerance(case):
    # All arithmetic on the way is fp32 (geometry and cutoff test fp64); row pointers and atoms are whole numbers and
    # exact.  Against the fp64 oracle, over these cases and fifty drawn ones: norm of the difference at most 2.6e-7 of
    # the norm, largest difference at most 2.6e-5 of the root mean square (single Jacobian entries many times larger
    # than their neighbours carry it).  Four times that.
    return {"rel": 1e-6, "max": 1e-4}
