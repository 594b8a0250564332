"""The work that users of this engine have it do: self-consistent energy + force evaluations,
of one structure or of a population, cold or warm started, in mixed precision or plain FP64.

A case is the evaluation of one structure (`members` 1, sgo_energy_forces) or of a population
(`members` > 1, sgo_energy_forces_batch, or its device-array form), and its sizes are those of
the structure: atoms, plane-wave cutoff, cell, k mesh.  One listed case is the H psi apply that
a program with its own eigensolver calls.

Positions come from the seed.  Crystals and population members are random structures with no
two atoms closer than 2.5 bohr, as the search has them before their relaxation (its own repair
distance is 2.0); the layer is a displaced honeycomb, the cluster a random compact one.

The mixed path computes its wavefunctions, transforms and products in FP32, and its results are
good to single precision; a program takes them as float32, and the plain path's as float64.
"""
import functools
import math
import types

import numpy as np
import torch

import paper_1603_02732_gb300 as sgo

Z4 = dict(z_val=4.0, rc=1.0, a_sr=0.5, sigma_sr=0.8, rp=0.9, d_nl=1.0)
Z4_P = dict(Z4, rp_p=1.0, d_p=0.6)
Z10 = dict(z_val=10.0, rc=1.2, a_sr=0.5, sigma_sr=1.0, rp=1.1, d_nl=0.8)

CASE = dict(kind="cell", atoms=8, ecut=10.0, precision="mixed", xc="lda", p_channel=False, mesh="1x1x1",
            members=1, first=0, warm=False, call="host", tol_rho=1e-5)


def _case(name=None, **kw):
    c = dict(CASE, **kw)
    if c["precision"] == "fp64":
        c["tol_rho"] = 1e-7
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: a 2-atom cell, a few hundred plane waves (launch latency counts)
        _case("cell2_mixed", atoms=2, ecut=3.0),
        # a crystal of the paper's table (8 atoms, 32^3 grid), on the plain FP64 path
        _case("crystal8_fp64", kind="diamond", precision="fp64"),
        # the 24-atom 2D layer with vacuum: a long cell, many SCF iterations
        _case("layer24_mixed", kind="layer", atoms=24, ecut=15.0, tol_rho=3e-6),
        # the same on the plain FP64 path
        _case("layer24_fp64", kind="layer", atoms=24, ecut=15.0, precision="fp64"),
        # a 13-atom metal cluster in a 20-bohr box with PBE (72^3 grid, 85 bands)
        _case("cluster13_pbe_mixed", kind="cluster", atoms=13, ecut=15.0, xc="pbe", tol_rho=3e-6),
        # a crystal's relaxation step on a rough 2 x 2 x 2 k mesh (folded: 64 atoms, 160 bands)
        _case("mesh222_mixed", kind="diamond", mesh="2x2x2"),
        # the largest population member on its own (32 atoms, 80 bands, ragged 60 x 50 x 54 grid),
        # with a p channel
        _case("member32_pchannel_mixed", kind="candidate", atoms=32, ecut=12.0, first=44, p_channel=True),
        # the paper's search population: 8 structures of 8 atoms in one cell
        _case("search8_mixed", kind="diamond", members=8),
        # a whole population, uneven cells of 8 to 32 atoms, positions and results on the device
        _case("population64_mixed", kind="candidate", ecut=12.0, members=64, call="device"),
        # one relaxation round of it: every member moved a little, started from its last state
        _case("population64_warm", kind="candidate", ecut=12.0, members=64, warm=True),
        # a small uneven population on the plain FP64 path
        _case("population6_fp64", kind="candidate", ecut=12.0, members=6, first=8, precision="fp64"),
        # H psi of every band of the layer, host arrays in and out
        _case("hpsi_layer24_mixed", kind="layer", atoms=24, ecut=15.0, call="hpsi"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    precision = "fp64" if rng.random() < 0.35 else "mixed"
    xc = "pbe" if rng.random() < 0.2 else "lda"
    what = rng.choice(["cell", "cell", "candidates", "candidates", "layer", "cluster", "mesh"])
    if what == "cell":
        return _case(atoms=log_int(2, 16 if precision == "fp64" else 32), ecut=round(rng.uniform(4.0, 13.0), 2),
                     precision=precision, xc=xc, p_channel=rng.random() < 0.3, first=rng.randrange(1000))
    if what == "candidates":
        # (a plain FP64 member takes about 0.1 s)
        n = log_int(2, 6 if precision == "fp64" else 64)
        return _case(kind="candidate", ecut=round(rng.uniform(8.0, 12.0), 2), members=n, precision=precision, xc=xc,
                     first=rng.randrange(1000), **rng.choice([{}, {}, dict(warm=True), dict(call="device")]))
    if what == "layer":
        return _case(kind="layer", atoms=24, ecut=round(rng.uniform(8.0, 14.0), 2), precision=precision, xc=xc,
                     tol_rho=3e-6, call="hpsi" if rng.random() < 0.3 else "host")
    if what == "cluster":
        return _case(kind="cluster", atoms=rng.randrange(3, 14), ecut=round(rng.uniform(8.0, 14.0), 2), xc=xc,
                     tol_rho=3e-6)
    return _case(kind="diamond", mesh=rng.choice(["2x1x1", "1x2x2", "2x2x1", "1x1x3"]),
                 ecut=round(rng.uniform(7.0, 10.0), 2), xc=xc, p_channel=rng.random() < 0.3)


def _fft_size(n):
    def smooth(k):
        for p in (2, 3, 5):
            while k % p == 0:
                k //= p
        return k == 1

    while not smooth(n):
        n += 1
    return n


def _grid(cell, ecut):
    m = np.floor(np.linalg.norm(cell, axis=1) * math.sqrt(2.0 * ecut) / (2.0 * math.pi)).astype(int)
    return tuple(_fft_size(4 * int(v) + 1) for v in m)


def _spread(cell, n, dmin, rng):
    """n random positions in the cell, no two (minimum image) closer than dmin."""
    inv = np.linalg.inv(cell)
    images = np.array([[a, b, c] for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)], dtype=float) @ cell
    pos = np.empty((0, 3))
    while len(pos) < n:
        p = rng.uniform(size=3) @ cell
        d = (p - pos) @ inv
        d = ((d - np.round(d)) @ cell)[:, None, :] + images
        if not len(pos) or np.sqrt((d * d).sum(axis=2)).min() >= dmin:
            pos = np.vstack([pos, p])
    return pos


@functools.lru_cache(maxsize=None)
def _population_member(i):
    """Cell and atom count of member i of the benchmark's population: a strained cell of 8 to
    32 atoms, 135 bohr^3 per atom within 20 %."""
    rng = np.random.default_rng(4000 + i)
    n = int(rng.integers(8, 33))
    return _strained(rng, n), n


def _strained(rng, n):
    e = rng.uniform(-0.1, 0.1, size=(3, 3))
    m = np.eye(3) + 0.5 * (e + e.T)
    vol = 135.0 * n * rng.uniform(0.8, 1.2)
    return (vol / abs(np.linalg.det(m))) ** (1.0 / 3.0) * m


@functools.lru_cache(maxsize=None)
def _honeycomb():
    """The flat 24-atom honeycomb: 2 sqrt3 x 2 sqrt3 R30 cell, a = 13, c = 26 bohr."""
    a, c = 13.0, 26.0
    cell = np.array([[a, 0.0, 0.0], [0.5 * a, 0.5 * math.sqrt(3.0) * a, 0.0], [0.0, 0.0, c]])
    a0 = a / (2.0 * math.sqrt(3.0))
    p = a0 * np.array([[math.cos(math.pi / 6), math.sin(math.pi / 6)], [0.0, 1.0]])
    inv = np.linalg.inv(cell[:2, :2])
    pts = []
    for i in range(-12, 13):
        for j in range(-12, 13):
            for b in (np.zeros(2), (p[0] + p[1]) / 3.0):
                f = (i * p[0] + j * p[1] + b) @ inv
                if np.all(f > -1e-9) and np.all(f < 1.0 - 1e-9):
                    pts.append(f @ cell[:2, :2])
    pos = np.concatenate([np.array(pts), np.full((len(pts), 1), 0.5 * c)], axis=1)
    return cell, pos


def _compact(rng, n, dmin, box):
    """n random positions in a sphere at the centre of the box, no two closer than dmin."""
    radius, fails, pos = 0.5 * dmin * (n / 0.35) ** (1.0 / 3.0), 0, []
    while len(pos) < n:
        u = rng.normal(size=3)
        p = 0.5 * box + u / np.linalg.norm(u) * radius * rng.uniform() ** (1.0 / 3.0)
        if all(np.linalg.norm(p - q) >= dmin for q in pos):
            pos.append(p)
            fails = 0
        else:
            fails += 1
            if fails >= 10000:
                radius, fails = 1.05 * radius, 0
    return np.array(pos)


def _size(case, k):
    """Cell, atom count, species, bands, grid of member k of a case."""
    kind, n, ecut = case["kind"], case["atoms"], case["ecut"]
    species = Z10 if kind == "cluster" else Z4_P if case["p_channel"] else Z4
    grid = None
    if kind == "cell":
        cell = _strained(np.random.default_rng(100 + case["first"]), n)
    elif kind == "diamond":
        cell = np.eye(3) * 10.26
        grid = (32, 32, 32) if ecut == 10.0 else None
    elif kind == "layer":
        cell, n = _honeycomb()[0], 24
        grid = (48, 48, 96) if ecut == 15.0 else None
    elif kind == "cluster":
        cell = np.eye(3) * 20.0
    else:
        cell, n = _population_member(case["first"] + k)
    nocc = n * species["z_val"] / 2.0
    bands = int(math.ceil((1.3 if kind == "cluster" else 1.25) * nocc))
    bands += bands % 2 if kind != "cluster" else 0
    if kind == "layer":
        bands = 64
    return cell, n, species, bands, grid or _grid(cell, ecut)


def _mesh(case):
    return tuple(int(v) for v in case["mesh"].split("x"))


def _structure(case, k, rng):
    cell, n, species, bands, grid = _size(case, k)
    if case["kind"] == "layer":
        pos = _honeycomb()[1] + rng.normal(scale=0.2, size=(n, 3))
    elif case["kind"] == "cluster":
        pos = _compact(rng, n, 3.0, 20.0)
    else:
        pos = _spread(cell, n, 2.5, rng)
    return types.SimpleNamespace(cell=cell, species=[species], species_of_atom=np.zeros(n, np.int32), pos=pos,
                                 ecut=case["ecut"], nbands=bands, fft=grid, kT=0.01, xc=case["xc"],
                                 kgrid=_mesh(case), natoms=n)


def prepare(case, seed):
    structures, rng, veff, psi = _inputs(case, seed)
    ctxs = []
    for st in structures:
        tol_e = 1e-8 if case["precision"] == "fp64" else 1e-7 * st.natoms
        ctxs.append(sgo.Context(st, precision=case["precision"], scf_tol_e=tol_e, scf_tol_rho=case["tol_rho"],
                                max_scf=150))
    s = dict(case=case, ctxs=ctxs, dtype=np.float64 if case["precision"] == "fp64" else np.float32)
    s["pos"] = [st.pos for st in structures]
    if case["call"] == "hpsi":
        s["veff"], s["psi"] = veff, psi
        return s
    if case["members"] > 1:
        s["batch"] = sgo.Batch(ctxs)
    if case["warm"]:
        s["moved"] = [p + rng.normal(scale=0.02, size=p.shape) for p in s["pos"]]
        s["batch"].energy_forces(s["pos"])
        for c in ctxs:
            c.set_warm(True)
    if case["call"] == "device":
        dev = torch.device("cuda")
        n = sum(st.natoms for st in structures)
        s["pos_dev"] = torch.as_tensor(np.concatenate(s["pos"]), dtype=torch.float64, device=dev)
        s["energies"] = torch.zeros(len(ctxs), dtype=torch.float64, device=dev)
        s["forces"] = torch.zeros((n, 3), dtype=torch.float64, device=dev)
        s["status"] = torch.zeros(len(ctxs), dtype=torch.int32, device=dev)
    return s


def run(s):
    case, dtype = s["case"], s["dtype"]
    if case["call"] == "hpsi":
        return s["ctxs"][0].apply_hamiltonian(s["veff"], s["psi"]).astype(dtype)
    if case["members"] == 1:
        energy, forces = s["ctxs"][0].energy_forces(s["pos"][0])
        return {"energy": dtype(energy), "forces": forces.astype(dtype)}
    if case["call"] == "device":
        s["batch"].energy_forces_device(s["pos_dev"].data_ptr(), s["energies"].data_ptr(), s["forces"].data_ptr(),
                                        s["status"].data_ptr())
        to = torch.float64 if dtype is np.float64 else torch.float32
        return {"energies": s["energies"].to(to), "forces": s["forces"].to(to), "status": s["status"].clone()}
    # (a warm pass is one relaxation round there and one back)
    out = {}
    for name in ("moved", "pos") if case["warm"] else ("pos",):
        energies, forces, status = s["batch"].energy_forces(s[name])
        out[name] = {"energies": energies.astype(dtype), "forces": np.concatenate(forces).astype(dtype),
                     "status": status}
    return out


# Self-consistent iterations of an evaluation, as measured over these inputs (each applies H
# three times to every band: once, and once in each of two CG steps).
_ITERATIONS = {"cell": 14, "diamond": 14, "candidate": 15, "layer": 36, "cluster": 31}


def work(case):
    """Per H apply of a band pair one inverse and one forward transform (the occupied columns
    along z, the occupied rows along y, all lines along x, 5 N log2 N each), the kinetic and
    nonlocal terms; per CG step and Rayleigh-Ritz step the products of the band block with
    itself and its rotations; per iteration the density and the grid transforms.  Bytes: the
    band block read and written once per H apply and per rotation, the grids once per
    iteration."""
    size = 8.0 if case["precision"] == "fp64" else 4.0
    mesh = _mesh(case)
    nk = mesh[0] * mesh[1] * mesh[2]
    total = {"bytes": 0.0, "flops": 0.0}
    for k in range(case["members"]):
        cell, n, species, bands, grid = _size(case, k)
        omega = abs(np.linalg.det(cell)) * nk
        n, bands = n * nk, bands * nk
        proj = n * (4 if species.get("d_p") else 1)
        n1, n2, n3 = (a * b for a, b in zip(grid, mesh))
        points = float(n1 * n2 * n3)
        gmax = math.sqrt(2.0 * case["ecut"])
        npw = omega * gmax ** 3 / (6.0 * math.pi ** 2)
        columns, rows = math.pi / 16.0 * n1 * n2, 0.5 * n1
        line = [5.0 * v * math.log2(v) for v in (n1, n2, n3)]
        one_way = columns * line[2] + n3 * (rows * line[1] + n2 * line[0])
        pair = 0.5 * bands
        h_flops = pair * (2.0 * one_way + 2.0 * points) + 4.0 * bands * npw * proj
        h_bytes = 2.0 * bands * npw * size + points * size
        if case["call"] == "hpsi":
            total["flops"] += h_flops
            total["bytes"] += 2.0 * bands * npw * 8.0 + points * 8.0
            continue
        it = _ITERATIONS[case["kind"]]
        it = 2 * 10 if case["warm"] else it
        block = 2.0 * bands * bands * npw
        rr = (2 * 3 + 2 * 2 + 4 * 2 + 2) * block + 3 * 9.0 * bands ** 3
        grids = (12 if case["xc"] == "pbe" else 2) * points / (n1 * n2 * n3) * (
            n2 * n3 * line[0] + n1 * n3 * line[1] + n1 * n2 * line[2])
        total["flops"] += it * (3 * h_flops + rr + pair * (one_way + 4.0 * points) + grids)
        total["bytes"] += it * (3 * h_bytes + 3 * 4.0 * bands * npw * size + 12.0 * points * 8.0)
    return total


def _miller(cell, ecut):
    """Half sphere |G|^2/2 <= ecut without G = 0: the (0, 0) column first, then the columns with
    m2 > 0, or m2 = 0 and m1 > 0, in order of (m1, m2); m3 ascending."""
    b = 2.0 * math.pi * np.linalg.inv(cell).T
    box = np.floor(np.linalg.norm(cell, axis=1) * math.sqrt(2.0 * ecut) / (2.0 * math.pi)).astype(int) + 1
    m = np.stack(np.meshgrid(*(np.arange(-v, v + 1) for v in box), indexing="ij"), axis=-1).reshape(-1, 3)
    first = (m[:, 0] == 0) & (m[:, 1] == 0)
    m = np.concatenate([m[first & (m[:, 2] > 0)], m[~first & ((m[:, 1] > 0) | ((m[:, 1] == 0) & (m[:, 0] > 0)))]])
    g = m @ b
    keep = 0.5 * (g * g).sum(axis=1) <= ecut
    return m[keep], g[keep]


def _inputs(case, seed):
    """The structures of a case, and veff and psi of an H psi case, from the seed."""
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 17])
    structures = [_structure(case, k, rng) for k in range(case["members"])]
    if case["call"] != "hpsi":
        return structures, rng, None, None
    st = structures[0]
    npw = 1 + 2 * len(_miller(st.cell, st.ecut)[0])
    return structures, rng, 0.2 * rng.normal(size=st.fft), rng.normal(size=(st.nbands, npw)) / math.sqrt(npw)


def exact(case, seed):
    """H psi in complex arithmetic over the whole sphere: |G|^2/2 + V on the grid + the s
    projectors.  None for the self-consistent evaluations: in plain numpy they take minutes."""
    if case["call"] != "hpsi":
        return None
    (st,), _, veff, psi = _inputs(case, seed)
    sp, m_, omega = st.species[0], _miller(st.cell, st.ecut), abs(np.linalg.det(st.cell))
    miller = np.concatenate([np.zeros((1, 3), int), m_[0], -m_[0]])
    g = np.concatenate([np.zeros((1, 3)), m_[1], -m_[1]])
    g2 = (g * g).sum(axis=1)
    half = (psi[:, 1::2] + 1j * psi[:, 2::2]) / math.sqrt(2.0)
    c = np.concatenate([psi[:, :1], half, half.conj()], axis=1)
    norm = (math.pi ** 1.5 * sp["rp"] ** 3) ** -0.5 * (2.0 * math.pi) ** 1.5 * sp["rp"] ** 3 / math.sqrt(omega)
    beta = norm * np.exp(-0.5 * g2 * sp["rp"] ** 2) * np.exp(-1j * (st.pos @ g.T))
    out = 0.5 * g2 * c + sp["d_nl"] * (c @ beta.conj().T) @ beta
    at = tuple(miller.T % np.array(st.fft)[:, None])
    for n in range(len(c)):
        box = np.zeros(st.fft, complex)
        box[at] = c[n]
        out[n] += np.fft.fftn(np.fft.ifftn(box) * veff)[at]
    h = out[:, 1:1 + half.shape[1]]
    packed = np.empty_like(psi)
    packed[:, 0], packed[:, 1::2], packed[:, 2::2] = out[:, 0].real, math.sqrt(2.0) * h.real, math.sqrt(2.0) * h.imag
    return packed
