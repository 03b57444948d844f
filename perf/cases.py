"""The workloads by which a change to this library's speed is judged.

Each case is one call sequence of a user's program: a lattice (or a batch of
them) in hand, its state set, `n` sweeps at one inverse temperature with the
per-sweep E / M moments accumulated, then the moments, a measurement of the
final state and the spins read back.  Launch configurations are the library's
automatic ones.  Sizes are those of the benchmark and the tests, plus odd and
ragged ones of the same kind.

`exact` repeats a case in 64 bits with plain torch: the Philox4x32-10 stream
of the documented schedules, the Metropolis rule of arXiv 2106.11286 (Eq. 1,
steps (i)-(iii)) colour class by colour class, and Eq. 2's moments.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2106_11286_gb300 import hs, inputs

BYTES = {"fp64": 8, "fp32": 4, "fp16": 2}
BASIS = {"sc": 1, "bcc": 2, "fcc": 4}
AXES = {"z": (0.0, 0.0, 1.0), "111": (1.0, 1.0, 1.0), "tilted": (0.3, -0.2, 1.0)}
FILM = (0.02, 0.03, -0.15, 0.01, 0.0, -0.02)  # the tensor of a thin film's effective shape anisotropy


def _sc(name, dims, precision, n, K=0.05, T=1.2, axis="z", tensor=False):
    return {"name": name, "kind": "sc", "Lx": dims[0], "Ly": dims[1], "Lz": dims[2], "precision": precision,
            "n": n, "K": K, "T": T, "axis": axis, "tensor": tensor, "periodic": True, "vacancies": 0.0}


def listed():
    return [
        # one sweep of a small lattice, measured after it: the inner step of a tempering or hybrid loop
        _sc("sc24_fp32_step", (24, 24, 24), "fp32", 1, K=0.0, T=1.4),
        # the small plain-FP64 workload of the paper's kind: a measurement block at 16^3
        _sc("sc16_fp64", (16, 16, 16), "fp64", 100, K=0.1, T=1.0),
        # a ragged box (an odd number of sites of one colour in a row) with an axis off the coordinate axes
        _sc("sc_ragged_fp32", (90, 62, 110), "fp32", 30, K=0.2, T=0.9, axis="111"),
        # a thin film with the shape-anisotropy tensor
        _sc("film_tensor_fp32", (256, 256, 16), "fp32", 30, K=0.05, T=1.0, tensor=True),
        # the benchmark's lattice, in its FP32 form ...
        _sc("sc256_fp32", (256, 256, 256), "fp32", 50),
        # ... and in plain FP64
        _sc("sc256_fp64", (256, 256, 256), "fp64", 10),
        # the largest lattice of the precision comparison, FP32 and FP16
        _sc("sc464_fp32", (464, 464, 464), "fp32", 10, K=0.1, T=1.0),
        _sc("sc464_fp16", (464, 464, 464), "fp16", 10, K=0.1, T=1.0),
        # a bcc nanoparticle with vacancies, as a neighbour list
        {"name": "nano_csr_fp32", "kind": "csr", "radius": 72, "precision": "fp32", "n": 20, "K": 0.2, "T": 0.9,
         "axis": "111", "tensor": False, "vacancies": 0.01},
        # an open fcc block with vacancies in FP64
        {"name": "fcc_open_fp64", "kind": "fcc", "Lx": 31, "Ly": 27, "Lz": 22, "precision": "fp64", "n": 20,
         "K": 0.1, "T": 2.4, "axis": "z", "tensor": False, "periodic": False, "vacancies": 0.01},
        # the temperature scan: 64 replicas of uneven size in one batch
        {"name": "scan64_fp32", "kind": "batch", "members": 64, "Lmin": 16, "Lmax": 96, "precision": "fp32",
         "n": 20, "K": 0.0, "axis": "z", "Tmin": 1.3, "Tmax": 1.6},
        # tempering: 48 plain-FP64 replicas of one small lattice
        {"name": "temper48_fp64", "kind": "batch", "members": 48, "Lmin": 16, "Lmax": 16, "precision": "fp64",
         "n": 20, "K": 0.01, "axis": "z", "Tmin": 1.3, "Tmax": 1.6},
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["sc", "sc", "sc", "sc", "table", "csr", "batch"])
    precision = rng.choice(["fp64", "fp32", "fp32", "fp16"])
    case = {"kind": kind, "precision": precision, "K": rng.choice([0.0, 0.01, 0.05, 0.2]),
            "axis": rng.choice(["z", "z", "111", "tilted"]), "T": round(rng.uniform(0.7, 1.7), 3)}
    most = 2.0e8 if precision == "fp64" else 1.0e9  # attempts of one pass: below the largest listed case
    if kind == "sc":
        dims = [_log_int(rng, 8, 320, 2) for _ in range(3)]
        if rng.random() < 0.5:  # a row that the widest vectors divide
            dims[0] = max(16, dims[0] // 16 * 16)
        case.update(Lx=dims[0], Ly=dims[1], Lz=dims[2], periodic=True, vacancies=0.0,
                    tensor=rng.random() < 0.15)
        sites = dims[0] * dims[1] * dims[2]
        case["n"] = max(1, min(_log_int(rng, 1, 200), int(most / sites)))
    elif kind == "table":
        case["kind"] = rng.choice(["sc", "bcc", "fcc"])
        dims = [_log_int(rng, 5, 60) for _ in range(3)]
        case.update(Lx=dims[0], Ly=dims[1], Lz=dims[2], periodic=case["kind"] != "sc" and rng.random() < 0.5,
                    vacancies=rng.choice([0.0, 0.01, 0.1]), tensor=rng.random() < 0.15)
        sites = dims[0] * dims[1] * dims[2] * BASIS[case["kind"]]
        case["n"] = max(1, min(_log_int(rng, 1, 100), int(most / sites)))
    elif kind == "csr":
        case.update(radius=_log_int(rng, 6, 60), vacancies=rng.choice([0.0, 0.01, 0.05]), tensor=False,
                    n=_log_int(rng, 1, 60))
    else:
        lo = 8 * rng.randint(1, 4)
        case.update(members=_log_int(rng, 2, 200), Lmin=lo, Lmax=lo + 8 * rng.choice([0, 0, 1, 3, 6]), Tmin=1.2,
                    Tmax=1.7)
        del case["T"]
        attempts = sum(L ** 3 for L in _sizes(case))
        case["n"] = max(1, min(_log_int(rng, 1, 100), int(most / attempts)))
    return case


def _sizes(case):
    """Edge lengths of a batch's members: cycling through Lmin ... Lmax in steps of 16 (or 8)."""
    span = case["Lmax"] - case["Lmin"]
    step = 16 if span % 16 == 0 and span else 8
    cycle = list(range(case["Lmin"], case["Lmax"] + 1, step))
    return [cycle[r % len(cycle)] for r in range(case["members"])]


def _temps(case):
    return np.linspace(case["Tmin"], case["Tmax"], case["members"])


@functools.lru_cache(maxsize=2)
def _particle(radius):
    return inputs.bcc_nanoparticle(radius, 2 * radius + 4)[:2]


def _mask(case, seed):
    """The sites present: bytes over the natural order, or None for all."""
    if not case.get("vacancies"):
        return None
    n = (len(_particle(case["radius"])[0]) - 1 if case["kind"] == "csr"
         else case["Lx"] * case["Ly"] * case["Lz"] * BASIS[case["kind"]])
    return inputs.vacancy_mask(n, case["vacancies"], seed)


def _state(n, seed, mask=None):
    """Unit spins about +z, disordered as a lattice somewhat below T_C is: (n, 3) FP64 on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s = torch.randn((n, 3), dtype=torch.float64, device="cuda", generator=g).mul_(0.75)
    s[:, 2] += 1.0
    s /= s.norm(dim=1, keepdim=True)
    if mask is not None:
        s[torch.from_numpy(mask == 0).cuda()] = 0.0
    return s


class _State:
    """The lattices of a case, the batch over them and the buffer that the spins come back in."""

    def __init__(self):
        self.lats, self.batch, self.betas, self.out = [], None, [], None

    def __del__(self):
        if self.batch is not None:
            hs.hs_batch_destroy(self.batch)
        for lat in self.lats:
            lat.close()


def prepare(case, seed):
    s = _State()
    common = dict(J=1.0, K=case["K"], e=AXES[case["axis"]], precision=case["precision"], seed=seed)
    if case["kind"] == "batch":
        for r, L in enumerate(_sizes(case)):
            s.lats.append(hs.Lattice("sc", dims=(L, L, L), replica=r, **common))
        s.betas = (1.0 / _temps(case)).tolist()
    else:
        mask, A = _mask(case, seed), FILM if case["tensor"] else None
        if case["kind"] == "csr":
            rp, col = _particle(case["radius"])
            s.lats.append(hs.Lattice("csr", A=A, row_ptr=rp, col_idx=col, site_mask=mask, **common))
        else:
            s.lats.append(hs.Lattice(case["kind"], A=A, dims=(case["Lx"], case["Ly"], case["Lz"]),
                                     periodic=case["periodic"], site_mask=mask, **common))
        s.betas = [1.0 / case["T"]]
    sizes = [lat.info.n_sites for lat in s.lats]
    first = _state(sum(sizes), seed, mask if case["kind"] != "batch" else None)
    s.out = list(torch.zeros_like(first).split(sizes))
    for lat, part in zip(s.lats, first.split(sizes)):
        hs.hs_set_spins_device(lat.h, part)
        lat.accumulate(True)
    torch.cuda.synchronize()
    if case["kind"] == "batch":
        s.batch = hs.hs_batch_create([lat.h for lat in s.lats])
    s.n = case["n"]
    return s


def run(s):
    for lat in s.lats:
        lat.reset_accumulator()
    if s.batch is not None:
        hs.hs_batch_run(s.batch, s.betas, s.n)
    else:
        s.lats[0].sweep(s.betas[0], s.n)
    got = {"spins": s.out[0]._base, "moments": [], "count": []}
    for lat, out in zip(s.lats, s.out):
        moments, count = lat.read_accumulator()
        got["moments"].append(moments)
        got["count"].append(count)
        hs.hs_get_spins_device(lat.h, out)
    got["moments"], got["count"] = np.array(got["moments"]), np.array(got["count"])
    if s.batch is None:
        m = s.lats[0].measure()
        got["E"], got["M"], got["accept_rate"] = m["E"], m["M"], m["accept_rate"]
    return got


def _sites(case):
    if case["kind"] == "batch":
        return sum(L ** 3 for L in _sizes(case))
    if case["kind"] == "csr":
        return len(_particle(case["radius"])[0]) - 1
    return case["Lx"] * case["Ly"] * case["Lz"] * BASIS[case["kind"]]


def work(case):
    """Per sweep the state read and written once (three components a spin); a neighbour list read once besides.
    At the end the spins widened to FP64.  About 72 operations an attempt: the field of the neighbours, the trial,
    the energy difference, the acceptance and the sums."""
    n, sites = case["n"], _sites(case)
    state = 3 * BYTES[case["precision"]] * sites
    table = 4 * 8 * sites if case["kind"] == "csr" else 0
    return {"bytes": n * (2 * state + table) + state + 24 * sites, "flops": 72 * n * sites}


# ---------------------------------------------------------------- 64 bits
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 over int64 tensors holding 32-bit words (two's complement products keep the low 64 bits)."""
    k0, k1 = key & _M32, (key >> 32) & _M32
    for _ in range(10):
        pa, pb = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((pb >> 32) & _M32) ^ c1 ^ k0, pb & _M32, ((pa >> 32) & _M32) ^ c3 ^ k1, pa & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _trial(precision, site, rank, sweep, colour, replica, key):
    """Trial spins and acceptance uniforms of the sites of one colour class."""
    full = lambda t, v: torch.full_like(t, v)  # noqa: E731
    if precision == "fp64":  # two blocks a site, 53-bit uniforms
        a = _philox(site, full(site, sweep), full(site, colour << 8), full(site, replica), key)
        z = ((((a[0] >> 5) << 26) | (a[1] >> 6)).double() - 2.0 ** 52) * 2.0 ** -52
        v = ((((a[2] >> 5) << 26) | (a[3] >> 6)).double() - 2.0 ** 52) * 2.0 ** -52
        b = _philox(site, full(site, sweep), full(site, (colour << 8) | 1), full(site, replica), key)
        u = (((b[0] >> 5) << 26) | (b[1] >> 6)).double() * 2.0 ** -53
    else:  # half a block a site, 21-, 21- and 22-bit uniforms
        pair = torch.arange((rank.numel() + 1) // 2, device=rank.device)
        w = _philox(pair, full(pair, sweep), full(pair, colour << 8), full(pair, replica), key)
        a = torch.stack((w[0], w[2]), 1).reshape(-1)[: rank.numel()]
        b = torch.stack((w[1], w[3]), 1).reshape(-1)[: rank.numel()]
        z = ((a >> 11).double() - 2.0 ** 20) * 2.0 ** -20
        v = ((b >> 11).double() - 2.0 ** 20) * 2.0 ** -20
        u = (((a & 0x7FF) << 11) | (b & 0x7FF)).double() * 2.0 ** -22
    r = ((1.0 - z) * (1.0 + z)).sqrt()
    t = torch.stack((r * torch.cos(math.pi * v), r * torch.sin(math.pi * v), z), 1)
    if precision == "fp16":  # the stored spin is the one tested
        t = (t / t.norm(dim=1, keepdim=True)).half().double()
    return t, u


_PARTNERS = {
    "sc": [[(-1, 0, 0, 0), (1, 0, 0, 0), (0, -1, 0, 0), (0, 1, 0, 0), (0, 0, -1, 0), (0, 0, 1, 0)]],
    "bcc": [[(x - 1, y - 1, z - 1, 1) for z in (0, 1) for y in (0, 1) for x in (0, 1)],
            [(x, y, z, 0) for z in (0, 1) for y in (0, 1) for x in (0, 1)]],
}


def _fcc_partners():
    corner = [(0, 0, 0), (0, 1, 1), (1, 0, 1), (1, 1, 0)]  # in half lattice constants
    rows = []
    for b in corner:
        row = []
        for d in [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]:
            if sum(v != 0 for v in d) == 2:
                q = [b[a] + d[a] for a in range(3)]
                row.append((q[0] // 2, q[1] // 2, q[2] // 2, corner.index(tuple(v % 2 for v in q))))
        rows.append(row)
    return rows


_PARTNERS["fcc"] = _fcc_partners()


def _neighbours(kind, dims, periodic, present):
    """[width][n] natural indices of each site's neighbours, n where there is none."""
    Lx, Ly, Lz = dims
    nb = BASIS[kind]
    n = Lx * Ly * Lz * nb
    i = torch.arange(n // nb, device="cuda")
    x, y, z = i % Lx, (i // Lx) % Ly, i // (Lx * Ly)
    width = len(_PARTNERS[kind][0])
    table = torch.empty((width, n), dtype=torch.int64, device="cuda")
    for b, row in enumerate(_PARTNERS[kind]):
        for k, (dx, dy, dz, o) in enumerate(row):
            X, Y, Z = x + dx, y + dy, z + dz
            j = (((Z % Lz) * Ly + Y % Ly) * Lx + X % Lx) * nb + o
            if not periodic:
                inside = (X >= 0) & (X < Lx) & (Y >= 0) & (Y < Ly) & (Z >= 0) & (Z < Lz)
                j = torch.where(inside, j, torch.full_like(j, n))
            table[k, b::nb] = j
    if present is not None:
        there = torch.cat((present, present.new_zeros(1)))
        table = torch.where(there[table], table, torch.full_like(table, n))
    if kind == "sc":
        colour = (x + y + z) % 2
    else:
        colour = torch.arange(n, device="cuda") % nb
    return table, colour


def _chain(kind, dims, periodic, mask, first, case, beta, seed, replica):
    """n sweeps from the state `first`: the final spins, the moments, E, M and the acceptance rate."""
    precision, J, K = case["precision"], 1.0, case["K"]
    e = torch.tensor(AXES[case["axis"]], dtype=torch.float64, device="cuda")
    e /= e.norm()
    A = None
    if case.get("tensor"):
        a = FILM
        A = torch.tensor([[a[0], a[3], a[4]], [a[3], a[1], a[5]], [a[4], a[5], a[2]]], dtype=torch.float64,
                         device="cuda")
    present = None if mask is None else torch.from_numpy(mask != 0).cuda()
    table, colour = _neighbours(kind, dims, periodic, present)
    n = first.shape[0]
    S = torch.cat((first, first.new_zeros((1, 3))))
    if precision != "fp64":
        S = S.to(torch.float32 if precision == "fp32" else torch.float16).double()
    classes = []
    for c in range(4 if kind == "fcc" else 2):
        own = colour == c if present is None else (colour == c) & present
        site = own.nonzero().reshape(-1)
        classes.append((site, table[:, site], torch.arange(site.numel(), device="cuda")))
    count = int(sum(c[0].numel() for c in classes))

    def quad(s):
        v = K * (s @ e) ** 2
        return v if A is None else v + ((s @ A) * s).sum(1)

    moments, accepted, E, M = np.zeros(9), 0, 0.0, np.zeros(3)
    for sweep in range(case["n"]):
        for c, (site, near, rank) in enumerate(classes):
            h = S[near[0]]
            for k in range(1, near.shape[0]):
                h += S[near[k]]
            t, u = _trial(precision, site, rank, sweep, c, replica, seed)
            s = S[site]
            dH = J * ((s - t) * h).sum(1) + quad(s) - quad(t)
            ok = (dH <= 0) | (u <= torch.exp(-beta * dH))
            S[site] = torch.where(ok[:, None], t, s)
            accepted += int(ok.sum())
        E, M = 0.0, np.zeros(3)
        for site, near, _ in classes:
            s = S[site]
            h = S[near[0]]
            for k in range(1, near.shape[0]):
                h += S[near[k]]
            E += float(-0.5 * J * (s * h).sum() - quad(s).sum())
            M += s.sum(0).cpu().numpy()
        M = M / count
        m2 = float(M @ M)
        moments += [E, E * E, math.sqrt(m2), m2, m2 * m2, M[0], M[1], M[2], abs(float(M @ e.cpu().numpy()))]
    return S[:n], moments, E, M, accepted / (case["n"] * count)


def exact(case, seed):
    if case["kind"] == "csr" or case["n"] * _sites(case) > 1.2e9:
        return None  # the greedy classes of a neighbour list come one site after the other; or too long
    if case["kind"] != "batch":
        mask, dims = _mask(case, seed), (case["Lx"], case["Ly"], case["Lz"])
        first = _state(_sites(case), seed, mask)
        S, moments, E, M, rate = _chain(case["kind"], dims, case["periodic"], mask, first, case, 1.0 / case["T"],
                                        seed, 0)
        return {"spins": S, "moments": moments[None], "count": np.array([case["n"]]), "E": E, "M": M,
                "accept_rate": rate}
    sizes = _sizes(case)
    first = _state(sum(L ** 3 for L in sizes), seed).split([L ** 3 for L in sizes])
    spins, rows = [], []
    for r, (L, T) in enumerate(zip(sizes, _temps(case))):
        S, moments, *_ = _chain("sc", (L, L, L), True, None, first[r], case, 1.0 / T, seed, r)
        spins.append(S)
        rows.append(moments)
    return {"spins": torch.cat(spins), "moments": np.array(rows), "count": np.full(len(sizes), case["n"])}
