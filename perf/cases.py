"""Workloads of the solver, as a user's program runs them.

A user holds a mesh handle for the chamber (it outlives every map and every
solve), builds a problem on it, and then asks for forward solves or for whole
steps of an inversion: new permittivities in, S-parameters, misfit, gradient
and fields out.  A case is one such call:

  forward   the solve of a set of transmitters on an assembled problem
  gradient  update_eps, forward_solve, misfit_and_gradient: one step with one
            complex permittivity per tet
  kappa     the same step with the nodal parameter, weights and the penalty
  steps     two consecutive steps on nearby maps with Krylov recycling

Sizes are those of this repository's benchmark, serving loop and tests: cubes
of a few hundred to a few thousand tets, chambers of 8 thousand to 402
thousand tets (order 1) and 53 thousand (order 2), 1 to 160 transmitters.
The FP64 path is solved to 1e-12 as the smoke run does.  The mixed path is
solved to 1e-11: an entry of S that lies X dB below the strongest one keeps
about rtol 10^(X/20) of relative accuracy, and the chamber's entries reach
down to about -116 dB, so this is what keeps five digits in the weakest
transmissions, which carry the image.
"""

import functools
import itertools
import math

import numpy as np
import torch

from paper_1607_02573_gb300 import mwi

FREQ = 1e9
GEL, HEAD, BLOOD, LOW = 44 - 20j, 45 - 18j, 60 - 25j, 38 - 15j


def listed():
    """cells: hexes per axis of a cube, or across the chamber (its height gets 14/15 as many)."""
    return [
        # the smallest call: the cube of the smoke run, plain FP64, latency-bound
        dict(name="cube_forward_fp64", kind="forward", cube=True, cells=8, order=1, precision=0, subs=4, tx=4, rx=4),
        # a whole inversion step at that size on the mixed path
        dict(name="cube_gradient", kind="gradient", cube=True, cells=8, order=1, precision=1, subs=4, tx=4, rx=4),
        # one transmitter against a ring of receivers on a small chamber (an interactive request)
        dict(name="chamber8k_one_tx", kind="forward", cube=False, cells=12, order=1, precision=1, subs=8, tx=1, rx=16),
        # a step of a coarse chamber with an odd, ragged set of transmitters
        dict(name="chamber19k_gradient_odd", kind="gradient", cube=False, cells=16, order=1, precision=1, subs=8,
             tx=13, rx=8),
        # one ring of transmitters on the medium chamber of the profiles
        dict(name="chamber120k_forward", kind="forward", cube=False, cells=30, order=1, precision=1, subs=32, tx=32,
             rx=32),
        # the reference precision: a step in plain FP64 with few transmitters
        dict(name="chamber46k_gradient_fp64", kind="gradient", cube=False, cells=22, order=1, precision=0, subs=16,
             tx=8, rx=16),
        # consecutive steps of an inversion with recycling
        dict(name="chamber120k_steps_recycled", kind="steps", cube=False, cells=30, order=1, precision=1, subs=32,
             tx=32, rx=32),
        # five rings merged by the serving loop on its 200k-tet mesh
        dict(name="chamber208k_forward_160", kind="forward", cube=False, cells=36, order=1, precision=1, subs=64,
             tx=160, rx=160),
        # the nodal parameter of the full objective, an odd number of transmitters
        dict(name="chamber208k_kappa_odd", kind="kappa", cube=False, cells=36, order=1, precision=1, subs=64, tx=31,
             rx=32),
        # second-order elements on the serving loop's 50k-tet mesh
        dict(name="chamber53k_gradient_order2", kind="gradient", cube=False, cells=23, order=2, precision=1, subs=16,
             tx=32, rx=32),
        # the benchmark's gradient step
        dict(name="chamber402k_gradient", kind="gradient", cube=False, cells=45, order=1, precision=1, subs=64, tx=32,
             rx=32),
    ]


def draw(rng):
    """One more call of the same ranges: sizes over their logarithm, what is dear (FP64, second order, many
    transmitters) on the meshes where a user can afford it."""
    kind = rng.choice(["forward", "forward", "gradient", "gradient", "kappa", "steps"])
    precision = rng.choice([1, 1, 1, 0])
    order = rng.choice([1, 1, 1, 2]) if kind in ("forward", "gradient") else 1
    cube = rng.random() < 0.25
    if cube:
        cells = rng.randint(4, 8) if order == 2 else rng.randint(5, 14)
    else:
        top = 22 if order == 2 else 44
        if precision == 0:
            top = 12 if order == 2 else 24
        cells = round(math.exp(rng.uniform(math.log(9), math.log(top))))
    tets = _tets(cube, cells)
    most = 160 if kind == "forward" else 32
    if precision == 0:
        most = max(1, min(most, int(8 * 30e3 / tets / (8 if order == 2 else 1))))
    tx = round(math.exp(rng.uniform(0, math.log(min(most, max(1, int(20e6 / tets)))))))
    subs = max(1, min(64, round(tets / rng.uniform(2500, 7000))))
    return dict(kind=kind, cube=cube, cells=cells, order=order, precision=precision, subs=subs, tx=tx,
                rx=rng.choice([4, 8, 16, 32]))


# ---------------------------------------------------------------- inputs
def _tets(cube, cells):
    return 6 * cells ** 3 if cube else round(6 * math.pi / 4 * cells ** 2 * (cells * 14 // 15))


@functools.lru_cache(maxsize=8)
def _grid(cube, cells):
    """xyz, tet and boundary tags: hexes split into six tets around their diagonal, ids and local order shuffled.
    The cube [0, 0.1]^3 has impedance faces all over; the chamber is the cylinder r < 0.15, 0 < z < 0.28 with a
    conducting wall and bottom and an impedance top, its interior vertices jittered."""
    n = np.array([cells, cells, cells if cube else cells * 14 // 15])
    lo, hi = (np.zeros(3), np.full(3, 0.1)) if cube else (np.array([-0.15, -0.15, 0]), np.array([0.15, 0.15, 0.28]))
    ijk = np.stack(np.meshgrid(*[np.arange(v) for v in n], indexing="ij"), axis=-1).reshape(-1, 3)
    h = (hi - lo) / n
    if not cube:
        c = lo + (ijk + 0.5) * h
        ijk = ijk[c[:, 0] ** 2 + c[:, 1] ** 2 < 0.15 ** 2]
    strides = np.array([1, n[0] + 1, (n[0] + 1) * (n[1] + 1)])
    first = ijk @ strides
    tet = np.concatenate([first[:, None] + np.cumsum([0] + [strides[a] for a in p])
                          for p in itertools.permutations(range(3))])
    used, tet = np.unique(tet, return_inverse=True)
    tet = tet.reshape(-1, 4)
    g = np.stack([used % (n[0] + 1), used // (n[0] + 1) % (n[1] + 1), used // strides[2]], axis=1)
    xyz = lo + (hi - lo) * (g / n)
    faces = np.sort(tet[:, [[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]]], axis=2)
    nv = len(used)
    key = (faces[..., 0] * nv + faces[..., 1]) * nv + faces[..., 2]
    _, at, count = np.unique(key.ravel(), return_inverse=True, return_counts=True)
    outer = (count[at] == 1).reshape(-1, 4)
    top = (g[faces, 2] == n[2]).all(axis=2)
    tag = np.where(outer, 2 if cube else np.where(top, 2, 1), 0).astype(np.int32)
    rng = np.random.default_rng(11)
    if not cube:
        inside = np.ones(nv, dtype=bool)
        inside[faces[outer]] = False
        xyz[inside] += rng.uniform(-0.15, 0.15, (int(inside.sum()), 3)) * h.min()
    names, order, local = rng.permutation(nv), rng.permutation(len(tet)), np.argsort(rng.random(tet.shape), axis=1)
    shuffled = np.empty_like(xyz)
    shuffled[names] = xyz
    tet = np.take_along_axis(names[tet], local, axis=1)[order]
    tag = np.take_along_axis(tag, local, axis=1)[order]
    return shuffled, np.ascontiguousarray(tet, dtype=np.int32), np.ascontiguousarray(tag)


@functools.lru_cache(maxsize=8)
def _mesh(cube, cells, order):
    xyz, tet, tag = _grid(cube, cells)
    return mwi.Mesh(xyz, tet, tag, order=order)


def _antennas(cube, cells, n):
    """n +z dipoles: on the lateral faces of the cube, or on up to five rings of 32 in the chamber (further from the
    staircase wall of a coarse one)."""
    a = np.zeros((n, 8))
    ring = 0.135 if cells > 26 else 0.1
    a[:, 5] = a[:, 6] = 1.0
    for k in range(n):
        if cube:
            face, up = k % 4, 0.05 + 0.0125 * (k // 4 % 3 - 1)
            a[k, :3] = [(0, 0.05, up), (0.1, 0.05, up), (0.05, 0, up), (0.05, 0.1, up)][face]
            a[k, face // 2 ^ 1] += 0.0125 * (k // 12 % 4)
        else:
            t = 2 * math.pi * (k % 32) / min(32, n)
            a[k, :3] = ring * math.cos(t), ring * math.sin(t), (0.14, 0.10, 0.18, 0.06, 0.22)[k // 32 % 5]
    return a


def _map(points, cube, rng, inclusions):
    """Gel, the head-sized ellipsoid of the chamber, and spheres of other tissue at random places inside."""
    e = np.full(len(points), GEL)
    axes, centre, r = np.array([0.09, 0.07, 0.10]), np.array([0, 0, 0.14]), 0.015
    if cube:
        axes, centre, r = np.full(3, 0.035), np.full(3, 0.05), 0.02
    else:
        e[(((points - centre) / axes) ** 2).sum(axis=1) < 1] = HEAD
    for value in inclusions:
        d = rng.standard_normal(3)
        c = centre + d / np.linalg.norm(d) * rng.random() ** (1 / 3) * (axes - r)
        e[((points - c) ** 2).sum(axis=1) < r * r] = value
    return e


def _inputs(case, seed):
    """Antennas, the map that was measured, the maps that are tried, the noise of the measurement, the weights."""
    cube, cells = case["cube"], case["cells"]
    xyz, tet, _ = _grid(cube, cells)
    rng = np.random.default_rng([seed, cells, case["tx"]])
    points = xyz if case["kind"] == "kappa" else xyz[tet].mean(axis=1)
    target = _map(points, cube, rng, (BLOOD, LOW))
    tried = _map(points, cube, rng, (BLOOD,))
    tried = [tried, tried * (1 + 0.01 * rng.random())] if case["kind"] == "steps" else [tried]
    tx, rx = (_antennas(cube, cells, case[k]) for k in ("tx", "rx"))
    tx[:, 6] += 0.1 * rng.standard_normal(len(tx))
    xi = rng.standard_normal((2, len(rx), len(tx)))
    noise = 1 + 0.01 * (xi[0] + 1j * xi[1]) / math.sqrt(2)
    weights = rng.uniform(0.5, 2.0, noise.shape) if case["kind"] == "kappa" else None
    return tx, rx, target, tried, noise, weights


ALPHA = 1e-4  # weight of the gradient penalty


class _View:
    """A borrowed device block as an object that torch can look at."""

    def __init__(self, problem, which):
        self.problem = problem  # the view keeps its owner
        p, n, m = problem.fields(which)
        self.__cuda_array_interface__ = dict(shape=(n, m), typestr="<c16", data=(p, False), version=3)


def _fields(problem, which):
    return torch.as_tensor(_View(problem, which), device="cuda")


def prepare(case, seed):
    tx, rx, target, tried, noise, weights = _inputs(case, seed)
    mesh = _mesh(case["cube"], case["cells"], case["order"])
    tried = [torch.from_numpy(e).cuda() for e in tried]
    options = dict(precision=case["precision"], rtol=1e-12 if case["precision"] == 0 else 1e-11, n_sub=case["subs"])
    if case["kind"] == "steps":
        options["recycle"] = 1
    s = dict(kind=case["kind"], tx=tx, rx=rx, tried=tried, weights=weights)
    if case["kind"] == "forward":
        s["problem"] = mwi.Problem(mesh, tried[0], FREQ, **options)
        return s
    if case["kind"] == "kappa":
        s["problem"] = mwi.Problem(mesh, np.full(mesh.nt, GEL), FREQ, **options)
        s["problem"].update_kappa(torch.from_numpy(target).cuda())
    else:
        s["problem"] = mwi.Problem(mesh, torch.from_numpy(target).cuda(), FREQ, **options)
    s["measured"] = s["problem"].forward_solve(tx, rx) * noise
    return s


def run(state):
    P, out = state["problem"], []
    if state["kind"] == "forward":
        return dict(S=P.forward_solve(state["tx"], state["rx"]), U=_fields(P, 0))
    for e in state["tried"]:
        if state["kind"] == "kappa":
            P.update_kappa(e)
            S = P.forward_solve(state["tx"], state["rx"])
            J, R, g = P.misfit_and_gradient_kappa(state["measured"], state["weights"], ALPHA)
            J = J + R
        else:
            P.update_eps(e)
            S = P.forward_solve(state["tx"], state["rx"])
            J, g = P.misfit_and_gradient_device(state["measured"])
        out.append(dict(S=S, J=J, grad=g))
    out[-1].update(U=_fields(P, 0), Lam=_fields(P, 1))
    return out


@functools.lru_cache(maxsize=64)
def _sizes(cube, cells, order):
    """Tets, unknowns and stored entries of the operator (with the removed ones of the wall: a few in a hundred)."""
    _, tet, _ = _grid(cube, cells)
    pairs = np.sort(tet[:, list(itertools.combinations(range(4), 2))].reshape(-1, 2), axis=1).astype(np.int64)
    edges = len(np.unique(pairs[:, 0] << 32 | pairs[:, 1]))
    nt, faces = len(tet), 2 * len(tet)
    # the unknowns of an edge see those of its tets: one tet, 6 x 6; a shared face, 3 x 3 once too often
    if order == 1:
        return nt, edges, 36 * nt - 9 * faces + edges
    return nt, 2 * (edges + faces), 400 * nt - 64 * faces + 4 * edges


def work(case):
    """Per system solved: the operator, its right-hand sides and solutions once, and one product with the operator;
    per step also the maps in and the gradient out."""
    nt, n, nnz = _sizes(case["cube"], case["cells"], case["order"])
    m = case["tx"]
    solves = {"forward": 1, "gradient": 2, "kappa": 2, "steps": 4}[case["kind"]]
    maps = 0 if case["kind"] == "forward" else (2 if case["kind"] == "steps" else 1) * 2 * 16 * nt
    return {"bytes": solves * (20 * nnz + 16 * n * m + 16 * case["rx"] * m) + maps, "flops": solves * 8 * nnz * m}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch
def exact(case, seed):
    """First-order elements only (None otherwise).  The fields come back in the library's own numbering of the
    unknowns and have no value here; S, J and the gradient depend on all of them."""
    if case["order"] != 1:
        return None
    tx, rx, target, tried, noise, weights = _inputs(case, seed)
    fem = _Whitney(case["cube"], case["cells"], tx, rx)
    nodal = case["kind"] == "kappa"
    if case["kind"] == "forward":
        return dict(S=fem.forward(tried[0])[0], U=None)
    measured = fem.forward(target, nodal)[0] * noise
    out = [dict(zip(("S", "J", "grad"), fem.step(e, measured, weights, nodal))) for e in tried]
    out[-1].update(U=None, Lam=None)
    return out


class _Whitney:
    """Lowest-order edge elements on sorted tets: N_ab = l_a grad l_b - l_b grad l_a, a < b; matrices by the integrals
    of products of barycentric coordinates, solves by conjugate orthogonal conjugate gradients (A = A^T)."""

    def __init__(self, cube, cells, tx, rx):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        xyz, tet, tag = _grid(cube, cells)
        by = np.argsort(tet, axis=1)
        self.tet, tag = np.take_along_axis(tet, by, axis=1).astype(np.int64), np.take_along_axis(tag, by, axis=1)
        self.xyz = xyz
        self.k0 = 2 * math.pi * FREQ / 299792458.0
        self.ab = np.array(list(itertools.combinations(range(4), 2)))
        pairs = self.tet[:, self.ab]
        keys, at = np.unique(pairs[..., 0] << 32 | pairs[..., 1], return_inverse=True)
        at = at.reshape(-1, 6)
        wall = np.zeros(len(keys), dtype=bool)
        for k in range(4):
            on = [i for i, (a, b) in enumerate(self.ab) if k not in (a, b)]
            wall[at[tag[:, k] == 1][:, on]] = True
        number = np.full(len(keys), -1)
        number[~wall] = np.arange(int((~wall).sum()))
        self.n = int((~wall).sum())
        self.tx, self.rx = (self._edges(a, keys, number) for a in (tx, rx))
        self.current = tx[:, 6] + 1j * tx[:, 7]
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(self.dev)  # noqa: E731
        self.dof, self.vert = t(number[at]), t(self.tet)
        x = t(xyz)[self.vert]
        d = x[:, 1:] - x[:, :1]
        self.vol = torch.linalg.det(d).abs() / 6
        g = torch.linalg.inv(d).transpose(1, 2)
        self.g = torch.cat([-g.sum(1, keepdim=True), g], 1)
        two, three = np.ones((4, 4)) + np.eye(4), np.zeros((4, 4, 4))
        for i in itertools.product(range(4), repeat=3):
            three[i] = math.prod(math.factorial(i.count(v)) for v in set(i))
        curl = 2 * torch.linalg.cross(self.g[:, self.ab[:, 0]], self.g[:, self.ab[:, 1]])
        self.K = self.vol[:, None, None] * curl @ curl.transpose(1, 2)
        self.M = self._mass(t(two / 20), self.g) * self.vol[:, None, None]
        self.Mw = [self._mass(t(three[w] / 120), self.g) * self.vol[:, None, None] for w in range(4)]
        owners, mats = [], []
        for k in range(4):
            own = np.nonzero(tag[:, k] == 2)[0]
            i = t(own)
            gk = self.g[i, k]
            nrm = gk / gk.norm(dim=1, keepdim=True)
            tang = self.g[i] - (self.g[i] * nrm[:, None]).sum(2, keepdim=True) * nrm[:, None]
            flat = two.copy() / 12
            flat[k, :] = flat[:, k] = 0
            owners.append(i)
            mats.append(self._mass(t(flat), tang) * (3 * self.vol[i] * gk.norm(dim=1))[:, None, None])
        self.own, self.B = torch.cat(owners), torch.cat(mats)

    def _edges(self, ants, keys, number):
        dof, sign = [], []
        lo, hi = keys >> 32, keys & 0xFFFFFFFF
        for row in ants:
            v = int(np.argmin(((self.xyz - row[:3]) ** 2).sum(axis=1)))
            at = np.nonzero((lo == v) | (hi == v))[0]
            vec = self.xyz[lo[at] + hi[at] - v] - self.xyz[v]
            e = at[np.argmax(vec @ row[3:6] / np.linalg.norm(vec, axis=1))]
            dof.append(number[e])
            sign.append(1.0 if (self.xyz[hi[e]] - self.xyz[lo[e]]) @ row[3:6] > 0 else -1.0)
        return np.array(dof), np.array(sign)

    def _mass(self, moments, g):
        """int N_ab . N_cd (per unit measure) for the moments of l_a l_c and gradients g [tets, 4, 3]."""
        G = g @ g.transpose(1, 2)
        (a, b), q = self.ab.T, lambda i, j, k, l: moments[i][:, j] * G[:, k][:, :, l]  # noqa: E741
        return q(a, a, b, b) - q(a, b, b, a) - q(b, a, a, b) + q(b, b, a, a)

    def _operator(self, eps, nodal):
        e = torch.from_numpy(eps).to(self.dev)
        if nodal:
            kv = e[self.vert]
            vol = sum(kv[:, w, None, None] * self.Mw[w] for w in range(4))
            e = kv.mean(1)
        else:
            vol = e[:, None, None] * self.M
        vals = self.K - self.k0 ** 2 * vol
        vals.index_add_(0, self.own, 1j * self.k0 * e[self.own].sqrt()[:, None, None] * self.B)
        r, c = self.dof[:, :, None].expand(-1, 6, 6), self.dof[:, None, :].expand(-1, 6, 6)
        keep = (r >= 0) & (c >= 0)
        A = torch.sparse_coo_tensor(torch.stack([r[keep], c[keep]]), vals[keep], (self.n, self.n)).coalesce()
        return A.to_sparse_csr(), e

    def _solve(self, A, b):
        i = A.crow_indices()
        rows = torch.repeat_interleave(torch.arange(self.n, device=self.dev), i[1:] - i[:-1])
        on = rows == A.col_indices()
        scale = A.values()[on][:, None]
        x, r = torch.zeros_like(b), b.clone()
        z = r / scale
        p, rho, end = z.clone(), (r * z).sum(0), 1e-14 * b.norm(dim=0)
        for k in range(4000):
            q = A @ p
            alpha = rho / (p * q).sum(0)
            alpha[torch.isnan(alpha.real)] = 0
            x += alpha * p
            r -= alpha * q
            if k % 10 == 9 and bool((r.norm(dim=0) <= end).all()):
                break
            z = r / scale
            new = (r * z).sum(0)
            beta = new / rho
            beta[torch.isnan(beta.real)] = 0
            rho, p = new, z + beta * p
        return x

    def _sources(self, edges, values):
        b = torch.zeros((self.n, values.shape[1]), dtype=torch.complex128, device=self.dev)
        b.index_add_(0, torch.from_numpy(edges[0]).to(self.dev),
                     torch.from_numpy(edges[1][:, None] * values).to(self.dev))
        return b

    def forward(self, eps, nodal=False):
        A, e = self._operator(eps, nodal)
        s = -1j * 2 * math.pi * FREQ * 4e-7 * math.pi
        U = self._solve(A, self._sources(self.tx, np.diag(s * self.current)))
        S = (U[torch.from_numpy(self.rx[0]).to(self.dev)].cpu().numpy() * self.rx[1][:, None]).conj()
        return S, U, A, e

    def step(self, eps, measured, weights, nodal):
        S, U, A, e = self.forward(eps, nodal)
        res = S - measured
        w = np.ones(res.shape) if weights is None else weights
        J = 0.5 * float((w * abs(res) ** 2).sum())
        L = self._solve(A, self._sources(self.rx, w * res))
        on = (self.dof >= 0)[:, :, None]
        G = torch.zeros((len(self.tet), 4 if nodal else 1), dtype=torch.complex128, device=self.dev)
        edge = torch.zeros(len(self.own), dtype=torch.complex128, device=self.dev)
        for c in range(U.shape[1]):
            u, v = (torch.where(on[..., 0], X[self.dof, c], 0) for X in (U, L))
            for j, M in enumerate(self.Mw if nodal else [self.M]):
                G[:, j] += self.k0 ** 2 * (v[:, None] @ (M + 0j) @ u[:, :, None])[:, 0, 0]
            edge += (v[self.own][:, None] @ (self.B + 0j) @ u[self.own][:, :, None])[:, 0, 0]
        edge *= -1j * self.k0 / (2 * e[self.own].sqrt())
        G.index_add_(0, self.own, edge[:, None].expand(-1, G.shape[1]) / G.shape[1])
        if not nodal:
            return S, J, G[:, 0].conj().resolve_conj()
        kappa = torch.from_numpy(eps).to(self.dev)
        grad = torch.zeros_like(kappa).index_add_(0, self.vert.reshape(-1), G.conj().resolve_conj().reshape(-1))
        stiff = (self.vol[:, None, None] * self.g @ self.g.transpose(1, 2)) @ kappa[self.vert][:, :, None].real \
            + 1j * ((self.vol[:, None, None] * self.g @ self.g.transpose(1, 2)) @ kappa[self.vert][:, :, None].imag)
        Kk = torch.zeros_like(kappa).index_add_(0, self.vert.reshape(-1), stiff.reshape(-1))
        R = 0.5 * ALPHA * float((kappa.conj() * Kk).sum().real)
        return S, J + R, grad + ALPHA * Kk
