"""The kernels' edges: column counts around the widths that pick another kernel
or leave a ragged chunk, trees from many tiny fronts to one large one, Krylov
bases longer than a warp, and columns that are not finite.

Tolerances are those of tests/test_gpu_parity.py: one ORAS application FP64
<= 1e-10, TF32 tensor-core sweeps <= 1e-2; solved fields FP64 (rtol 1e-12) <= 1e-8,
mixed (rtol 1e-9) <= 1e-6.  A column's operations do not depend on the width of
the block it is solved in, so those comparisons are bit for bit.
"""

import numpy as np
import pytest

import oracle as O
from oracle import dd
from synthetic import antenna_array, ring_antennas
from tests._helpers import FREQ, chamber_case, col_rel_err, cube_case, key_perm, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1607_02573_gb300 import mwi
    return mwi


@pytest.fixture(scope="module")
def chamber(lib):
    mesh, eps, _, _ = chamber_case(12, 11)
    M = lib.Mesh(mesh.xyz, mesh.tet, mesh.bface_tag)
    topo = O.build_topology(mesh.tet, mesh.bface_tag, mesh.nv, 1)
    kind, verts = M.dof_keys()
    return mesh, eps, M, topo, key_perm(kind, verts, topo)


_ORAS = {}


def _oracle_apply(chamber, n_sub, X):
    mesh, eps, M, topo, perm = chamber
    if n_sub not in _ORAS:
        part = dd.rcb_partition(mesh.xyz, mesh.tet, n_sub)
        dec = dd.Decomposition(mesh.xyz, mesh.tet, topo, part, 1)
        _ORAS[n_sub] = part, dd.ORAS(dec, dd.local_matrices(mesh.xyz, topo, dec, eps, FREQ))
    part, oras = _ORAS[n_sub]
    return part, oras.apply(X[np.argsort(perm)])[perm]


@pytest.mark.parametrize("n_sub,leaf", [(1, 9), (1, 300), (7, 33), (7, 128)])
@pytest.mark.parametrize("precision,widths,tol", [(0, (1, 2, 3, 8, 9, 17), 1e-10), (1, (1, 2, 5, 31, 34, 68), 1e-2)])
def test_oras_over_trees_and_widths(lib, chamber, precision, widths, tol, n_sub, leaf):
    """Fronts of a few pivots in a deep tree, fronts beyond one 128-row tile and one
    64-row factorisation tile, odd and ragged column counts."""
    mesh, eps, M, topo, perm = chamber
    rng = np.random.default_rng(3)
    X = rng.standard_normal((M.ndof, 68)) + 1j * rng.standard_normal((M.ndof, 68))
    part, ref = _oracle_apply(chamber, n_sub, X)
    P = lib.Problem(M, eps, FREQ, n_sub=n_sub, part=part, precision=precision, nd_leaf=leaf)
    for m in widths:
        Y = P.oras_apply(torch.from_numpy(X[:, :m].copy()).cuda()).cpu().numpy()
        assert rel_err(Y, ref[:, :m]) <= tol, m
    P.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_columns_that_are_not_finite_stay_alone(lib, chamber, precision):
    """NaN and infinity in some columns leave the others bit for bit as they are, in
    both column chunks, and nothing of them is left for the next call."""
    mesh, eps, M, topo, perm = chamber
    P = lib.Problem(M, eps, FREQ, n_sub=7, precision=precision)
    rng = np.random.default_rng(4)
    X = rng.standard_normal((M.ndof, 40)) + 1j * rng.standard_normal((M.ndof, 40))
    ref = P.oras_apply(torch.from_numpy(X).cuda()).cpu().numpy()
    bad = X.copy()
    bad[:, 3] = np.nan
    bad[::7, 35] = np.inf
    got = P.oras_apply(torch.from_numpy(bad).cuda()).cpu().numpy()
    keep = [c for c in range(40) if c not in (3, 35)]
    assert np.array_equal(got[:, keep], ref[:, keep])
    assert not np.isfinite(got[:, 3]).any() and not np.isfinite(got[:, 35]).all()
    assert np.array_equal(P.oras_apply(torch.from_numpy(X).cuda()).cpu().numpy(), ref)
    P.close()


@pytest.mark.parametrize("precision,widths", [(0, (1, 2, 9)), (1, (2, 5, 7, 13, 17, 31, 33))])
def test_solves_do_not_depend_on_the_block_width(lib, chamber, precision, widths):
    mesh, eps, M, topo, perm = chamber
    ants = antenna_array(ring_antennas(40, radius=0.1))
    ref = None
    for mb in (40,) + widths:
        P = lib.Problem(M, eps, FREQ, n_sub=7, precision=precision, rtol=1e-9, max_block=mb)
        S = P.forward_solve(ants, ants[:8])
        U = P.fields_host(0)
        P.close()
        ref = ref or (S, U)
        assert np.array_equal(S, ref[0]) and np.array_equal(U, ref[1]), mb


@pytest.mark.parametrize("precision,rtol,tol", [(0, 1e-12, 1e-8), (1, 1e-9, 1e-6)])
@pytest.mark.parametrize("cells,restart,least", [(8, 400, 150), (5, 3100, 1)])
def test_long_krylov_bases(lib, precision, rtol, tol, cells, restart, least):
    """More steps than a warp has lanes in one cycle (a nearly lossless medium over
    many subdomains without overlap: the oracle's FGMRES is at 5e-6 after 150
    steps), and a restart length whose back substitution does not fit in shared
    memory."""
    mesh, eps, tx, rx = cube_case(cells)
    if least > 1:
        eps = np.full(mesh.nt, 30 - 0.3j)
    M = lib.Mesh(mesh.xyz, mesh.tet, mesh.bface_tag)
    topo = O.build_topology(mesh.tet, mesh.bface_tag, mesh.nv, 1)
    perm = key_perm(*M.dof_keys(), topo)
    P = lib.Problem(M, eps, FREQ, n_sub=24 if least > 1 else 4, overlap=-1 if least > 1 else 1, precision=precision,
                    rtol=rtol, restart=restart, max_iter=4000)
    S = P.forward_solve(tx, rx)
    info = P.info.as_dict()
    ref = O.forward(mesh.xyz, topo, eps, FREQ, tx, rx)
    assert info["iters_max"] >= least, info
    assert col_rel_err(P.fields_host(0), ref["U"][perm]).max() <= tol
    assert rel_err(S, ref["S"]) <= tol
    P.close()
    M.close()
