"""The one-launch tensor-core sweeps (sweep_engine 4): what their tiles hand to
each other inside the launch, their rounding, and their bounded waits.
"""

import numpy as np
import pytest

from synthetic import antenna_array, ring_antennas
from tests._helpers import FREQ, chamber_case, cube_case, rel_err

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
    return lib.Mesh(mesh.xyz, mesh.tet, mesh.bface_tag), eps


def _block(n, m, seed):
    rng = np.random.default_rng(seed)
    return torch.from_numpy(rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m))).cuda()


@pytest.mark.parametrize("n_sub,leaf,m", [(1, 9, 68), (7, 33, 96), (7, 128, 31)])
def test_repeated_applications_agree_bit_for_bit(lib, chamber, n_sub, leaf, m):
    """A tile reads rows that other tiles of the launch have just written; the
    sums have a fixed order, so a read that came too early would show as a
    difference between applications.  Deep trees, one to three column chunks;
    every chunk also as a block of its own."""
    M, eps = chamber
    P = lib.Problem(M, eps, FREQ, n_sub=n_sub, precision=1, nd_leaf=leaf)
    X = _block(M.ndof, m, 5)
    ref = P.oras_apply(X).cpu()
    assert torch.isfinite(torch.view_as_real(ref)).all()
    for _ in range(12):
        assert torch.equal(P.oras_apply(X).cpu(), ref)
    for c in range(0, m, 32):
        assert torch.equal(P.oras_apply(X[:, c:c + 32].contiguous()).cpu(), ref[:, c:c + 32])
    P.close()


def test_an_expired_wait_is_reported_and_the_problem_stays_usable(lib, chamber):
    """No looks at the dependencies' counts: every tile that depends on another
    one gives up at once, the launch returns, the host reads the status, and the
    next call with the default limit gives the earlier result bit for bit."""
    M, eps = chamber
    P = lib.Problem(M, eps, FREQ, n_sub=7, precision=1, rtol=1e-9, max_iter=60)
    ants = antenna_array(ring_antennas(5, radius=0.1))
    X = _block(M.ndof, 40, 6)
    ref, S = P.oras_apply(X).cpu(), P.forward_solve(ants, ants)
    for _ in range(2):
        P.set_sweep_polls(0)
        for call in (lambda: P.oras_apply(X), lambda: P.forward_solve(ants, ants)):
            with pytest.raises(lib.MwiError) as err:
                call()
            assert err.value.status == lib.MWI_ETIMEOUT
        P.set_sweep_polls(-1)
        assert torch.equal(P.oras_apply(X).cpu(), ref)
        assert np.array_equal(P.forward_solve(ants, ants), S)
    P.close()


def test_a_failed_solve_leaves_no_fields_behind(lib, chamber):
    """A forward solve that gives up has overwritten the fields of the one
    before: asking for a gradient of them is a call out of order, and the next
    solve is not recycled from them."""
    M, eps = chamber
    P = lib.Problem(M, eps, FREQ, n_sub=7, precision=1, rtol=1e-9, max_iter=60, recycle=1)
    ants = antenna_array(ring_antennas(5, radius=0.1))
    S = P.forward_solve(ants, ants)
    P.misfit_and_gradient(S * 1.1)
    P.set_sweep_polls(0)
    with pytest.raises(lib.MwiError) as err:
        P.forward_solve(ants, ants)
    assert err.value.status == lib.MWI_ETIMEOUT
    P.set_sweep_polls(-1)
    for call in (lambda: P.misfit_and_gradient(S * 1.1), lambda: P.fields(0), lambda: P.fields(1)):
        with pytest.raises(lib.MwiError) as err:
            call()
        assert err.value.status == lib.MWI_ESTATE
    assert np.array_equal(P.forward_solve(ants, ants), S)
    P.close()


@pytest.mark.parametrize("leaf", [10 ** 6, 16])
def test_operands_are_rounded_to_nearest(lib, leaf):
    """Where the forward sweep's operands are TF32 values already, the engine
    rounds what engine 2 (mma.sync) rounds, both to nearest, so their errors
    against FP64 are the same up to FP32 summation: right-hand sides of 8-bit
    integers on the root front alone -- one front over all rows, and a tree of
    small fronts, whose backward products then read the ancestors' rows.  An
    operand truncated instead has four times the mean square error (a factor
    of sqrt((1 + 4) / 2) = 1.58 with one of a product's two): the bound of 1.25
    lies between."""
    mesh, eps, _, _ = cube_case(6)
    M = lib.Mesh(mesh.xyz, mesh.tet, mesh.bface_tag)
    info = lib.fronts_host(mesh, 1, nd_leaf=leaf)["info"]
    l2g = lib.decomposition_host(mesh, 1, nd_leaf=leaf)["loc2glob"]
    root = [r for _, start, p, _, parent in info if parent < 0 for r in range(start, start + p)]
    rng = np.random.default_rng(8)
    X = np.zeros((M.ndof, 64), dtype=np.complex128)
    X[l2g[root]] = (rng.integers(-127, 128, (len(root), 64)) + 1j * rng.integers(-127, 128, (len(root), 64)))
    out = {}
    for engine, precision in ((0, 0), (2, 1), (4, 1)):
        P = lib.Problem(M, eps, FREQ, n_sub=1, precision=precision, sweep_engine=engine, nd_leaf=leaf)
        out[engine] = P.oras_apply(torch.from_numpy(X).cuda()).cpu().numpy()
        P.close()
    assert 0 < rel_err(out[4], out[0]) <= 1.25 * rel_err(out[2], out[0])


def test_a_failed_adjoint_solve_leaves_no_adjoint_fields_behind(lib, chamber):
    M, eps = chamber
    P = lib.Problem(M, eps, FREQ, n_sub=7, precision=1, rtol=1e-9, max_iter=60)
    ants = antenna_array(ring_antennas(5, radius=0.1))
    S_meas = P.forward_solve(ants, ants) * 1.1
    J, grad = P.misfit_and_gradient(S_meas)
    P.set_sweep_polls(0)
    with pytest.raises(lib.MwiError) as err:
        P.misfit_and_gradient(S_meas)
    assert err.value.status == lib.MWI_ETIMEOUT
    P.set_sweep_polls(-1)
    with pytest.raises(lib.MwiError) as err:
        P.fields(1)
    assert err.value.status == lib.MWI_ESTATE
    P.fields(0)  # the forward fields are still there, and the gradient can be asked for again
    J2, grad2 = P.misfit_and_gradient(S_meas)
    assert J2 == J and np.array_equal(grad2, grad)
    P.close()
