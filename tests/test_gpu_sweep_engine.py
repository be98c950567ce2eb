"""The one-launch tensor-core sweeps (sweep_engine 4): what their tiles hand to
each other inside the launch, their rounding, and their bounded waits.
"""

import numpy as np
import pytest

from synthetic import antenna_array, ring_antennas
from tests._helpers import FREQ, chamber_case

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
