"""GPU: kernels and dispatch branches at the sizes where they can go wrong (tile edges, remainders,
partly filled groups), against the oracle or an exact identity."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1303_1377_gb300 import synth  # noqa: E402


def _solver(dims, **kw):
    from paper_1303_1377_gb300 import ddamg

    U = synth.gauge_field(dims, 0.4, seed=5)
    return ddamg.Solver(dims, U, -0.4, 1.0, ddamg.default_params(**kw), setup=False), U


@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((8, 4, 4, 12), (4, 2, 2, 2)), ((8, 8, 16, 24), (4, 4, 4, 4))])
def test_layout_round_trip_is_exact(dims, block):
    """ABI -> internal -> ABI permutes FP64 fields without changing a bit."""
    from paper_1303_1377_gb300 import ddamg

    s, _ = _solver(dims, n_vec=4, block=block, precision=ddamg.PREC_DOUBLE)
    with s:
        v = synth.random_test_vectors(dims, 4, seed=3)
        s.setup_from_vectors(v)
        assert np.array_equal(s.vectors(), v)


@pytest.mark.parametrize("prec,tol", [("single", 1e-6), ("half", 2e-3)])
@pytest.mark.parametrize("dims,nrhs,mr", [((8, 8, 8, 8), 1, 4), ((8, 8, 8, 8), 3, 1), ((16, 8, 8, 8), 2, 0), ((8, 8, 16, 8), 5, 4)])
def test_sap_on_4x4x4x4_blocks_by_right_hand_sides(prec, tol, dims, nrhs, mr):
    """Pairs of right-hand sides: one, an odd last one, full pairs; the stated FP32 / FP16-storage bounds."""
    from oracle.dirac import DiracOperator
    from oracle.sap import SAP
    from paper_1303_1377_gb300 import ddamg

    s, U = _solver(dims, n_vec=4, precision={"single": ddamg.PREC_SINGLE, "half": ddamg.PREC_HALF}[prec], mr_steps=mr)
    with s:
        b = synth.gaussian_spinors(dims, nrhs, seed=21)
        got = s.apply_sap(b, 2)
    sap = SAP(DiracOperator(U, dims, -0.4, 1.0), (4, 4, 4, 4), mr_steps=mr)
    ref = np.stack([sap.apply(b[r], 2) for r in range(nrhs)])
    for r in range(nrhs):
        assert np.max(np.abs(got[r] - ref[r])) < tol * np.max(np.abs(ref[r]))
