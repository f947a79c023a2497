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
