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


@pytest.mark.parametrize("n_vec", [8, 12, 20])
def test_level1_sap_on_tensor_cores(n_vec):
    """The half-precision level-1 SAP (FP16 D_1 and D_ee^{-1}, split right-hand sides) against the
    oracle's SAP on the operator rounded as stored: a product errs by about 2^-22 (split) +
    sqrt(9 * 2N) 2^-24 (FP32 accumulation) <= 1.4e-6 of the field maximum, and two iterations with MR(4)
    amplify a rounding error by less than 10, so 1e-5 is asserted.  Every right-hand side is
    independent of its group: full, partial and many-group batches agree bit for bit."""
    from oracle.lattice import Lattice
    from oracle.multilevel import StencilOperator, StencilSAP
    from paper_1303_1377_gb300 import ddamg

    dims, blk = (8, 8, 8, 8), (2, 2, 2, 2)
    s, _ = _solver(dims, n_vec=n_vec, block=blk, precision=ddamg.PREC_HALF)
    with s:
        s.setup_from_vectors(synth.random_test_vectors(dims, n_vec, seed=31))
        s.ml_build(synth.gaussian_coarse(256, 2 * n_vec, 3, seed=32), ddamg.ml_default_params(n_vec1=3))
        B = s.coarse_stencil()
        x = synth.gaussian_coarse(256, 2 * n_vec, 77, seed=33)
        all77 = s.ml_apply_sap1(x, 2)
        for a, b in ((0, 1), (1, 6), (6, 18)):
            assert np.array_equal(s.ml_apply_sap1(x[a:b], 2), all77[a:b])

    def r16(v):
        return v.real.astype(np.float32).astype(np.float16) + 1j * v.imag.astype(np.float32).astype(np.float16).astype(np.float64)

    op = StencilOperator(Lattice((4, 4, 4, 4)), r16(B))
    sap = StencilSAP(op, (2, 2, 2, 2), mr_steps=4)
    inv = r16(np.linalg.inv(B[:, 0]))
    sap.apply_Aee_inv = lambda f: np.einsum("xij,xj->xi", inv, f)
    for r in (0, 41):
        ref = sap.apply(x[r], 2)
        assert np.max(np.abs(all77[r] - ref)) < 1e-5 * np.max(np.abs(ref))


@pytest.mark.parametrize("dims,nrhs", [((8, 8, 8, 8), 1), ((8, 8, 8, 8), 2), ((8, 16, 8, 8), 3), ((8, 8, 8, 16), 13)])
def test_fp32_dslash_by_right_hand_sides_and_alignment(dims, nrhs):
    """FP32 D on 4^4 blocks: one field, pairs, an odd last one, more than one CTA row of pairs, against the
    oracle at the stated 1e-6; an output that is only 8-byte aligned takes the other route and gives the
    same bits."""
    import ctypes as C

    import torch

    from oracle.dirac import DiracOperator
    from paper_1303_1377_gb300 import ddamg

    s, U = _solver(dims, n_vec=4, precision=ddamg.PREC_SINGLE)
    with s:
        x = synth.gaussian_spinors(dims, nrhs, seed=41).astype(np.complex64)
        xt = torch.from_numpy(x).cuda()
        got = s.apply_D_f32(xt)
        buf = torch.zeros(got.numel() + 1, dtype=torch.complex64, device="cuda")
        torch.cuda.synchronize()
        assert ddamg.lib.ddamg_apply_D_f32(s.h, C.c_void_p(xt.data_ptr()), C.c_void_p(buf.data_ptr() + 8), nrhs) == 0
        assert torch.equal(torch.view_as_real(buf[1:]).flatten(), torch.view_as_real(got).flatten())
    D = DiracOperator(U, dims, -0.4, 1.0)
    for r in range(nrhs):
        ref = D.apply(x[r].astype(np.complex128))
        assert np.max(np.abs(got[r].cpu().numpy() - ref)) < 1e-6 * np.max(np.abs(ref))


@pytest.mark.parametrize("dims,block,nrhs", [((8, 8, 8, 8), (4, 4, 4, 4), 1), ((8, 4, 4, 12), (4, 2, 2, 2), 2), ((8, 8, 8, 16), (4, 4, 4, 4), 9)])
def test_double_word_dslash_by_right_hand_sides(dims, block, nrhs):
    """D in double-word arithmetic, one field and pairs (odd and even batches): the stated 1e-13 against the
    oracle's FP64."""
    from oracle.dirac import DiracOperator
    from paper_1303_1377_gb300 import ddamg

    s, U = _solver(dims, n_vec=4, block=block, precision=ddamg.PREC_SINGLE)
    with s:
        x = synth.gaussian_spinors(dims, nrhs, seed=51).astype(np.complex64)
        got = s.apply_D_mixed(x)
    D = DiracOperator(U, dims, -0.4, 1.0)
    for r in range(nrhs):
        ref = D.apply(x[r].astype(np.complex128))
        assert np.max(np.abs(got[r] - ref)) < 1e-13 * np.max(np.abs(ref))


@pytest.mark.parametrize("dims,block,n_vec,nrhs,steps", [((4, 4, 4, 4), (2, 2, 2, 2), 1, 3, 5), ((4, 4, 4, 8), (2, 2, 2, 2), 3, 1, 9),
                                                         ((8, 8, 8, 16), (2, 2, 2, 4), 5, 13, 35), ((16, 16, 16, 8), (2, 2, 2, 2), 10, 2, 12)])
def test_coarse_gmres_steps_by_vector_length(dims, block, n_vec, nrhs, steps):
    """A fixed number of FP32 coarse GMRES steps on vectors of 16 to 20480 numbers (slices with idle CTAs, a
    ragged last slice, a restart, and beyond the one-kernel step) against FP64 steps on the same operator, to
    the stated 1e-6.  Random test vectors keep the coarse operator well conditioned."""
    from paper_1303_1377_gb300 import ddamg

    v = synth.random_test_vectors(dims, n_vec, seed=61)
    out = {}
    for prec in ("DOUBLE", "SINGLE"):
        s, _ = _solver(dims, n_vec=n_vec, block=block, precision=getattr(ddamg, "PREC_" + prec))
        with s:
            s.setup_from_vectors(v)
            e = synth.gaussian_coarse(s.n_coarse, s.coarse_dof, nrhs, seed=62)
            out[prec] = s.coarse_solve(e, steps)
    for r in range(nrhs):
        assert np.max(np.abs(out["SINGLE"][r] - out["DOUBLE"][r])) < 1e-6 * np.max(np.abs(out["DOUBLE"][r]))


@pytest.mark.parametrize("dims,n_vec,nrhs", [((8, 8, 8, 8), 4, 1), ((8, 8, 16, 8), 12, 17), ((16, 8, 8, 24), 20, 5)])
def test_half_restriction_of_fields_of_very_different_size(dims, n_vec, nrhs):
    """P^H on half-precision handles scales every field by its own maximum: fields from 1e-30 to 1e30 and a zero
    field, each to the stated 4e-3 of its own result's maximum."""
    from oracle.aggregation import Aggregation
    from oracle.dirac import DiracOperator
    from paper_1303_1377_gb300 import ddamg

    s, U = _solver(dims, n_vec=n_vec, precision=ddamg.PREC_HALF)
    v = synth.random_test_vectors(dims, n_vec, seed=71)
    x = synth.gaussian_spinors(dims, nrhs, seed=72)
    x *= 10.0 ** np.linspace(-30, 30, nrhs)[:, None, None, None]
    x[nrhs // 2] = 0
    with s:
        s.setup_from_vectors(v)
        got = s.restrict(x)
    agg = Aggregation(DiracOperator(U, dims, -0.4, 1.0).lat, (4, 4, 4, 4), v)
    for r in range(nrhs):
        ref = agg.restrict(x[r])
        assert np.max(np.abs(got[r] - ref)) <= 4e-3 * np.max(np.abs(ref))


@pytest.mark.parametrize("prec,tol", [("single", 1e-6), ("half", 2e-3)])
@pytest.mark.parametrize("nrhs", [2, 3])
def test_sap_on_both_sides_of_the_line_between_its_kernels(prec, tol, nrhs):
    """16^4 has 128 blocks per colour: two and three fields lie on either side of the line between one field per
    CTA and pairs of fields.  The first and the last field against the oracle, at the stated bounds."""
    from oracle.dirac import DiracOperator
    from oracle.sap import SAP
    from paper_1303_1377_gb300 import ddamg

    dims = (16, 16, 16, 16)
    s, U = _solver(dims, n_vec=4, precision={"single": ddamg.PREC_SINGLE, "half": ddamg.PREC_HALF}[prec], mr_steps=2)
    with s:
        b = synth.gaussian_spinors(dims, nrhs, seed=25)
        got = s.apply_sap(b, 1)
    sap = SAP(DiracOperator(U, dims, -0.4, 1.0), (4, 4, 4, 4), mr_steps=2)
    for r in (0, nrhs - 1):
        ref = sap.apply(b[r], 1)
        assert np.max(np.abs(got[r] - ref)) < tol * np.max(np.abs(ref))


@pytest.mark.parametrize("prec,tol", [("DOUBLE", 1e-13), ("SINGLE", 1e-6)])
@pytest.mark.parametrize("dims,block,n_vec,nrhs", [((4, 4, 4, 4), (2, 2, 2, 2), 1, 1), ((8, 8, 8, 8), (4, 4, 4, 4), 3, 3),
                                                   ((16, 8, 8, 8), (2, 2, 4, 4), 7, 1), ((16, 16, 16, 16), (2, 4, 4, 4), 2, 5)])
def test_transfers_with_shared_aggregates(prec, tol, dims, block, n_vec, nrhs):
    """P^H and P with several CTAs per aggregate (few aggregates, fewer vectors than CTAs) and with one, odd and
    even batches, against the oracle at the stated bounds."""
    from oracle.aggregation import Aggregation
    from oracle.dirac import DiracOperator
    from paper_1303_1377_gb300 import ddamg

    s, U = _solver(dims, n_vec=n_vec, block=block, precision=getattr(ddamg, "PREC_" + prec))
    v = synth.random_test_vectors(dims, n_vec, seed=81)
    x = synth.gaussian_spinors(dims, nrhs, seed=82)
    agg = Aggregation(DiracOperator(U, dims, -0.4, 1.0).lat, block, v)
    with s:
        s.setup_from_vectors(v)
        e = synth.gaussian_coarse(s.n_coarse, s.coarse_dof, nrhs, seed=83)
        c, f = s.restrict(x), s.prolong(e)
    for r in range(nrhs):
        for got, ref in ((c[r], agg.restrict(x[r])), (f[r], agg.prolong(e[r]))):
            assert np.max(np.abs(got - ref)) < tol * np.max(np.abs(ref))


@pytest.mark.parametrize("dims,block,n_vec,nrhs", [((4, 4, 4, 4), (2, 2, 2, 2), 4, 3), ((8, 4, 4, 12), (4, 2, 2, 2), 8, 1),
                                                   ((8, 8, 16, 8), (4, 4, 4, 4), 20, 17)])
def test_half_prolongation_by_block_and_right_hand_sides(dims, block, n_vec, nrhs):
    """P on half-precision handles: blocks of 16 sites (result through the internal layout), of 32 and of 256 sites
    (written in the caller's layout), one field and a second launch of five, fields from 1e-30 to 1e30, each to the
    stated 4e-3 of its own result's maximum."""
    from oracle.aggregation import Aggregation
    from oracle.dirac import DiracOperator
    from paper_1303_1377_gb300 import ddamg

    s, U = _solver(dims, block=block, n_vec=n_vec, precision=ddamg.PREC_HALF)
    v = synth.random_test_vectors(dims, n_vec, seed=73)
    agg = Aggregation(DiracOperator(U, dims, -0.4, 1.0).lat, block, v)
    rng = np.random.default_rng(74)
    nb = int(np.prod(dims)) // int(np.prod(block))
    e = rng.standard_normal((nrhs, nb, 2 * n_vec)) + 1j * rng.standard_normal((nrhs, nb, 2 * n_vec))
    e *= 10.0 ** np.linspace(-30, 30, nrhs)[:, None, None]
    with s:
        s.setup_from_vectors(v)
        got = s.prolong(e)
    for r in range(nrhs):
        ref = agg.prolong(e[r])
        assert np.max(np.abs(np.reshape(got[r], ref.shape) - ref)) <= 4e-3 * np.max(np.abs(ref))


@pytest.mark.parametrize("dims,n_vec,block1,mr", [((8, 8, 8, 8), 8, (2, 2, 2, 2), 4), ((8, 8, 8, 8), 16, (2, 2, 2, 2), 1),
                                                  ((8, 8, 8, 8), 20, (2, 2, 2, 2), 4), ((8, 8, 8, 8), 24, (2, 2, 2, 1), 4),
                                                  ((8, 8, 8, 16), 8, (2, 2, 2, 4), 0)])
def test_level1_sap_of_fields_of_very_different_size(dims, n_vec, block1, mr):
    """The half-precision level-1 SAP is homogeneous in its right-hand side: fields from 1e-30 to 1e30, a zero
    field and a field that is tiny on all sites but one, each to the 1e-5 of its own result's maximum that
    test_level1_sap_on_tensor_cores derives; level-1 blocks of 8, 16 and 32 sites, 0, 1 and 4 MR steps."""
    from oracle.lattice import Lattice
    from oracle.multilevel import StencilOperator, StencilSAP
    from paper_1303_1377_gb300 import ddamg

    l1 = tuple(d // 2 for d in dims)
    nb = int(np.prod(l1))
    s, _ = _solver(dims, n_vec=n_vec, block=(2, 2, 2, 2), precision=ddamg.PREC_HALF)
    x = synth.gaussian_coarse(nb, 2 * n_vec, 7, seed=35)
    x[:5] *= 10.0 ** np.array([-30, -12, 6, 20, 30])[:, None, None]
    x[5] = 0
    x[6, 1:] *= 1e-12
    with s:
        s.setup_from_vectors(synth.random_test_vectors(dims, n_vec, seed=31))
        s.ml_build(synth.gaussian_coarse(nb, 2 * n_vec, 3, seed=32), ddamg.ml_default_params(n_vec1=3, block1=block1, mr_steps1=mr))
        B = s.coarse_stencil()
        got = s.ml_apply_sap1(x, 2)

    def r16(v):
        return v.real.astype(np.float32).astype(np.float16) + 1j * v.imag.astype(np.float32).astype(np.float16).astype(np.float64)

    sap = StencilSAP(StencilOperator(Lattice(l1), r16(B)), block1, mr_steps=mr)
    inv = r16(np.linalg.inv(B[:, 0]))
    sap.apply_Aee_inv = lambda f: np.einsum("xij,xj->xi", inv, f)
    for r in range(7):
        ref = sap.apply(x[r], 2)
        assert np.max(np.abs(got[r] - ref)) <= 1e-5 * np.max(np.abs(ref))


@pytest.mark.parametrize("n_vec", [8, 12, 20])
def test_level1_sap_on_tensor_cores_is_as_accurate_as_in_fp32(n_vec):
    """The same level-1 SAP on a SINGLE handle (FP32 operator, vectors and accumulation on the CUDA cores) sets the
    bound: the half-precision handle's error against 64 bits on the operator as it stores it is no larger."""
    from oracle.lattice import Lattice
    from oracle.multilevel import StencilOperator, StencilSAP
    from paper_1303_1377_gb300 import ddamg

    def r32(v):
        return v.astype(np.complex64).astype(np.complex128)

    def r16(v):
        return v.real.astype(np.float32).astype(np.float16) + 1j * v.imag.astype(np.float32).astype(np.float16).astype(np.float64)

    dims, err = (8, 8, 8, 8), {}
    x = synth.gaussian_coarse(256, 2 * n_vec, 6, seed=33)
    for prec, stored in ((ddamg.PREC_SINGLE, r32), (ddamg.PREC_HALF, r16)):
        s, _ = _solver(dims, n_vec=n_vec, block=(2, 2, 2, 2), precision=prec)
        with s:
            s.setup_from_vectors(synth.random_test_vectors(dims, n_vec, seed=31))
            s.ml_build(synth.gaussian_coarse(256, 2 * n_vec, 3, seed=32), ddamg.ml_default_params(n_vec1=3))
            B = s.coarse_stencil()
            got = s.ml_apply_sap1(x, 2)
        sap = StencilSAP(StencilOperator(Lattice((4, 4, 4, 4)), stored(B)), (2, 2, 2, 2), mr_steps=4)
        inv = stored(np.linalg.inv(B[:, 0]))
        sap.apply_Aee_inv = lambda f: np.einsum("xij,xj->xi", inv, f)
        err[prec] = np.linalg.norm(got - np.stack([sap.apply(x[r], 2) for r in range(6)]))
    assert err[ddamg.PREC_HALF] <= err[ddamg.PREC_SINGLE]


@pytest.mark.parametrize("prec,tol", [("DOUBLE", 1e-13), ("SINGLE", 1e-6)])
@pytest.mark.parametrize("dims,block,n_vec", [((16, 16, 16, 8), (2, 2, 2, 2), 5), ((16, 16, 16, 8), (2, 2, 4, 4), 3),
                                              ((16, 16, 16, 16), (4, 4, 4, 4), 8), ((16, 16, 16, 16), (4, 4, 4, 4), 24)])
def test_coarse_stencil_of_one_field_by_sites_and_columns(prec, tol, dims, block, n_vec):
    """D_c of one field on 256 (short and long columns), 512 and 2048 sites, on both sides of the lines between the forms
    of the stencil kernel, against the handle's own stencil in FP64, at the stated bounds."""
    from oracle.lattice import Lattice
    from oracle.multilevel import StencilOperator
    from paper_1303_1377_gb300 import ddamg

    s, _ = _solver(dims, n_vec=n_vec, block=block, precision=getattr(ddamg, "PREC_" + prec))
    with s:
        s.setup_from_vectors(synth.random_test_vectors(dims, n_vec, seed=91))
        x = synth.gaussian_coarse(s.n_coarse, s.coarse_dof, 1, seed=92)
        got, B = s.apply_Dc(x)[0], s.coarse_stencil()
    ref = StencilOperator(Lattice(tuple(d // b for d, b in zip(dims, block))), B).apply(x[0])
    assert np.max(np.abs(got - ref)) < tol * np.max(np.abs(ref))


def test_half_prolongation_gives_the_same_bits_by_either_route():
    """Few aggregates: up to four fields leave the kernel in the caller's layout, larger batches go through the internal
    one; the same products either way."""
    from paper_1303_1377_gb300 import ddamg

    dims, n_vec = (8, 8, 8, 8), 8
    s, _ = _solver(dims, n_vec=n_vec, precision=ddamg.PREC_HALF)
    with s:
        s.setup_from_vectors(synth.random_test_vectors(dims, n_vec, seed=75))
        e = synth.gaussian_coarse(s.n_coarse, s.coarse_dof, 13, seed=76)
        got = s.prolong(e)
        for a, b in ((0, 4), (4, 8), (8, 12), (12, 13)):
            assert np.array_equal(s.prolong(e[a:b]), got[a:b])


@pytest.mark.parametrize("prec,n_vec", [("SINGLE", 1), ("HALF", 24)])
def test_level1_calls_with_more_fields_than_a_grid_row(prec, n_vec):
    """262145 fields, more groups of four than grid.y may have: the last fields come out as in a batch of their own."""
    import torch

    from paper_1303_1377_gb300 import ddamg

    s, _ = _solver((4, 4, 4, 8), n_vec=n_vec, block=(2, 2, 2, 2), precision=getattr(ddamg, "PREC_" + prec))
    with s:
        s.setup_from_vectors(synth.random_test_vectors((4, 4, 4, 8), n_vec, seed=1))
        s.ml_build(synth.gaussian_coarse(32, 2 * n_vec, 1, seed=2), ddamg.ml_default_params(n_vec1=1, block1=(1, 1, 1, 2)))
        x = torch.zeros((262145, 32, 2 * n_vec), dtype=torch.complex128, device="cuda")
        x[-3:] = torch.from_numpy(synth.gaussian_coarse(32, 2 * n_vec, 3, seed=3))
        last = x[-3:].contiguous()
        assert torch.equal(s.ml_restrict1(x)[-3:], s.ml_restrict1(last))
        assert torch.equal(s.ml_apply_sap1(x, 1)[-3:], s.ml_apply_sap1(last, 1))
