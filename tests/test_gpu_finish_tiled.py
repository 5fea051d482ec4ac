"""The mixed forms' second half above 32 AO at the edges of its 8 x 8 blocks and
pair groups (marked gpu): AO counts around multiples of 4 and 8 (slices that
16-byte copies can and cannot move), one pair and more pairs than a group or a
task, one set of slices (128 AO) and two, very unequal monomers.

Against the oracle at the FP32 forms' bound for few-term random dimers, 2e-6 of
|E_J|, in both epilogues; the two agree within 2e-12 |E_J| as in
test_gpu_epilogue."""
import numpy as np
import pytest

import oracle
from helpers import rand_dimer

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")

SIZES = [(33, 33, 1, 1), (34, 40, 3, 5), (41, 35, 7, 6), (64, 36, 10, 9), (72, 5, 12, 1), (8, 100, 2, 16),
         (128, 128, 2, 1), (126, 33, 5, 4)]


@pytest.mark.parametrize("nX,nY,oX,oY", SIZES)
def test_finish_above_32_ao(nX, nY, oX, oY):
    rng = np.random.default_rng(nX + 200 * nY)
    A, K, CX, eX, CY, eY = rand_dimer(rng, nX, nY, oX, oY)
    ref = oracle.dimer(A, K, CX, eX, CY, eY, oX, oY)
    out = []
    for fp64_epilogue in (False, True):
        with M.Context(precision="fp32c", fp64_epilogue=fp64_epilogue) as ctx:
            ctx.add_monomer(CX, eX, oX)
            ctx.add_monomer(CY, eY, oY)
            ctx.add_dimer(0, 1, np.concatenate([A.ravel(), K.ravel()]), M.MCPT_AO_BLOCKS)
            ctx.run()
            out.append(ctx.energies()[2][0].copy())
        assert np.all(np.abs(out[-1] - ref) <= 2e-6 * abs(ref[0])), (out[-1], ref)
    assert np.all(np.abs(out[0] - out[1]) <= 2e-12 * abs(ref[0]))


@pytest.mark.parametrize("prec", ["bf16x2", "fp32c"])
def test_energies_do_not_depend_on_the_wave(prec):
    """Twelve dimers of different sizes above 32 AO in one run, whose tasks are
    whole groups, and one by one, whose pairs are dealt to every SM: the same
    bits."""
    rng = np.random.default_rng(9)
    sizes = [(34, 5), (40, 7), (64, 9), (16, 3), (56, 8), (48, 6)]
    with M.Context(precision=prec) as ctx:
        mono = [rand_dimer(rng, n, n, o, o)[2:4] for n, o in sizes]
        for k in range(24):
            ctx.add_monomer(*mono[k % 6], sizes[k % 6][1])
        for d in range(12):
            nX, nY = sizes[2 * d % 6][0], sizes[(2 * d + 1) % 6][0]
            ctx.add_dimer(2 * d, 2 * d + 1, rng.standard_normal(2 * nX * nX * nY * nY) * 1e-3, M.MCPT_AO_BLOCKS)
        ctx.run()
        whole = ctx.energies()[2].copy()
        for d in range(12):
            ctx.run(d, 1)
        assert np.array_equal(ctx.energies()[2], whole)
