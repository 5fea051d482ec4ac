"""The 32-AO second half deals a dimer's occupied pairs to one or several CTAs
by the size of the wave; the energies do not depend on how (marked gpu).

A chain of more dimers than the one-CTA rule's line (six per SM), run at once,
against the same dimers run as short ranges, whose pairs are spread over CTAs:
the same bits.  Sizes: odd slices (their pair sums are kept at 4-byte aligned
places), one pair, and more pairs (81) than the CTA keeps in shared memory.
The first dimers also against the oracle, at the forms' bounds for few-term
dimers (test_gpu_parity); the lattice total and the monomer sums against the
exact sums of the dimers' terms."""
import math

import numpy as np
import pytest

import oracle
from helpers import rand_dimer

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")

SIZES = {"fp64": [(3, 1), (5, 2), (12, 9), (7, 3)], "fp32c": [(3, 1), (5, 2), (12, 9), (7, 3)],
         "tf32": [(4, 1), (6, 2), (14, 9), (8, 3)], "fp64e": [(4, 1), (6, 2), (14, 5), (8, 3)]}
TOL = {"fp64": 1e-12, "fp32c": 2e-6, "tf32": 2e-3, "fp64e": 5e-12}
ND = 6 * 160 + 8


@pytest.mark.parametrize("prec", list(SIZES))
def test_energies_do_not_depend_on_the_split(prec):
    sizes = SIZES[prec]
    rng = np.random.default_rng(11)
    kinds = [rand_dimer(rng, sizes[k][0], sizes[(k + 1) % 4][0], sizes[k][1], sizes[(k + 1) % 4][1]) for k in range(4)]
    mono = [(kinds[k][2], kinds[k][3], sizes[k][1]) for k in range(4)]
    with M.Context(precision=prec) as ctx:
        for m in range(ND + 1):
            ctx.add_monomer(*mono[m % 4])
        for d in range(ND):
            A, K = kinds[d % 4][:2]
            s = 1.0 + d / ND
            ctx.add_dimer(d, d + 1, np.concatenate([A.ravel() * s, K.ravel() * s]), M.MCPT_AO_BLOCKS)
        ctx.run()
        mj, mk, pd, tot = ctx.energies()
        whole = pd.copy()
        # the compensated sums, over many blocks of dimers: one FP64 rounding
        # of the exact sum (2^-53) and of the lanes' error terms, within 2^-51
        for f, mon in ((0, mj), (1, mk)):
            assert abs(tot[f] - math.fsum(pd[:, f])) <= 2.0 ** -51 * np.abs(pd[:, f]).sum()
            both = np.zeros(ND + 1)
            both[:-1] += 0.5 * pd[:, f]
            both[1:] += 0.5 * pd[:, f]
            assert np.all(np.abs(mon - both) <= 2.0 ** -51 * np.abs(pd[:, f]).max())
        ctx.run(0, 6)
        ctx.run(6, 1)
        ctx.run(7, 30)
        parts = ctx.energies()[2]
        assert np.array_equal(parts, whole)
    for d in range(4):
        A, K = kinds[d][:2]
        CX, eX, oX = mono[d]
        CY, eY, oY = mono[(d + 1) % 4]
        s = 1.0 + d / ND
        ref = oracle.dimer(A * s, K * s, CX, eX, CY, eY, oX, oY)
        assert np.all(np.abs(whole[d] - ref) <= TOL[prec] * abs(ref[0])), (d, whole[d], ref)


def test_results_after_monomers_are_added():
    """The results of a run stay those of the run when monomers are added after
    it (they belong to no dimer: zero sums), and follow the next run, also of a
    part, with more dimers and on a replayed graph."""
    rng = np.random.default_rng(4)
    A, K, CX, eX, CY, eY = rand_dimer(rng, 10, 12, 2, 3)
    blocks = np.concatenate([A.ravel(), K.ravel()])
    with M.Context(precision="fp64") as ctx:
        ctx.add_monomer(CX, eX, 2)
        ctx.add_monomer(CY, eY, 3)
        ctx.add_dimer(0, 1, blocks, M.MCPT_AO_BLOCKS)
        ctx.run()
        mj, mk, pd, tot = ctx.energies()
        for k in range(5):
            ctx.add_monomer(CX, eX, 2)
        mj2, mk2, pd2, tot2 = ctx.energies()
        assert np.array_equal(pd2, pd) and np.array_equal(tot2, tot)
        assert np.array_equal(mj2[:2], mj) and np.array_equal(mk2[:2], mk)
        assert not mj2[2:].any() and not mk2[2:].any()
        for k in range(4):
            ctx.add_dimer(1, 2 + k, np.concatenate([rand_dimer(rng, 12, 10, 3, 2)[q].ravel() for q in (0, 1)]),
                          M.MCPT_AO_BLOCKS)
        for _ in range(3):
            ctx.run(1, 4)
            mj3, mk3, pd3, tot3 = ctx.energies()
            assert np.array_equal(pd3[0], pd[0]) and pd3.shape == (5, 2) and np.all(pd3[1:, 0] < 0)
            assert abs(tot3[0] - math.fsum(pd3[:, 0])) <= 2.0 ** -51 * np.abs(pd3[:, 0]).sum()
            assert mj3[6] == 0.0 and abs(mj3[1] - 0.5 * pd3[:, 0].sum()) <= 1e-15 * abs(pd3[:, 0].sum()) * 4
