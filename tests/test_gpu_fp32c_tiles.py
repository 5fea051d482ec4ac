"""The FP32C first half's two kernels (64-row tiles with scratch slots, and
the one without scratch that runs when the scratch limit leaves no room for
the slots) at the edges of tiles, passes and blocks (marked gpu).

Both against the oracle at the form's bound for few-term random dimers, 2e-6
of |E_J| (FP32 inputs and second half).  Against each other: both round the
same pair sum to FP32, so an element of the first-half result differs by at
most one FP32 rounding (2^-23), which moves a term of the energies by at most
2^-22 relative; the bound is 2^-21 of |E_J| (|E_K| terms are no larger than
about |E_J|'s)."""
import numpy as np
import pytest

import oracle
from helpers import rand_dimer

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")

# tiles of 64 rows: 4, 63, 64, 65, ... rows; passes and blocks of at most 10 occupied orbitals
SIZES = [(2, 2, 1, 1), (7, 9, 3, 2), (8, 8, 6, 7), (13, 5, 4, 3), (33, 17, 10, 11), (22, 31, 21, 9), (12, 66, 8, 25)]


@pytest.mark.parametrize("nX,nY,oX,oY", SIZES)
def test_fp32c_tiles_against_oracle_and_scratch_free_kernel(nX, nY, oX, oY):
    rng = np.random.default_rng(nX * 1000 + nY)
    A, K, CX, eX, CY, eY = rand_dimer(rng, nX, nY, oX, oY)
    ref = oracle.dimer(A, K, CX, eX, CY, eY, oX, oY)
    out = []
    for wave_bytes in (0, 1):          # default scratch; no room for slots
        with M.Context(precision="fp32c", wave_bytes=wave_bytes) as ctx:
            ctx.add_monomer(CX, eX, oX)
            ctx.add_monomer(CY, eY, oY)
            ctx.add_dimer(0, 1, np.concatenate([A.ravel(), K.ravel()]), M.MCPT_AO_BLOCKS)
            ctx.run()
            out.append(ctx.energies()[2][0].copy())
            ctx.run()                  # the tile counter starts over
            assert np.array_equal(out[-1], ctx.energies()[2][0])
        assert np.all(np.abs(out[-1] - ref) <= 2e-6 * abs(ref[0])), (out[-1], ref)
    assert np.all(np.abs(out[0] - out[1]) <= 2.0 ** -21 * abs(ref[0]))
