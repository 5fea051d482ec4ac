"""mcpt_update_dimers' finiteness check over several host threads and beside
the first copies (marked gpu): a non-finite value anywhere refuses the whole
call with the first offending dimer named, nothing of it reaches the dimers'
integrals, and the caller's buffer is free afterwards."""
import numpy as np
import pytest

import synth
from helpers import rand_dimer

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")

ND, N = 6, 32          # 6 x 6.4 MB: several pieces per dimer, several threads


@pytest.mark.parametrize("bad", [[(0, 0)], [(ND - 1, -1)], [(2, 70000), (4, 3)], [(3, 65535)], [(3, 65536)]])
@pytest.mark.parametrize("value", [np.nan, -np.inf])
def test_refused_update_leaves_the_integrals(bad, value):
    rng = np.random.default_rng(3)
    A, K, CX, eX, CY, eY = rand_dimer(rng, N, N, 4, 5)
    one = synth.pack_blocks(A, K)
    flat = np.concatenate([one * (1.0 + 0.1 * d) for d in range(ND)])
    offs = (np.arange(ND) * one.size).astype(np.uint64)
    with M.Context(precision="bf16x2") as ctx:
        for d in range(ND):
            ctx.add_monomer(CX, eX, 4)
            ctx.add_monomer(CY, eY, 5)
            ctx.add_dimer(2 * d, 2 * d + 1, flat[d * one.size:(d + 1) * one.size], M.MCPT_AO_PACKED)
        ctx.run()
        ref = ctx.energies()[2].copy()
        new = 2.0 * flat
        for d, k in bad:
            new[d * one.size + k % one.size] = value
        for asynchronous in (False, True):
            with pytest.raises(M.McptError) as ei:
                ctx.update_dimers(0, ND, new, offs, M.MCPT_AO_PACKED, asynchronous=asynchronous)
            assert ei.value.status == M.MCPT_EINVAL
            assert "(dimer %d)" % min(d for d, _ in bad) in str(ei.value)
        ctx.run()
        assert np.array_equal(ctx.energies()[2], ref)
        ctx.update_dimers(0, ND, 2.0 * flat, offs, M.MCPT_AO_PACKED)
        ctx.run()
        assert np.array_equal(ctx.energies()[2], 4.0 * ref)
