"""The 32-AO second half's split of a dimer's occupied pairs over CTAs, at the
edges of its rule (marked gpu): the same bits whether a dimer runs in a wave
of one CTA per dimer (the FP32 forms and FP64E), in one of five-warp CTAs, or
with few others over one CTA per four pairs.

Dimers of one pair, of 9 (FP64E 5) and of 81 (FP64E 25): more than the 64 a CTA
keeps in shared memory, so that a single CTA's sums also go through the H
slices.  The lines of the rule, and so the ranges, follow from the device's SMs.
Each kind also against the oracle, at test_gpu_finish_split's bounds."""
import numpy as np
import pytest

import oracle
from helpers import rand_dimer

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")
torch = pytest.importorskip("torch")

SIZES = {"fp64": [(3, 1), (5, 1), (12, 9), (13, 9)], "fp32c": [(3, 1), (5, 1), (12, 9), (13, 9)],
         "tf32": [(4, 1), (6, 1), (14, 9), (12, 9)], "fp64e": [(4, 1), (6, 1), (14, 5), (12, 5)]}
TOL = {"fp64": 1e-12, "fp32c": 2e-6, "tf32": 2e-3, "fp64e": 5e-12}


@pytest.mark.parametrize("prec", list(SIZES))
def test_same_bits_for_every_split(prec):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sizes = SIZES[prec]
    pairs = sizes[2][1] * sizes[3][1]            # of the largest kind
    p4, p5 = -(-pairs // 4), -(-pairs // 5)
    n5 = sms // p5                               # a range of five-warp CTAs, one per SM
    assert n5 * p5 <= sms < n5 * p4
    nd = 6 * sms + 8                             # FP32: above the one-CTA line
    if prec == "fp64e":                          # whole sets of two CTAs per SM: one per dimer fills them
        nd = 6 * sms
        assert 3 * (p4 + 0.18) < -(-nd * p4 // (2 * sms)) * 1.18
    rng = np.random.default_rng(23)
    kinds = [rand_dimer(rng, sizes[k][0], sizes[(k + 1) % 4][0], sizes[k][1], sizes[(k + 1) % 4][1]) for k in range(4)]
    mono = [(kinds[k][2], kinds[k][3], sizes[k][1]) for k in range(4)]
    with M.Context(precision=prec) as ctx:
        for m in range(nd + 1):
            ctx.add_monomer(*mono[m % 4])
        bufs = [torch.from_numpy(np.concatenate([A.ravel(), K.ravel()])).cuda() for A, K, *_ in kinds]
        torch.cuda.synchronize()
        for d in range(nd):
            ctx.add_dimer(d, d + 1, bufs[d % 4].data_ptr(), M.MCPT_AO_BLOCKS, on_device=1)
        ctx.run()
        whole = ctx.energies()[2].copy()
        # one pair alone; the 81 pairs alone; five warps; several CTAs of four; the rest
        for first, count in ((0, 1), (1, 1), (2, 1), (3, n5), (3 + n5, 2 * n5)):
            ctx.run(first, count)
            assert np.array_equal(ctx.energies()[2], whole), (first, count)
    for k in range(4):
        assert np.all(whole[k::4] == whole[k]), k
        A, K = kinds[k][:2]
        CX, eX, oX = mono[k]
        CY, eY, oY = mono[(k + 1) % 4]
        ref = oracle.dimer(A, K, CX, eX, CY, eY, oX, oY)
        assert np.all(np.abs(whole[k] - ref) <= TOL[prec] * abs(ref[0])), (k, whole[k], ref)
