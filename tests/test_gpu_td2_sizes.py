"""The doubles iteration's FP32 kernels at the edges of their tiles (marked gpu).

Many small dimers, so that every launch has the tiles its larger kernels ask
for, of sizes that leave ragged rows, columns and chunks: o v of 2 to 78, v_X v_Y
of 4 to 169 (ladder rows 128 + 41), occupied pairs from 1 to 42 (more than one
tile of 32 columns), n odd and even.  Against the oracle at the FP32 form's
bound, 5e-7 of |E_J| (test_gpu_td2); the same dimers one by one, which take the
other kernels, give the same bits (every output is one chain over k in order)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")

SIZES = [(3, 1), (12, 6), (13, 7), (17, 4), (8, 2), (19, 6)]
ND, NIT = 300, 4


def test_td2_sizes_large_and_small_batches():
    rng = np.random.default_rng(8)
    mons = []
    for n, o in SIZES:
        C = np.linalg.qr(rng.standard_normal((n, n)))[0]
        e = np.concatenate([np.sort(rng.uniform(-1.5, -0.5, o)), np.sort(rng.uniform(0.2, 3.0, n - o))])
        mons.append((C, e, o))
    kinds = [(0, 1), (1, 2), (2, 3), (3, 4), (4, 5), (5, 1)]
    blocks, ref = [], []
    for X, Y in kinds:
        nX, nY = SIZES[X][0], SIZES[Y][0]
        B = rng.standard_normal((6, nX + nY, nX + nY)) * 0.02
        A, K = synth.eri_blocks(B + np.transpose(B, (0, 2, 1)), nX, 0.6)
        gX, gY = synth.monomer_doubles(X, *SIZES[X]), synth.monomer_doubles(Y, *SIZES[Y])
        _, e, _ = oracle.td2(A, K, mons[X][0], mons[X][1], mons[Y][0], mons[Y][1], mons[X][2], mons[Y][2], NIT,
                             gX[0], gY[0], gX[1], gY[1])
        blocks.append(np.concatenate([A.ravel(), K.ravel()]))
        ref.append(e)
    ref = np.array(ref)

    def run(count):
        with M.Context(precision="fp32c") as ctx:
            for d in range(count):
                for m in kinds[d % 6]:
                    i = ctx.add_monomer(*mons[m])
                    ctx.set_monomer_doubles(i, *synth.monomer_doubles(m, *SIZES[m]))
                ctx.add_dimer(2 * d, 2 * d + 1, blocks[d % 6], M.MCPT_AO_BLOCKS)
            return ctx.td2(NIT)

    many, dmany = run(ND)
    few, dfew = run(6)
    assert np.all(np.abs(many[:6] - ref) <= 5e-7 * np.abs(ref[:, :1])), np.abs(many[:6] - ref) / np.abs(ref[:, :1])
    assert np.array_equal(many.reshape(ND // 6, 6, 2), np.broadcast_to(few, (ND // 6, 6, 2)))
    assert np.array_equal(dmany, dfew)
