"""The density-fitted route's FP32 kernels as a large lattice launches them
(marked gpu): several hundred dimers, so that a CTA of the half-transformation
takes several rounds of four factors with a short last one (and the next
batch's loads cross the rounds' barriers), and one of the pair kernel up to
five j.  Batches whose largest occupation is 4, 6 and 11 take the three
register blocks; occupations of 3 to 11 give j blocks of 3, 4 and 5, near-equal
ones among them.  Ragged sizes, even and odd (no paired loads).

A batch holds nine kinds of dimer over three kinds of monomer.  Each kind
against the oracle's factor route at the FP32 form's bound, 5e-7 of |E_J|
(test_gpu_df, test_gpu_df_sizes); its repeats bit for bit."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")
torch = pytest.importorskip("torch")

N = 40                                           # monomers: 780 dimers
NAUX = [37, 52, 70, 41, 64, 38, 67, 49, 70]      # of the nine kinds


@pytest.mark.parametrize("kinds", [((9, 3), (14, 4), (11, 1)), ((12, 5), (17, 6), (10, 3)), ((15, 7), (24, 11), (34, 4))],
                         ids=["occ4", "occ6", "occ11"])
def test_df_many_dimers(kinds):
    rng = np.random.default_rng(29)
    mons = []
    for n, o in kinds:
        C = np.linalg.qr(rng.standard_normal((n, n)))[0]
        mons.append((C, np.concatenate([np.sort(rng.uniform(-1.5, -0.5, o)), np.sort(rng.uniform(0.2, 3.0, n - o))]), o))
    ref, bufs = {}, {}
    for a in range(3):
        for b in range(3):
            (CX, eX, oX), (CY, eY, oY) = mons[a], mons[b]
            n = len(eX) + len(eY)
            B = rng.standard_normal((NAUX[3 * a + b], n, n)) * 0.1
            V, W = oracle.factor_route(B, 0.7, CX, CY, oX, oY)
            ref[a, b] = np.array(oracle.energy_from_mo(V, W, eX, eY, oX, oY))
            bufs[a, b] = torch.from_numpy(B).cuda()
    torch.cuda.synchronize()
    which = []
    with M.Context(precision="bf16x2") as ctx:
        for m in range(N):
            ctx.add_monomer(*mons[m % 3])
        for X in range(N):
            for Y in range(X + 1, N):
                k = (X % 3, Y % 3)
                ctx.add_dimer_df(X, Y, bufs[k].data_ptr(), NAUX[3 * k[0] + k[1]], 0.7, on_device=1)
                which.append(k)
        ctx.run_df()
        pd = ctx.df_energies()[2].copy()
        ctx.run_df()
        assert np.array_equal(ctx.df_energies()[2], pd)
    for k in ref:
        rows = pd[[q for q, w in enumerate(which) if w == k]]
        assert np.all(rows == rows[0]), k
        assert np.all(np.abs(rows[0] - ref[k]) <= 5e-7 * abs(ref[k][0])), (k, rows[0], ref[k])
