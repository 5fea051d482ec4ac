"""The density-fitted route's FP32 kernels at the edges of their tiles: odd AO
counts and factors that are only 8-byte aligned (no paired loads), ragged
32-column groups and 16-AO batches, more occupied orbitals than one register
block or j block, one auxiliary function, one dimer and several (marked gpu).

Against the oracle's factor route at the FP32 form's bound, 5e-7 of |E_J|
(test_gpu_df): sums of a few tens of FP32 products per stage, each rounding
2^-24 of its largest term, with E_J summing at least oX oY vX vY squares."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")
torch = pytest.importorskip("torch")

# (nX, oX), (nY, oY), naux
SIZES = [((5, 1), (9, 2), 1), ((16, 3), (15, 3), 17), ((33, 9), (20, 11), 33), ((36, 6), (44, 7), 20),
         ((64, 5), (18, 4), 16)]


@pytest.mark.parametrize("prec", ["bf16x2", "fp64"])
@pytest.mark.parametrize("shift", [0, 1])
def test_df_sizes_and_alignment(prec, shift):
    rng = np.random.default_rng(5 + shift)
    tol = {"bf16x2": 5e-7, "fp64": 1e-12}[prec]
    with M.Context(precision=prec) as ctx:
        ref, keep = [], []
        for (nX, oX), (nY, oY), naux in SIZES:
            mons = []
            for n, o in ((nX, oX), (nY, oY)):
                C = np.linalg.qr(rng.standard_normal((n, n)))[0]
                e = np.concatenate([np.sort(rng.uniform(-1.5, -0.5, o)), np.sort(rng.uniform(0.2, 3.0, n - o))])
                mons.append((ctx.add_monomer(C, e, o), C, e, o))
            (X, CX, eX, _), (Y, CY, eY, _) = mons
            B = rng.standard_normal((naux, nX + nY, nX + nY)) * 0.1
            V, W = oracle.factor_route(B, 0.7, CX, CY, oX, oY)
            ref.append(oracle.energy_from_mo(V, W, eX, eY, oX, oY))
            buf = torch.zeros(B.size + 1, dtype=torch.float64, device="cuda")
            buf[shift:shift + B.size] = torch.from_numpy(B.ravel())
            keep.append(buf)
            torch.cuda.synchronize()
            ctx.add_dimer_df(X, Y, buf.data_ptr() + 8 * shift, naux, 0.7, on_device=1)
        ref = np.array(ref)
        ctx.run_df()
        pd = ctx.df_energies()[2]
        assert np.all(np.abs(pd - ref) <= tol * np.abs(ref[:, :1])), np.abs(pd - ref) / np.abs(ref[:, :1])
        ctx.run_df()
        assert np.array_equal(ctx.df_energies()[2], pd)
