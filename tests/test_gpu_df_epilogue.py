"""The density-fitted route's energy epilogue: FP64 denominators, products and
sums, whatever the arithmetic of the integrals, and any scale of the factors
(marked gpu).

Precision: C the identity and one auxiliary function of small integers, so
that (ia|jb) and (ib|ja) are exact integers in FP32 and the energies' only
roundings are the epilogue's.  With one occupied orbital each and v x v virtual
ones, an energy is a sum of n = v^2 terms.  A term's relative error: the
denominator's three subtractions of values that do not cancel (3 u, u = 2^-53),
its reciprocal (2 u allowed) and the two products (2 u); the sums of more than
one term add at most n + 13 roundings (a thread's terms, 5 tree steps, 8 warps),
and the scalings by 4 and s (1 here) none: 7 u of a single term, (20 + n) u of
the sum of |terms| otherwise.  FP32 pairs leave 2^-45, 256 u.

Range: factors of 1e-12, 1 and 1e10 with the scale s that brings the
integrals back to order one: the same energies, at the FP32 route's 5e-7 of
|E_J| (test_gpu_df), also where s^2 or the products of unscaled integrals
leave FP32's range."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")


@pytest.mark.parametrize("v", [1, 4])
@pytest.mark.parametrize("prec", ["bf16x2", "fp32c", "fp64"])
def test_epilogue_is_fp64(prec, v):
    rng = np.random.default_rng(17)
    n, nd = v + 1, 100
    ref, mag = [], []
    with M.Context(precision=prec) as ctx:
        for d in range(nd):
            e = [np.concatenate([[-rng.uniform(0.5, 1.5)], np.sort(rng.uniform(0.2, 3.0, v))]) for _ in range(2)]
            X, Y = (ctx.add_monomer(np.eye(n), x, 1) for x in e)
            B = rng.integers(1, 32, (1, 2 * n, 2 * n)).astype(np.float64)
            ctx.add_dimer_df(X, Y, B, 1, 1.0)
            g = B[0].astype(np.longdouble)
            V = np.outer(g[0, 1:n], g[n, n + 1:])               # B_{ia} B_{jb}
            W = np.outer(g[n, 1:n], g[0, n + 1:])               # B_{ja} B_{ib}
            x = [y.astype(np.longdouble) for y in e]
            D = 1 / (x[0][0] + x[1][0] - x[0][1:, None] - x[1][None, 1:])
            ref.append([4 * (V * V * D).sum(), -2 * (V * W * D).sum()])
            mag.append([4 * abs(V * V * D).sum(), 2 * abs(V * W * D).sum()])
        ctx.run_df()
        pd = ctx.df_energies()[2]
    err = np.abs(pd - np.array(ref)) / np.array(mag)
    print(f"{prec}: worst relative error {float(err.max()):.2e}")
    assert np.all(err <= (7 if v == 1 else 20 + v * v) * 2.0 ** -53)


@pytest.mark.parametrize("prec", ["bf16x2", "fp64"])
@pytest.mark.parametrize("scale", [1e-12, 1.0, 1e10])
def test_any_scale_of_the_factors(prec, scale):
    rng = np.random.default_rng(3)
    (nX, oX), (nY, oY), naux = (12, 3), (17, 6), 20
    C = [np.linalg.qr(rng.standard_normal((n, n)))[0] for n in (nX, nY)]
    e = [np.concatenate([np.sort(rng.uniform(-1.5, -0.5, o)), np.sort(rng.uniform(0.2, 3.0, n - o))])
         for n, o in ((nX, oX), (nY, oY))]
    B = rng.standard_normal((naux, nX + nY, nX + nY)) * 0.1
    V, W = oracle.factor_route(B, 0.7, C[0], C[1], oX, oY)
    ref = oracle.energy_from_mo(V, W, e[0], e[1], oX, oY)
    with M.Context(precision=prec) as ctx:
        X, Y = (ctx.add_monomer(C[k], e[k], o) for k, o in ((0, oX), (1, oY)))
        ctx.add_dimer_df(X, Y, B * scale, naux, 0.7 / scale / scale)
        ctx.run_df()
        pd = ctx.df_energies()[2][0]
    assert np.all(np.abs(pd - ref) <= {"bf16x2": 5e-7, "fp64": 1e-12}[prec] * abs(ref[0])), (pd, ref)
