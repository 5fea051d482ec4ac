"""The dimer -> monomer doubles coupling over enough monomers that the output
tiles keep their own edges (three tiles per SM or more; with fewer every
monomer takes edge 32): o v of 120, 80 and 28 take edges 64, 48 and 32, the
first two ragged (marked gpu).

A chain of three kinds of monomer, so that all monomers of a kind with the same
neighbours have the same R: the first, the last and one interior monomer of each
kind against the oracle, at test_gpu_coupling's bounds, the others bit for bit.
The chain's first five monomers alone (edge 32 throughout) add the same terms
over the same rows in the same order: the same bits as in the long chain."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")
torch = pytest.importorskip("torch")

TOL = {"fp64": 1e-11, "fp32c": 1e-5, "bf16x3": 1e-5}      # of the largest |R_X| element
SIZES = [(26, 6), (24, 4), (16, 2)]                       # o v = 120, 80, 28: 3, 3 and 1 tiles


@pytest.mark.parametrize("prec", list(TOL))
def test_edges_of_many_monomers(prec):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 3 * (-(-3 * sms // 7) + 2)                        # 7 tiles per three monomers
    rng = np.random.default_rng(37)
    mons = []
    for k, o in SIZES:
        C = np.linalg.qr(rng.standard_normal((k, k)))[0]
        mons.append((C, np.concatenate([np.sort(rng.uniform(-1.5, -0.5, o)), np.sort(rng.uniform(0.2, 3.0, k - o))]), o))
    m = [o * (k - o) for k, o in SIZES]
    left = [np.zeros((m[(a + 1) % 3],) * 2) for a in range(3)]     # of the dimer (a, a + 1): its share of R_Y
    right = [np.zeros((m[a],) * 2) for a in range(3)]              # and of R_X
    bufs = []
    for a in range(3):
        (CX, eX, oX), (CY, eY, oY) = mons[a], mons[(a + 1) % 3]
        nX, nY = len(eX), len(eY)
        A, K = rng.standard_normal((nX, nX, nY, nY)) * 1e-3, rng.standard_normal((nX, nY, nY, nX)) * 1e-3
        oracle.coupling_add(oracle.transform_J(A, CX, CY, oX, oY), eX, eY, oX, oY, right[a], left[a])
        bufs.append(torch.from_numpy(np.concatenate([A.ravel(), K.ravel()])).cuda())
    torch.cuda.synchronize()

    def chain(count):
        with M.Context(precision=prec, coupling=True) as ctx:
            for X in range(count):
                ctx.add_monomer(*mons[X % 3])
            for X in range(count - 1):
                ctx.add_dimer(X, X + 1, bufs[X % 3].data_ptr(), M.MCPT_AO_BLOCKS, on_device=1)
            ctx.run()
            return [ctx.coupling(X, *SIZES[X % 3]) for X in range(count)]

    R = chain(n)
    for X in range(n):
        assert np.array_equal(R[X], R[X].T)
        if 1 <= X < n - 1 and X > 3:
            assert np.array_equal(R[X], R[X % 3 + 3 if X % 3 == 0 else X % 3]), X
    for X in (0, 1, 2, 3, n - 1):
        ref = (left[(X - 1) % 3] if X else 0) + (right[X % 3] if X < n - 1 else 0)
        err = np.abs(R[X] - ref).max() / np.abs(ref).max()
        print(f"{prec} monomer {X}: rel err {err:.2e}")
        assert err <= TOL[prec], X
    few = chain(5)
    for X in range(4):                                    # the fifth has another neighbour in the long chain
        assert np.array_equal(few[X], R[X]), X
