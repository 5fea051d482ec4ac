"""A run that fails while its plan is built leaves the results of the last
completed run in place (marked gpu): mcpt_energies then returns them bit for
bit, with a zero for a monomer added since.

The failure is the memory cap: the second run's plan adds a monomer whose
coupling matrix (o v)^2 does not fit under a cap that the first run fits."""
import numpy as np
import pytest

from helpers import rand_dimer

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_1409_2700_gb300")
torch = pytest.importorskip("torch")


def _context(prec, cap, dimer, buf):
    A, K, CX, eX, CY, eY = dimer
    ctx = M.Context(precision=prec, coupling=True, mem_cap_bytes=cap)
    ctx.add_monomer(CX, eX, 2)
    ctx.add_monomer(CY, eY, 3)
    ctx.add_dimer(0, 1, buf.data_ptr(), M.MCPT_AO_BLOCKS, on_device=1)
    return ctx


@pytest.mark.parametrize("prec", ["bf16x2", "fp64"])
def test_energies_after_a_failed_run(prec):
    rng = np.random.default_rng(41)
    dimer = rand_dimer(rng, 8, 10, 2, 3)
    buf = torch.from_numpy(np.concatenate([dimer[0].ravel(), dimer[1].ravel()])).cuda()
    torch.cuda.synchronize()
    # the smallest cap, in steps of 32 KB, that the first run fits
    for cap in range(1 << 15, 1 << 24, 1 << 15):
        ctx = _context(prec, cap, dimer, buf)
        try:
            ctx.run()
            break
        except M.McptError as e:
            assert e.status == M.MCPT_ENOMEM
            ctx.close()
    with _context(prec, cap + (128 << 10), dimer, buf) as ctx:
        ctx.run()
        mj, mk, pd, tot = ctx.energies()
        n, o = 32, 16
        C = np.linalg.qr(rng.standard_normal((n, n)))[0]
        ctx.add_monomer(C, np.linspace(-2.0, 2.0, n), o)      # (o v)^2 doubles: 512 KB
        with pytest.raises(M.McptError) as ei:
            ctx.run()
        assert ei.value.status == M.MCPT_ENOMEM
        mj2, mk2, pd2, tot2 = ctx.energies()
        assert np.array_equal(pd2, pd) and np.array_equal(tot2, tot)
        assert np.array_equal(mj2, np.append(mj, 0.0)) and np.array_equal(mk2, np.append(mk, 0.0))
