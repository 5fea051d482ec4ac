"""Workloads of the MCPT(2) dimer library that its speed is measured on.

Each case is one call sequence a program makes through the package's public
entry points, on inputs it already holds: the four-index run in each precision
form that is used, the steps that follow it (coupling, singles), the doubles
iteration, the density-fitted route and the host-data update of a sequence of
geometries.  The integrals are B^Q products over seeded symmetric Gaussian
factors (kappa 0.01, 192 auxiliary functions, cross-monomer factor
exp(-R/2 Angstrom), cubic sites 3 Angstrom apart), as in the package's
synthetic workloads.

A case:
  entry      "run" (run + energies), "coupling" (run + energies + every
             monomer's coupling matrix + the singles term), "td2" (the doubles
             iteration), "df" (the density-fitted route) or "update" (new host
             integrals, then run + energies)
  precision  the context's arithmetic form
  layout     "blocks", "full" or "packed" integrals ("factors" for df)
  box, cheb  "LxMxN" sites of a cubic lattice with every pair within that
             Chebyshev distance; box "pairs:D" is D separate dimers
  nao        "lo-hi/step" AO functions per monomer, nocc 0 = nao / 6 rounded
  sizes      seed of the monomers' sizes (lo < hi)
  steps      Jacobi steps of td2
"""
import itertools
import math
import random

import numpy as np
import torch

import paper_1409_2700_gb300 as mcpt

NAUX = 192
KAPPA = 0.01
SPACING = 3.0


def _case(name, entry, precision, layout, box, cheb=1, nao="32-32/1", nocc=0, sizes=0, steps=0):
    c = {"entry": entry, "precision": precision, "layout": layout, "box": box, "cheb": cheb, "nao": nao,
         "nocc": nocc, "sizes": sizes, "steps": steps}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # one dimer of a geometry scan: the smallest call, launches and latency
        _case("one-dimer-bf16x2", "run", "bf16x2", "blocks", "2x1x1"),
        # the plain FP64 form on a small lattice given as full 64^4 tensors
        _case("lattice-2x2x2-fp64-full", "run", "fp64", "full", "2x2x2"),
        # a mid-size lattice in FP64 accuracy from the tensor cores
        _case("lattice-3x3x4-fp64e", "run", "fp64e", "blocks", "3x3x4"),
        # the 125-monomer lattice in TF32
        _case("lattice-5x5x5-tf32", "run", "tf32", "blocks", "5x5x5"),
        # a wave of a large lattice, second shell included, in the form a production run takes
        _case("wave-8x8x2-cheb2-bf16x2", "run", "bf16x2", "blocks", "8x8x2", cheb=2),
        # a batch of unequal dimers, 16 to 96 AO
        _case("uneven-bf16x2", "run", "bf16x2", "blocks", "pairs:96", nao="16-96/8", sizes=20141409),
        # large monomers, 20 occupied: the two forms they are run in
        _case("ao128-fp32c", "run", "fp32c", "blocks", "4x1x1", nao="128-128/1", nocc=20),
        _case("ao128-bf16x3", "run", "bf16x3", "blocks", "4x1x1", nao="128-128/1", nocc=20),
        # the doubles iteration over a small lattice, FP32 arithmetic
        _case("td2-3x3x3", "td2", "bf16x3", "blocks", "3x3x3", steps=10),
        # the density-fitted route on the 125-monomer lattice
        _case("df-5x5x5", "df", "bf16x2", "factors", "5x5x5"),
        # first-order run with the doubles coupling and singles terms it feeds
        _case("coupling-3x3x3-bf16x3", "coupling", "bf16x3", "blocks", "3x3x3"),
        # the next geometry of a sequence: packed integrals from pinned host memory
        _case("update-3x3x3-packed", "update", "bf16x2", "packed", "3x3x3"),
    ]


# ------------------------------------------------------------------- shapes
def _range(case):
    span, step = case["nao"].split("/")
    lo, hi = (int(x) for x in span.split("-"))
    return lo, hi, int(step)


def _monomers(case):
    """[(nao, nocc)] of every monomer and [(X, Y, R)] of every dimer."""
    lo, hi, step = _range(case)
    pairs = []
    if case["box"].startswith("pairs:"):
        nd = int(case["box"][6:])
        count = 2 * nd
        pairs = [(2 * k, 2 * k + 1, SPACING * math.sqrt(1 + k % 3)) for k in range(nd)]
    else:
        box = [int(x) for x in case["box"].split("x")]
        sites = list(itertools.product(*(range(b) for b in box)))
        count = len(sites)
        for X in range(count):
            for Y in range(X + 1, count):
                d = [abs(p - q) for p, q in zip(sites[X], sites[Y])]
                if max(d) <= case["cheb"]:
                    pairs.append((X, Y, SPACING * math.sqrt(sum(x * x for x in d))))
    rng = random.Random(case["sizes"])
    nao = [lo + step * rng.randrange((hi - lo) // step + 1) for _ in range(count)]
    return [(n, case["nocc"] or max(1, int(math.floor(n / 6.0 + 0.5)))) for n in nao], pairs


def _block_elems(nX, nY):
    return 2 * nX * nX * nY * nY


def _packed_elems(nX, nY):
    return (nX * (nX + 1) // 2) * (nY * (nY + 1) // 2) + nX * nY * (nX * nY + 1) // 2


def draw(rng):
    """One more case of the listed ranges."""
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(most):
        # a box of sites with at most `most` dimers within Chebyshev distance 1
        while True:
            b = sorted(logint(1, 6) for _ in range(3))
            sites = b[0] * b[1] * b[2]
            near = math.prod(3 * x - 2 for x in b)
            if sites > 1 and (near - sites) // 2 <= most:
                return "x".join(str(x) for x in b)

    kind = rng.choice(["mixed", "mixed", "mixed", "fp64", "fp64e", "fp32c", "uneven", "uneven", "large", "td2", "df",
                       "coupling", "update"])
    form = rng.choice(["bf16x2", "tf32", "bf16x3"])
    even = 2 * rng.randrange(8, 25)               # 16 .. 48 AO, what the tensor-core forms take
    if kind == "mixed":
        return _case(None, "run", form, rng.choice(["blocks", "blocks", "full"]) if even <= 32 else "blocks",
                     box(40 if even > 32 else 160), nao="%d-%d/1" % (even, even))
    if kind == "fp64":
        n = rng.randrange(13, 41)
        return _case(None, "run", "fp64", "blocks", box(120), nao="%d-%d/1" % (n, n))
    if kind == "fp64e":
        return _case(None, "run", "fp64e", "blocks", box(150), nao="%d-%d/2" % (even // 2 * 2 - 2, even), nocc=rng.randrange(1, 6),
                     sizes=rng.randrange(1 << 20))
    if kind == "fp32c":
        n = rng.randrange(15, 65)
        return _case(None, "run", "fp32c", "blocks", box(20 if n > 40 else 100), nao="%d-%d/1" % (n, n + 3),
                     sizes=rng.randrange(1 << 20))
    if kind == "uneven":
        return _case(None, "run", rng.choice(["bf16x2", "bf16x3"]), "blocks", "pairs:%d" % logint(4, 80),
                     nao="16-96/8", sizes=rng.randrange(1 << 20))
    if kind == "large":
        n = 2 * rng.randrange(50, 65)
        return _case(None, "run", form, "blocks", rng.choice(["2x1x1", "3x1x1"]), nao="%d-%d/1" % (n, n),
                     nocc=rng.randrange(14, 21))
    if kind == "td2":
        n = rng.randrange(16, 35)
        return _case(None, "td2", rng.choice(["fp32c", "bf16x3"]), "blocks", box(60), nao="%d-%d/1" % (n, n + 2),
                     sizes=rng.randrange(1 << 20), steps=rng.randrange(4, 11))
    if kind == "df":
        n = rng.randrange(16, 41)
        return _case(None, "df", rng.choice(["bf16x2", "bf16x2", "fp64"]), "factors", box(200),
                     nao="%d-%d/1" % (n, n + 4), sizes=rng.randrange(1 << 20))
    if kind == "coupling":
        return _case(None, "coupling", form, "blocks", rng.choice(["2x2x2", "1x3x4", "2x2x5", "2x3x4"]),
                     nao="%d-%d/2" % (even - 4, even), sizes=rng.randrange(1 << 20))
    return _case(None, "update", form, "packed", box(100), nao="%d-%d/1" % (min(even, 36), min(even, 36)))


# ------------------------------------------------------------------- inputs
def _orbitals(mons, seed):
    """Orthonormal C and orbital energies (occupied, then virtual, ascending)."""
    rng = np.random.default_rng([seed, 1])
    out = []
    for n, o in mons:
        C = np.linalg.qr(rng.standard_normal((n, n)))[0]
        e = np.concatenate([np.sort(rng.uniform(-1.5, -0.5, o)), np.sort(rng.uniform(0.2, 3.0, n - o))])
        out.append((np.ascontiguousarray(C), e))
    return out


def _doubles(mons, seed):
    """The monomers' ring and amplitude matrices of the doubles iteration."""
    rng = np.random.default_rng([seed, 2])
    out = []
    for n, o in mons:
        m = o * (n - o)
        r = [rng.standard_normal((m, m)) for _ in range(2)]
        out.append((2e-3 * (r[0] + r[0].T) / math.sqrt(2.0), 1e-3 * (r[1] + r[1].T) / math.sqrt(2.0)))
    return out


def _singles(mons, seed):
    rng = np.random.default_rng([seed, 3])
    return [0.01 * rng.standard_normal((o, n - o)) for n, o in mons]


def _all_factors(mons, pairs, seed):
    """Each dimer's B[naux][n][n] in turn."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    for X, Y, R in pairs:
        n = mons[X][0] + mons[Y][0]
        G = torch.randn((NAUX, n, n), dtype=torch.float64, device="cuda", generator=gen)
        yield (G + G.transpose(1, 2)).mul_(KAPPA / math.sqrt(2.0))


def _write_blocks(B, nX, s, out):
    """[A | K]: A = (XX|YY), K = (XY|YX)."""
    n = B.shape[1]
    nY = n - nX
    half = nX * nX * nY * nY
    xx, yy = B[:, :nX, :nX].reshape(NAUX, -1), B[:, nX:, nX:].reshape(NAUX, -1)
    xy, yx = B[:, :nX, nX:].reshape(NAUX, -1), B[:, nX:, :nX].reshape(NAUX, -1)
    torch.mm((s * xx).T, yy, out=out[:half].view(nX * nX, nY * nY))
    torch.mm((s * xy).T, yx, out=out[half:].view(nX * nY, nY * nX))


def _write_full(B, nX, s, out):
    """The dimer's whole tensor: every integral not on one monomer alone scaled by s."""
    n = B.shape[1]
    G = out.view(n, n, n, n)
    F = B.reshape(NAUX, n * n)
    torch.mm((s * F).T, F, out=out.view(n * n, n * n))
    for a in (slice(0, nX), slice(nX, n)):
        G[a, a, a, a] /= s


def _pack_index(nX, nY):
    """Indices into [A | K] of the packed layout's elements, in its order."""
    def low(n):
        return torch.tril_indices(n, n, device="cuda")
    ix, iy, ip = low(nX), low(nY), low(nX * nY)
    a = ((ix[0] * nX + ix[1]) * nY * nY)[:, None] + (iy[0] * nY + iy[1])[None, :]
    mu, la, nu, sg = ip[0] // nY, ip[0] % nY, ip[1] // nY, ip[1] % nY
    k = nX * nX * nY * nY + ((mu * nY + la) * nY + sg) * nX + nu
    return torch.cat([a.reshape(-1), k])


def _scale(R):
    return math.exp(-R / 2.0)


class State:
    """A context with its monomers and dimers, and the buffers they live in."""


def prepare(case, seed):
    mons, pairs = _monomers(case)
    s = State()
    s.entry, s.mons, s.steps, s.count = case["entry"], mons, case["steps"], len(pairs)
    s.ctx = mcpt.Context(precision=case["precision"], coupling=case["entry"] == "coupling")
    for (C, e), (n, o) in zip(_orbitals(mons, seed), mons):
        s.ctx.add_monomer(C, e, o)
    if case["entry"] == "df":
        s.keep = list(_all_factors(mons, pairs, seed))
        torch.cuda.synchronize()
        for (X, Y, R), B in zip(pairs, s.keep):
            s.ctx.add_dimer_df(X, Y, B, NAUX, _scale(R))
        return s
    full, packed = case["layout"] == "full", case["layout"] == "packed"
    elems = [(mons[X][0] + mons[Y][0]) ** 4 if full else _block_elems(mons[X][0], mons[Y][0]) for X, Y, R in pairs]
    at = [0]
    for n in elems:
        at.append(at[-1] + (n + 31) // 32 * 32)
    buf = torch.empty(max(elems) if packed else at[-1], dtype=torch.float64, device="cuda")
    if packed:
        sizes = [_packed_elems(mons[X][0], mons[Y][0]) for X, Y, R in pairs]
        s.offsets = np.concatenate([[0], np.cumsum(sizes)[:-1]]).astype(np.uint64)
        s.host = torch.empty(sum(sizes), dtype=torch.float64, pin_memory=True)
        index = {}
    for d, ((X, Y, R), B) in enumerate(zip(pairs, _all_factors(mons, pairs, seed))):
        nX, nY = mons[X][0], mons[Y][0]
        out = buf[:elems[d]] if packed else buf[at[d]:at[d] + elems[d]]
        (_write_full if full else _write_blocks)(B, nX, _scale(R), out)
        if packed:
            if (nX, nY) not in index:
                index[nX, nY] = _pack_index(nX, nY)
            o = int(s.offsets[d])
            s.host[o:o + sizes[d]].copy_(out[index[nX, nY]])
    torch.cuda.synchronize()
    for d, (X, Y, R) in enumerate(pairs):
        if packed:
            o = int(s.offsets[d])
            s.ctx.add_dimer(X, Y, s.host[o:o + sizes[d]].numpy(), mcpt.MCPT_AO_PACKED)
        else:
            s.ctx.add_dimer(X, Y, buf[at[d]:at[d] + elems[d]], mcpt.MCPT_AO_FULL if full else mcpt.MCPT_AO_BLOCKS)
    s.keep = None if packed else buf
    if packed:
        s.host_np = s.host.numpy()
    if case["entry"] == "td2":
        for X, (G, U) in enumerate(_doubles(mons, seed)):
            s.ctx.set_monomer_doubles(X, G, U)
    if case["entry"] == "coupling":
        s.t = _singles(mons, seed)
    return s


# --------------------------------------------------------------------- pass
def run(s):
    ctx = s.ctx
    if s.entry == "td2":
        return list(ctx.td2(s.steps))
    if s.entry == "df":
        ctx.run_df()
        return list(ctx.df_energies())
    if s.entry == "update":
        ctx.update_dimers(0, s.count, s.host_np, s.offsets, mcpt.MCPT_AO_PACKED, asynchronous=True)
    ctx.run()
    out = list(ctx.energies())
    if s.entry == "coupling":
        out.append([ctx.coupling(X, n, o) for X, (n, o) in enumerate(s.mons)])
        out.append(ctx.singles(s.t))
    return out


# --------------------------------------------------------------------- work
def work(case):
    mons, pairs = _monomers(case)
    b = f = 0
    for X, Y, R in pairs:
        (nX, oX), (nY, oY) = mons[X], mons[Y]
        vX, vY = nX - oX, nY - oY
        mX, mY = oX * vX, oY * vY
        first = 2 * 2 * (nX * nX * nY * nY * oY + oX * nX * nX * nY * oY + oX * nX * oY * nY * vY + oX * vX * oY * vY * nX)
        if case["entry"] == "df":
            n = nX + nY
            b += 8 * NAUX * n * n
            f += 2 * NAUX * ((oX * nX + oY * nY) * n + (oX + oY) * (nX * vX + nY * vY)) + 4 * NAUX * mX * mY
        elif case["entry"] == "td2":
            b += 8 * _block_elems(nX, nY)
            f += first // 2 + 2 * (2 * nX * nX * nY * nY * (nX + nY))
            f += case["steps"] * 2 * mX * mY * (vX * vY + oX * oY + oX * vY + vX * oY + mX + mY) + 2 * mX * mY * (mX + mY)
        else:
            b += 8 * (_packed_elems(nX, nY) if case["layout"] == "packed" else _block_elems(nX, nY))
            f += first
            if case["entry"] == "coupling":
                f += 2 * (mX * mX * mY + mY * mY * mX) + 4 * mX * mY
        b += 16
    for n, o in mons:
        m = o * (n - o)
        b += 8 * (n * n + n) + 16
        if case["entry"] == "coupling":
            b += 8 * (m * m + 2 * m)
        if case["entry"] == "td2":
            b += 16 * m * m
    return {"bytes": float(b), "flops": float(f)}


# -------------------------------------------------------------------- exact
def _to_gpu(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _contract(T, C, axis):
    """Index `axis` of T transformed by C's columns."""
    return torch.movedim(torch.tensordot(T, C, dims=([axis], [0])), -1, axis)


def _denominators(eX, eY, oX, oY):
    return 1.0 / (eX[:oX, None, None, None] - eX[None, oX:, None, None] + eY[None, None, :oY, None] - eY[None, None, None, oY:])


def exact(case, seed):
    """The same outputs from torch FP64 contractions."""
    mons, pairs = _monomers(case)
    orb = [(_to_gpu(C), _to_gpu(e)) for C, e in _orbitals(mons, seed)]
    N, entry = len(mons), case["entry"]
    pd = torch.zeros((len(pairs), 2), dtype=torch.float64, device="cuda")
    if entry == "coupling":
        R_ = [torch.zeros((o * (n - o),) * 2, dtype=torch.float64, device="cuda") for n, o in mons]
        t_ = [_to_gpu(t) for t in _singles(mons, seed)]
        s_ = [torch.zeros_like(t) for t in t_]
    if entry == "td2":
        gu = [(_to_gpu(G), _to_gpu(U)) for G, U in _doubles(mons, seed)]
        delta = torch.zeros(case["steps"], dtype=torch.float64, device="cuda")
    for d, ((X, Y, R), B) in enumerate(zip(pairs, _all_factors(mons, pairs, seed))):
        (nX, oX), (nY, oY) = mons[X], mons[Y]
        vX, vY = nX - oX, nY - oY
        (CX, eX), (CY, eY) = orb[X], orb[Y]
        D = _denominators(eX, eY, oX, oY)
        if entry == "df":
            def half(rows, cols, Cr, Cc, r, c):
                return torch.einsum("qmn,mi,na->qia", B[:, rows, cols], Cr[:, :r], Cc[:, c:])
            x, y = slice(0, nX), slice(nX, nX + nY)
            V = _scale(R) * torch.einsum("qia,qjb->iajb", half(x, x, CX, CX, oX, oX), half(y, y, CY, CY, oY, oY))
            W = _scale(R) * torch.einsum("qib,qja->ibja", half(x, y, CX, CY, oX, oY), half(y, x, CY, CX, oY, oX))
        else:
            buf = torch.empty(_block_elems(nX, nY), dtype=torch.float64, device="cuda")
            _write_blocks(B, nX, _scale(R), buf)
            A = buf[:buf.numel() // 2].view(nX, nX, nY, nY)
            K = buf[buf.numel() // 2:].view(nX, nY, nY, nX)
            W = _contract(_contract(_contract(_contract(K, CX[:, :oX], 0), CY[:, :oY], 2), CX[:, oX:], 3), CY[:, oY:], 1)
            if entry == "td2":
                g = _contract(_contract(_contract(_contract(A, CX, 0), CY, 2), CX, 1), CY, 3)
                V = g[:oX, oX:, :oY, oY:]
            else:
                V = _contract(_contract(_contract(_contract(A, CX[:, :oX], 0), CY[:, :oY], 2), CX[:, oX:], 1), CY[:, oY:], 3)
        T = V * D
        if entry == "td2":
            (GX, UX), (GY, UY) = gu[X], gu[Y]
            mX, mY = oX * vX, oY * vY
            v2 = V.reshape(mX, mY)
            S = (UX @ v2 + v2 @ UY.T).view(V.shape)
            T = torch.zeros_like(V)
            for it in range(case["steps"]):
                t2 = T.reshape(mX, mY)
                r = V + S + (GX @ t2 + t2 @ GY.T).view(V.shape)
                r = r + torch.einsum("acbd,icjd->iajb", g[oX:, oX:, oY:, oY:], T)
                r = r + torch.einsum("kilj,kalb->iajb", g[:oX, :oX, :oY, :oY], T)
                r = r - torch.einsum("kibd,kajd->iajb", g[:oX, :oX, oY:, oY:], T)
                r = r - torch.einsum("aclj,iclb->iajb", g[oX:, oX:, :oY, :oY], T)
                Tn = r * D
                delta[it] = torch.maximum(delta[it], (Tn - T).abs().max())
                T = Tn
        pd[d, 0] = 4.0 * (V * T).sum()
        pd[d, 1] = -2.0 * (W.permute(0, 3, 2, 1) * T).sum()
        if entry == "coupling":
            mX, mY = oX * vX, oY * vY
            v2, t2 = V.reshape(mX, mY), T.reshape(mX, mY)
            R_[X] += t2 @ v2.T + v2 @ t2.T
            R_[Y] += t2.T @ v2 + v2.T @ t2
            s_[X] += (v2 @ t_[Y].reshape(-1)).view(oX, vX)
            s_[Y] += (v2.T @ t_[X].reshape(-1)).view(oY, vY)
    if entry == "td2":
        return [pd.cpu().numpy(), delta.cpu().numpy()]
    mon = torch.zeros((N, 2), dtype=torch.float64, device="cuda")
    for which in (0, 1):
        mon.index_add_(0, torch.tensor([p[which] for p in pairs], device="cuda"), 0.5 * pd)
    mon, pd = mon.cpu().numpy(), pd.cpu().numpy()
    out = [np.ascontiguousarray(mon[:, 0]), np.ascontiguousarray(mon[:, 1]), pd, pd.sum(axis=0)]
    if entry == "coupling":
        out += [[r.cpu().numpy() for r in R_], [x.cpu().numpy() for x in s_]]
    return out
