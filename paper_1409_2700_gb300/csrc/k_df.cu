// k_df.cu -- the density-fitted route to the dimer terms: (ia|jb) and
// (ib|ja) from three-index factors B^Q over the dimer's AO space instead of
// the four-index blocks,
//   (ia|jb) = s sum_Q (C_X^T B^Q_XX C_X)_{ia} (C_Y^T B^Q_YY C_Y)_{jb}
//   (ib|ja) = s sum_Q (C_X^T B^Q_XY C_Y)_{ib} (C_Y^T B^Q_YX C_X)_{ja},
// then the same denominators and energies as the four-index path.
//
// k_df_half: a CTA takes a range of Q of one dimer.  It forms the occupied rows
// of each factor, u_X = C_X,occ^T B^Q[X rows] and u_Y = C_Y,occ^T B^Q[Y rows]
// (over all n columns), then the four o x v half-transformed blocks.
// k_df_pair: a CTA takes one occupied i and up to five j of a dimer, sums
// their vX x vY tiles over Q, staged in chunks, and applies the epilogue; the
// CTAs' partial energies are added per dimer in fixed order (k_df_sum).
#include "internal.h"
#include "convert.h"

#include <algorithm>

namespace mcpt {
namespace {

__host__ __device__ constexpr int up4(int x) { return (x + 3) / 4 * 4; }

constexpr int kHWarps = 8;
constexpr int kHQ = 4;                         // most Q values of a round
constexpr int kHRows = 5;                      // occupied rows per warp task of the second product

// FP32.  A round is hq <= kHQ factors.  First product: a warp takes 32 columns
// of one half (X or Y rows), two per lane; its two half-warps sum the even and
// the odd AO, RB occupied orbitals in registers, every factor element loaded
// straight into registers and converted once; the two chains meet in a
// shuffle.  A batch covers 16 AO, and the next batch's eight 16-byte loads per
// lane (also across the round's barriers) are in flight while one is summed.  Second product: a lane per
// virtual column, five occupied rows of u per warp read as broadcasts, the even
// and the odd AO as the two chains of the packed multiply-add.  C stays in
// shared memory for all of the CTA's Q.  Bound by the factors' HBM reads (naux
// n^2 doubles per dimer).  The kernel before it staged B^Q and both C in
// shared memory, one Q per CTA: 3.10 ms for 1036 dimers of 32 + 32 AO and naux
// 192 against 1.34 ms (0.96 ms at the measured copy rate).
template <int RB>
__global__ void __launch_bounds__(kHWarps * 32, 2)
k_df_half(const DfDim* __restrict__ dims, const double* __restrict__ C, float* __restrict__ half, int qper, int hq)
{
    const DfDim& d = dims[blockIdx.y];
    const int naux = d.naux;
    const int q0 = blockIdx.x * qper, q1 = min(q0 + qper, naux);
    if (q0 >= q1) return;
    const int nX = d.nX, nY = d.nY, n = nX + nY, oX = d.oX, oY = d.oY, vX = nX - oX, vY = nY - oY;
    const int nXp = up4(nX), nYp = up4(nY), uw = nXp + nYp, vXq = up4(vX), vYq = up4(vY), ot = oX + oY;
    const int sX = (oX + RB - 1) / RB * RB, sY = (oY + RB - 1) / RB * RB;   // padded occupied rows of C
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* U = reinterpret_cast<float*>(smem_raw);       // [hq][ot][X part, Y part], the parts zero padded
    float2* VX = reinterpret_cast<float2*>(U + hq * ot * uw);   // [AO pair][vXq]: virtual columns, zero padded
    float2* VY = VX + nXp / 2 * vXq;
    float* OX = reinterpret_cast<float*>(VY + nYp / 2 * vYq);   // [AO][sX]: occupied columns, zero padded
    float* OY = OX + nX * sX;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, par = lane >> 4;
    const int ng = (n + 31) / 32;              // column groups of a half
    const double* const Bd = d.B;
    const bool vec = (n & 1) == 0 && ((size_t)Bd & 15) == 0;   // a lane's column pair is one 16-byte load
    // step of a warp: task t of the round at qb (factor, half, columns), r0 first occupied, m0 first AO
    struct Step { int qb, t, r0, m0; };
    auto advance = [&](Step s) {
        const bool hy = s.t % (2 * ng) >= ng;
        s.m0 += 16;
        if (s.m0 < (hy ? nY : nX)) return s;
        s.m0 = 0;
        s.r0 += RB;
        if (s.r0 < (hy ? oY : oX)) return s;
        s.r0 = 0;
        s.t += kHWarps;
        if (s.t < min(hq, q1 - s.qb) * 2 * ng) return s;
        s.t = warp;
        s.qb += hq;
        return s;
    };
    auto fetch = [&](Step s, double2 (&x)[8]) {
        const int qn = min(hq, q1 - s.qb);
        const bool ok = s.t < qn * 2 * ng;     // past the last round, or a warp without a task in it
        const int qq = s.t / (2 * ng), g = s.t % (2 * ng), hy = g >= ng;
        const int c = (hy ? g - ng : g) * 32 + 2 * (lane & 15), len = hy ? nY : nX;
        const double* B = Bd + (long long)(s.qb + qq) * n * n + ((hy ? nX : 0) + s.m0 + par) * n + c;
        if (ok && vec && s.m0 + 16 <= len && c + 1 < n) {
#pragma unroll
            for (int k = 0; k < 8; k++) x[k] = __ldg(reinterpret_cast<const double2*>(B + 2 * k * n));
        } else {
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const bool row = ok && s.m0 + par + 2 * k < len;
                x[k].x = row && c < n ? __ldg(B + 2 * k * n) : 0.0;
                x[k].y = row && c + 1 < n ? __ldg(B + 2 * k * n + 1) : 0.0;
            }
        }
    };
    Step cur{q0, warp, 0, 0};
    double2 x[8];
    fetch(cur, x);
    for (int e = tid; e < hq * ot * uw; e += kHWarps * 32) U[e] = 0.f;
    auto stage = [&](float2* V, float* O, const double* Cm, int m, int o, int mp, int vq, int so) {
        for (int e = tid; e < mp / 2 * vq; e += kHWarps * 32) {
            const int k = e / vq * 2, c = o + e % vq;
            const double a = k < m && c < m ? Cm[k * m + c] : 0.0, b = k + 1 < m && c < m ? Cm[(k + 1) * m + c] : 0.0;
            V[e] = make_float2(f32_from_f64(a), f32_from_f64(b));
        }
        for (int e = tid; e < m * so; e += kHWarps * 32) {
            const int k = e / so, r = e % so;
            O[e] = r < o ? f32_from_f64(Cm[k * m + r]) : 0.f;
        }
    };
    stage(VX, OX, C + d.cX, nX, oX, nXp, vXq, sX);
    stage(VY, OY, C + d.cY, nY, oY, nYp, vYq, sY);
    // the four blocks (32-bit indices below count rows of four: naux o v alone
    // passes 2^31 above 64 GB of factors, a quarter of it not within the device)
    float* xx = half + d.h_off;
    float* yy = xx + (long long)naux * oX * vXq;
    float* xy = yy + (long long)naux * oY * vYq;
    float* yx = xy + (long long)naux * oX * vYq;
    const int cbX = (vXq + 31) / 32, cbY = (vYq + 31) / 32;
    for (int qb = q0; qb < q1; qb += hq) {
        const int qn = min(hq, q1 - qb);
        __syncthreads();                       // C and the zeros staged; the previous round's u consumed
        float2 acc[2][RB / 2];                 // a lane's two columns
        while (cur.qb == qb && cur.t < qn * 2 * ng) {
            const Step next = advance(cur);
            double2 y[8];
            fetch(next, y);
            const int qq = cur.t / (2 * ng), g = cur.t % (2 * ng), hy = g >= ng;
            const int len = hy ? nY : nX, so = hy ? sY : sX;
            const float* O = (hy ? OY : OX) + (cur.m0 + par) * so + cur.r0;
            if (cur.m0 == 0)
#pragma unroll
                for (int r = 0; r < RB / 2; r++) acc[0][r] = acc[1][r] = make_float2(0.f, 0.f);
            auto add = [&](int k) {
                const float b0 = f32_from_f64(x[k].x), b1 = f32_from_f64(x[k].y);
                const float2* w = reinterpret_cast<const float2*>(O + 2 * k * so);
#pragma unroll
                for (int r = 0; r < RB / 2; r++) {
                    acc[0][r] = __ffma2_rn(w[r], make_float2(b0, b0), acc[0][r]);
                    acc[1][r] = __ffma2_rn(w[r], make_float2(b1, b1), acc[1][r]);
                }
            };
            if (cur.m0 + 16 <= len) {
#pragma unroll
                for (int k = 0; k < 8; k++) add(k);
            } else {
#pragma unroll
                for (int k = 0; k < 8; k++)
                    if (cur.m0 + par + 2 * k < len) add(k);
            }
            if (cur.m0 + 16 >= len) {
                const int o = hy ? oY : oX, c = (hy ? g - ng : g) * 32 + 2 * (lane & 15);
                float* u = U + (qq * ot + (hy ? oX : 0) + cur.r0) * uw;
                const int c0 = c < nX ? c : nXp + c - nX, c1 = c + 1 < nX ? c + 1 : nXp + c + 1 - nX;
#pragma unroll
                for (int r = 0; r < RB / 2; r++) {
                    float2 a[2];
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        a[h].x = acc[h][r].x + __shfl_xor_sync(0xffffffffu, acc[h][r].x, 16);
                        a[h].y = acc[h][r].y + __shfl_xor_sync(0xffffffffu, acc[h][r].y, 16);
                    }
                    // the lower half-warp writes the first column, the upper the second
                    const float2 v = par ? a[1] : a[0];
                    const int cc = par ? c1 : c0;
                    if (c + par < n) {
                        if (cur.r0 + 2 * r < o) u[2 * r * uw + cc] = v.x;
                        if (cur.r0 + 2 * r + 1 < o) u[(2 * r + 1) * uw + cc] = v.y;
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 8; k++) x[k] = y[k];
            cur = next;
        }
        if (cur.qb == qb) {                    // no task for this warp in the round
            cur = Step{qb + hq, warp, 0, 0};
            if (cur.qb < q1) fetch(cur, x);
        }
        __syncthreads();
        const int rows = qn * ot, ngr = (rows + kHRows - 1) / kHRows;
        for (int t = warp; t < ngr * (cbX + cbY); t += kHWarps) {
            const int gr = t / (cbX + cbY), cb = t % (cbX + cbY), hy = cb >= cbX;
            const int c = (hy ? cb - cbX : cb) * 32 + lane, vq = hy ? vYq : vXq;
            const float2* V = (hy ? VY : VX) + min(c, vq - 1);
            const float* u[kHRows];
            float2 a2[kHRows];
#pragma unroll
            for (int r = 0; r < kHRows; r++) {
                u[r] = U + min(gr * kHRows + r, rows - 1) * uw + (hy ? nXp : 0);
                a2[r] = make_float2(0.f, 0.f);
            }
            const int np = (hy ? nYp : nXp) / 2;
#pragma unroll 2
            for (int k = 0; k < np; k += 2) {
                const float2 c0 = V[k * vq], c1 = V[(k + 1) * vq];
#pragma unroll
                for (int r = 0; r < kHRows; r++) {
                    const float4 z = *reinterpret_cast<const float4*>(u[r] + 2 * k);
                    a2[r] = __ffma2_rn(make_float2(z.x, z.y), c0, a2[r]);
                    a2[r] = __ffma2_rn(make_float2(z.z, z.w), c1, a2[r]);
                }
            }
            if (c < vq) {
                int q = gr * kHRows / ot, o = gr * kHRows - q * ot;
#pragma unroll
                for (int r = 0; r < kHRows; r++) {
                    if (gr * kHRows + r < rows) {
                        float4* out = o < oX ? reinterpret_cast<float4*>(hy ? xy : xx) + ((qb + q) * oX + o) * (vq / 4)
                                             : reinterpret_cast<float4*>(hy ? yy : yx) + ((qb + q) * oY + o - oX) * (vq / 4);
                        reinterpret_cast<float*>(out)[c] = a2[r].x + a2[r].y;
                    }
                    if (++o == ot) { o = 0; q++; }
                }
            }
        }
    }
}

constexpr int kDQ = 16;                        // Q values per staged chunk
constexpr int kDJ = 5;                         // most j of a CTA

// FP64 from FP32, exact for every value: normal ones on the integer pipes, the
// rest (zeros, subnormals, infinities, NaN) by the conversion unit, out of line
// so that it does not issue for the others.
__device__ __noinline__ double convert(float f) { return (double)f; }

__device__ __forceinline__ double widen(float f)
{
    const unsigned e = (__float_as_uint(f) >> 23) & 0xFFu;
    return e - 1u < 254u ? f64_from_f32(f) : convert(f);
}

__device__ __noinline__ double divide(double v, double x) { return v / x; }

// One energy term in FP64, v and w the unscaled (ia|jb) and (ib|ja), x the
// denominator: v / x to FP64 rounding by two Newton steps (convert.h) where |x|
// lies in 2^+-124, as the differences of orbital energies do, else by division.
// On FP32 pairs (2^-45) with the squares formed in FP32 the terms were less
// accurate and overflowed where s v does not.  (Out of line the rare paths cost
// no registers of the loop above.)
__device__ __forceinline__ void df_term(double& sj, double& sk, float v, float w, double x)
{
    const double vd = widen(v);
    const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7FFu;
    const double t = e - 899u < 249u ? div_newton<2>(vd, x) : divide(vd, x);
    sj = fma(t, vd, sj);
    sk = fma(t, widen(w), sk);
}

// The j block [j0, j0 + JB) of occupied i: a thread holds 4 a x 4 b x JB values of
// (ia|jb) and of (ib|ja), two per packed multiply-add; per Q, 2 + 2 JB 16-byte
// shared loads feed 32 JB multiply-adds.  Bound by latency at two warps per
// scheduler (231 registers; FMA pipe 32 % busy, shared memory 23 % of its
// wavefronts), then by the FP64 pipe in the epilogue.  The kernel before it took
// one (i, j) per CTA with one element per thread (4 shared loads per 2
// multiply-adds) and an FP64 division per term: 2.08 ms for 1036 dimers of
// 32 + 32 AO and naux 192 against 0.75 ms (0.24 of it the epilogue).
template <int JB>
__device__ __forceinline__ void df_pairs(const DfDim& d, const double* __restrict__ eps,
                                         const float* __restrict__ half, int i, int j0, float* buf, double& ej,
                                         double& ek)
{
    const int nX = d.nX, nY = d.nY, oX = d.oX, oY = d.oY, vX = nX - oX, vY = nY - oY;
    const int vXq = up4(vX), vYq = up4(vY), nb = vYq / 4, nt = vXq / 4 * nb;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const float* xx = half + d.h_off + i * vXq;
    const float* yy = half + d.h_off + (long long)d.naux * oX * vXq + j0 * vYq;
    const float* xy = half + d.h_off + (long long)d.naux * (oX * vXq + oY * vYq) + i * vYq;
    const float* yx = half + d.h_off + (long long)d.naux * (oX * vXq + oY * vYq + oX * vYq) + j0 * vXq;
    // a staged Q is one row: xx, xy, yy[JB], yx[JB]
    const int oxy = vXq, oyy = vXq + vYq, oyx = oyy + JB * vYq, per = oyx + JB * vXq;
    auto stage = [&](int q0, int b) {          // a thread copies its 16-byte columns of every row
        const int qn = min(kDQ, d.naux - q0);
        for (int c = 4 * tid; c < per; c += 4 * nthr) {
            const float* src = c < oxy ? xx + c : c < oyy ? xy + c - oxy : c < oyx ? yy + c - oyy : yx + c - oyx;
            const int ld = c < oxy ? oX * vXq : c < oyy ? oX * vYq : c < oyx ? oY * vYq : oY * vXq;
            src += (long long)q0 * ld;
            unsigned dst = (unsigned)__cvta_generic_to_shared(buf + b * kDQ * per + c);
            for (int q = 0; q < qn; q++, src += ld, dst += per * sizeof(float))
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto ld = [](const float* p, float (&x)[4]) {
        const float4 y = *reinterpret_cast<const float4*>(p);
        x[0] = y.x; x[1] = y.y; x[2] = y.z; x[3] = y.w;
    };
    const double ei = eps[d.eX + i];
    for (int t0 = 0; t0 < nt; t0 += nthr) {
        const int t = min(t0 + tid, nt - 1), a0 = t / nb * 4, b0 = t % nb * 4;
        float2 v[JB][4][2], w[JB][4][2];       // (ia|jb): [j][a][b pair]; (ib|ja): [j][b][a pair]
#pragma unroll
        for (int j = 0; j < JB; j++)
#pragma unroll
            for (int x = 0; x < 4; x++)
#pragma unroll
                for (int y = 0; y < 2; y++) v[j][x][y] = w[j][x][y] = make_float2(0.f, 0.f);
        __syncthreads();                       // the previous pass has consumed the buffers
        stage(0, 0);
        int b = 0;
        for (int q0 = 0; q0 < d.naux; q0 += kDQ, b ^= 1) {
            const int qn = min(kDQ, d.naux - q0);
            if (q0 + kDQ < d.naux) {
                stage(q0 + kDQ, b ^ 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            const float* row = buf + b * kDQ * per;
            for (int q = 0; q < qn; q++, row += per) {
                float xa[4], xb[4];
                ld(row + a0, xa);
                ld(row + oxy + b0, xb);
#pragma unroll
                for (int j = 0; j < JB; j++) {
                    float yb[4], ya[4];
                    ld(row + oyy + j * vYq + b0, yb);
                    ld(row + oyx + j * vXq + a0, ya);
#pragma unroll
                    for (int x = 0; x < 4; x++)
#pragma unroll
                        for (int y = 0; y < 2; y++) {
                            v[j][x][y] = __ffma2_rn(make_float2(xa[x], xa[x]), make_float2(yb[2 * y], yb[2 * y + 1]),
                                                    v[j][x][y]);
                            w[j][x][y] = __ffma2_rn(make_float2(xb[x], xb[x]), make_float2(ya[2 * y], ya[2 * y + 1]),
                                                    w[j][x][y]);
                        }
                }
            }
            __syncthreads();                   // chunk consumed before its buffer is refilled
        }
        if (t0 + tid >= nt) continue;
        double eb[4];
#pragma unroll
        for (int y = 0; y < 4; y++) eb[y] = b0 + y < vY ? eps[d.eY + oY + b0 + y] : 0.0;
#pragma unroll
        for (int x = 0; x < 4; x++) {
            if (a0 + x >= vX) break;
            const double ea = eps[d.eX + oX + a0 + x];
#pragma unroll
            for (int j = 0; j < JB; j++) {
                const double eija = ei + eps[d.eY + j0 + j] - ea;
#pragma unroll
                for (int y = 0; y < 4; y++) {
                    if (b0 + y >= vY) break;
                    df_term(ej, ek, y & 1 ? v[j][x][y / 2].y : v[j][x][y / 2].x,
                            x & 1 ? w[j][y][x / 2].y : w[j][y][x / 2].x, eija - eb[y]);
                }
            }
        }
    }
}

// CTAs of a dimer: i-major, near-equal j blocks of at most jmax <= kDJ.
__global__ void __launch_bounds__(256)
k_df_pair(const DfDim* __restrict__ dims, const double* __restrict__ eps, const float* __restrict__ half,
          double* __restrict__ part, int jmax)
{
    const DfDim& d = dims[blockIdx.y];
    const int njb = (d.oY + jmax - 1) / jmax, k = blockIdx.x;
    if (k >= d.oX * njb) return;
    const int i = k / njb, jb = k % njb;
    const int j0 = jb * d.oY / njb, jn = (jb + 1) * d.oY / njb - j0;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* buf = reinterpret_cast<float*>(smem_raw);
    double ej = 0.0, ek = 0.0;
    switch (jn) {
    case 1: df_pairs<1>(d, eps, half, i, j0, buf, ej, ek); break;
    case 2: df_pairs<2>(d, eps, half, i, j0, buf, ej, ek); break;
    case 3: df_pairs<3>(d, eps, half, i, j0, buf, ej, ek); break;
    case 4: df_pairs<4>(d, eps, half, i, j0, buf, ej, ek); break;
    default: df_pairs<5>(d, eps, half, i, j0, buf, ej, ek); break;
    }
    // fixed-order block reduction
    __shared__ double red[2][8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ej += __shfl_down_sync(0xffffffffu, ej, o);
        ek += __shfl_down_sync(0xffffffffu, ek, o);
    }
    if (lane == 0) { red[0][warp] = ej; red[1][warp] = ek; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sj = 0.0, sk = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) { sj += red[0][w]; sk += red[1][w]; }
        // s and s again: its square alone may leave FP64's range where s v does not
        part[2 * (d.p_off + k)] = d.s * (d.s * (4.0 * sj));
        part[2 * (d.p_off + k) + 1] = d.s * (d.s * (-2.0 * sk));
    }
}

// ---- the FP64 form: bound by the FP64 pipe in both kernels (29 GFLOP, 23.4 of
// the 25 ms of 1036 dimers of 32 + 32 AO), so that operands may come from shared
// memory one by one, and padding -- the FP32 kernels' 4 x 4 blocks and padded
// rows measured 1.39 times slower here -- is what costs.  Rows unpadded.
// A CTA per (dimer, Q).
__global__ void __launch_bounds__(256)
k_df_half_fp64(const DfDim* __restrict__ dims, const double* __restrict__ C, double* __restrict__ half)
{
    const DfDim d = dims[blockIdx.y];
    const int q = blockIdx.x;
    if (q >= d.naux) return;
    const int nX = d.nX, nY = d.nY, n = nX + nY, oX = d.oX, oY = d.oY, vX = nX - oX, vY = nY - oY;
    const double* B = d.B + (long long)q * n * n;
    // shared: B^Q [n][n], C_X [nX][nX], C_Y [nY][nY], then u_X [oX][n], u_Y [oY][n]
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* sB = reinterpret_cast<double*>(smem_raw);
    double* sCX = sB + n * n;
    double* sCY = sCX + nX * nX;
    double* uX = sCY + nY * nY;
    double* uY = uX + oX * n;
    // eight loads in flight per thread
    for (int e0 = threadIdx.x; e0 < n * n; e0 += 8 * blockDim.x) {
        double x[8];
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int e = e0 + u * blockDim.x;
            x[u] = e < n * n ? B[e] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int e = e0 + u * blockDim.x;
            if (e < n * n) sB[e] = x[u];
        }
    }
    for (int e = threadIdx.x; e < nX * nX; e += blockDim.x) sCX[e] = C[d.cX + e];
    for (int e = threadIdx.x; e < nY * nY; e += blockDim.x) sCY[e] = C[d.cY + e];
    __syncthreads();
    for (int e = threadIdx.x; e < (oX + oY) * n; e += blockDim.x) {
        const int r = e / n, c = e % n;
        double a0 = 0.0, a1 = 0.0;                // two chains for latency
        if (r < oX) {
            int mu = 0;
            for (; mu + 1 < nX; mu += 2) {
                a0 = fma(sCX[mu * nX + r], sB[mu * n + c], a0);
                a1 = fma(sCX[(mu + 1) * nX + r], sB[(mu + 1) * n + c], a1);
            }
            if (mu < nX) a0 = fma(sCX[mu * nX + r], sB[mu * n + c], a0);
        } else {
            const int j = r - oX;
            int la = 0;
            for (; la + 1 < nY; la += 2) {
                a0 = fma(sCY[la * nY + j], sB[(nX + la) * n + c], a0);
                a1 = fma(sCY[(la + 1) * nY + j], sB[(nX + la + 1) * n + c], a1);
            }
            if (la < nY) a0 = fma(sCY[la * nY + j], sB[(nX + la) * n + c], a0);
        }
        uX[e] = a0 + a1;                       // uY follows uX contiguously
    }
    __syncthreads();
    const long long mX = (long long)oX * vX, mY = (long long)oY * vY, xb = (long long)oX * vY, yb = (long long)oY * vX;
    double* xx = half + d.h_off + (long long)q * mX;
    double* yy = half + d.h_off + (long long)d.naux * mX + (long long)q * mY;
    double* xy = half + d.h_off + (long long)d.naux * (mX + mY) + (long long)q * xb;
    double* yx = half + d.h_off + (long long)d.naux * (mX + mY + xb) + (long long)q * yb;
    // the four o x v blocks: out[r][c] = sum_k u[r][k0 + k] C[k][o + c]
    const int tot = (int)(mX + mY + xb + yb);
    for (int e = threadIdx.x; e < tot; e += blockDim.x) {
        const double* u;
        const double* Cm;
        int len, ldc, co, r, c;
        double* out;
        if (e < mX) {
            r = e / vX; c = e % vX; u = uX + r * n; Cm = sCX; len = nX; ldc = nX; co = oX; out = xx + e;
        } else if (e < mX + mY) {
            const int f = e - (int)mX;
            r = f / vY; c = f % vY; u = uY + r * n + nX; Cm = sCY; len = nY; ldc = nY; co = oY; out = yy + f;
        } else if (e < mX + mY + xb) {
            const int f = e - (int)(mX + mY);
            r = f / vY; c = f % vY; u = uX + r * n + nX; Cm = sCY; len = nY; ldc = nY; co = oY; out = xy + f;
        } else {
            const int f = e - (int)(mX + mY + xb);
            r = f / vX; c = f % vX; u = uY + r * n; Cm = sCX; len = nX; ldc = nX; co = oX; out = yx + f;
        }
        double a0 = 0.0, a1 = 0.0;
        int k = 0;
        for (; k + 1 < len; k += 2) {
            a0 = fma(u[k], Cm[k * ldc + co + c], a0);
            a1 = fma(u[k + 1], Cm[(k + 1) * ldc + co + c], a1);
        }
        if (k < len) a0 = fma(u[k], Cm[k * ldc + co + c], a0);
        *out = a0 + a1;
    }
}

constexpr int kDQ64 = 32;                      // Q values per staged chunk

// A CTA per (dimer, occupied pair i, j).
__global__ void __launch_bounds__(256)
k_df_pair_fp64(const DfDim* __restrict__ dims, const double* __restrict__ eps, const double* __restrict__ half,
               double* __restrict__ part)
{
    const DfDim d = dims[blockIdx.y];
    const int nX = d.nX, nY = d.nY, oX = d.oX, oY = d.oY, vX = nX - oX, vY = nY - oY;
    const int pr = blockIdx.x;                 // occupied pair i * oY + j
    if (pr >= oX * oY) return;
    const int i = pr / oY, j = pr % oY;
    const long long mX = (long long)oX * vX, mY = (long long)oY * vY, xb = (long long)oX * vY, yb = (long long)oY * vX;
    const double* xx = half + d.h_off;
    const double* yy = xx + (long long)d.naux * mX;
    const double* xy = yy + (long long)d.naux * mY;
    const double* yx = xy + (long long)d.naux * xb;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* sxx = reinterpret_cast<double*>(smem_raw);   // [kDQ64][vX]: xx[Q][i][.]
    double* syy = sxx + kDQ64 * vX;                   // [kDQ64][vY]: yy[Q][j][.]
    double* sxy = syy + kDQ64 * vY;                   // [kDQ64][vY]: xy[Q][i][.]
    double* syx = sxy + kDQ64 * vY;                   // [kDQ64][vX]: yx[Q][j][.]
    double* red = reinterpret_cast<double*>(syx + kDQ64 * vX + (kDQ64 * vX) % 2);
    const int nab = vX * vY;
    double ej = 0.0, ek = 0.0;
    // the thread owns the (a, b) elements e0 + tid + 256 u of each block of 1024
    for (int e0 = 0; e0 < nab; e0 += 256 * 4) {
        double v[4] = {0.0, 0.0, 0.0, 0.0}, w[4] = {0.0, 0.0, 0.0, 0.0};
        for (int q0 = 0; q0 < d.naux; q0 += kDQ64) {
            const int qn = min(kDQ64, d.naux - q0);
            __syncthreads();
            for (int e = threadIdx.x; e < qn * vX; e += blockDim.x) {
                const int qq = e / vX, a = e % vX;
                sxx[qq * vX + a] = xx[(long long)(q0 + qq) * mX + i * vX + a];
                syx[qq * vX + a] = yx[(long long)(q0 + qq) * yb + j * vX + a];
            }
            for (int e = threadIdx.x; e < qn * vY; e += blockDim.x) {
                const int qq = e / vY, b = e % vY;
                syy[qq * vY + b] = yy[(long long)(q0 + qq) * mY + j * vY + b];
                sxy[qq * vY + b] = xy[(long long)(q0 + qq) * xb + i * vY + b];
            }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int e = e0 + threadIdx.x + 256 * u;
                if (e < nab) {
                    const int a = e / vY, b = e % vY;
                    double vv = v[u], ww = w[u];
                    for (int qq = 0; qq < qn; qq++) {
                        vv = fma(sxx[qq * vX + a], syy[qq * vY + b], vv);
                        ww = fma(sxy[qq * vY + b], syx[qq * vX + a], ww);
                    }
                    v[u] = vv;
                    w[u] = ww;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int e = e0 + threadIdx.x + 256 * u;
            if (e < nab) {
                const int a = e / vY, b = e % vY;
                const double D = 1.0 / (eps[d.eX + i] + eps[d.eY + j] - eps[d.eX + oX + a] - eps[d.eY + oY + b]);
                const double vs = d.s * v[u], ws = d.s * w[u];
                ej += 4.0 * vs * vs * D;
                ek += -2.0 * vs * ws * D;
            }
        }
    }
    red[threadIdx.x] = ej;
    red[256 + threadIdx.x] = ek;
    __syncthreads();
    for (int h = 128; h; h >>= 1) {
        if (threadIdx.x < h) {
            red[threadIdx.x] += red[threadIdx.x + h];
            red[256 + threadIdx.x] += red[256 + threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[2 * (d.p_off + pr)] = red[0];
        part[2 * (d.p_off + pr) + 1] = red[256];
    }
}

// A dimer's partial energies in order, jmax its CTAs' j block: one warp, lanes
// strided, fixed tree.
__global__ void __launch_bounds__(32)
k_df_sum(const DfDim* __restrict__ dims, const double* __restrict__ part, double* __restrict__ E2, int jmax)
{
    const DfDim& d = dims[blockIdx.x];
    const int n = d.oX * ((d.oY + jmax - 1) / jmax);
    double ej = 0.0, ek = 0.0;
    for (int p = threadIdx.x; p < n; p += 32) {
        ej += part[2 * (d.p_off + p)];
        ek += part[2 * (d.p_off + p) + 1];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ej += __shfl_down_sync(0xffffffffu, ej, o);
        ek += __shfl_down_sync(0xffffffffu, ek, o);
    }
    if (threadIdx.x == 0) {
        E2[2 * d.id] = ej;
        E2[2 * d.id + 1] = ek;
    }
}

template <int RB>
cudaError_t launch_half(const DfDim* dims, int nd, const DfMax& m, const double* C, float* half, int sms,
                        cudaStream_t s)
{
    // four factors per round where two CTAs then fit an SM, else one or two
    int hq = kHQ;
    while (hq > 1 && ((size_t)hq * m.u_elems + m.c_elems) * sizeof(float) > 110 * 1024) hq /= 2;
    const size_t sh = ((size_t)hq * m.u_elems + m.c_elems) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(k_df_half<RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    if (e != cudaSuccess) return e;
    // Q per CTA: C staged once (about one Q's work) for up to 32, fewer where
    // the dimers are few, so that every SM gets about sixteen CTAs, two at a time
    const long long want = (long long)nd * m.naux / (16 * sms);
    const int qper = (int)std::min<long long>(32, std::max<long long>(1, want));
    k_df_half<RB><<<dim3((m.naux + qper - 1) / qper, nd), kHWarps * 32, sh, s>>>(dims, C, half, qper, std::min(hq, qper));
    return cudaGetLastError();
}

cudaError_t launch_df_fp32(const DfDim* dims, int nd, const DfMax& m, const double* C, const double* eps, float* half,
                           double* part, double* E2, int sms, cudaStream_t s)
{
    cudaError_t e = m.occ <= 4   ? launch_half<4>(dims, nd, m, C, half, sms, s)
                    : m.occ <= 6 ? launch_half<6>(dims, nd, m, C, half, sms, s)
                                 : launch_half<8>(dims, nd, m, C, half, sms, s);
    if (e != cudaSuccess) return e;
    // five j per CTA, fewer where that leaves SMs without one
    int jmax = std::min(kDJ, m.occ);
    while (jmax > 1 && (long long)nd * m.occ * ((m.occ + jmax - 1) / jmax) < 2 * sms) jmax--;
    const int vq = up4(m.v), tiles = (vq / 4) * (vq / 4), thr = std::min(256, std::max(32, (tiles + 31) / 32 * 32));
    const size_t sp = (size_t)2 * kDQ * (1 + jmax) * 2 * vq * sizeof(float);
    e = cudaFuncSetAttribute(k_df_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sp);
    if (e != cudaSuccess) return e;
    k_df_pair<<<dim3(m.occ * ((m.occ + jmax - 1) / jmax), nd), thr, sp, s>>>(dims, eps, half, part, jmax);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_df_sum<<<nd, 32, 0, s>>>(dims, part, E2, jmax);
    return cudaGetLastError();
}

cudaError_t launch_df_fp64(const DfDim* dims, int nd, const DfMax& m, const double* C, const double* eps, double* half,
                           double* part, double* E2, cudaStream_t s)
{
    const size_t sh = (size_t)m.b_elems * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(k_df_half_fp64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    if (e != cudaSuccess) return e;
    k_df_half_fp64<<<dim3(m.naux, nd), 256, sh, s>>>(dims, C, half);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const size_t sp = (size_t)4 * kDQ64 * m.v * sizeof(double) + 16 + 512 * sizeof(double);
    e = cudaFuncSetAttribute(k_df_pair_fp64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sp);
    if (e != cudaSuccess) return e;
    k_df_pair_fp64<<<dim3(m.occ * m.occ, nd), 256, sp, s>>>(dims, eps, half, part);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_df_sum<<<nd, 32, 0, s>>>(dims, part, E2, 1);
    return cudaGetLastError();
}

}  // namespace

void df_smem_elems(int nX, int nY, int oX, int oY, int* u_elems, int* c_elems)
{
    *u_elems = (oX + oY) * (up4(nX) + up4(nY));
    // virtual columns, and occupied ones padded to a register block (at most 7 more)
    *c_elems = up4(nX) * up4(nX - oX) + up4(nY) * up4(nY - oY) + nX * (oX + 7) + nY * (oY + 7);
}

long long df_half_elems(bool fp64, int naux, int nX, int nY, int oX, int oY)
{
    const long long vX = nX - oX, vY = nY - oY;
    return (long long)naux * (oX + oY) * (fp64 ? vX + vY : up4((int)vX) + up4((int)vY));
}

cudaError_t launch_df(bool fp64, const DfDim* dims, int nd, const DfMax& m, const double* C, const double* eps,
                      void* half, double* part, double* E2, int sms, cudaStream_t s)
{
    if (nd <= 0) return cudaSuccess;
    return fp64 ? launch_df_fp64(dims, nd, m, C, eps, static_cast<double*>(half), part, E2, s)
                : launch_df_fp32(dims, nd, m, C, eps, static_cast<float*>(half), part, E2, sms, s);
}

}  // namespace mcpt
