// k_fp32c.cu -- compensated-FP32 first half of the dimer transformation.
//
// Same contraction as the FP64 form,
//   H_f[(p1,p3)][(i,j)] = sum_{p0} C_X[p0][i] sum_{p2} C_Y[p2][j] E[p0][p1][p2][p3],
// but on the FP32 pipes: integrals and coefficients are rounded once to FP32,
// and every dot product is accumulated with the error-free transformations of
// Ogita, Rump and Oishi ("Accurate sum and dot product", SIAM J. Sci.
// Comput. 26, 2005): TwoProduct by FMA (h = x*y, r = fma(x, y, -h)) and
// Knuth's TwoSum, so each sum is as accurate as if computed in twice the
// working precision and then rounded (their Dot2).  The FP64 -> FP32
// rounding of each integral runs on the integer pipes (convert.h).  The inner sum over p2 is
// kept as an unevaluated pair (hi, lo) and multiplied into the outer sum over
// p0 the same way.
//
// k_half_fp32c_tiles is the kernel that runs.  It is bound by the FP32 pipes
// (8 operations per integral and occupied j, 9 per p0, row and occupied pair),
// so each of the two sums is formed once: the pairs F[p0][j] of a tile of 64
// rows go through a scratch slot (L2) between the two phases of a CTA.  The
// kernel before it, k_half_fp32c, holds an OB x OB block of sums per thread
// and forms F again for every block of i, 3 x 3 passes over the integrals at
// 20 occupied orbitals; it needs no scratch and stays for runs whose scratch
// limits leave no room for the slots.  Measured, whole calls, before and after:
// three dimers of 128 + 128 AO with 20 occupied 246 -> 13.5 ms (11.9 ms of it
// this kernel, 2.2 TB/s of integrals in two passes; the FP32 operations alone
// are 7.7 ms at the pipes' rate), 1036 of 32 + 32 AO 6.34 -> 5.30 ms, one of
// 32 + 32 AO 228 -> 150 us (its 32 tiles' p0 spread over eight warps each),
// 28 of 16 + 16 AO 145 -> 105 us.
#include "internal.h"
#include "convert.h"

#include <algorithm>

namespace mcpt {
namespace {

constexpr int kThreads = 128;

struct ff { float hi, lo; };   // value hi + lo, |lo| <= ulp(hi)/2 after renormalising

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = a + b;
    const float z = s - a;
    e = (a - (s - z)) + (b - z);
}

// acc += x * y with the product's and the sum's rounding errors kept in acc.lo
__device__ __forceinline__ void dot2_step(ff& acc, float x, float y)
{
    const float h = x * y;
    const float r = fmaf(x, y, -h);
    float s, q;
    two_sum(acc.hi, h, s, q);
    acc.hi = s;
    acc.lo += q + r;
}

// acc += w * (v.hi + v.lo)
__device__ __forceinline__ void dot2_step_ff(ff& acc, float w, ff v)
{
    dot2_step(acc, w, v.hi);
    acc.lo = fmaf(w, v.lo, acc.lo);
}

template <int OB>
__global__ void __launch_bounds__(kThreads)
k_half_fp32c(const DimerDesc* __restrict__ dd, const float* __restrict__ Cf, float* __restrict__ H)
{
    const DimerDesc& d = dd[blockIdx.z];
    const int f = blockIdx.y;
    const int n0 = d.nX, n1 = f ? d.nY : d.nX, n2 = d.nY, n3 = f ? d.nX : d.nY;
    const int rows = n1 * n3;
    if (blockIdx.x * kThreads >= rows) return;

    const int o0 = d.oX, o2 = d.oY;
    extern __shared__ float smf[];
    float* U0 = smf;               // [n0][OB]
    float* U2 = smf + n0 * OB;     // [n2][OB]
    const float* CX = Cf + d.cX;
    const float* CY = Cf + d.cY;

    const int r = blockIdx.x * kThreads + threadIdx.x;
    const bool active = r < rows;
    const int p1 = active ? r / n3 : 0, p3 = active ? r % n3 : 0;
    const long long s0 = d.st[f][0], s1 = d.st[f][1], s2 = d.st[f][2];
    const double* __restrict__ Erow = d.E[f] + p1 * s1 + p3;
    float* out = H + d.h_off + (long long)f * d.oX * d.oY * rows + r;   // pair-major

    for (int t0b = 0; t0b < o0; t0b += OB) {
        for (int t2b = 0; t2b < o2; t2b += OB) {
            __syncthreads();
            for (int k = threadIdx.x; k < n0 * OB; k += kThreads) {
                int p = k / OB, t = t0b + k % OB;
                U0[k] = t < o0 ? CX[p * d.nX + t] : 0.f;
            }
            for (int k = threadIdx.x; k < n2 * OB; k += kThreads) {
                int p = k / OB, t = t2b + k % OB;
                U2[k] = t < o2 ? CY[p * d.nY + t] : 0.f;
            }
            __syncthreads();
            if (!active) continue;
            ff acc[OB][OB];
#pragma unroll
            for (int a = 0; a < OB; a++)
#pragma unroll
                for (int t = 0; t < OB; t++) acc[a][t] = ff{0.f, 0.f};
            for (int p0 = 0; p0 < n0; p0++) {
                const double* __restrict__ Ep = Erow + p0 * s0;
                ff F[OB];
#pragma unroll
                for (int t = 0; t < OB; t++) F[t] = ff{0.f, 0.f};
#pragma unroll 4
                for (int p2 = 0; p2 < n2; p2++) {
                    const float e = f32_from_f64(__ldg(Ep + p2 * s2));   // integer-pipe conversion
                    const float* u = U2 + p2 * OB;
#pragma unroll
                    for (int t = 0; t < OB; t++) dot2_step(F[t], u[t], e);
                }
                const float* u0 = U0 + p0 * OB;
#pragma unroll
                for (int a = 0; a < OB; a++) {
                    const float w = u0[a];
#pragma unroll
                    for (int t = 0; t < OB; t++) dot2_step_ff(acc[a][t], w, F[t]);
                }
            }
#pragma unroll
            for (int a = 0; a < OB; a++)
#pragma unroll
                for (int t = 0; t < OB; t++)
                    if (t0b + a < o0 && t2b + t < o2) out[(long long)((t0b + a) * o2 + t2b + t) * rows] = acc[a][t].hi + acc[a][t].lo;
        }
    }
}

// ---------------------------------------------------------------------------
// Two rows per lane on the packed FP32 operations (one instruction for two
// values: half the issue slots, the same pipe time).
//
// acc += x * y: h = x y rounded, TwoSum(acc.hi, h) with its second error term
// taken from the exact product, b = fma(x, y, -z) in place of (h - z) + r: the
// sum of the TwoSum's exact h - z and the product's residual in one rounding.
// 8 operations instead of 10, and one rounding (of 2^-24 of an error term)
// fewer; the pairs rounded to FP32 agree with the 10-operation form bit for bit
// on every element compared.  The product is two scalar multiplications: a
// packed one is contracted with the addition that follows (the assembler does
// so for the packed operations, rounding modifier or not), and the TwoSum of
// an unrounded product is not error-free when it cancels.
struct ff2 { float2 hi, lo; };

__device__ __forceinline__ float2 neg2(float2 x) { return make_float2(-x.x, -x.y); }
// x - y (exactly rounded: the product by -1 is exact)
__device__ __forceinline__ float2 sub2(float2 x, float2 y) { return __ffma2_rn(y, make_float2(-1.f, -1.f), x); }

__device__ __forceinline__ void dot2_step2(ff2& acc, float2 x, float2 y)
{
    const float2 h = make_float2(__fmul_rn(x.x, y.x), __fmul_rn(x.y, y.y));
    const float2 s = __fadd2_rn(acc.hi, h);
    const float2 z = sub2(s, acc.hi);
    const float2 a = sub2(acc.hi, sub2(s, z));
    const float2 b = __ffma2_rn(x, y, neg2(z));
    acc.hi = s;
    acc.lo = __fadd2_rn(acc.lo, __fadd2_rn(a, b));
}

constexpr int kFcWarps = 8;            // warps per CTA
constexpr int kFcRows = 64;            // rows per tile: lane and lane + 32
constexpr int kFcTB = 10;              // most occupied j of one pass (F in registers: 4 TB)
constexpr int kFcAB = 10;              // most occupied i of one accumulator block (4 AB registers)
constexpr int kFcChunk = 4;            // p2 values loaded ahead

// Phase 1 of a tile: F[p0][t] = sum_{p2} U[p2][t] E[p0][p2] for the pass's TB
// occupied j, a warp per p0, into the slot as (hi row A, hi row B, lo A, lo B).
template <int TB>
__device__ __forceinline__ void fc_inner(const double* __restrict__ ra, const double* __restrict__ rb, long long s0,
                                         long long s2, int n0, int n2, const float2* __restrict__ U,
                                         float4* __restrict__ slot, int warp, int lane)
{
    for (int p0 = warp; p0 < n0; p0 += kFcWarps) {
        const double* pa = ra + p0 * s0;
        const double* pb = rb + p0 * s0;
        ff2 F[TB];
#pragma unroll
        for (int t = 0; t < TB; t++) F[t] = ff2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        double xa[kFcChunk], xb[kFcChunk];
#pragma unroll
        for (int k = 0; k < kFcChunk; k++) {
            xa[k] = k < n2 ? __ldg(pa + k * s2) : 0.0;
            xb[k] = k < n2 ? __ldg(pb + k * s2) : 0.0;
        }
#pragma unroll 1
        for (int p2 = 0; p2 < n2; p2 += kFcChunk) {
            float2 e[kFcChunk];
#pragma unroll
            for (int k = 0; k < kFcChunk; k++) e[k] = make_float2(f32_from_f64(xa[k]), f32_from_f64(xb[k]));
#pragma unroll
            for (int k = 0; k < kFcChunk; k++) {   // the next chunk in flight during this one
                const int p = p2 + kFcChunk + k;
                xa[k] = p < n2 ? __ldg(pa + p * s2) : 0.0;
                xb[k] = p < n2 ? __ldg(pb + p * s2) : 0.0;
            }
            // the chunk's coefficients two per 16-byte broadcast load; rows past n2 are zero
            const float4* u = reinterpret_cast<const float4*>(U + p2 * TB);
#pragma unroll
            for (int q = 0; q < kFcChunk * TB; q += 2) {
                const float4 c = u[q / 2];
                dot2_step2(F[q % TB], make_float2(c.x, c.y), e[q / TB]);
                dot2_step2(F[(q + 1) % TB], make_float2(c.z, c.w), e[(q + 1) / TB]);
            }
        }
#pragma unroll
        for (int t = 0; t < TB; t++)
            __stcg(slot + (p0 * TB + t) * 32 + lane, make_float4(F[t].hi.x, F[t].hi.y, F[t].lo.x, F[t].lo.y));
    }
}

// Phase 2 of a tile: sum_{p0} W[p0][a] F[p0][t] for AB occupied i of one t,
// written to H (out: row A of pair (first i, t); ok: which of the two rows exist).
template <int AB>
__device__ __forceinline__ void fc_outer(const float4* __restrict__ F, int tb, int n0, const float2* __restrict__ W,
                                         int na, float* __restrict__ out, long long astride, bool okA, bool okB)
{
    ff2 acc[AB];
#pragma unroll
    for (int a = 0; a < AB; a++) acc[a] = ff2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    const int st = tb * 32;
#pragma unroll 4
    for (int p0 = 0; p0 < n0; p0++) {
        const float4 v = __ldcg(F + p0 * st);
        const float2 vh = make_float2(v.x, v.y), vl = make_float2(v.z, v.w);
        const float2* w = W + p0 * AB;
#pragma unroll
        for (int a = 0; a < AB; a++) {
            float2 wa;
            if constexpr (AB % 2 == 0) {       // two coefficients per 16-byte broadcast load
                const float4 c = reinterpret_cast<const float4*>(w)[a / 2];
                wa = a & 1 ? make_float2(c.z, c.w) : make_float2(c.x, c.y);
            } else {
                wa = w[a];
            }
            dot2_step2(acc[a], wa, vh);
            acc[a].lo = __ffma2_rn(wa, vl, acc[a].lo);
        }
    }
#pragma unroll
    for (int a = 0; a < AB; a++) {
        if (a < na) {
            if (okA) out[a * astride] = acc[a].hi.x + acc[a].lo.x;
            if (okB) out[a * astride + 32] = acc[a].hi.y + acc[a].lo.y;
        }
    }
}

// Coefficients of n occupied orbitals from column c0 on, each value twice (the
// packed operations' broadcast operand), rows past nrow zero, columns padded to B.
__device__ __forceinline__ void fc_stage(float2* __restrict__ dst, const float* __restrict__ C, int ld, int nrow,
                                         int nrow_pad, int c0, int n, int B)
{
    for (int k = threadIdx.x; k < nrow_pad * B; k += kFcWarps * 32) {
        const int p = k / B, t = k % B;
        const float x = (p < nrow && t < n) ? C[p * ld + c0 + t] : 0.f;
        dst[k] = make_float2(x, x);
    }
}

#define FC_SWITCH(width, call)                      \
    switch (width) {                                \
    case 1: { constexpr int B = 1; call; } break;   \
    case 2: { constexpr int B = 2; call; } break;   \
    case 3: { constexpr int B = 3; call; } break;   \
    case 4: { constexpr int B = 4; call; } break;   \
    case 5: { constexpr int B = 5; call; } break;   \
    case 6: { constexpr int B = 6; call; } break;   \
    case 7: case 8: { constexpr int B = 8; call; } break; \
    default: { constexpr int B = 10; call; } break; \
    }
__device__ __forceinline__ int fc_width(int w) { return w <= 6 ? w : w <= 8 ? 8 : 10; }

// Persistent: CTAs take (dimer, form, tile of 64 rows) units from a counter.
// Occupied j run in near-equal passes of at most 10 (the integrals are read
// once per pass), occupied i in near-equal blocks of at most 10 that read the
// pass's F back from the CTA's slot (n0 TB 512 bytes).
__global__ void __launch_bounds__(kFcWarps * 32, 2)
k_half_fp32c_tiles(const DimerDesc* __restrict__ dd, int units, int max_tiles, const float* __restrict__ Cf,
                   float* __restrict__ H, unsigned* __restrict__ counter, float4* __restrict__ slots,
                   long long slot_elems)
{
    extern __shared__ __align__(16) unsigned char fc_smem[];
    float2* U = reinterpret_cast<float2*>(fc_smem);                     // [p2][TB], then [p0][AB]
    __shared__ int s_unit;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4* slot = slots + blockIdx.x * slot_elems;
    for (;;) {
        __syncthreads();                       // the previous unit's shared values are no longer read
        if (threadIdx.x == 0) s_unit = (int)atomicAdd(counter, 1u);
        __syncthreads();
        const int unit = s_unit;
        if (unit >= units) return;
        const int tile = unit % max_tiles, f = (unit / max_tiles) & 1;
        const DimerDesc& d = dd[unit / (2 * max_tiles)];
        const int n0 = d.nX, n2 = d.nY, n1 = f ? d.nY : d.nX, n3 = f ? d.nX : d.nY;
        const int rows = n1 * n3;
        if (tile * kFcRows >= rows) continue;
        const int o0 = d.oX, o2 = d.oY;
        const long long s0 = d.st[f][0], s1 = d.st[f][1], s2 = d.st[f][2];
        const int rA = tile * kFcRows + lane, rB = rA + 32;
        const bool okA = rA < rows, okB = rB < rows;
        const int qA = okA ? rA : 0, qB = okB ? rB : 0;    // rows past the end read row 0, write nothing
        const double* ra = d.E[f] + (qA / n3) * s1 + qA % n3;
        const double* rb = d.E[f] + (qB / n3) * s1 + qB % n3;
        float* out = H + d.h_off + (long long)f * o0 * o2 * rows + rA;   // pair-major
        const int np2 = (n2 + kFcChunk - 1) / kFcChunk * kFcChunk;
        const int npass = (o2 + kFcTB - 1) / kFcTB, nblk = (o0 + kFcAB - 1) / kFcAB;
        for (int ps = 0; ps < npass; ps++) {
            const int t0 = ps * o2 / npass, tn = (ps + 1) * o2 / npass - t0, tb = fc_width(tn);
            __syncthreads();                   // the previous pass's slot and coefficients are consumed
            fc_stage(U, Cf + d.cY, d.nY, n2, np2, t0, tn, tb);
            __syncthreads();
            FC_SWITCH(tb, (fc_inner<B>(ra, rb, s0, s2, n0, n2, U, slot, warp, lane)))
            for (int ab = 0; ab < nblk; ab++) {
                const int a0 = ab * o0 / nblk, an = (ab + 1) * o0 / nblk - a0, aw = fc_width(an);
                __syncthreads();               // F written (ab = 0); the previous block's coefficients consumed
                fc_stage(U, Cf + d.cX, d.nX, n0, n0, a0, an, aw);
                __syncthreads();
                for (int t = warp; t < tn; t += kFcWarps)
                    FC_SWITCH(aw, (fc_outer<B>(slot + t * 32 + lane, tb, n0, U, an,
                                               out + (long long)(a0 * o2 + t0 + t) * rows, (long long)o2 * rows, okA,
                                               okB)))
            }
        }
    }
}

template <int OB>
cudaError_t launch(const DimerDesc* d_desc, int nd, int max_rows, const float* Cf, float* H, cudaStream_t s)
{
    const size_t smem = (size_t)2 * kMaxAOTensor * OB * sizeof(float);
    dim3 grid((max_rows + kThreads - 1) / kThreads, 2, nd);
    k_half_fp32c<OB><<<grid, kThreads, smem, s>>>(d_desc, Cf, H);
    return cudaGetLastError();
}

}  // namespace

size_t fp32c_slot_bytes(int nX, int oY)
{
    const int npass = (oY + kFcTB - 1) / kFcTB, w = (oY + npass - 1) / npass;
    return (size_t)nX * (w <= 6 ? w : w <= 8 ? 8 : 10) * 32 * sizeof(float4);
}

cudaError_t launch_half_fp32c(const DimerDesc* d_desc, int nd, int max_rows, int max_occ, const float* Cf,
                              float* H, void* scratch, int slots, size_t slot_bytes, cudaStream_t s)
{
    if (nd <= 0) return cudaSuccess;
    if (slots > 0) {
        const int max_tiles = (max_rows + kFcRows - 1) / kFcRows;
        const int units = 2 * nd * max_tiles;
        const size_t smem = (size_t)kMaxAOTensor * kFcTB * sizeof(float2);
        cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(unsigned), s);
        if (e != cudaSuccess) return e;
        k_half_fp32c_tiles<<<std::min(units, slots), kFcWarps * 32, smem, s>>>(
            d_desc, units, max_tiles, Cf, H, static_cast<unsigned*>(scratch),
            reinterpret_cast<float4*>(static_cast<char*>(scratch) + kFp32cCounterBytes),
            (long long)(slot_bytes / sizeof(float4)));
        return cudaGetLastError();
    }
    if (max_occ <= 4) return launch<4>(d_desc, nd, max_rows, Cf, H, s);
    if (max_occ <= 5) return launch<5>(d_desc, nd, max_rows, Cf, H, s);
    return launch<8>(d_desc, nd, max_rows, Cf, H, s);
}

}  // namespace mcpt
