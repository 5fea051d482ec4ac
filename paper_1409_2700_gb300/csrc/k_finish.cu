// k_finish.cu -- second half of the dimer transformation, the FP64 energy
// epilogue, and the per-monomer accumulation.
//
// For each occupied pair (i, j) the first half left two nX x nY matrices
//   H_0[(nu,sig)][(i,j)]   (nu in X, sig in Y)   from the (XX|YY) block
//   H_1[(lam,nu)][(i,j)]   (lam in Y, nu in X)   from the (XY|YX) block
// and the virtual quarter transformations of Eq. (dp2e) finish them:
//   (i a|j b) = sum_nu C_X[nu][a] sum_sig H_0[nu][sig] C_Y[sig][b]
//   (i b|j a) = sum_lam C_Y[lam][b] sum_nu H_1[lam][nu] C_X[nu][a]
// Then, at FP64 accuracy (Sec. II.C energy tensor, Eq. (ed2) with T = vD):
//   D = 1/(e_i + e_j - e_a - e_b),  E_J += 4 (ia|jb)^2 D,  E_K += -2 (ia|jb)(ib|ja) D.
// GB300's FP64 unit runs at 1/64 of its FP32 rate.  The FP64 form keeps every
// step on it at the fewest operations per term: v D from an FP32 reciprocal
// seed and two Newton steps in FP64, the last folded into the product
// (convert.h), then one FMA each for E_J and E_K.  The mixed forms take
// e_i + e_j - e_a in FP64 once per (pair, a) and the rest on FP32 pairs
// (48-bit double-length arithmetic, below): the last subtraction, D to ~2^-45
// relative (the accuracy of one FP64 Newton step from an FP32 seed), the
// products with D and the sums over b, added to the FP64 sums once per pair --
// no FP64 operation per term.  The FP64-pipe variant of that epilogue (five
// FP64 operations per term) stays selectable for comparison.
// Monomers of at most 32 AO: one warp per occupied pair, a dimer's pairs over
// one or more CTAs; the last of them to arrive adds the pairs' sums.
// Larger ones: register-tiled GEMMs, one CTA per range of a dimer's pairs; one
// partial sum per range in FP64, one per pair in FP32, added per dimer with
// strided lanes and a fixed tree.  Every sum has a fixed order, so the energies
// are deterministic run to run: the only atomics are arrival counters (zero
// before a launch and after it) that pick the block which does the last pass.
#include "internal.h"
#include "convert.h"
#include "ff.h"

#include <algorithm>

namespace mcpt {
namespace {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// FP64 to the storage type (FP32 through the integer pipes)
template <typename T> __device__ __forceinline__ T narrow(double x);
template <> __device__ __forceinline__ double narrow<double>(double x) { return x; }
template <> __device__ __forceinline__ float narrow<float>(double x) { return f32_from_f64(x); }

// The mixed forms' terms of one (i, a, j, b) on FP32 pairs: x = e_ija - e_b,
// D = 1/x, E_J += v^2 D, E_K += v vk D into the pair accumulators sj, sk;
// returns v D (FP32) for the coupling store.  v^2 and v vk are FP32 products
// as in the FP64 variant; D, the products with D and the sums keep ~2^-45.
__device__ __forceinline__ float energy_terms_ff(float v, float vk, FF eija, FF eb, FF& sj, FF& sk)
{
    const FF D = ff_rcp(ff_sub(eija, eb));
    ff_acc(sj, __fmul_rn(v, v), D);
    ff_acc(sk, __fmul_rn(v, vk), D);
    return fmaf(v, D.l, __fmul_rn(v, D.h));
}

// The energy terms of one (i, a, j, b) with v = (ia|jb), vk = (ib|ja) and the
// FP64 denominator x = e_i + e_j - e_a - e_b: D = 1/x in FP64, then
// E_J += v^2 D and E_K += v vk D as FP64 sums; *vd (may be null) gets v D.
// FP64 form: v D by two Newton steps from an FP32 seed, the last folded into
// the product (full FP64 accuracy).  Mixed forms: D = r + r (1 - x r) from
// the FP32 seed r (relative error ~2^-46), v^2 and v vk as FP32 products (one
// rounding of 2^-24, far below the error these forms carry into v): five
// FP64 operations per term, the fewest that keep D and the sums in FP64.
template <typename T>
__device__ __forceinline__ void energy_terms(T v, T vk, double x, double& ej, double& ek, double* vd)
{
    if constexpr (sizeof(T) == 8) {
        const double t = div_newton<2>(v, x);
        ej = fma(t, v, ej);
        ek = fma(t, vk, ek);
        if (vd) *vd = t;
    } else {
        const double r = rcp_seed_f64(x);
        const double D = fma(r, fma(-x, r, 1.0), r);
        ej = fma(f64_from_f32(v * v), D, ej);
        ek = fma(f64_from_f32(v * vk), D, ek);
        if (vd) *vd = f64_from_f32(v) * D;
    }
}

// ---------------------------------------------------------------------------
// Monomers of at most 32 AO: one warp per occupied pair (i, j).
//   lane b:  tm[nu] = sum_sig H0[nu][sig] C_Y[sig][b]         (C_Y column b in registers)
//            VA[a][b] = sum_nu C_X[nu][a] tm[nu]              (C_X rows broadcast from smem)
//   lane a:  tk[lam] = sum_nu H1[lam][nu] C_X[nu][a]
//            VK[b][a] = sum_lam C_Y[lam][b] tk[lam]           (FP32: all b, into a third slab;
//                                                              FP64: b by b in the energy loop)
//            for each b, with VA[a][b], VK and the FP64 denominator, the two
//            energy terms of (a, b)
// Two slice buffers per warp swap roles every pair and are filled by cp.async
// one step ahead: H1 of this pair streams in during the H0 work, H0 of the
// next pair during the H1 work, so the warp rarely waits on memory.  VA
// takes the place of H0 in its buffer.  Per-lane sums reduce in a fixed order.
// A dimer's pairs are dealt to `parts` CTAs of W warps (finish_w32_split).
constexpr int kW32Slab = 32 * 33;      // one padded 32 x 32 tile (row stride 33)
constexpr int kCS = 36;                // row stride of the staged C columns: 16-byte rows for vector
                                       // loads, lane rows 4 banks apart (4-way instead of 32-way)

// FP32 (the mixed forms) adds a third slab per warp: the pair's (ib|ja),
// formed for all b before the energy loop, which then runs no multiply-add
// chain of its own (the FP64 form keeps two slabs, for its occupancy).
template <typename T>
__host__ __device__ constexpr int w32_slabs() { return sizeof(T) == 4 ? 3 : 2; }

template <typename T>
constexpr size_t w32_smem_bytes(int W)
{
    return 32 * sizeof(double) + 32 * sizeof(FF) + 2 * 32 * kCS * sizeof(T) +
           W * w32_slabs<T>() * kW32Slab * sizeof(T);
}

// sum_{m < 32} a[m] x[m], a a 16-byte aligned row in shared memory (read as
// broadcasts), x in registers.  FP64 (the FP64 form): one chain in m order.
__device__ __forceinline__ double dot32(const double* a, const double (&x)[32])
{
    double acc = 0;
#pragma unroll
    for (int m = 0; m < 32; m++) acc = fma(a[m], x[m], acc);
    return acc;
}

// FP32: the sums of R rows at once, rows a + r * stride (16-byte aligned),
// each as two chains (even and odd m) advanced together by the packed FP32
// multiply-add (one instruction per two products) and added at the end; the
// R rows' chains interleave in issue order, so that a warp has R
// multiply-adds in flight instead of one dependent chain.
template <int R>
__device__ __forceinline__ void dots32(const float* a, int stride, const float (&x)[32], float (&out)[R])
{
    float2 acc[R];
#pragma unroll
    for (int r = 0; r < R; r++) acc[r] = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < 8; q++) {
        float4 v[R];
#pragma unroll
        for (int r = 0; r < R; r++) v[r] = reinterpret_cast<const float4*>(a + r * stride)[q];
#pragma unroll
        for (int r = 0; r < R; r++)
            acc[r] = __ffma2_rn(make_float2(v[r].x, v[r].y), make_float2(x[4 * q], x[4 * q + 1]), acc[r]);
#pragma unroll
        for (int r = 0; r < R; r++)
            acc[r] = __ffma2_rn(make_float2(v[r].z, v[r].w), make_float2(x[4 * q + 2], x[4 * q + 3]), acc[r]);
    }
#pragma unroll
    for (int r = 0; r < R; r++) out[r] = __fadd_rn(acc[r].x, acc[r].y);
}

// The same sum as two chains (even and odd m), for the FP64 form.
__device__ __forceinline__ double dot32_2(const double* a, const double (&x)[32])
{
    double v0 = 0, v1 = 0;
#pragma unroll
    for (int m = 0; m < 32; m += 2) {
        v0 = fma(a[m], x[m], v0);
        v1 = fma(a[m + 1], x[m + 1], v1);
    }
    return v0 + v1;
}

// One warp starts the asynchronous copy of an nr x nc (<= 32 x 32) row-major
// slice into a zero-padded 32 x 32 tile (lane c copies column c of every
// row; padding is written as zeros by the copy itself) and commits it as one
// group of this lane's cp.async operations.
template <typename T>
__device__ __forceinline__ void prefetch_slice(T* S, const T* __restrict__ h, int nr, int nc, int lane)
{
    const T* p = h + lane;
    const bool col = lane < nc;
    const unsigned dst0 = (unsigned)__cvta_generic_to_shared(S + lane);
#pragma unroll 4
    for (int r = 0; r < 32; r++) {
        const bool ok = r < nr && col;
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst0 + (unsigned)(r * 32 * sizeof(T))),
                     "l"(ok ? p : h), "n"(sizeof(T)), "r"(ok ? (int)sizeof(T) : 0)
                     : "memory");
        p += nc;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Wait until at most N of this lane's copy groups are in flight, then make
// the whole warp's copies visible to the warp.
template <int N>
__device__ __forceinline__ void slice_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
    __syncwarp();
}

// A warp's lanes' E_J and E_K sums by a fixed tree: the halves swap a sum
// first, so that lanes 0-15 reduce E_J while 16-31 reduce E_K (five FP64
// additions, not ten).  Lane 0 returns E_J, lane 16 E_K.
__device__ __forceinline__ double pair_tree(double ej, double ek, int lane)
{
    const bool hi = lane >= 16;
    double s = (hi ? ek : ej) + __shfl_xor_sync(0xffffffffu, hi ? ej : ek, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// Where the sums of a dimer's pairs meet.  A CTA that has the whole dimer
// keeps them in shared memory (up to kPairSums pairs).  Otherwise each pair's
// two sums go into the first 16 bytes of the pair's own H_0 slice, which its
// warp has read and nobody reads again (a slice has at least 2 x 2 elements;
// written as words: slices of odd sizes are 4-byte aligned).
constexpr int kPairSums = 64;

__device__ __forceinline__ void put_pair_sums(double (*ps)[2], void* slice, int pr, bool local, double ej, double ek,
                                              int lane)
{
    const double s = pair_tree(ej, ek, lane);
    if ((lane & 15) != 0) return;
    if (local) {
        ps[pr][lane >> 4] = s;
    } else {
        unsigned* w = static_cast<unsigned*>(slice) + (lane >> 3);
        const unsigned long long a = (unsigned long long)__double_as_longlong(s);
        __stcg(w, (unsigned)a);
        __stcg(w + 1, (unsigned)(a >> 32));
    }
}

__device__ __forceinline__ void get_pair_sums(const void* slice, double& ej, double& ek)
{
    const unsigned* w = static_cast<const unsigned*>(slice);
    const unsigned long long a = ((unsigned long long)__ldcg(w + 1) << 32) | __ldcg(w);
    const unsigned long long b = ((unsigned long long)__ldcg(w + 3) << 32) | __ldcg(w + 2);
    ej = __longlong_as_double((long long)a);
    ek = __longlong_as_double((long long)b);
}

// End of one of a dimer's `parts` CTAs: the last to arrive (any of them: the
// result does not depend on which) adds the dimer's pair sums -- lane l pairs
// l, l + 32, ... in order, then the fixed tree -- so the energies are the same
// bits however the pairs were dealt to warps and CTAs.  slices: the dimer's
// first H_0 slice; stride: bytes from one to the next.  cnt: the dimer's
// arrival counter, zero before the launch and again after it.
__device__ __forceinline__ void finish_dimer(const double (*ps)[2], const char* slices, size_t stride, int pairs,
                                             bool local, int parts, unsigned* cnt, double* E2)
{
    __shared__ int last;
    if (parts > 1) {
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(cnt, 1u) == (unsigned)parts - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
    } else {
        __syncthreads();
    }
    if (threadIdx.x >= 32) return;
    double ej = 0.0, ek = 0.0;
    for (int p = threadIdx.x; p < pairs; p += 32) {
        double a, b;
        if (local) {
            a = ps[p][0];
            b = ps[p][1];
        } else {
            get_pair_sums(slices + p * stride, a, b);
        }
        ej += a;
        ek += b;
    }
    const double s = pair_tree(ej, ek, threadIdx.x);
    if (threadIdx.x == 0) {
        E2[0] = 4.0 * s;
        if (parts > 1) *cnt = 0;
    }
    if (threadIdx.x == 16) E2[1] = -2.0 * s;
}

// STORE: also write the dimer's (ia|jb) and T for the coupling (a separate
// instantiation keeps the plain path's registers).  PAIRS (mixed forms only):
// the energy terms on FP32 pairs, summed per (pair, a) and added to the FP64
// sums once per pair; otherwise on the FP64 pipe term by term.
template <typename T, bool STORE, bool PAIRS, int W>
__global__ void __launch_bounds__(W * 32, W == 4 ? 3 : 2)
k_finish_w32(const DimerDesc* __restrict__ dd, const T* __restrict__ C, const double* __restrict__ Epool,
             T* H, double* __restrict__ E2, T* __restrict__ VT, int parts, unsigned* __restrict__ cnt)
{
    const int dimer = blockIdx.y, cta = blockIdx.x;
    const DimerDesc& d = dd[dimer];
    const int nX = d.nX, nY = d.nY, oX = d.oX, oY = d.oY;
    const int vX = d.vX, vY = d.vY;
    const int rows = nX * nY, pairs = oX * oY;
    const int pr0 = cta * pairs / parts, pr1 = (cta + 1) * pairs / parts;   // this CTA's pairs
    __shared__ double ps[kPairSums][2];
    const bool local = parts == 1 && pairs <= kPairSums;
    const T* CXv = C + d.cXv;                 // virtual columns
    const T* CYv = C + d.cYv;
    const double* eX = Epool + d.eX;          // occupied energies of this block
    const double* eY = Epool + d.eY;
    T* H0 = H + d.h_off;
    const T* H1 = H + d.h_off + (long long)pairs * rows;

    extern __shared__ __align__(16) unsigned char smraw[];
    static_assert(!PAIRS || sizeof(T) == 4, "FP32 pairs serve the mixed forms");
    double* eYv = reinterpret_cast<double*>(smraw);          // [b]: e_b (read as a broadcast)
    FF* eYs = reinterpret_cast<FF*>(eYv + 32);                // [b]: e_b as an FP32 pair
    T* CXT = reinterpret_cast<T*>(eYs + 32);                  // [a][nu], zero padded, row stride kCS
    T* CYT = CXT + 32 * kCS;                                  // [b][sig]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T* const buf = CYT + 32 * kCS + warp * (w32_slabs<T>() * kW32Slab);   // two slice buffers of kW32Slab
    [[maybe_unused]] T* const SV = buf + 2 * kW32Slab;        // FP32: (ib|ja) as [b][a] (stride 33)

    // the warp's first pair streams in while the block stages C and the energies
    if (pr0 + warp < pr1) {
        prefetch_slice(buf, H0 + (long long)(pr0 + warp) * rows, nX, nY, lane);
        prefetch_slice(buf + kW32Slab, H1 + (long long)(pr0 + warp) * rows, nY, nX, lane);
    }
    {
        // all loads first (independent, in flight together), then the stores;
        // lanes run along a, the contiguous index of the coefficient rows
        constexpr int kPer = (32 * 32 + W * 32 - 1) / (W * 32);
        T cxv[kPer], cyv[kPer];
#pragma unroll
        for (int t = 0; t < kPer; t++) {
            const int k = threadIdx.x + t * W * 32;
            const int m = k >> 5, a = k & 31;
            cxv[t] = (a < vX && m < nX) ? CXv[m * nX + a] : T(0);   // k >= 1024 gives m >= 32 > nX
            cyv[t] = (a < vY && m < nY) ? CYv[m * nY + a] : T(0);
        }
#pragma unroll
        for (int t = 0; t < kPer; t++) {
            const int k = threadIdx.x + t * W * 32;
            if (k < 32 * 32) {
                CXT[(k & 31) * kCS + (k >> 5)] = cxv[t];
                CYT[(k & 31) * kCS + (k >> 5)] = cyv[t];
            }
        }
        if (threadIdx.x < 32) {
            const double e = threadIdx.x < vY ? Epool[d.eYv + threadIdx.x] : 0.0;
            eYv[threadIdx.x] = e;
            eYs[threadIdx.x] = ff_split(e);
        }
    }
    __syncthreads();

    const bool live = lane < vX;
    const double ea = live ? Epool[d.eXv + lane] : 0.0;   // this lane's virtual orbital a
    // coupling storage: (ia|jb) and T = vD as [(j,b)][(i,a)] over the whole dimer
    const bool store = STORE && d.vt_off >= 0;
    const long long mXc = (long long)d.oXt * vX, mYc = (long long)d.oYt * vY;
    T* const Vst = store ? VT + d.vt_off : nullptr;
    int x = 0;                                   // buffer holding this pair's H0
    for (int pr = pr0 + warp; pr < pr1; pr += W, x ^= 1) {
        const int i = pr / oY, j = pr % oY;
        double ej = 0.0, ek = 0.0;               // this pair's sums
        const double eija = (eX[i] + eY[j]) - ea;  // e_i + e_j - e_a of this lane
        [[maybe_unused]] const FF eijas = PAIRS ? ff_split(eija) : FF{0.f, 0.f};
        [[maybe_unused]] FF sj{0.f, 0.f}, sk{0.f, 0.f};   // this pair's sums over even b (PAIRS)
        [[maybe_unused]] FF sj1{0.f, 0.f}, sk1{0.f, 0.f}; // and over odd b
        const int nx = pr + W;                   // next pair of this warp
        T* SX = x ? buf + kW32Slab : buf;        // H0, then VA [a][b] (stride 33)
        T* SY = x ? buf : buf + kW32Slab;        // H1, then the next pair's H0
        // ---- (i a|j b): SX[nu][sig] = H0 slice; lane b
        slice_wait<1>();
        {
            T cy[32], tm[32];
#pragma unroll
            for (int m = 0; m < 32; m++) cy[m] = CYT[lane * kCS + m];
            if constexpr (sizeof(T) == 4) {
#pragma unroll
                for (int nu = 0; nu < 32; nu += 2) {
                    float o[2];
                    dots32<2>(SX + nu * 32, 32, cy, o);
                    tm[nu] = o[0];
                    tm[nu + 1] = o[1];
                }
            } else {
#pragma unroll
                for (int nu = 0; nu < 32; nu++) tm[nu] = dot32(SX + nu * 32, cy);
            }
            __syncwarp();                        // H0 consumed: VA takes its place
            // rows a >= vX of VA are never read (only lanes a < vX form terms)
            if constexpr (sizeof(T) == 4) {
#pragma unroll 1
                for (int a = 0; a < vX; a += 4) {   // CXT rows up to 32 are zero padded
                    float o[4];
                    dots32<4>(CXT + a * kCS, kCS, tm, o);
#pragma unroll
                    for (int r = 0; r < 4; r++) SX[(a + r) * 33 + lane] = o[r];
                }
            } else {
#pragma unroll 4
                for (int a = 0; a < vX; a++) SX[a * 33 + lane] = dot32(CXT + a * kCS, tm);
            }
        }
        // ---- (i b|j a): SY[lam][nu] = H1 slice; lane a
        slice_wait<0>();
        {
            T cx[32], tk[32];
#pragma unroll
            for (int m = 0; m < 32; m++) cx[m] = CXT[lane * kCS + m];
            if constexpr (sizeof(T) == 4) {
#pragma unroll
                for (int lam = 0; lam < 32; lam += 2) {
                    float o[2];
                    dots32<2>(SY + lam * 32, 32, cx, o);
                    tk[lam] = o[0];
                    tk[lam + 1] = o[1];
                }
            } else {
#pragma unroll
                for (int lam = 0; lam < 32; lam++) tk[lam] = dot32(SY + lam * 32, cx);
            }
            __syncwarp();                        // H1 consumed: the next pair's H0 streams into SY
            if (nx < pr1) prefetch_slice(SY, H0 + (long long)nx * rows, nX, nY, lane);
            // ---- FP32: (ib|ja) of every b into this lane's column of SV, four
            // independent multiply-add chains at a time (each lane reads back
            // only its own column)
            if constexpr (sizeof(T) == 4) {
#pragma unroll 1
                for (int b = 0; b < vY; b += 4) {   // CYT rows up to 32 are zero padded
                    float o[4];
                    dots32<4>(CYT + b * kCS, kCS, tk, o);
#pragma unroll
                    for (int r = 0; r < 4; r++) SV[(b + r) * 33 + lane] = o[r];
                }
            }
            // ---- denominators and energy sums, lane a over b
            if constexpr (PAIRS) {
                // two b at a time, even b into (sj, sk) and odd b into (sj1, sk1):
                // independent chains for the FP32 pipes; an odd vY's last odd b
                // adds exact zeros
#pragma unroll 1
                for (int b = 0; b < vY; b += 2) {
                    const bool has1 = b + 1 < vY;
                    if (live) {
                        const T v0 = SX[lane * 33 + b], vk0 = SV[b * 33 + lane];
                        const T v1 = has1 ? SX[lane * 33 + b + 1] : T(0);
                        const T vk1 = has1 ? SV[(b + 1) * 33 + lane] : T(0);
                        const T tv0 = energy_terms_ff(v0, vk0, eijas, eYs[b], sj, sk);
                        const T tv1 = energy_terms_ff(v1, vk1, eijas, eYs[b + 1], sj1, sk1);
                        if (store) {
                            const long long e = ((long long)(d.jY0 + j) * vY + b) * mXc + (long long)(d.iX0 + i) * vX + lane;
                            Vst[e] = v0;
                            Vst[mXc * mYc + e] = tv0;
                            if (has1) {
                                Vst[e + mXc] = v1;
                                Vst[mXc * mYc + e + mXc] = tv1;
                            }
                        }
                    }
                }
            } else {
#pragma unroll 1
                for (int b = 0; b < vY; b++) {
                    T vk;
                    if constexpr (sizeof(T) == 4) vk = SV[b * 33 + lane];
                    else vk = dot32_2(CYT + b * kCS, tk);   // two chains of 16
                    if (live) {
                        const T vab = SX[lane * 33 + b];
                        double t;
                        energy_terms<T>(vab, vk, eija - eYv[b], ej, ek, store ? &t : nullptr);
                        if (store) {
                            const long long e = ((long long)(d.jY0 + j) * vY + b) * mXc + (long long)(d.iX0 + i) * vX + lane;
                            Vst[e] = vab;
                            Vst[mXc * mYc + e] = narrow<T>(t);
                        }
                    }
                }
            }
        }
        if constexpr (PAIRS) {
            ej = ff_f64(sj) + ff_f64(sj1);
            ek = ff_f64(sk) + ff_f64(sk1);
        }
        __syncwarp();                            // VA consumed: the next pair's H1 streams into SX
        if (nx < pr1) prefetch_slice(SX, H1 + (long long)nx * rows, nY, nX, lane);
        put_pair_sums(ps, H0 + (long long)pr * rows, pr, local, ej, ek, lane);
    }
    finish_dimer(ps, reinterpret_cast<const char*>(H0), (size_t)rows * sizeof(T), pairs, local, parts, cnt + dimer,
                 E2 + 2 * d.slot);
}

// ---------------------------------------------------------------------------
// FP64E second half, monomers of at most 32 AO: the structure of
// k_finish_w32 with every value an FP32 pair (ff.h) -- the H slices written
// as pairs by the first half, C, the virtual quarter transformations as pair
// multiply-adds, and the energy terms with v^2 and v vk as pair products and
// D = 1/x on pairs -- so that the FP64 form's accuracy (~2^-45 per step) is
// kept off the FP64 pipe, whose rate a multiply-add per (row, pair) term
// would otherwise set.  The C columns stay in shared memory (a lane's column
// as pairs would take 64 registers); four outputs accumulate at once so that
// each lane runs independent chains.  Per-lane sums over b go into FP64 sums
// once per occupied pair; with STORE the dimer's (ia|jb) and T = vD are
// written as FP64 for the coupling.
constexpr int kFFSlab = 32 * 33;   // one padded 32 x 32 tile of pairs (row stride 33)
constexpr int kFFChains = 4;       // independent pair multiply-add chains per lane (eight measured slower)

size_t w32_ff_smem_bytes(int W) { return (32 + 2 * (size_t)kFFSlab + 2 * (size_t)W * kFFSlab) * sizeof(FF); }

template <bool STORE, int W>
__global__ void __launch_bounds__(W * 32, 2)
k_finish_w32_ff(const DimerDesc* __restrict__ dd, const double* __restrict__ C, const double* __restrict__ Epool,
                FF* H, double* __restrict__ E2, double* __restrict__ VT, int parts, unsigned* __restrict__ cnt)
{
    const int dimer = blockIdx.y, cta = blockIdx.x;
    const DimerDesc& d = dd[dimer];
    const int nX = d.nX, nY = d.nY, oX = d.oX, oY = d.oY;
    const int vX = d.vX, vY = d.vY;
    const int rows = nX * nY, pairs = oX * oY;
    const int pr0 = cta * pairs / parts, pr1 = (cta + 1) * pairs / parts;   // this CTA's pairs
    __shared__ double ps[kPairSums][2];
    const bool local = parts == 1 && pairs <= kPairSums;
    const double* CXv = C + d.cXv;            // virtual columns
    const double* CYv = C + d.cYv;
    const double* eX = Epool + d.eX;          // occupied energies of this block
    const double* eY = Epool + d.eY;
    FF* H0 = H + d.h_off;
    const FF* H1 = H + d.h_off + (long long)pairs * rows;

    extern __shared__ __align__(16) unsigned char smraw[];
    FF* eYs = reinterpret_cast<FF*>(smraw);   // [b]: e_b
    FF* CXT = eYs + 32;                       // [a][nu], row stride 33, zero padded
    FF* CYT = CXT + kFFSlab;                  // [b][sig]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    FF* const buf = CYT + kFFSlab + warp * (2 * kFFSlab);   // two slice buffers

    if (pr0 + warp < pr1) {
        prefetch_slice(buf, H0 + (long long)(pr0 + warp) * rows, nX, nY, lane);
        prefetch_slice(buf + kFFSlab, H1 + (long long)(pr0 + warp) * rows, nY, nX, lane);
    }
    for (int k = threadIdx.x; k < 32 * 32; k += W * 32) {
        const int m = k >> 5, a = k & 31;       // lanes along the contiguous index a
        CXT[a * 33 + m] = (a < vX && m < nX) ? ff_split(CXv[m * nX + a]) : FF{0.f, 0.f};
        CYT[a * 33 + m] = (a < vY && m < nY) ? ff_split(CYv[m * nY + a]) : FF{0.f, 0.f};
    }
    if (threadIdx.x < 32) eYs[threadIdx.x] = threadIdx.x < vY ? ff_split(Epool[d.eYv + threadIdx.x]) : FF{0.f, 0.f};
    __syncthreads();

    const bool live = lane < vX;
    const double ea = live ? Epool[d.eXv + lane] : 0.0;   // this lane's virtual orbital a
    const bool store = STORE && d.vt_off >= 0;
    const long long mXc = (long long)d.oXt * vX, mYc = (long long)d.oYt * vY;
    double* const Vst = store ? VT + d.vt_off : nullptr;
    int x = 0;                                   // buffer holding this pair's H0
    for (int pr = pr0 + warp; pr < pr1; pr += W, x ^= 1) {
        const int i = pr / oY, j = pr % oY;
        const FF eija = ff_split((eX[i] + eY[j]) - ea);   // e_i + e_j - e_a of this lane
        FF sj{0.f, 0.f}, sk{0.f, 0.f};
        const int nx = pr + W;
        FF* SX = x ? buf + kFFSlab : buf;        // H0 (row stride 32), then VA [a][b] (stride 33)
        FF* SY = x ? buf : buf + kFFSlab;        // H1, then the next pair's H0
        // ---- (i a|j b): lane b, tm[nu] = sum_sig H0[nu][sig] C_Y[sig][b]
        slice_wait<1>();
        {
            FF tm[32];
            const FF* cy = CYT + lane * 33;
#pragma unroll
            for (int nu = 0; nu < 32; nu += kFFChains) {
                FF acc[kFFChains];
#pragma unroll
                for (int q = 0; q < kFFChains; q++) acc[q] = FF{0.f, 0.f};
#pragma unroll 4
                for (int m = 0; m < 32; m++) {
                    const FF c = cy[m];
#pragma unroll
                    for (int q = 0; q < kFFChains; q++) ff_mac(acc[q], SX[(nu + q) * 32 + m], c);
                }
#pragma unroll
                for (int q = 0; q < kFFChains; q++) tm[nu + q] = acc[q];
            }
            __syncwarp();                        // H0 consumed: VA takes its place
#pragma unroll 1
            for (int a = 0; a < 32; a += kFFChains) {
                FF acc[kFFChains];
#pragma unroll
                for (int q = 0; q < kFFChains; q++) acc[q] = FF{0.f, 0.f};
#pragma unroll
                for (int nu = 0; nu < 32; nu++)
#pragma unroll
                    for (int q = 0; q < kFFChains; q++) ff_mac(acc[q], CXT[(a + q) * 33 + nu], tm[nu]);
#pragma unroll
                for (int q = 0; q < kFFChains; q++) SX[(a + q) * 33 + lane] = acc[q];
            }
        }
        // ---- (i b|j a): lane a, tk[lam] = sum_nu H1[lam][nu] C_X[nu][a]
        slice_wait<0>();
        {
            FF tk[32];
            const FF* cx = CXT + lane * 33;
#pragma unroll
            for (int lam = 0; lam < 32; lam += kFFChains) {
                FF acc[kFFChains];
#pragma unroll
                for (int q = 0; q < kFFChains; q++) acc[q] = FF{0.f, 0.f};
#pragma unroll 4
                for (int m = 0; m < 32; m++) {
                    const FF c = cx[m];
#pragma unroll
                    for (int q = 0; q < kFFChains; q++) ff_mac(acc[q], SY[(lam + q) * 32 + m], c);
                }
#pragma unroll
                for (int q = 0; q < kFFChains; q++) tk[lam + q] = acc[q];
            }
            __syncwarp();                        // H1 consumed: the next pair's H0 streams into SY
            if (nx < pr1) prefetch_slice(SY, H0 + (long long)nx * rows, nX, nY, lane);
            // ---- denominators and energy sums, lane a over b
#pragma unroll 1
            for (int b = 0; b < vY; b++) {
                FF v0{0.f, 0.f}, v1{0.f, 0.f};   // two chains of 16
#pragma unroll
                for (int lam = 0; lam < 32; lam += 2) {
                    ff_mac(v0, CYT[b * 33 + lam], tk[lam]);
                    ff_mac(v1, CYT[b * 33 + lam + 1], tk[lam + 1]);
                }
                if (live) {
                    const FF v = SX[lane * 33 + b];
                    const FF vk = ff_add(v0, v1);
                    const FF D = ff_rcp(ff_sub(eija, eYs[b]));
                    ff_mac(sj, ff_mul(v, v), D);
                    ff_mac(sk, ff_mul(v, vk), D);
                    if (store) {
                        const long long e = ((long long)(d.jY0 + j) * vY + b) * mXc + (long long)(d.iX0 + i) * vX + lane;
                        Vst[e] = ff_f64(v);
                        Vst[mXc * mYc + e] = ff_f64(ff_mul(v, D));
                    }
                }
            }
        }
        __syncwarp();                            // VA consumed: the next pair's H1 streams into SX
        if (nx < pr1) prefetch_slice(SX, H1 + (long long)nx * rows, nY, nX, lane);
        put_pair_sums(ps, H0 + (long long)pr * rows, pr, local, ff_f64(sj), ff_f64(sk), lane);
    }
    finish_dimer(ps, reinterpret_cast<const char*>(H0), (size_t)rows * sizeof(FF), pairs, local, parts, cnt + dimer,
                 E2 + 2 * d.slot);
}

// ---------------------------------------------------------------------------
// Monomers above 32 AO: the virtual quarter transformations of one occupied
// pair are four small GEMMs,
//   Tm  [nu][b]  = sum_sig H0[nu][sig]  C_Y[sig][oY+b]      (nX x vY, K = nY)
//   TmK [lam][a] = sum_nu  H1[lam][nu]  C_X[nu][oX+a]       (nY x vX, K = nX)
//   VA  [a][b]   = sum_nu  C_X[nu][oX+a] Tm[nu][b]          (vX x vY, K = nX)
//   VKT [a][b]   = sum_lam TmK[lam][a]  C_Y[lam][oY+b]      (vX x vY, K = nY)
// Each GEMM's M x N outputs are cut into 8 x 4 blocks dealt round-robin to the
// 256 threads, so small and ragged shapes keep the threads on useful work;
// a thread accumulates its block in registers (per K step 12 loads feed 32
// FMAs).  FP64 here; the FP32 forms' kernel follows.  H slices and Tm/TmK live in shared memory, the C columns are read
// through L1.  VA and VKT use the same blocks, so each thread meets its own
// (a, b) terms for the FP64 epilogue (VA goes through shared memory to free
// its registers).  One CTA runs a range of pairs of one dimer; its FP64
// partial sums are written per task and added in task order by k_finish_sum.
constexpr int kTThreads = 256;
constexpr int kTM = 8, kTN = 4;

size_t tiled_smem_bytes(int max_ao)
{
    const size_t n = (size_t)max_ao;
    return (n * n + 2 * n * n) * sizeof(double) + 2 * n * sizeof(double) + 64;
}

// acc[i][j] = sum_k A(m0 + i, k) B(k, n0 + j) over rows < M, columns < N.
template <typename FA, typename FB>
__device__ __forceinline__ void mm_block(double (&acc)[kTM][kTN], int m0, int n0, int M, int N, int K, FA A, FB B)
{
#pragma unroll
    for (int i = 0; i < kTM; i++)
#pragma unroll
        for (int j = 0; j < kTN; j++) acc[i][j] = 0.0;
    bool mok[kTM], nok[kTN];
#pragma unroll
    for (int i = 0; i < kTM; i++) mok[i] = m0 + i < M;
#pragma unroll
    for (int j = 0; j < kTN; j++) nok[j] = n0 + j < N;
#pragma unroll 2
    for (int k = 0; k < K; k++) {
        double a[kTM], b[kTN];
#pragma unroll
        for (int i = 0; i < kTM; i++) a[i] = mok[i] ? A(m0 + i, k) : 0.0;
#pragma unroll
        for (int j = 0; j < kTN; j++) b[j] = nok[j] ? B(k, n0 + j) : 0.0;
#pragma unroll
        for (int i = 0; i < kTM; i++)
#pragma unroll
            for (int j = 0; j < kTN; j++) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
}

__device__ __forceinline__ void copy_slice(double* S, const double* __restrict__ src, int n, int tid)
{
    for (int k0 = 0; k0 < n; k0 += 4 * kTThreads) {
        double v[4];
#pragma unroll
        for (int t = 0; t < 4; t++) {
            const int k = k0 + t * kTThreads + tid;
            v[t] = k < n ? src[k] : 0.0;
        }
#pragma unroll
        for (int t = 0; t < 4; t++) {
            const int k = k0 + t * kTThreads + tid;
            if (k < n) S[k] = v[t];
        }
    }
}

__global__ void __launch_bounds__(kTThreads, 2)
k_finish_tiled(const DimerDesc* __restrict__ dd, const FinTask* __restrict__ tasks, const double* __restrict__ C,
               const double* __restrict__ Epool, const double* __restrict__ H, double* __restrict__ part,
               int smem_elems, double* __restrict__ VT)
{
    const FinTask tk = tasks[blockIdx.x];
    const DimerDesc& d = dd[tk.dimer];
    const int nX = d.nX, nY = d.nY, oY = d.oY;
    const int vX = d.vX, vY = d.vY;
    const int rows = nX * nY, pairs = d.oX * oY;
    const double* __restrict__ CXv = C + d.cXv;    // virtual columns
    const double* __restrict__ CYv = C + d.cYv;
    const double* eX = Epool + d.eX;          // occupied energies of this block
    const double* eY = Epool + d.eY;
    const double* H0 = H + d.h_off;
    const double* H1 = H + d.h_off + (long long)pairs * rows;

    extern __shared__ __align__(16) unsigned char smraw[];
    double* eXv = reinterpret_cast<double*>(smraw);           // [vX]
    double* eYv = eXv + nX;                                   // [vY]
    double* base = eYv + nY;
    // a group of np pairs runs each phase together (one barrier per phase for
    // the group): as many as the launch's shared memory holds
    const int per_pair = rows + nX * vY + nY * vX;
    const int gmax = max(1, min(tk.pr1 - tk.pr0, smem_elems / per_pair));
    double* S = base;                                              // H slices [np][rows], then VA [np][vX][vY]
    double* Tm = S + gmax * rows;                                  // [np][nX][vY]
    double* TmK = Tm + gmax * nX * vY;                             // [np][nY][vX]
    const int tid = threadIdx.x;
    for (int k = tid; k < vX; k += kTThreads) eXv[k] = Epool[d.eXv + k];
    for (int k = tid; k < vY; k += kTThreads) eYv[k] = Epool[d.eYv + k];
    // 8 x 4 output blocks of each GEMM shape, per pair
    const int bn_vY = (vY + kTN - 1) / kTN, bn_vX = (vX + kTN - 1) / kTN;
    const int nb1 = ((nX + kTM - 1) / kTM) * bn_vY;          // Tm
    const int nb3 = ((nY + kTM - 1) / kTM) * bn_vX;          // TmK
    const int nb2 = ((vX + kTM - 1) / kTM) * bn_vY;          // VA, VKT

    const bool store = VT != nullptr && d.vt_off >= 0;
    const long long mXc = (long long)d.oXt * vX, mYc = (long long)d.oYt * vY;
    double* const Vst = store ? VT + d.vt_off : nullptr;
    double ej = 0.0, ek = 0.0;
    for (int g0 = tk.pr0; g0 < tk.pr1; g0 += gmax) {
        const int np = min(gmax, tk.pr1 - g0);
        double acc[kTM][kTN];
        // ---- Tm = H0 C_Y(virtual), every pair of the group
        copy_slice(S, H0 + (long long)g0 * rows, np * rows, tid);
        __syncthreads();
        for (int blk = tid; blk < np * nb1; blk += kTThreads) {
            const int p = blk / nb1, q = blk - p * nb1;
            const int m0 = (q / bn_vY) * kTM, n0 = (q % bn_vY) * kTN;
            const double* Sp = S + p * rows;
            double* Tp = Tm + p * nX * vY;
            mm_block(acc, m0, n0, nX, vY, nY, [&](int m, int k) { return Sp[m * nY + k]; },
                        [&](int k, int n) { return __ldg(CYv + k * nY + n); });
#pragma unroll
            for (int a = 0; a < kTM; a++)
#pragma unroll
                for (int b = 0; b < kTN; b++)
                    if (m0 + a < nX && n0 + b < vY) Tp[(m0 + a) * vY + n0 + b] = acc[a][b];
        }
        __syncthreads();
        // ---- TmK = H1 C_X(virtual)
        copy_slice(S, H1 + (long long)g0 * rows, np * rows, tid);
        __syncthreads();
        for (int blk = tid; blk < np * nb3; blk += kTThreads) {
            const int p = blk / nb3, q = blk - p * nb3;
            const int m0 = (q / bn_vX) * kTM, n0 = (q % bn_vX) * kTN;
            const double* Sp = S + p * rows;
            double* Kp = TmK + p * nY * vX;
            mm_block(acc, m0, n0, nY, vX, nX, [&](int m, int k) { return Sp[m * nX + k]; },
                        [&](int k, int n) { return __ldg(CXv + k * nX + n); });
#pragma unroll
            for (int a = 0; a < kTM; a++)
#pragma unroll
                for (int b = 0; b < kTN; b++)
                    if (m0 + a < nY && n0 + b < vX) Kp[(m0 + a) * vX + n0 + b] = acc[a][b];
        }
        __syncthreads();
        // ---- VA, VKT and the FP64 epilogue, block by block
        for (int blk = tid; blk < np * nb2; blk += kTThreads) {
            const int p = blk / nb2, q = blk - p * nb2;
            const int m0 = (q / bn_vY) * kTM, n0 = (q % bn_vY) * kTN;
            const int pr = g0 + p, i = pr / oY, j = pr - i * oY;
            const double eij = eX[i] + eY[j];
            const double* Tp = Tm + p * nX * vY;
            const double* Kp = TmK + p * nY * vX;
            double* Vp = S + p * rows;                                 // VA of pair p (own elements)
            mm_block(acc, m0, n0, vX, vY, nX, [&](int m, int k) { return __ldg(CXv + k * nX + m); },
                        [&](int k, int n) { return Tp[k * vY + n]; });
#pragma unroll
            for (int a = 0; a < kTM; a++)
#pragma unroll
                for (int b = 0; b < kTN; b++)
                    if (m0 + a < vX && n0 + b < vY) Vp[(m0 + a) * vY + n0 + b] = acc[a][b];
            mm_block(acc, m0, n0, vX, vY, nY, [&](int m, int k) { return Kp[k * vX + m]; },
                        [&](int k, int n) { return __ldg(CYv + k * nY + n); });
#pragma unroll
            for (int a = 0; a < kTM; a++) {
                const int m = m0 + a;
#pragma unroll
                for (int b = 0; b < kTN; b++) {
                    const int n = n0 + b;
                    if (m < vX && n < vY) {
                        const double vab = Vp[m * vY + n];
                        double tv;
                        energy_terms<double>(vab, acc[a][b], eij - (eXv[m] + eYv[n]), ej, ek, store ? &tv : nullptr);
                        if (store) {
                            const long long e =
                                ((long long)(d.jY0 + j) * vY + n) * mXc + (long long)(d.iX0 + i) * vX + m;
                            Vst[e] = vab;
                            Vst[mXc * mYc + e] = tv;
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
    // fixed-order block reduction
    __shared__ double red[2][kTThreads / 32];
    ej = warp_sum(ej);
    ek = warp_sum(ek);
    if ((tid & 31) == 0) { red[0][tid >> 5] = ej; red[1][tid >> 5] = ek; }
    __syncthreads();
    if (tid == 0) {
        double sj = 0.0, sk = 0.0;
        for (int w = 0; w < kTThreads / 32; w++) { sj += red[0][w]; sk += red[1][w]; }
        part[2 * blockIdx.x + 0] = sj;
        part[2 * blockIdx.x + 1] = sk;
    }
}

// FP32 (mixed forms).  The same four products on 8 x 8 blocks, two columns per
// packed multiply-add, every operand in shared memory: both virtual coefficient
// blocks for the whole task, the pairs' H slices, and Tm / TmK in the slices'
// place (written from registers once the slice is consumed).  A thread has one
// block of each product -- as many pairs as fill 256 threads run together --
// and keeps its (ia|jb) block in registers until it meets (ib|ja) in the
// epilogue.  A second set of slices, where it fits, is filled while the first
// is used.  A block's columns are 4 nb .. 4 nb + 3 and the same in the upper half, so
// that a warp's 16-byte loads are contiguous.  Every output is one chain over k
// in order.  Bound by the FP32 pipes at eight warps per SM (64 accumulators
// twice): 1200 pairs of 128 + 128 AO in 0.63 ms, 25 TFLOP/s; the FP64 kernel's
// scheme above (8 x 4 blocks, scalar loads, C through L1) took 1.55 ms there in
// FP32, and 1.41 ms against 0.78 for 96 dimers of 16 to 96 AO.
constexpr int kF32Cap = 220 * 1024;   // shared bytes a launch may use

struct TiledShape {
    int bmX, bmY, bnX, bnY;            // 8-blocks of nX, nY, vX, vY
    int kX, kY;                        // nX, nY padded to 4
    int np, nbuf, slab;                // pairs of a group, slice sets, elements of a pair's slice
    int c_elems;
};

// The shape for a dimer within `elems` shared floats.
__host__ __device__ inline TiledShape tiled_shape(int nX, int nY, int vX, int vY, int elems)
{
    TiledShape t;
    t.bmX = (nX + 7) / 8; t.bmY = (nY + 7) / 8; t.bnX = (vX + 7) / 8; t.bnY = (vY + 7) / 8;
    t.kX = (nX + 3) / 4 * 4; t.kY = (nY + 3) / 4 * 4;
    const int rX = 8 * t.bmX * (t.kY + 4 > 8 * t.bnY ? t.kY + 4 : 8 * t.bnY);
    const int rY = 8 * t.bmY * (t.kX + 4 > 8 * t.bnX ? t.kX + 4 : 8 * t.bnX);
    t.slab = rX > rY ? rX : rY;
    t.c_elems = t.kX * 8 * t.bnX + t.kY * 8 * t.bnY;
    int nb = t.bmX * t.bnY;
    if (t.bmY * t.bnX > nb) nb = t.bmY * t.bnX;
    t.np = kTThreads / nb;
    const int fit = (elems - t.c_elems) / t.slab;
    if (t.np > fit) t.np = fit;
    t.nbuf = 2 * t.np <= fit ? 2 : 1;
    return t;
}

// Copy np slices (rows x cols, contiguous, `rows * cols` apart) into
// S[p][up8(rows)][ld], zero beyond the rows and columns (up to colsp), by cp.async.
__device__ __forceinline__ void load_slices(float* S, const float* __restrict__ src, int np, int rows, int cols,
                                            int rowsp, int colsp, int ld, int slab, int tid)
{
    if ((cols & 3) == 0 && ((size_t)src & 15) == 0) {
        const int pc = cols / 4, per = rowsp * pc;
        for (int e = tid; e < np * per; e += kTThreads) {
            const int p = e / per, r = (e - p * per) / pc, c = (e - p * per - r * pc) * 4;
            const bool ok = r < rows;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                             (unsigned)__cvta_generic_to_shared(S + p * slab + r * ld + c)),
                         "l"(ok ? src + ((long long)p * rows + r) * cols + c : src), "r"(ok ? 16 : 0)
                         : "memory");
        }
    } else {
        const int per = rowsp * colsp;
        for (int e = tid; e < np * per; e += kTThreads) {
            const int p = e / per, r = (e - p * per) / colsp, c = e - p * per - r * colsp;
            const bool ok = r < rows && c < cols;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                             (unsigned)__cvta_generic_to_shared(S + p * slab + r * ld + c)),
                         "l"(ok ? src + ((long long)p * rows + r) * cols + c : src), "r"(ok ? 4 : 0)
                         : "memory");
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void zero8(float2 (&acc)[8][4])
{
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = make_float2(0.f, 0.f);
}

// acc[i] += a[i] b, b the block's eight columns.
__device__ __forceinline__ void outer8(float2 (&acc)[8][4], const float (&a)[8], const float* b, int half)
{
    const float4 lo = *reinterpret_cast<const float4*>(b), hi = *reinterpret_cast<const float4*>(b + half);
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const float2 x = make_float2(a[i], a[i]);
        acc[i][0] = __ffma2_rn(x, make_float2(lo.x, lo.y), acc[i][0]);
        acc[i][1] = __ffma2_rn(x, make_float2(lo.z, lo.w), acc[i][1]);
        acc[i][2] = __ffma2_rn(x, make_float2(hi.x, hi.y), acc[i][2]);
        acc[i][3] = __ffma2_rn(x, make_float2(hi.z, hi.w), acc[i][3]);
    }
}

// acc = sum_k A[i][k] B[k][.], A row-major (four k per 16-byte load), K a multiple of 4.
__device__ __forceinline__ void mm_rows(float2 (&acc)[8][4], const float* A, int lda, const float* B, int ldb, int K)
{
    zero8(acc);
#pragma unroll 1
    for (int k = 0; k < K; k += 4) {
        float4 a[8];
#pragma unroll
        for (int i = 0; i < 8; i++) a[i] = *reinterpret_cast<const float4*>(A + i * lda + k);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            float x[8];
#pragma unroll
            for (int i = 0; i < 8; i++) x[i] = u == 0 ? a[i].x : u == 1 ? a[i].y : u == 2 ? a[i].z : a[i].w;
            outer8(acc, x, B + (k + u) * ldb, ldb / 2);
        }
    }
}

// acc = sum_k A[k][i] B[k][.], both k-major.
__device__ __forceinline__ void mm_cols(float2 (&acc)[8][4], const float* A, int lda, const float* B, int ldb, int K)
{
    zero8(acc);
#pragma unroll 2
    for (int k = 0; k < K; k++) {
        const float4 p = *reinterpret_cast<const float4*>(A + k * lda), q = *reinterpret_cast<const float4*>(A + k * lda + 4);
        const float x[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
        outer8(acc, x, B + k * ldb, ldb / 2);
    }
}

__device__ __forceinline__ void put8(float* T, int ld, const float2 (&acc)[8][4])
{
#pragma unroll
    for (int i = 0; i < 8; i++) {
        *reinterpret_cast<float4*>(T + i * ld) = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
        *reinterpret_cast<float4*>(T + i * ld + ld / 2) = make_float4(acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y);
    }
}

template <bool PAIRS>
__global__ void __launch_bounds__(kTThreads, 1)
k_finish_tiled_f32(const DimerDesc* __restrict__ dd, const FinTask* __restrict__ tasks, const float* __restrict__ C,
                   const double* __restrict__ Epool, const float* __restrict__ H, double* __restrict__ part,
                   int smem_elems, float* __restrict__ VT)
{
    const FinTask tk = tasks[blockIdx.x];
    const DimerDesc& d = dd[tk.dimer];
    const int nX = d.nX, nY = d.nY, oY = d.oY, vX = d.vX, vY = d.vY;
    const int rows = nX * nY, pairs = d.oX * oY;
    const TiledShape t = tiled_shape(nX, nY, vX, vY, smem_elems);
    const int vX8 = 8 * t.bnX, vY8 = 8 * t.bnY, ldY = t.kY + 4, ldX = t.kX + 4;
    const float* H0 = H + d.h_off;
    const float* H1 = H0 + (long long)pairs * rows;
    extern __shared__ __align__(16) unsigned char smraw[];
    float* sCX = reinterpret_cast<float*>(smraw);              // [kX][vX8], zero padded
    float* sCY = sCX + t.kX * vX8;                             // [kY][vY8]
    float* S0 = sCY + t.kY * vY8;
    float* S1 = t.nbuf == 2 ? S0 + t.np * t.slab : S0;
    const int tid = threadIdx.x;
    for (int e = tid; e < t.c_elems; e += kTThreads) {
        const bool y = e >= t.kX * vX8;
        const int f = y ? e - t.kX * vX8 : e, w = y ? vY8 : vX8, n = y ? nY : nX, k = f / w, c = f - k * w;
        const bool ok = k < n && c < (y ? vY : vX);
        const float* src = C + (y ? d.cYv : d.cXv);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(sCX + e)),
                     "l"(ok ? src + k * n + c : src), "r"(ok ? 4 : 0)
                     : "memory");
    }
    load_slices(S0, H0 + (long long)tk.pr0 * rows, min(t.np, tk.pr1 - tk.pr0), nX, nY, 8 * t.bmX, t.kY, ldY, t.slab, tid);
    const int nb1 = t.bmX * t.bnY, nb3 = t.bmY * t.bnX, nb2 = t.bnX * t.bnY;
    // this thread's block of each product: pair p, row block m, column block n
    const int p1 = tid / nb1, m1 = (tid - p1 * nb1) / t.bnY, n1 = tid - p1 * nb1 - m1 * t.bnY;
    const int p3 = tid / nb3, m3 = (tid - p3 * nb3) / t.bnX, n3 = tid - p3 * nb3 - m3 * t.bnX;
    const int p2 = tid / nb2, m2 = (tid - p2 * nb2) / t.bnY, n2 = tid - p2 * nb2 - m2 * t.bnY;
    const bool store = VT != nullptr && d.vt_off >= 0;
    const long long mXc = (long long)d.oXt * vX, mYc = (long long)d.oYt * vY;
    float* const Vst = store ? VT + d.vt_off : nullptr;
    __shared__ double red[2][kTThreads];       // the threads' sums of a group
    for (int g0 = tk.pr0; g0 < tk.pr1; g0 += t.np) {
        const int np = min(t.np, tk.pr1 - g0);
        double ej = 0.0, ek = 0.0;
        float2 acc[8][4], v[8][4];
        if (t.nbuf == 2) {
            load_slices(S1, H1 + (long long)g0 * rows, np, nY, nX, 8 * t.bmY, t.kX, ldX, t.slab, tid);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        // ---- Tm[nu][b] = sum_sig H0[nu][sig] C_Y[sig][b], then in the slice's place
        if (p1 < np) mm_rows(acc, S0 + p1 * t.slab + 8 * m1 * ldY, ldY, sCY + 4 * n1, vY8, t.kY);
        __syncthreads();
        if (p1 < np) put8(S0 + p1 * t.slab + 8 * m1 * vY8 + 4 * n1, vY8, acc);
        __syncthreads();
        // ---- (ia|jb) = sum_nu C_X[nu][a] Tm[nu][b]
        if (p2 < np) mm_cols(v, sCX + 8 * m2, vX8, S0 + p2 * t.slab + 4 * n2, vY8, t.kX);
        __syncthreads();
        const int nn = min(t.np, tk.pr1 - g0 - t.np);   // the next group's pairs
        if (t.nbuf == 1) {
            load_slices(S1, H1 + (long long)g0 * rows, np, nY, nX, 8 * t.bmY, t.kX, ldX, t.slab, tid);
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        } else if (nn > 0) {
            load_slices(S0, H0 + (long long)(g0 + t.np) * rows, nn, nX, nY, 8 * t.bmX, t.kY, ldY, t.slab, tid);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        // ---- TmK[lam][a] = sum_nu H1[lam][nu] C_X[nu][a]
        if (p3 < np) mm_rows(acc, S1 + p3 * t.slab + 8 * m3 * ldX, ldX, sCX + 4 * n3, vX8, t.kX);
        __syncthreads();
        if (p3 < np) put8(S1 + p3 * t.slab + 8 * m3 * vX8 + 4 * n3, vX8, acc);
        __syncthreads();
        // ---- (ib|ja) = sum_lam TmK[lam][a] C_Y[lam][b], and the epilogue
        if (p2 < np) {
            mm_cols(acc, S1 + p2 * t.slab + 8 * m2, vX8, sCY + 4 * n2, vY8, t.kY);
            const int pr = g0 + p2, i = pr / oY, j = pr - i * oY;
            const double eij = Epool[d.eX + i] + Epool[d.eY + j];
            const int b0 = 4 * n2, b1 = b0 + vY8 / 2;
            [[maybe_unused]] FF sj{0.f, 0.f}, sk{0.f, 0.f}, ebs[8];
            [[maybe_unused]] const FF eijs = ff_split(eij);
            if constexpr (PAIRS) {
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    const int b = (c < 4 ? b0 : b1 - 4) + c;
                    ebs[c] = b < vY ? ff_split(Epool[d.eYv + b]) : FF{0.f, 0.f};
                }
            }
#pragma unroll
            for (int r = 0; r < 8; r++) {
                const int a = 8 * m2 + r;
                if (a >= vX) break;
                const double ea = Epool[d.eXv + a];
                [[maybe_unused]] FF eijas{0.f, 0.f};
                if constexpr (PAIRS) eijas = ff_sub(eijs, ff_split(ea));
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    const int b = (c < 4 ? b0 : b1 - 4) + c;
                    if (b < vY) {
                        const float vab = c & 1 ? v[r][c / 2].y : v[r][c / 2].x;
                        const float vk = c & 1 ? acc[r][c / 2].y : acc[r][c / 2].x;
                        float tv;
                        if constexpr (PAIRS) {
                            tv = energy_terms_ff(vab, vk, eijas, ebs[c], sj, sk);
                        } else {
                            double x;
                            energy_terms<float>(vab, vk, eij - (ea + Epool[d.eYv + b]), ej, ek, store ? &x : nullptr);
                            tv = store ? narrow<float>(x) : 0.f;
                        }
                        if (store) {
                            const long long e = ((long long)(d.jY0 + j) * vY + b) * mXc + (long long)(d.iX0 + i) * vX + a;
                            Vst[e] = vab;
                            Vst[mXc * mYc + e] = tv;
                        }
                    }
                }
            }
            if constexpr (PAIRS) {
                ej = ff_f64(sj);
                ek = ff_f64(sk);
            }
            red[0][tid] = ej;
            red[1][tid] = ek;
        }
        __syncthreads();                         // sums written; S1 consumed
        if (t.nbuf == 1 && nn > 0)
            load_slices(S0, H0 + (long long)(g0 + t.np) * rows, nn, nX, nY, 8 * t.bmX, t.kY, ldY, t.slab, tid);
        // w lanes per pair (w fixed by its block count): its blocks' sums, lanes strided, then
        // a fixed tree, so that a pair's sums do not depend on the pairs that ran with it
        // (the largest power of two within it: a group's pairs then take one pass)
        const int w = nb2 >= 32 ? 32 : nb2 >= 16 ? 16 : nb2 >= 8 ? 8 : nb2 >= 4 ? 4 : nb2 >= 2 ? 2 : 1;
        for (int q = tid; q < (np * w + 31) / 32 * 32; q += kTThreads) {   // whole warps
            const int p = q / w, l = q - p * w;
            double sj = 0.0, sk = 0.0;
            if (p < np)
                for (int k = l; k < nb2; k += w) {
                    sj += red[0][p * nb2 + k];
                    sk += red[1][p * nb2 + k];
                }
            for (int o = w >> 1; o > 0; o >>= 1) {
                sj += __shfl_xor_sync(0xffffffffu, sj, o);
                sk += __shfl_xor_sync(0xffffffffu, sk, o);
            }
            if (p < np && l == 0) {
                part[2 * (tk.first + g0 + p)] = sj;
                part[2 * (tk.first + g0 + p) + 1] = sk;
            }
        }
    }
}

// Per dimer: its partials (one per task, FP32 one per pair) -> {4 sum, -2 sum}; a
// warp each, lane l partials l, l + 32, ... in order, then the fixed tree (400
// of a 128-AO dimer added by one thread took 23 to 40 us).
__global__ void __launch_bounds__(32)
k_finish_sum(const DimerDesc* __restrict__ dd, const FinTask* __restrict__ tasks, const int* __restrict__ first_task,
             const double* __restrict__ part, double* __restrict__ E2)
{
    const int k = blockIdx.x, lane = threadIdx.x;
    const FinTask t0 = tasks[first_task[k]];
    double ej = 0.0, ek = 0.0;
    for (int t = t0.first + lane; t < t0.first + t0.nparts; t += 32) {
        ej += part[2 * t];
        ek += part[2 * t + 1];
    }
    const double s = pair_tree(ej, ek, lane);
    if ((lane & 15) == 0) E2[2 * dd[k].slot + (lane >> 4)] = lane ? -2.0 * s : 4.0 * s;
}

template <typename T, bool PAIRS, int W>
cudaError_t launch_w32(const DimerDesc* d_desc, int nd, const T* C, const double* Epool, T* H, double* E2,
                       T* VT, FinSplit sp, cudaStream_t s)
{
    const size_t smem = w32_smem_bytes<T>(W);
    auto fn = VT ? k_finish_w32<T, true, PAIRS, W> : k_finish_w32<T, false, PAIRS, W>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    // all of the unified L1 as shared memory, so that the CTAs the registers
    // allow are also resident by shared memory
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    fn<<<dim3(sp.parts, nd), W * 32, smem, s>>>(d_desc, C, Epool, H, E2, VT, sp.parts, sp.cnt);
    return cudaGetLastError();
}

template <typename T, bool PAIRS>
cudaError_t launch_finish(const DimerDesc* d_desc, int nd, int max_ao, const T* C, const double* Epool,
                          T* H, double* E2, const FinTask* tasks, int ntasks, double* part, T* VT,
                          FinSplit sp, cudaStream_t s)
{
    if (nd <= 0) return cudaSuccess;
    if (max_ao <= 32)
        return sp.warps == 5 ? launch_w32<T, PAIRS, 5>(d_desc, nd, C, Epool, H, E2, VT, sp, s)
                             : launch_w32<T, PAIRS, 4>(d_desc, nd, C, Epool, H, E2, VT, sp, s);
    if (!tasks || ntasks <= 0 || !part) return cudaErrorInvalidValue;
    cudaError_t e;
    if constexpr (sizeof(T) == 4) {
        e = cudaFuncSetAttribute(k_finish_tiled_f32<PAIRS>, cudaFuncAttributeMaxDynamicSharedMemorySize, kF32Cap);
        if (e != cudaSuccess) return e;
        k_finish_tiled_f32<PAIRS><<<ntasks, kTThreads, kF32Cap, s>>>(d_desc, tasks, C, Epool, H, part,
                                                                      kF32Cap / (int)sizeof(float), VT);
    } else {
        const size_t smem = tiled_smem_bytes(max_ao);
        if (smem > 227 * 1024) return cudaErrorInvalidValue;
        e = cudaFuncSetAttribute(k_finish_tiled, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        const int smem_elems = (int)((smem - 2 * max_ao * sizeof(double) - 64) / sizeof(double));
        k_finish_tiled<<<ntasks, kTThreads, smem, s>>>(d_desc, tasks, C, Epool, H, part, smem_elems, VT);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // the dimers' first-task indices follow the task array
    const int* first = reinterpret_cast<const int*>(tasks + ntasks);
    k_finish_sum<<<nd, 32, 0, s>>>(d_desc, tasks, first, part, E2);
    return cudaGetLastError();
}

template <int W>
cudaError_t launch_finish_ff_t(const DimerDesc* d_desc, int nd, const double* C, const double* Epool, FF* H,
                               double* E2, double* VT, FinSplit sp, cudaStream_t s)
{
    if (nd <= 0) return cudaSuccess;
    const size_t smem = w32_ff_smem_bytes(W);
    auto fn = VT ? k_finish_w32_ff<true, W> : k_finish_w32_ff<false, W>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    fn<<<dim3(sp.parts, nd), W * 32, smem, s>>>(d_desc, C, Epool, H, E2, VT, sp.parts, sp.cnt);
    return cudaGetLastError();
}

// Split dimers: the blocks' terms added in block order.
__global__ void k_fold(const int* __restrict__ fold, int nfold, double* __restrict__ E2)
{
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= nfold) return;
    const int d = fold[3 * f], first = fold[3 * f + 1], n = fold[3 * f + 2];
    double sj = 0.0, sk = 0.0;
    for (int b = 0; b < n; b++) {
        sj += E2[2 * (first + b)];
        sk += E2[2 * (first + b) + 1];
    }
    E2[2 * d] = sj;
    E2[2 * d + 1] = sk;
}

// ------------------------------------------------------------ reduction
__device__ __forceinline__ void neumaier_add(double& s, double& c, double v)
{
    const double t = s + v;
    if (fabs(s) >= fabs(v)) c += (s - t) + v;
    else                    c += (v - t) + s;
    s = t;
}

// Knuth's TwoSum of two compensated sums (s, c) and (s2, c2) into (s, c).
__device__ __forceinline__ void twosum_pair(double& s, double& c, double s2, double c2)
{
    const double t = s + s2;
    const double bp = t - s;
    const double err = (s - (t - bp)) + (s2 - bp);
    c = c + c2 + err;
    s = t;
}

// The 32 lanes' compensated sums of J and K, (sj, cj) and (sk, ck), merged by
// a fixed tree of TwoSums: the halves of the warp swap a sum first, so that
// lanes 0-15 merge J while lanes 16-31 merge K (one dependent TwoSum per level
// instead of two).  Returns J's sum in lanes 0-15, K's in 16-31.
__device__ __forceinline__ void warp_merge(double sj, double cj, double sk, double ck, int lane, double& s, double& c)
{
    const bool hi = lane >= 16;
    s = hi ? sk : sj;
    c = hi ? ck : cj;
    const double s2 = __shfl_xor_sync(0xffffffffu, hi ? sj : sk, 16);
    const double c2 = __shfl_xor_sync(0xffffffffu, hi ? cj : ck, 16);
    twosum_pair(s, c, s2, c2);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
        const double s3 = __shfl_xor_sync(0xffffffffu, s, o), c3 = __shfl_xor_sync(0xffffffffu, c, o);
        twosum_pair(s, c, s3, c3);
    }
}

// One warp per block.  Blocks [0, n_mon): a monomer each; lane l sums half of
// the terms of the monomer's dimers l, l + 32, ... of its list (Neumaier), and
// the warp tree merges the lanes: the list's loads are in flight together.
// Blocks [n_mon, n_mon + nbt): the lattice total, block b over a fixed
// contiguous range of the dimer list, its lanes over fixed strides (Neumaier),
// merged by the warp tree; the last of several blocks to arrive merges the
// block sums the same way (cnt: zero before the launch and again after it).
// Bound by dependent FP64 additions and loads.  An SM's FP64 pipe takes 16
// cycles for one warp's addition, so warps that share an SM wait on each
// other: single-warp blocks spread them over the chip.  One launch instead of
// two with shared-memory trees of both sums over 256 threads.  The partition
// depends only on the dimer and monomer counts, so every run gives the same
// bits.  With a mirror the results also go to mapped host memory as they are
// formed, which spares the caller five device-to-host copies (one dimer's call
// 93 -> 48 us).
__global__ void __launch_bounds__(32)
k_reduce(const double* __restrict__ E2, int nd, MonomerLists L, double* __restrict__ mon, int nbt,
         double* __restrict__ partials, double* __restrict__ total, unsigned* __restrict__ cnt, ResultMirror mir)
{
    const int lane = threadIdx.x;
    double sj = 0, cj = 0, sk = 0, ck = 0, s, c;
    if ((int)blockIdx.x < L.n_mon) {
        const int m = blockIdx.x;
        for (int k = L.start[m] + lane; k < L.start[m + 1]; k += 32) {
            const int dslot = L.list[k];
            neumaier_add(sj, cj, 0.5 * E2[2 * dslot]);
            neumaier_add(sk, ck, 0.5 * E2[2 * dslot + 1]);
        }
        warp_merge(sj, cj, sk, ck, lane, s, c);
        if ((lane & 15) == 0) {
            mon[(lane >> 4) * L.n_mon + m] = s + c;
            if (mir.out) mir.out[(lane >> 4) * L.n_mon + m] = s + c;
        }
        return;
    }
    const int b = blockIdx.x - L.n_mon;
    const int per = (nd + nbt - 1) / nbt;
    const int b0 = b * per, b1 = min(nd, b0 + per);
    double2* const out2 = reinterpret_cast<double2*>(mir.out + 2 * L.n_mon + 2);
    for (int k = b0 + lane; k < b1; k += 32) {
        const double2 e = *reinterpret_cast<const double2*>(E2 + 2 * k);
        if (mir.out) out2[k] = e;
        neumaier_add(sj, cj, e.x);
        neumaier_add(sk, ck, e.y);
    }
    warp_merge(sj, cj, sk, ck, lane, s, c);
    if (nbt > 1) {
        unsigned arrived = 0;
        if ((lane & 15) == 0) {
            __stcg(partials + 4 * b + (lane >> 3), s);
            __stcg(partials + 4 * b + (lane >> 3) + 1, c);
            __threadfence();
        }
        __syncwarp();
        if (lane == 0) arrived = atomicAdd(cnt, 1u);
        if (__shfl_sync(0xffffffffu, arrived, 0) != (unsigned)nbt - 1) return;
        __threadfence();
        sj = cj = sk = ck = 0;
        for (int k = lane; k < nbt; k += 32) {
            twosum_pair(sj, cj, __ldcg(partials + 4 * k), __ldcg(partials + 4 * k + 1));
            twosum_pair(sk, ck, __ldcg(partials + 4 * k + 2), __ldcg(partials + 4 * k + 3));
        }
        warp_merge(sj, cj, sk, ck, lane, s, c);
        if (lane == 0) *cnt = 0;
    }
    if ((lane & 15) == 0) {
        total[lane >> 4] = s + c;
        if (mir.out) mir.out[2 * L.n_mon + (lane >> 4)] = s + c;
    }
    if (lane == 0 && mir.out) *reinterpret_cast<int*>(mir.out + 2 * L.n_mon + 2 + 2 * nd) = mir.status ? *mir.status : 0;
}

__global__ void k_check_finite(const double* __restrict__ x, long long n, int* flag)
{
    bool bad = false;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x)
        bad |= !isfinite(x[k]);
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
}

__global__ void k_check_finite4(const double* __restrict__ x, int d0, int d1, int d2, int d3,
                                long long s0, long long s1, long long s2, int* flag)
{
    const long long n = (long long)d0 * d1 * d2 * d3;
    bool bad = false;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        long long r = k;
        const int i3 = r % d3; r /= d3;
        const int i2 = r % d2; r /= d2;
        const int i1 = r % d1; r /= d1;
        const int i0 = (int)r;
        bad |= !isfinite(x[i0 * s0 + i1 * s1 + i2 * s2 + i3]);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
}

}  // namespace

cudaError_t launch_finish_fp64(const DimerDesc* d_desc, int nd, int max_ao, const double* Cpool,
                               const double* Epool, double* H, double* E2, const FinTask* tasks,
                               int ntasks, double* part, double* VT, FinSplit sp, cudaStream_t s)
{
    return launch_finish<double, false>(d_desc, nd, max_ao, Cpool, Epool, H, E2, tasks, ntasks, part, VT, sp, s);
}

cudaError_t launch_finish_fp32(const DimerDesc* d_desc, int nd, int max_ao, const float* Cf,
                               const double* Epool, float* H, double* E2, const FinTask* tasks,
                               int ntasks, double* part, float* VT, bool fp64_epilogue, FinSplit sp,
                               cudaStream_t s)
{
    return fp64_epilogue
               ? launch_finish<float, false>(d_desc, nd, max_ao, Cf, Epool, H, E2, tasks, ntasks, part, VT, sp, s)
               : launch_finish<float, true>(d_desc, nd, max_ao, Cf, Epool, H, E2, tasks, ntasks, part, VT, sp, s);
}

cudaError_t launch_finish_ff(const DimerDesc* d_desc, int nd, int max_ao, const double* Cpool, const double* Epool,
                             void* H, double* E2, double* VT, FinSplit sp, cudaStream_t s)
{
    if (max_ao > 32) return cudaErrorInvalidValue;
    FF* Hf = static_cast<FF*>(H);
    return sp.warps == 5 ? launch_finish_ff_t<5>(d_desc, nd, Cpool, Epool, Hf, E2, VT, sp, s)
                         : launch_finish_ff_t<4>(d_desc, nd, Cpool, Epool, Hf, E2, VT, sp, s);
}

// One round (a warp per pair) per CTA of four warps: the CTAs of a dimer run
// on different SMs, so a wave of few dimers fills the chip instead of one SM
// per dimer, and the CTAs' fine grain evens out the end of a larger wave.
// Measured in us, one CTA of four warps per dimer against this: FP32, 1 / 28 /
// 158 / 227 dimers 62 / 62 / 84 / 87 -> 17 / 22 / 54 / 70; FP64 (31 us of FP64
// pipe per pair) 1 / 158 / 1036 dimers 1026 / 1682 / 5965 -> 154 / 952 / 5574;
// FP64E 364 / 531 / 2117 -> 66 / 346 / 2065.  Five warps where they keep a
// wave at one CTA per SM and four do not (28 dimers of 25 pairs: FP64 265 ->
// 176).  FP32 waves of more than six dimers per SM are bound by the FP32
// pipes either way, and staging the coefficients once per dimer is then the
// cheaper: 1036 dimers 256 against 266, 2248 dimers 513 against 557.
// FP64E (two CTAs per SM, 74 us of pair arithmetic per round of four pairs, 0.18
// of that to stage the coefficients) takes whichever of the two fills its last
// set of CTAs better: 25 pairs, one CTA per dimer against seven, 158 dimers 530 /
// 350, 304 554 / 630, 1036 2129 / 2104, 1216 2153 / 2466, 2216 4230 / 4460; 9
// pairs against three, 158 187 / 153, 1036 736 / 804; two to five CTAs for 25
// pairs were slower than the better of these at every size.
FinSplit finish_w32_split(const DimerDesc* h, int nd, int form, int sms)
{
    int pairs = 1;
    for (int k = 0; k < nd; k++) pairs = std::max(pairs, h[k].oX * h[k].oY);
    if ((form == FIN_F32_PAIRS || form == FIN_F32_F64EPI) && nd > 6 * sms) return FinSplit{4, 1, nullptr};
    const int p4 = (pairs + 3) / 4, p5 = (pairs + 4) / 5;
    if (form == FIN_FF) {                      // in hundredths of a round
        auto sets = [&](long long ctas) { return (ctas + 2 * sms - 1) / (2 * sms); };
        if (sets(nd) * (100 * p4 + 18) < sets((long long)nd * p4) * 118) return FinSplit{4, 1, nullptr};
    }
    const bool five = (long long)nd * p5 <= sms && (long long)nd * p4 > sms;
    return five ? FinSplit{5, p5, nullptr} : FinSplit{4, p4, nullptr};
}

int finish_tasks(const DimerDesc* h, int nd, bool fp32, int sms, std::vector<FinTask>* out)
{
    out->clear();
    constexpr long long kTaskFma = 1 << 22;
    auto fma_of = [](const DimerDesc& d) {     // multiply-adds of one pair, both forms
        const long long nX = d.nX, nY = d.nY, vX = d.vX, vY = d.vY;
        return std::max(1LL, 2 * (nX * nY * vY + vX * vY * nX));
    };
    if (!fp32) {
        for (int k = 0; k < nd; k++) {
            const int pairs = h[k].oX * h[k].oY;
            const int ppt = (int)std::max<long long>(1, std::min<long long>(pairs, kTaskFma / fma_of(h[k])));
            const int ntasks = (pairs + ppt - 1) / ppt, first = (int)out->size();
            for (int t = 0; t < ntasks; t++)
                out->push_back(FinTask{k, t * ppt, std::min(pairs, (t + 1) * ppt), first, ntasks});
        }
        return (int)out->size();
    }
    // FP32: whole groups of the pairs that run together, about kTaskFma multiply-adds;
    // a wave with less than a quarter of one per SM gives each SM its share (the
    // energies do not depend on it): one dimer of 48 AO, 64 pairs, 53 -> 40 us
    long long total = 0;
    for (int k = 0; k < nd; k++) total += fma_of(h[k]) * h[k].oX * h[k].oY;
    const bool few = total / sms < kTaskFma / 4;
    const long long per_task = few ? total / sms : kTaskFma;
    int pairs_before = 0;
    for (int k = 0; k < nd; k++) {
        const int pairs = h[k].oX * h[k].oY;
        const int grp = tiled_shape(h[k].nX, h[k].nY, h[k].vX, h[k].vY, kF32Cap / (int)sizeof(float)).np;
        const long long want = std::max(1LL, (per_task + (few ? fma_of(h[k]) - 1 : 0)) / fma_of(h[k]));
        const int ppt = (int)std::min<long long>(pairs, want >= grp ? want / grp * grp : few ? want : grp);
        for (int p = 0; p < pairs; p += ppt)
            out->push_back(FinTask{k, p, std::min(pairs, p + ppt), pairs_before, pairs});
        pairs_before += pairs;
    }
    return pairs_before;
}

cudaError_t launch_fold(const int* fold, int nfold, double* E2, cudaStream_t s)
{
    if (nfold <= 0) return cudaSuccess;
    k_fold<<<(nfold + 127) / 128, 128, 0, s>>>(fold, nfold, E2);
    return cudaGetLastError();
}

cudaError_t launch_reduce(const double* E2, int nd, MonomerLists lists, double* mon, double* total,
                          double* scratch, unsigned* cnt, ResultMirror mir, cudaStream_t s)
{
    // two dimers per lane of a total block, at most kReduceBlocks blocks
    const int nbt = std::max(1, std::min(kReduceBlocks, (nd + 63) / 64));
    k_reduce<<<lists.n_mon + nbt, 32, 0, s>>>(E2, nd, lists, mon, nbt, scratch, total, cnt, mir);
    return cudaGetLastError();
}

cudaError_t launch_check_finite(const double* x, long long n, int* flag, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    long long blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    k_check_finite<<<(int)blocks, 256, 0, s>>>(x, n, flag);
    return cudaGetLastError();
}

cudaError_t launch_check_finite4(const double* x, const int dims[4], const long long st[3], int* flag,
                                 cudaStream_t s)
{
    const long long n = (long long)dims[0] * dims[1] * dims[2] * dims[3];
    if (n <= 0) return cudaSuccess;
    long long blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    k_check_finite4<<<(int)blocks, 256, 0, s>>>(x, dims[0], dims[1], dims[2], dims[3], st[0], st[1], st[2], flag);
    return cudaGetLastError();
}

}  // namespace mcpt
