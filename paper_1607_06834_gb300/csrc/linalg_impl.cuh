// Vector kernels of the ROK step (Sec. 2.2.2): inner products, the
// modified-Gram-Schmidt passes of the Arnoldi process, the projected stage
// solves of Eq. ROK, stage vectors and combines.
//
// Compiled twice like the stencil (linalg_fast.cu, linalg_strict.cu with
// --fmad=false), each time inside namespace ROK_NS.
//
// Every inner product is the pairwise sum of the rounded entrywise products: a
// balanced binary tree over the natural index order, zero-padded to a power of
// two.  The GPU evaluates exactly that tree:
//   - every lane owns 8 consecutive entries and adds them as a 3-level tree in
//     registers (vector loads when aligned);
//   - the 32 lanes of a warp own 256 consecutive entries; an xor butterfly of
//     increasing distance (1, 2, 4, 8, 16) adds the lane sums as the next 5
//     tree levels;
//   - the 8 warps of a CTA own 2048 consecutive entries, added as 3 levels;
//   - the CTA partials are added as a tree again by the consumer (one warp,
//     contiguous chunks per lane, then a butterfly).
// Addition is commutative in IEEE arithmetic, so both partners of a butterfly
// hold the same sum; the result is deterministic and independent of the launch
// configuration (extra zero leaves change nothing).
//
// On GB300 the FP64 pipe is the scarce unit (2 FP64 lanes per SM per clock):
// summing in registers first keeps the tree at about 1.5 additions per entry
// (a butterfly over strided entries would cost 5), which puts a fused MGS pass
// (1 FMA, 1 product, the tree) at the HBM/FP64 balance point.
#pragma once
#include <math.h>
#include <stdint.h>

#include "intdot.cuh"
#include "linalg.cuh"

namespace rok {
namespace ROK_NS {

constexpr int RT = 256;            // threads per CTA
constexpr int EPL = 8;             // consecutive entries per lane
constexpr int RB = RT * EPL;       // entries per CTA (2048)

__device__ __forceinline__ bool aligned16(const void *p) { return ((uintptr_t)p & 15) == 0; }

// x[0..8) = p[e0 .. e0+8) (zero beyond n); 16-byte vector loads when aligned
__device__ __forceinline__ void load8(const double *__restrict__ p, size_t e0, size_t n, double (&x)[EPL])
{
    if (e0 + EPL <= n && aligned16(p)) {
        const double2 *q = reinterpret_cast<const double2 *>(p + e0);
#pragma unroll
        for (int k = 0; k < EPL / 2; ++k) {
            double2 t = q[k];
            x[2 * k] = t.x;
            x[2 * k + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < EPL; ++k) x[k] = e0 + k < n ? p[e0 + k] : 0.0;
    }
}

__device__ __forceinline__ void load8(const float *__restrict__ p, size_t e0, size_t n, float (&x)[EPL])
{
    if (e0 + EPL <= n && aligned16(p + e0)) {
        const float4 *q = reinterpret_cast<const float4 *>(p + e0);
#pragma unroll
        for (int k = 0; k < EPL / 4; ++k) {
            float4 t = q[k];
            x[4 * k] = t.x;
            x[4 * k + 1] = t.y;
            x[4 * k + 2] = t.z;
            x[4 * k + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < EPL; ++k) x[k] = e0 + k < n ? p[e0 + k] : 0.0f;
    }
}

__device__ __forceinline__ void store8(double *__restrict__ p, size_t e0, size_t n, const double (&x)[EPL])
{
    if (e0 + EPL <= n && aligned16(p)) {
        double2 *q = reinterpret_cast<double2 *>(p + e0);
#pragma unroll
        for (int k = 0; k < EPL / 2; ++k) q[k] = make_double2(x[2 * k], x[2 * k + 1]);
    } else {
#pragma unroll
        for (int k = 0; k < EPL; ++k)
            if (e0 + k < n) p[e0 + k] = x[k];
    }
}

__device__ __forceinline__ void store8(float *__restrict__ p, size_t e0, size_t n, const float (&x)[EPL])
{
    if (e0 + EPL <= n && aligned16(p + e0)) {
        float4 *q = reinterpret_cast<float4 *>(p + e0);
#pragma unroll
        for (int k = 0; k < EPL / 4; ++k) q[k] = make_float4(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < EPL; ++k)
            if (e0 + k < n) p[e0 + k] = x[k];
    }
}

// tree over the 8 consecutive entries of a lane
template <class T>
__device__ __forceinline__ T tree8(const T (&x)[EPL])
{
    return ((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7]));
}

template <class T>
__device__ __forceinline__ T lane_tree(T v)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// tree over the 8 warp sums of a CTA; sh >= 9 values; result in every thread
template <class T>
__device__ __forceinline__ T cta_tree(T wsum, T *sh)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = wsum;
    __syncthreads();
    if (wid == 0) {
        T v = lane < 8 ? sh[lane] : T(0);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        if (lane == 0) sh[8] = v;
    }
    __syncthreads();
    return sh[8];
}

// CTA sum of one 8-entry chunk per lane: the lane's entries, the lane
// butterfly, then the warp tree
template <class T>
__device__ __forceinline__ T chunk_sum(const T (&x)[EPL], T *sh)
{
    return cta_tree(lane_tree(tree8(x)), sh);
}

// The lane's part of a dot product, sum_k a_k b_k over its 8 entries (in T).
// Strict build: the 8 products, then the aligned tree (the order of a plain
// pairwise evaluation).  FMA build (ROK_LINALG_FAST): one chain of fused
// multiply-adds in entry order, 8 FP64 operations instead of 11 (deterministic,
// other rounding).
template <class T, class U>
__device__ __forceinline__ T lane_dot(const U (&a)[EPL], const T (&b)[EPL])
{
#ifdef ROK_LINALG_FAST
    T s = (T)a[0] * b[0];
#pragma unroll
    for (int k = 1; k < EPL; ++k) s = (T)a[k] * b[k] + s;
    return s;
#else
    T x[EPL];
#pragma unroll
    for (int k = 0; k < EPL; ++k) x[k] = (T)a[k] * b[k];
    return tree8(x);
#endif
}

// CTA sum from the lanes' parts v (lane butterfly, then the warp tree)
template <class T>
__device__ __forceinline__ T chunk_sumv(T v, T *sh)
{
    return cta_tree(lane_tree(v), sh);
}

// Aligned tree over the C consecutive leaves p[lo .. lo + C) (zero beyond P),
// C a power of two: up to 32 leaves are loaded at once (independent loads) and
// added level by level; longer runs use a carry stack over the leaves in order.
template <int L, class T>
__device__ __forceinline__ T leaf_tree_fixed(const T *__restrict__ p, int lo, int P)
{
    T x[L];
#pragma unroll
    for (int k = 0; k < L; ++k) x[k] = lo + k < P ? p[lo + k] : T(0);
#pragma unroll
    for (int len = L; len > 1; len >>= 1)
#pragma unroll
        for (int i = 0; i < len / 2; ++i) x[i] = x[2 * i] + x[2 * i + 1];
    return x[0];
}

template <class T>
__device__ __forceinline__ T leaf_tree(const T *__restrict__ p, int lo, int C, int P)
{
    switch (C) {
    case 1: return lo < P ? p[lo] : T(0);
    case 2: return leaf_tree_fixed<2>(p, lo, P);
    case 4: return leaf_tree_fixed<4>(p, lo, P);
    case 8: return leaf_tree_fixed<8>(p, lo, P);
    case 16: return leaf_tree_fixed<16>(p, lo, P);
    case 32: return leaf_tree_fixed<32>(p, lo, P);
    default: break;
    }
    T stack[24];
    for (int k = 0; k < C; ++k) {
        T s = lo + k < P ? p[lo + k] : T(0);
        int lvl = 0;
        for (int m = k; m & 1; m >>= 1, ++lvl) s = stack[lvl] + s;
        stack[lvl] = s;
    }
    int top = 0;
    while ((1 << top) < C) ++top;
    return stack[top];
}

__device__ __forceinline__ int pow2_ceil(int P)
{
    int P2 = 1;
    while (P2 < P) P2 <<= 1;
    return P2;
}

// Tree sum of p[0..P) (zero-padded to a power of two) by one warp: lane l owns
// the C = P2/32 consecutive leaves [lC, lC + C), then the lane butterfly.
template <class T>
__device__ __forceinline__ T warp_tree_partials(const T *__restrict__ p, int P)
{
    const int P2 = pow2_ceil(P);
    const int lane = threadIdx.x & 31;
    const int C = P2 > 32 ? P2 / 32 : 1;
    return lane_tree(leaf_tree(p, lane * C, C, P));
}

// The same tree by the CTA's first four warps, one per scheduler (thread
// t < 128 owns C = P2/128 leaves; the four warp sums are added by one thread),
// result in every thread; sh >= 5 values.  Half the FP64 instructions of a
// tree spread over all eight warps, whose lane butterflies would repeat on
// every warp.
template <class T>
__device__ __forceinline__ T tree_partials(const T *__restrict__ p, int P, T *sh)
{
    const int P2 = pow2_ceil(P);
    const int C = P2 > 128 ? P2 / 128 : 1;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (wid < 4) {
        const T v = lane_tree(leaf_tree(p, threadIdx.x * C, C, P));
        if (lane == 0) sh[wid] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) sh[4] = (sh[0] + sh[1]) + (sh[2] + sh[3]);
    __syncthreads();
    return sh[4];
}

__device__ __forceinline__ size_t lane_e0() { return ((size_t)blockIdx.x * RT + threadIdx.x) * EPL; }

// ---- persistent kernels: arrival counters and paired chunk sums -----------------

constexpr int kColChunks = 2;                  // chunks of 2048 entries per CTA (max)
constexpr long long kBarrierSpins = 1LL << 22; // 4M polls (~0.3 s or more), then give up

// gpu-scope acquire / release accesses of the arrival counters
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_add_release_gpu(unsigned *p, unsigned x)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
}

// The sums of two 2048-entry chunks at once from the lanes' parts a and b
// (lane_dot), each the same tree as chunk_sumv: even lanes finish the first
// chunk's butterfly and odd lanes the second's (one exchange and five
// additions per lane instead of ten); then the two 8-warp trees together.
// Results in thread 0 (first) and thread 8 (second).  sh needs 16 entries.
template <class T>
__device__ __forceinline__ void chunk_sum2v(const T a, const T b, T *sh, T &sa, T &sb)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool odd = lane & 1;
    const T recv = __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
    T v = odd ? recv + b : a + recv;   // a_l + a_{l+1} on even lanes, b_{l-1} + b_l on odd lanes
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    __syncthreads();
    if (lane < 2) sh[lane * 8 + wid] = v;
    __syncthreads();
    if (wid == 0) {
        T u = lane < 16 ? sh[lane] : T(0);
        u += __shfl_xor_sync(0xffffffffu, u, 1);
        u += __shfl_xor_sync(0xffffffffu, u, 2);
        u += __shfl_xor_sync(0xffffffffu, u, 4);
        if (lane == 0) sa = u;
        if (lane == 8) sb = u;
    }
}

// Per-generation arrival counters (the persistent Arnoldi column): after
// writing its partials of a generation, a CTA adds one to that generation's
// counter (release, no reply awaited); a CTA that needs the generation waits
// (thread 0, acquire, bounded) until the counter reaches the grid size.  Each
// counter serves one generation and is zeroed before the launch, so the
// arrivals neither wait for an atomic's reply nor need a release by the last
// one.
__device__ __forceinline__ void gen_arrive(unsigned *cnt)
{
    __syncthreads();
    if (threadIdx.x == 0) red_add_release_gpu(cnt, 1u);
}

__device__ __forceinline__ bool gen_wait(const unsigned *cnt, unsigned nblocks, int *status,
                                         long long max_spins = kBarrierSpins)
{
    __shared__ int ok;
    if (threadIdx.x == 0) {
        ok = 1;
        long long spins = 0;
        while (ld_acquire_gpu(cnt) < nblocks) {
            if (++spins > max_spins) {
                atomicOr(status, kStatusTimeout);
                ok = 0;
                break;
            }
            __nanosleep(32);
        }
    }
    __syncthreads();
    return ok != 0;
}

// Hint: fetch the 128-byte line holding this thread's entries of p (from e0)
// into L2; one thread per line issues it.
template <class T>
__device__ __forceinline__ void prefetch_l2(const T *p, size_t e0, size_t n)
{
    constexpr int kThreadsPerLine = 128 / (EPL * (int)sizeof(T));
    if (e0 < n && threadIdx.x % kThreadsPerLine == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + e0));
}

#ifndef ROK_LINALG_DEVICE_ONLY
// partials[b] = <a0, b0> and partials[P + b] = <a1, b1> (if a1) over CTA b's range
__global__ void __launch_bounds__(RT) dot2_kernel(const double *__restrict__ a0, const double *__restrict__ b0,
                                                  const double *__restrict__ a1, const double *__restrict__ b1,
                                                  size_t n, double *__restrict__ partials, int P,
                                                  const int *active)
{
    if (active && *active == 0) return;
    __shared__ double sh[10];
    const size_t e0 = lane_e0();
    double x[EPL], y[EPL];
    load8(a0, e0, n, x);
    load8(b0, e0, n, y);
    double s0 = chunk_sumv(lane_dot(x, y), sh);
    double s1 = 0.0;
    if (a1) {
        load8(a1, e0, n, x);
        load8(b1, e0, n, y);
        s1 = chunk_sumv(lane_dot(x, y), sh);
    }
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = s0;
        partials[P + blockIdx.x] = s1;
    }
}

// h = tree(pin); H entry <- h; w <- w - h vprev; pout[b] = <vnext, w> (or <w, w>)
__global__ void __launch_bounds__(RT) mgs_kernel(double *__restrict__ w, const double *__restrict__ vprev,
                                                 const double *__restrict__ vnext, size_t n,
                                                 const double *__restrict__ pin, int P, double *hout,
                                                 double *__restrict__ pout, int first, StepState *st)
{
    if (st->active == 0) return;
    __shared__ double sh[10];
    const size_t e0 = lane_e0();
    double wv[EPL], vp[EPL], vn[EPL];
    load8(w, e0, n, wv);
    load8(vprev, e0, n, vp);
    if (vnext) load8(vnext, e0, n, vn);
    const double h = tree_partials(pin, P, sh);
    if (first) {
        double wn2 = tree_partials(pin + P, P, sh);
        if (blockIdx.x == 0 && threadIdx.x == 0) st->wnorm0 = sqrt(wn2);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *hout = h;
#pragma unroll
    for (int k = 0; k < EPL; ++k) wv[k] = wv[k] - h * vp[k];
    store8(w, e0, n, wv);
    double s = chunk_sumv(vnext ? lane_dot(vn, wv) : lane_dot(wv, wv), sh);
    if (threadIdx.x == 0) pout[blockIdx.x] = s;
}

#ifndef ROK_LINALG_FAST
// hn = sqrt(tree(pin)); breakdown test; v = w * (1/hn)
__global__ void __launch_bounds__(RT) normalize_kernel(const double *__restrict__ w, double *__restrict__ v,
                                                       size_t n, const double *__restrict__ pin, int P,
                                                       double *hsub, int column, StepState *st)
{
    // block 0 may clear st->active below while other CTAs start: read it once
    // per CTA so that every thread of a CTA takes the same branch
    __shared__ int act;
    __shared__ double sh[10];
    if (threadIdx.x == 0) act = st->active;
    __syncthreads();
    if (act == 0) return;
    const double hn = sqrt(tree_partials(pin, P, sh));
    // column 0: v_1 = f(y_n)/beta, beta = 0 leaves an empty basis; later columns
    // stop when h_{j+1,j} <= 1e-12 ||J v_j|| (also catches NaN)
    const bool brk = column == 0 ? !(hn > 0.0) : !(hn > 1e-12 * st->wnorm0);
    if (brk) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->active = 0;
            st->meff = column;
        }
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (hsub) *hsub = hn;
        if (column == 0) st->beta = hn;
    }
    const double r = 1.0 / hn;
    const size_t e0 = lane_e0();
    double x[EPL];
    load8(w, e0, n, x);
#pragma unroll
    for (int k = 0; k < EPL; ++k) x[k] = x[k] * r;
    store8(v, e0, n, x);
}

#endif

// Lane trees of 16 values at once by recursive halving across the lanes: at
// level l (exchange with lane ^ 2^l) each lane keeps half of its remaining
// values and adds the partner's copy of them, so every value's sum over the 32
// lanes is the same aligned pairwise tree as lane_tree, for 16 additions per
// lane instead of 80.  Lane l (and l ^ 16) ends with the sum of value
// 8 b0 + 4 b1 + 2 b2 + b3, b_k the bits of l.
template <class T>
__device__ __forceinline__ T lane_tree16(T (&t)[16], int lane)
{
#pragma unroll
    for (int lev = 0; lev < 4; ++lev) {
        const int half = 8 >> lev;
        const bool upper = (lane >> lev) & 1;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const T recv = __shfl_xor_sync(0xffffffffu, upper ? t[k] : t[k + half], 1 << lev);
            t[k] = upper ? recv + t[k + half] : t[k] + recv;
        }
    }
    T v = t[0];
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    return v;
}

__device__ __forceinline__ int lane_tree16_value(int lane)
{
    return ((lane & 1) << 3) | ((lane & 2) << 1) | ((lane & 4) >> 1) | ((lane & 8) >> 3);
}

// 8 warp sums of one CTA added as the warp tree of cta_tree does
__device__ __forceinline__ double warp8_tree(const double *w)
{
    return ((w[0] + w[1]) + (w[2] + w[3])) + ((w[4] + w[5]) + (w[6] + w[7]));
}

#ifdef ROK_LINALG_FAST
// the exponent field of a lane's entries and their limbs (idot)
__device__ __forceinline__ int lane_limbs(const double (&w)[EPL], idot::Limb (&wl)[EPL])
{
    int ew = 0;
#pragma unroll
    for (int k = 0; k < EPL; ++k) ew = max(ew, idot::magnitude(w[k]));
    ew = idot::top(ew);
#pragma unroll
    for (int k = 0; k < EPL; ++k) wl[k] = idot::limbs(w[k], ew);
    return ew;
}

// <v, w> of one lane's 8 entries on the integer pipe, w given as limbs (and in
// memory, for the operands that idot leaves out)
__device__ __forceinline__ double lane_idot(const double (&v)[EPL], const idot::Limb (&wl)[EPL], int ew,
                                            const double *w, size_t e0, size_t n)
{
    int ev = 0;
#pragma unroll
    for (int k = 0; k < EPL; ++k) ev = max(ev, idot::magnitude(v[k]));
    ev = idot::top(ev);
    if (!idot::usable(ev) || !idot::usable(ew)) {
        double x[EPL];
        load8(w, e0, n, x);
        return lane_dot(v, x);
    }
    idot::Acc s{0, 0, 0};
#pragma unroll
    for (int k = 0; k < EPL; ++k) idot::mad(s, idot::limbs(v[k], ev), wl[k]);
    return idot::finish(s, ev, ew);
}
#endif

// pout[m * P + b] = <V_m, F> over CTA b's range, m < meff (basis entries read
// exactly as binary64; products and tree in binary64).  The m CTA sums are
// formed together: every warp keeps its lane-tree sums in shared memory and
// one barrier later each sum is finished with the warp tree of chunk_sum.
template <class T>
__global__ void __launch_bounds__(RT) multidot_kernel(const double *__restrict__ F, const T *__restrict__ V,
                                                      size_t ldv, size_t n, double *__restrict__ pout, int P,
                                                      const StepState *st)
{
    const int m = st->meff;
    __shared__ double ws[kMaxKrylov][8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t e0 = lane_e0();
    double f[EPL];
    load8(F, e0, n, f);
    for (int g = 0; g < m; g += 16) {
        double t[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            t[q] = 0.0;
            if (g + q < m) {
                T v[EPL];
                load8(V + (size_t)(g + q) * ldv, e0, n, v);
                t[q] = lane_dot(v, f);
            }
        }
        const double s = lane_tree16(t, lane);
        const int q = lane_tree16_value(lane);
        if (lane < 16 && g + q < m) ws[g + q][wid] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += RT) pout[(size_t)i * P + blockIdx.x] = warp8_tree(ws[i]);
}

// ---- persistent Arnoldi column ------------------------------------------------

// One Arnoldi column in one cooperative launch.  T is the basis type: double
// (plain path) or float (mixed path: basis storage and Gram-Schmidt in binary32;
// the binary64 JVP result w is rounded to T on load; H is stored in binary64).
template <class T>
__global__ void __launch_bounds__(RT, 2) arnoldi_column_kernel(const double *__restrict__ w, T *__restrict__ V,
                                                               size_t ldv, size_t n, int j, int next, int P,
                                                               T *partA, T *partB, unsigned *cnt,
                                                               StepState *st, double brk_tol)
{
    static_assert(kColChunks == 2, "the CTA sums are formed for two chunks at once");
    __shared__ T sh[16];
    __shared__ int act;
    if (threadIdx.x == 0) act = st->active;
    __syncthreads();
    if (act == 0) return;
    const unsigned G = gridDim.x;
    T wv[kColChunks][EPL], vn[kColChunks][EPL];
    size_t e0[kColChunks];
    bool have[kColChunks];
#pragma unroll
    for (int c = 0; c < kColChunks; ++c) {
        const int b = blockIdx.x + c * G;
        have[c] = b < P;
        e0[c] = ((size_t)b * RT + threadIdx.x) * EPL;
        if (have[c]) {
            double wd[EPL];
            load8(w, e0[c], n, wd);
#pragma unroll
            for (int k = 0; k < EPL; ++k) wv[c][k] = (T)wd[k];
            load8(V, e0[c], n, vn[c]);     // v_0
            if (j >= 1) prefetch_l2(V + ldv, e0[c], n);   // v_1, read after the first wait
        }
    }
    // pass 0 partials: <v_0, w> and <w, w> (a missing second chunk sums zeros)
    {
        T x[kColChunks], y[kColChunks];
#pragma unroll
        for (int c = 0; c < kColChunks; ++c) {
            x[c] = have[c] ? lane_dot(vn[c], wv[c]) : T(0);
            y[c] = have[c] ? lane_dot(wv[c], wv[c]) : T(0);
        }
        T s0a, s0b, s1a, s1b;
        if (have[1]) {   // uniform per CTA
            chunk_sum2v(x[0], x[1], sh, s0a, s0b);
            chunk_sum2v(y[0], y[1], sh, s1a, s1b);
        } else {
            s0a = chunk_sumv(x[0], sh);
            s1a = chunk_sumv(y[0], sh);
        }
        if (threadIdx.x == 0) {
            partA[blockIdx.x] = s0a;
            partA[P + blockIdx.x] = s1a;
        }
        if (threadIdx.x == 8 && have[1]) {
            partA[blockIdx.x + G] = s0b;
            partA[P + blockIdx.x + G] = s1b;
        }
    }
    gen_arrive(cnt);
    T *pin = partA, *pout = partB;
    T wnorm0 = T(0);
    for (int i = 0; i <= j; ++i) {
        // generation i complete; the buffer written next (i + 1) was last read
        // for generation i - 1, which every CTA finished before its arrival at i
        if (!gen_wait(cnt + i, G, &st->status)) return;
        const T h = tree_partials(pin, P, sh);
        if (i == 0) wnorm0 = sqrt(tree_partials(pin + P, P, sh));
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->H[i * kMaxKrylov + j] = (double)h;
            if (i == 0) st->wnorm0 = (double)wnorm0;
        }
        const T *vnext = i < j ? V + (size_t)(i + 1) * ldv : nullptr;
        T x[kColChunks];
#pragma unroll
        for (int c = 0; c < kColChunks; ++c) {
            if (!have[c]) {   // uniform per CTA
                x[c] = T(0);
                continue;
            }
#pragma unroll
            for (int k = 0; k < EPL; ++k) wv[c][k] = wv[c][k] - h * vn[c][k];
            if (vnext) load8(vnext, e0[c], n, vn[c]);
            if (i + 2 <= j) prefetch_l2(V + (size_t)(i + 2) * ldv, e0[c], n);   // the next pass's vector
            x[c] = vnext ? lane_dot(vn[c], wv[c]) : lane_dot(wv[c], wv[c]);
        }
        T sa, sb;
        if (have[1]) chunk_sum2v(x[0], x[1], sh, sa, sb);
        else sa = chunk_sumv(x[0], sh);
        if (threadIdx.x == 0) pout[blockIdx.x] = sa;
        if (threadIdx.x == 8 && have[1]) pout[blockIdx.x + G] = sb;
        gen_arrive(cnt + i + 1);
        T *t = pin;
        pin = pout;
        pout = t;
    }
    if (!next) return;   // last column: the orthogonalised w is not needed further
    if (!gen_wait(cnt + j + 1, G, &st->status)) return;
    const T hn = sqrt(tree_partials(pin, P, sh));
    const bool brk = !((double)hn > brk_tol * (double)wnorm0);
    if (brk) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->active = 0;
            st->meff = j + 1;
        }
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) st->H[(j + 1) * kMaxKrylov + j] = (double)hn;
    const T r = T(1) / hn;
    T *vout = V + (size_t)(j + 1) * ldv;
#pragma unroll
    for (int c = 0; c < kColChunks; ++c) {
        if (!have[c]) continue;
        T x[EPL];
#pragma unroll
        for (int k = 0; k < EPL; ++k) x[k] = wv[c][k] * r;
        store8(vout, e0[c], n, x);
    }
}

#ifdef ROK_LINALG_FAST
// ---- mixed-precision Arnoldi column by classical Gram-Schmidt, twice (CGS2) -----
// The binary32 Gram-Schmidt of the mixed-precision form is cheap arithmetic but
// pays one grid-wide wait per modified-Gram-Schmidt pass (j + 2 per column).
// CGS2 forms all j + 1 projections of a pass at once: h1 = V^T w, w' = w - V h1,
// h2 = V^T w' (the second projection restores orthogonality to binary32
// rounding), ||w'||^2 in the same reduction, h_{j+1,j}^2 = ||w'||^2 - ||h2||^2
// (w'' = w' - V h2 is orthogonal to V), H[:, j] = h1 + h2, v_{j+1} = w'' / h.
// Two waits per column.  It spans the same Krylov space and equals MGS up to
// rounding (classical Gram-Schmidt twice is as stable as MGS here); the strict
// build keeps MGS, whose every rounding the oracle repeats.
constexpr int kCgsVals = kMaxKrylov + 1;   // j + 1 projections and one squared norm

// out[i * G + blockIdx.x] = the CTA's part of <v_i, w> for i <= j and of
// ||w||^2 for i = j + 1 (nv = j + 2 values).  Per slot the thread loads eight
// basis vectors at once (one L2 latency per eight vectors), forms their dots
// with its entries, and the values go 16 at a time through lane_tree16.
__device__ __forceinline__ void cgs_values(const float (&wv)[kColChunks][EPL], const bool (&have)[kColChunks],
                                           const size_t (&e0)[kColChunks], const float *__restrict__ V,
                                           size_t ldv, size_t n, int j, float (*ws)[8], float *out, unsigned G)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nv = j + 2;
    for (int g = 0; g < nv; g += 16) {
        float t[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) t[q] = 0.0f;
#pragma unroll
        for (int c = 0; c < kColChunks; ++c) {
            if (!have[c]) continue;
#pragma unroll
            for (int q0 = 0; q0 < 16; q0 += 8) {
                float v[8][EPL];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int i = g + q0 + q;
                    if (i <= j) {
                        load8(V + (size_t)i * ldv, e0[c], n, v[q]);
                    } else {
#pragma unroll
                        for (int k = 0; k < EPL; ++k) v[q][k] = i == j + 1 ? wv[c][k] : 0.0f;
                    }
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) t[q0 + q] += lane_dot(v[q], wv[c]);
            }
        }
        const float sum = lane_tree16(t, lane);
        const int q = lane_tree16_value(lane);
        if (lane < 16 && g + q < nv) ws[g + q][wid] = sum;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nv; i += RT) {
        const float *w8 = ws[i];
        out[(size_t)i * G + blockIdx.x] = ((w8[0] + w8[1]) + (w8[2] + w8[3])) + ((w8[4] + w8[5]) + (w8[6] + w8[7]));
    }
}

// hs[i] = sum over the G CTA partials of value i, i < nv (one warp per value;
// a lane issues all its loads of a value before adding: one L2 latency per
// value instead of one per load)
constexpr int kCgsMaxCtasPerLane = 32;   // G <= 1024
__device__ __forceinline__ void grid_values(int nv, const float *part, unsigned G, float *hs)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int i = wid; i < nv; i += RT / 32) {
        const float *p = part + (size_t)i * G;
        float x[kCgsMaxCtasPerLane];
#pragma unroll
        for (int q = 0; q < kCgsMaxCtasPerLane; ++q) {
            const unsigned b = lane + 32u * q;
            x[q] = b < G ? p[b] : 0.0f;
        }
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < kCgsMaxCtasPerLane; ++q) s += x[q];
        s = lane_tree(s);
        if (lane == 0) hs[i] = s;
    }
    __syncthreads();
}

// w -= sum_{i <= j} h[i] v_i over the thread's entries, four basis vectors at a
// time with their loads issued together
__device__ __forceinline__ void cgs_update(float (&wv)[kColChunks][EPL], const bool (&have)[kColChunks],
                                           const size_t (&e0)[kColChunks], const float *__restrict__ V, size_t ldv,
                                           size_t n, int j, const float *h)
{
#pragma unroll
    for (int c = 0; c < kColChunks; ++c) {
        if (!have[c]) continue;
        int i = 0;
        for (; i + 4 <= j + 1; i += 4) {
            float v[4][EPL];
#pragma unroll
            for (int q = 0; q < 4; ++q) load8(V + (size_t)(i + q) * ldv, e0[c], n, v[q]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float hq = h[i + q];
#pragma unroll
                for (int k = 0; k < EPL; ++k) wv[c][k] = wv[c][k] - hq * v[q][k];
            }
        }
        for (; i <= j; ++i) {
            float v[EPL];
            load8(V + (size_t)i * ldv, e0[c], n, v);
            const float hi = h[i];
#pragma unroll
            for (int k = 0; k < EPL; ++k) wv[c][k] = wv[c][k] - hi * v[k];
        }
    }
}

__global__ void __launch_bounds__(RT, 2) cgs2_column_kernel(const double *__restrict__ w, float *__restrict__ V,
                                                            size_t ldv, size_t n, int j, int next, int P,
                                                            float *part, unsigned *cnt, StepState *st,
                                                            double brk_tol)
{
    __shared__ float ws[kCgsVals][8];
    __shared__ float h1[kCgsVals], h2[kCgsVals];
    __shared__ int act;
    if (threadIdx.x == 0) act = st->active;
    __syncthreads();
    if (act == 0) return;
    const unsigned G = gridDim.x;
    float wv[kColChunks][EPL];
    size_t e0[kColChunks];
    bool have[kColChunks];
#pragma unroll
    for (int c = 0; c < kColChunks; ++c) {
        const int b = blockIdx.x + c * G;
        have[c] = b < P;
        e0[c] = ((size_t)b * RT + threadIdx.x) * EPL;
        if (have[c]) {
            double wd[EPL];
            load8(w, e0[c], n, wd);
#pragma unroll
            for (int k = 0; k < EPL; ++k) wv[c][k] = (float)wd[k];
        } else {
#pragma unroll
            for (int k = 0; k < EPL; ++k) wv[c][k] = 0.0f;
        }
    }
    const int nv = j + 2;
    float *partA = part, *partB = part + (size_t)kCgsVals * G;
    // first projection h1 = V^T w and ||w||^2
    cgs_values(wv, have, e0, V, ldv, n, j, ws, partA, G);
    gen_arrive(cnt);
    if (!gen_wait(cnt, G, &st->status)) return;
    grid_values(nv, partA, G, h1);
    const float wnorm0 = sqrt(h1[j + 1]);
    // w' = w - V h1, then h2 = V^T w' and ||w'||^2
    cgs_update(wv, have, e0, V, ldv, n, j, h1);
    __syncthreads();   // ws is reused
    cgs_values(wv, have, e0, V, ldv, n, j, ws, partB, G);
    gen_arrive(cnt + 1);
    if (!gen_wait(cnt + 1, G, &st->status)) return;
    grid_values(nv, partB, G, h2);
    float hn2 = h2[j + 1];
    for (int i = 0; i <= j; ++i) hn2 -= h2[i] * h2[i];
    const float hn = hn2 > 0.0f ? sqrt(hn2) : 0.0f;
    const bool brk = !((double)hn > brk_tol * (double)wnorm0);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        for (int i = 0; i <= j; ++i) st->H[i * kMaxKrylov + j] = (double)h1[i] + (double)h2[i];
        st->wnorm0 = (double)wnorm0;
        if (next) {
            if (brk) {
                st->active = 0;
                st->meff = j + 1;
            } else {
                st->H[(j + 1) * kMaxKrylov + j] = (double)hn;
            }
        }
    }
    if (!next || brk) return;
    // v_{j+1} = (w' - V h2) / h_{j+1,j}
    cgs_update(wv, have, e0, V, ldv, n, j, h2);
    const float r = 1.0f / hn;
    float *vout = V + (size_t)(j + 1) * ldv;
#pragma unroll
    for (int c = 0; c < kColChunks; ++c) {
        if (!have[c]) continue;
        float x[EPL];
#pragma unroll
        for (int k = 0; k < EPL; ++k) x[k] = wv[c][k] * r;
        store8(vout, e0[c], n, x);
    }
}

// ---- binary64 Arnoldi column, FMA build: even split, two basis vectors a pass ----
// The strict build's pairwise tree fixes 2048-entry chunks, and 512 of them
// (512^2) do not divide over 152 SMs: some SMs would hold 4, the others 3.
// The FMA build is free in its summation order, so this kernel gives CTA b the
// contiguous range [b L, (b + 1) L) of L = ceil(n / G) entries (at most
// kEvenPerThread per thread, strided by the CTA width so that loads stay
// coalesced) and one partial per CTA and value.
//
// Orthogonalisation (Sec. 2.3.3, Arnoldi; the modified Gram-Schmidt
// projections taken two basis vectors at a time).  For the pair (a, b) =
// (v_{2p}, v_{2p+1}) and the current w, one grid-wide reduction gives
// alpha = <a, w> and beta = <b, w>; then h_{2p} = alpha and
// h_{2p+1} = beta - g alpha with g = <b, a>, and w -= h_{2p} a + h_{2p+1} b.
// This is exactly the product (I - b b^T)(I - a a^T) w of the two MGS
// projections, for any a and b: the term g alpha is what the second
// projection sees of the first.  g is reduced once, when b is formed (its
// partials at the end of the column that made b, its sum in the next
// column's first reduction), and kept in StepState::gram.  So a pair costs
// the same 2 FMAs per entry and vector as two MGS passes but one grid-wide
// wait instead of two; the results agree with one-vector MGS to rounding (the
// two differ only in where the dot product of b is rounded).  The scale of
// the breakdown test, ||w|| before the projections, is taken as
// (sum_i h_ij^2 + h_{j+1,j}^2)^(1/2) (Pythagoras for the orthonormal basis)
// instead of a dot product of its own.
//
// One CTA of kEvenThreads threads per SM (the register file holds 512 threads
// of this kernel): one set of reductions and one arrival per SM and pass,
// each reduction spread over quads of four warps, one warp per SM
// sub-partition (a warp-wide FP64 instruction keeps a sub-partition's FP64
// unit busy for 64 cycles, so a reduction's latency is its dependent FP64
// instructions on the busiest sub-partition).  The next pair is staged into
// shared memory by two bulk copies (the CTA's contiguous ranges, completing
// on an mbarrier) while the current pair is in registers; the copy is issued
// after a CTA barrier has ordered every thread's reads of the buffer.
constexpr int kEvenThreads = 512;
constexpr int kEvenPerThread = 16;    // 8192 entries per CTA at most (E <= 16)
constexpr int kEvenMaxGrid = 256;     // grid sums: 4 warps, 2 partials a lane

template <int E>
constexpr size_t pair_stage_bytes() { return 2 * (size_t)E * kEvenThreads * sizeof(double); }

// named barrier ID of NT threads (immediate operands)
template <int ID, int NT>
__device__ __forceinline__ void bar_named()
{
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(NT) : "memory");
}

// bulk copies global -> shared completing on an mbarrier (one phase a stage)
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity)
{
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// bytes (a multiple of 16) from global src to shared dst, both 16-byte aligned
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, unsigned long long *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// the stage's reads of the buffer (generic proxy) before the bulk copy that overwrites it
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// bounded wait of every thread for the phase of the stage buffer; false after
// kStageSpins polls (the caller then gives up together, see pair_stage_wait)
constexpr long long kStageSpins = 1LL << 20;
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long *bar, unsigned parity)
{
    for (long long s = 0; s < kStageSpins; ++s)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// the first kmax terms (kmax uniform over the CTA: the slots no thread of the
// CTA holds are skipped, not multiplied by zero)
template <int E>
__device__ __forceinline__ double even_dot(const double (&a)[E], const double (&b)[E], int kmax)
{
    double s = a[0] * b[0];
#pragma unroll
    for (int k = 1; k < E; ++k)
        if (k < kmax) s = a[k] * b[k] + s;
    return s;
}

// this thread's entries of a range are base[k kEvenThreads], k < kv (a prefix
// of the k); slots kv <= k < kmax hold zeros
template <int E>
__device__ __forceinline__ void even_load(double (&x)[E], const double *__restrict__ base, int kv, int kmax)
{
#pragma unroll
    for (int k = 0; k < E; ++k)
        if (k < kmax) x[k] = k < kv ? base[k * kEvenThreads] : 0.0;
}

// Stage the CTA's ranges of a (and b, if not null), cnt entries each, into
// sa (sb) by bulk copies completing on bar; by one thread, after the CTA's
// reads of the previous contents (a barrier) and the proxy fence.  The slots
// past cnt keep the zeros written at the start.
__device__ __forceinline__ void pair_stage_issue(double *sa, double *sb, const double *a, const double *b, size_t cnt,
                                                 unsigned long long *bar)
{
    const unsigned bytes = (unsigned)(cnt * sizeof(double));
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, b ? 2 * bytes : bytes);
    if (bytes) {
        bulk_g2s(sa, a, bytes, bar);
        if (b) bulk_g2s(sb, b, bytes, bar);
    }
}

template <int E>
__device__ __forceinline__ void pair_unstage(double (&x)[E], const double *s, int kmax)
{
#pragma unroll
    for (int k = 0; k < E; ++k)
        if (k < kmax) x[k] = s[k * kEvenThreads + threadIdx.x];
}

// CTA sums of the nsum arrays s + q kEvenThreads by quads q < nsum (warps
// 4q .. 4q + 3): warp k of a quad adds 128 consecutive values, four a lane,
// then the lane butterfly, into sh4[4q + k]; then a barrier of the quads.
// quad_total gives a sum from its four warp sums.
template <int nsum>
__device__ __forceinline__ void quads_cta(const double *s, double *sh4)
{
    const int q = threadIdx.x >> 7;
    if (q < nsum) {
        const int k = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
        const double *v = s + q * kEvenThreads + k * 128 + lane * 4;
        const double a = lane_tree((v[0] + v[1]) + (v[2] + v[3]));
        if (lane == 0) sh4[4 * q + k] = a;
        bar_named<1, 128 * nsum>();
    }
}

__device__ __forceinline__ double quad_total(const double *sh4, int q)
{
    return (sh4[4 * q] + sh4[4 * q + 1]) + (sh4[4 * q + 2] + sh4[4 * q + 3]);
}

// Wait (thread 0, bounded) until generation counter *cnt reaches G, then the
// grid sums of the nsum partial arrays p + q G (G <= kEvenMaxGrid) by quads
// q < nsum: warp k of a quad adds the k-th quarter (two partials a lane, then
// the butterfly) into sh4[4q + k].  Every CTA forms the same sums in the same
// order.  After it, thread 0 reads the sums with quad_total.  False (status
// set) on timeout, in every thread of the quads (the others learn it from
// the caller's barrier).
template <int nsum>
__device__ __forceinline__ bool pair_wait(const unsigned *cnt, unsigned G, int *status, const double *p, double *sh4,
                                          int *ok)
{
    const int q = threadIdx.x >> 7;
    if (q < nsum) {
        if (threadIdx.x == 0) {
            int good = 1;
            long long spins = 0;
            while (ld_acquire_gpu(cnt) < G) {
                if (++spins > kBarrierSpins) {
                    atomicOr(status, kStatusTimeout);
                    good = 0;
                    break;
                }
                __nanosleep(32);
            }
            *ok = good;
        }
        bar_named<2, 128 * nsum>();
        if (!*ok) return false;
        const int k = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
        const int Q = ((int)G + 3) >> 2;
        const int b0 = k * Q + lane, e = min((int)G, (k + 1) * Q);
        const double *pq = p + (size_t)q * G;
        const double x0 = b0 < e ? pq[b0] : 0.0;
        const double x1 = b0 + 32 < e ? pq[b0 + 32] : 0.0;
        const double a = lane_tree(x0 + x1);
        if (lane == 0) sh4[4 * q + k] = a;
        bar_named<1, 128 * nsum>();
    }
    return true;
}
// Two sums in one warp butterfly: lanes < 16 keep a and send b to lane ^ 16,
// lanes >= 16 the reverse, so after one exchange the low half carries a and
// the high half b, each summed over two lanes; four more levels finish both.
// Lane 0 ends with the warp sum of a, lane 16 with that of b (one FP64
// instruction a level for both sums).
__device__ __forceinline__ double lane_tree2(double a, double b)
{
    const bool low = (threadIdx.x & 16) == 0;
    double v = (low ? a : b) + __shfl_xor_sync(0xffffffffu, low ? b : a, 16);
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The CTA sums of s[0 .. T) and s[T .. 2T) together by quad 0: warp k adds
// the values of threads 128 k .. 128 k + 127 of both arrays (four a lane,
// then lane_tree2) into sh4[k] and sh4[4 + k]; then the quad's barrier.
__device__ __forceinline__ void quad0_cta2(const double *s, double *sh4)
{
    if (threadIdx.x < 128) {
        const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const double *u = s + k * 128 + lane * 4, *v = u + kEvenThreads;
        const double x = lane_tree2((u[0] + u[1]) + (u[2] + u[3]), (v[0] + v[1]) + (v[2] + v[3]));
        if (lane == 0) sh4[k] = x;
        if (lane == 16) sh4[4 + k] = x;
        bar_named<1, 128>();
    }
}

// pair_wait for the two partial arrays p and p + G, both by quad 0 (warp k:
// the k-th quarter of each, two partials a lane, then lane_tree2).
__device__ __forceinline__ bool pair_wait2(const unsigned *cnt, unsigned G, int *status, const double *p,
                                           double *sh4, int *ok)
{
    if (threadIdx.x < 128) {
        if (threadIdx.x == 0) {
            int good = 1;
            long long spins = 0;
            while (ld_acquire_gpu(cnt) < G) {
                if (++spins > kBarrierSpins) {
                    atomicOr(status, kStatusTimeout);
                    good = 0;
                    break;
                }
                __nanosleep(32);
            }
            *ok = good;
        }
        bar_named<2, 128>();
        if (!*ok) return false;
        const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int Q = ((int)G + 3) >> 2;
        const int b0 = k * Q + lane, e = min((int)G, (k + 1) * Q);
        const double *pb = p + G;
        const double a = (b0 < e ? p[b0] : 0.0) + (b0 + 32 < e ? p[b0 + 32] : 0.0);
        const double b = (b0 < e ? pb[b0] : 0.0) + (b0 + 32 < e ? pb[b0 + 32] : 0.0);
        const double x = lane_tree2(a, b);
        if (lane == 0) sh4[k] = x;
        if (lane == 16) sh4[4 + k] = x;
        bar_named<1, 128>();
    }
    return true;
}

// In warp 0, lane q (q < 4) forms total q from sh4[4q .. 4q + 4): all the
// totals of a pass in one set of three FP64 instructions.
__device__ __forceinline__ double warp0_totals(const double *sh4) { return quad_total(sh4, threadIdx.x & 3); }

template <int E>
__global__ void __launch_bounds__(kEvenThreads, 1)
    arnoldi_pair_kernel(const double *__restrict__ w, double *__restrict__ V, size_t ldv, size_t n, int j, int next,
                        size_t L, double *partA, double *partB, unsigned *cnt, StepState *st, double brk_tol)
{
    constexpr int T = kEvenThreads;
    extern __shared__ __align__(16) double stage_buf[];   // 2 E T: the staged pair
    double *sa = stage_buf, *sb = stage_buf + E * T;
    __shared__ double sred[4 * T];
    __shared__ double sh4[16];
    __shared__ double sh[2];
    __shared__ double sgram[kMaxKrylov];
    __shared__ __align__(8) unsigned long long stage_bar;   // one phase per staged pair
    __shared__ int act, ok, brk;
    if (threadIdx.x == 0) {
        act = st->active;
        mbar_init(&stage_bar);
    }
    if (threadIdx.x + 1 < (unsigned)j) sgram[threadIdx.x] = st->gram[threadIdx.x];   // <v_{i+1}, v_i>, i < j - 1
    __syncthreads();
    if (act == 0) return;
    const unsigned G = gridDim.x;
    const size_t lo = (size_t)blockIdx.x * L;
    const size_t hi = lo + L < n ? lo + L : n;
    const size_t my = lo + threadIdx.x;   // this thread's first entry
    const int kv = my < hi ? (int)((hi - my + T - 1) / T) : 0;
    const int kmax = (int)((hi - lo + T - 1) / T);   // uniform over the CTA
    const int P = (j + 2) >> 1;   // passes: pairs (v_{2p}, v_{2p+1}); the last is v_j alone when j is even
    double *gpart = partA + 2 * (size_t)G;   // partials of <v_{j+1}, v_j> for the next column
#pragma unroll
    for (int k = 0; k < E; ++k)
        if (k >= kv && k < kmax) sa[k * T + threadIdx.x] = sb[k * T + threadIdx.x] = 0.0;
    double wv[E], va[E], vb[E];
    even_load(wv, w + my, kv, kmax);
    even_load(va, V + my, kv, kmax);   // v_0
    if (j >= 1) even_load(vb, V + ldv + my, kv, kmax);   // v_1
    if (P >= 2 && threadIdx.x == 0)   // pair 1 (the zeros above lie past its bytes)
        pair_stage_issue(sa, sb, V + 2 * ldv + lo, j >= 3 ? V + 3 * ldv + lo : nullptr, hi - lo, &stage_bar);
    // first partials: <v_0, w> and (j >= 1) <v_1, w>
    sred[threadIdx.x] = even_dot(va, wv, kmax);
    if (j >= 1) sred[T + threadIdx.x] = even_dot(vb, wv, kmax);
    __syncthreads();
    if (j >= 1) quad0_cta2(sred, sh4);
    else quads_cta<1>(sred, sh4);
    if (threadIdx.x < 32) {
        const double t = warp0_totals(sh4);
        const double t1 = __shfl_sync(0xffffffffu, t, 1);
        if (threadIdx.x == 0) {
            partA[blockIdx.x] = t;
            if (j >= 1) partA[G + blockIdx.x] = t1;
            red_add_release_gpu(cnt, 1u);   // the same thread stored the partials
        }
    }
    double *pin = partA, *pout = partB;
    // warp 0: sum of the squares of the column's projections so far; with the
    // final h_{j+1,j}^2 it is ||w||^2 of the JVP result for an orthonormal
    // basis (Pythagoras), the scale of the breakdown test
    double ssq = 0.0, gfresh = 0.0;
    for (int p = 0; p < P; ++p) {
        const bool pair = 2 * p + 1 <= j;
        bool good;
        if (p == 0)   // with j >= 1 also <v_j, v_{j-1}> from the previous column's partials
            good = j >= 1 ? pair_wait<3>(cnt, G, &st->status, pin, sh4, &ok)
                          : pair_wait<1>(cnt, G, &st->status, pin, sh4, &ok);
        else
            good = pair ? pair_wait2(cnt + p, G, &st->status, pin, sh4, &ok)
                        : pair_wait<1>(cnt + p, G, &st->status, pin, sh4, &ok);
        if (threadIdx.x < 32 && good) {   // warp 0: the totals in lanes 0 .. 3 at once
            const double t = warp0_totals(sh4);
            const double alpha = __shfl_sync(0xffffffffu, t, 0), beta = __shfl_sync(0xffffffffu, t, 1);
            if (p == 0) gfresh = __shfl_sync(0xffffffffu, t, 2);
            double h1 = 0.0;
            if (pair) {
                const double g = 2 * p + 1 == j ? gfresh : sgram[2 * p];
                h1 = fma(-g, alpha, beta);
            }
            ssq = fma(alpha, alpha, ssq);
            if (pair) ssq = fma(h1, h1, ssq);
            if (threadIdx.x == 0) {
                sh[0] = alpha;
                sh[1] = h1;
            }
            if (threadIdx.x == 0 && blockIdx.x == 0) {
                st->H[2 * p * kMaxKrylov + j] = alpha;
                if (pair) st->H[(2 * p + 1) * kMaxKrylov + j] = h1;
                if (p == 0 && j >= 1) st->gram[j - 1] = gfresh;
            }
        }
        __syncthreads();
        if (!ok) {
            if (p + 1 < P) mbar_wait_bounded(&stage_bar, p & 1);   // the staged pair in flight
            return;
        }
        const double h0 = sh[0], h1 = sh[1];
        if (pair) {
#pragma unroll
            for (int k = 0; k < E; ++k)
                if (k < kmax) wv[k] = wv[k] - h0 * va[k] - h1 * vb[k];
        } else {
#pragma unroll
            for (int k = 0; k < E; ++k)
                if (k < kmax) wv[k] = wv[k] - h0 * va[k];
        }
        if (p + 1 < P) {
            const bool npair = 2 * p + 3 <= j;
            const bool late = !mbar_wait_bounded(&stage_bar, p & 1);   // pair p + 1 staged
            pair_unstage(va, sa, kmax);
            if (npair) pair_unstage(vb, sb, kmax);
            sred[threadIdx.x] = even_dot(va, wv, kmax);
            if (npair) sred[T + threadIdx.x] = even_dot(vb, wv, kmax);
            if (__syncthreads_or(late)) {   // every thread gives up together
                if (threadIdx.x == 0) atomicOr(&st->status, kStatusTimeout);
                mbar_wait_bounded(&stage_bar, p & 1);
                return;
            }
            if (p + 2 < P && threadIdx.x == 0)   // the buffer is read: stage pair p + 2
                pair_stage_issue(sa, sb, V + (size_t)(2 * p + 4) * ldv + lo,
                                 2 * p + 5 <= j ? V + (size_t)(2 * p + 5) * ldv + lo : nullptr, hi - lo,
                                 &stage_bar);
            if (npair) quad0_cta2(sred, sh4);
            else quads_cta<1>(sred, sh4);
            if (threadIdx.x < 32) {
                const double t = warp0_totals(sh4);
                const double tb = __shfl_sync(0xffffffffu, t, 1);
                if (threadIdx.x == 0) {
                    pout[blockIdx.x] = t;
                    if (npair) pout[G + blockIdx.x] = tb;
                    red_add_release_gpu(cnt + p + 1, 1u);
                }
            }
        } else {
            sred[threadIdx.x] = even_dot(wv, wv, kmax);
            __syncthreads();
            quads_cta<1>(sred, sh4);
            if (threadIdx.x == 0) {
                pout[blockIdx.x] = quad_total(sh4, 0);
                red_add_release_gpu(cnt + p + 1, 1u);
            }
        }
        double *t = pin;
        pin = pout;
        pout = t;
    }
    if (!next) return;
    const bool good = pair_wait<1>(cnt + P, G, &st->status, pin, sh4, &ok);
    // the norm, the breakdown test and the reciprocal by thread 0 (in every warp
    // they would cost each sub-partition): the test on the squares and one reciprocal
    // square root, a chain of half a dozen FP64 instructions where two square roots
    // and a division were some sixty (0.5 us a column)
    double hn2 = 0.0;
    if (threadIdx.x == 0 && good) {
        hn2 = quad_total(sh4, 0);
        brk = !(hn2 > (brk_tol * brk_tol) * (ssq + hn2));
        sh[0] = rsqrt(hn2);
    }
    __syncthreads();
    if (threadIdx.x == 0 && blockIdx.x == 0 && ok) {
        st->wnorm0 = sqrt(ssq + hn2);   // ||J v_j||
        if (brk) {
            st->active = 0;
            st->meff = j + 1;
        } else {
            const double hn = hn2 * sh[0];   // and one Newton step: the rounding of the square root
            st->H[(j + 1) * kMaxKrylov + j] = fma(fma(-hn, hn, hn2), 0.5 * sh[0], hn);
        }
    }
    if (!ok || brk) return;
    const double r = sh[0];
    // v_{j+1}, and the partials of <v_{j+1}, v_j> (v_j: the last vector used)
    const bool last_pair = (j & 1) != 0;
    double *vout = V + (size_t)(j + 1) * ldv + my;
    double g = 0.0;
#pragma unroll
    for (int k = 0; k < E; ++k)
        if (k < kmax) {
            const double x = wv[k] * r;
            if (k < kv) vout[k * T] = x;
            g = x * (last_pair ? vb[k] : va[k]) + g;
        }
    sred[threadIdx.x] = g;
    __syncthreads();
    quads_cta<1>(sred, sh4);
    if (threadIdx.x == 0) gpart[blockIdx.x] = quad_total(sh4, 0);   // read by the next launch
}

// ---- projections <V_i, F>, FMA build: the entries split evenly ------------------
// The chunked multidot gives the 2048-entry chunks to 512 CTAs, so on 152 SMs
// some SMs hold 4 chunks and the others 3; the FP64 work (m FMAs per entry)
// runs at the pace of the 4-chunk SMs.  Here CTA b of G = one per SM owns the
// contiguous range [b L, (b + 1) L), each thread E slots strided by the CTA
// width, and the m values of a group are summed across the lanes by recursive
// halving sized to the group (R = 16, 8 or 4 values: R - 1 + 5 - log2 R
// additions a lane, not 16 for every group).  The partials keep the layout of
// the chunked kernel, pout[i P + b], with zeros for G <= b < P, so the stage
// solve reads them unchanged.

// lane sums of R values at once (R = 16, 8, 4): LV halving levels, then the
// plain butterfly; lane l ends with the sum of value lane_treeR_value<R>(l)
template <int R>
__device__ __forceinline__ double lane_treeR(double (&t)[16], int lane)
{
    constexpr int LV = R == 16 ? 4 : R == 8 ? 3 : 2;
#pragma unroll
    for (int lev = 0; lev < LV; ++lev) {
        const int half = (R / 2) >> lev;
        const bool upper = (lane >> lev) & 1;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const double recv = __shfl_xor_sync(0xffffffffu, upper ? t[k] : t[k + half], 1 << lev);
            t[k] = upper ? recv + t[k + half] : t[k] + recv;
        }
    }
    double v = t[0];
#pragma unroll
    for (int o = 1 << LV; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int R>
__device__ __forceinline__ int lane_treeR_value(int lane)
{
    constexpr int LV = R == 16 ? 4 : R == 8 ? 3 : 2;
    int v = 0;
#pragma unroll
    for (int lev = 0; lev < LV; ++lev)
        if ((lane >> lev) & 1) v += (R / 2) >> lev;
    return v;
}

template <int R>
__device__ __forceinline__ void multidot_group(double (&t)[16], int g, int m, double (*ws)[kEvenThreads / 32])
{
    const int lane = threadIdx.x & 31;
    const double s = lane_treeR<R>(t, lane);
    const int q = lane_treeR_value<R>(lane);
    if (lane < R && g + q < m) ws[g + q][threadIdx.x >> 5] = s;
}

// four consecutive binary64 values (one 32-byte load; p 32-byte aligned)
struct Quad {
    double x, y, z, w;
};
__device__ __forceinline__ Quad ld_quad(const double *p)
{
    Quad q;
    asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(q.x), "=d"(q.y), "=d"(q.z), "=d"(q.w) : "l"(p));
    return q;
}
// binary32 to binary64 on the integer pipe: the conversion instruction runs at
// the FP64 rate (2 lanes per SM and clock) and cost as much as the product it
// feeds.  A normal number's exponent is rebiased by 896 and its fraction moved up
// by 29 bits; zeros keep their sign; subnormals, infinities and NaN take the
// instruction (out of line: a predicated conversion would be issued for all).
// 512^2, 20 vectors: projections 97 -> 66 us, stage vectors 83 -> 43 us a launch.
__device__ __noinline__ double widen_special(float x) { return (double)x; }
__device__ __forceinline__ double widen(float x)
{
    const unsigned b = __float_as_uint(x);
    const unsigned m = b & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u && m != 0u) return widen_special(x);
    const unsigned hi = (b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
    return __hiloint2double((int)hi, (int)(b << 29));
}

// four consecutive binary32 basis values (one 16-byte load), exactly as binary64
__device__ __forceinline__ Quad ld_quad(const float *p)
{
    const float4 f = __ldg(reinterpret_cast<const float4 *>(p));
    return Quad{widen(f.x), widen(f.y), widen(f.z), widen(f.w)};
}

template <int E, class T>
__global__ void __launch_bounds__(kEvenThreads, 1)
    multidot_even_kernel(const double *__restrict__ F, const T *__restrict__ V, size_t ldv, size_t n, size_t L,
                         double *__restrict__ pout, int P, const StepState *st)
{
    // quads of consecutive entries (32-byte loads of binary64, 16-byte of a
    // binary32 basis): thread t holds quads t + k TH, k < E / 4
    constexpr int TH = kEvenThreads, NW = kEvenThreads / 32, E4 = E / 4;
    static_assert(NW == 16, "the CTA sum below adds 16 warp sums");
    __shared__ double ws[kMaxKrylov][NW];
    const int m = st->meff;
    const size_t lo = (size_t)blockIdx.x * L;
    const size_t hi = lo + L < n ? lo + L : n;
    const size_t nq = (hi - lo) / 4;   // quads of this CTA (L, n multiples of 4)
    const int kv = threadIdx.x < nq ? (int)((nq - threadIdx.x + TH - 1) / TH) : 0;
    const double *F4 = F + lo + 4 * (size_t)threadIdx.x;
    if ((threadIdx.x & ~31u) >= nq) {   // a warp without entries: its share is zero (see pair_kernel)
        for (int i = threadIdx.x & 31; i < m; i += 32) ws[i][threadIdx.x >> 5] = 0.0;
    }
    Quad f[E4];
#pragma unroll
    for (int k = 0; k < E4; ++k) f[k] = k < kv ? ld_quad(F4 + (size_t)4 * k * TH) : Quad{0.0, 0.0, 0.0, 0.0};
    for (int g = 0; g < m && (threadIdx.x & ~31u) < nq; g += 16) {
        const int cnt = m - g < 16 ? m - g : 16;   // uniform
        double t[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            double s = 0.0;
            if (q < cnt) {
                const T *v = V + (size_t)(g + q) * ldv + lo + 4 * (size_t)threadIdx.x;
#pragma unroll
                for (int k = 0; k < E4; ++k)
                    if (k < kv) {
                        const Quad x = ld_quad(v + (size_t)4 * k * TH);
                        s = x.x * f[k].x + s;
                        s = x.y * f[k].y + s;
                        s = x.z * f[k].z + s;
                        s = x.w * f[k].w + s;
                    }
            }
            t[q] = s;
        }
        if (cnt > 8) multidot_group<16>(t, g, m, ws);
        else if (cnt > 4) multidot_group<8>(t, g, m, ws);
        else multidot_group<4>(t, g, m, ws);
    }
    __syncthreads();
    if (threadIdx.x < m) {
        const double *w = ws[threadIdx.x];
        const double s = (((w[0] + w[1]) + (w[2] + w[3])) + ((w[4] + w[5]) + (w[6] + w[7]))) +
                         (((w[8] + w[9]) + (w[10] + w[11])) + ((w[12] + w[13]) + (w[14] + w[15])));
        pout[(size_t)threadIdx.x * P + blockIdx.x] = s;
    }
    if (blockIdx.x == 0)   // the chunk slots past the grid
        for (int i = threadIdx.x; i < m * (P - (int)gridDim.x); i += TH)
            pout[(size_t)(i / (P - (int)gridDim.x)) * P + gridDim.x + i % (P - (int)gridDim.x)] = 0.0;
}

// The same for longer ranges: the CTA's range in tiles of E entries a thread, the
// lanes' sums of a group of vectors kept over the tiles and reduced once (the
// chunked kernel adds a lane tree of 16 FP64 instructions to every 128
// multiply-adds).  F is read once a group.  1024^2, 20 vectors: 196 -> 161 us a launch
// (HBM 104, FP64 140).
template <int E>
__global__ void __launch_bounds__(kEvenThreads, 1)
    multidot_long_kernel(const double *__restrict__ F, const double *__restrict__ V, size_t ldv, size_t n, size_t L,
                         double *__restrict__ pout, int P, const StepState *st)
{
    constexpr int TH = kEvenThreads, NW = kEvenThreads / 32, E4 = E / 4;
    static_assert(NW == 16, "the CTA sum below adds 16 warp sums");
    __shared__ double ws[kMaxKrylov][NW];
    const int m = st->meff;
    const size_t lo = (size_t)blockIdx.x * L;
    const size_t hi = lo + L < n ? lo + L : n;
    const size_t nq = (hi - lo) / 4;   // quads of this CTA (L, n multiples of 4)
    for (int g = 0; g < m; g += 16) {
        const int cnt = m - g < 16 ? m - g : 16;   // uniform
        double t[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) t[q] = 0.0;
        for (size_t q0 = threadIdx.x; q0 < nq; q0 += (size_t)E4 * TH) {
            Quad f[E4];
#pragma unroll
            for (int k = 0; k < E4; ++k)
                f[k] = q0 + (size_t)k * TH < nq ? ld_quad(F + lo + 4 * (q0 + (size_t)k * TH)) : Quad{0.0, 0.0, 0.0, 0.0};
#pragma unroll
            for (int q = 0; q < 16; ++q)
                if (q < cnt) {
                    const double *v = V + (size_t)(g + q) * ldv + lo;
                    double s = t[q];
#pragma unroll
                    for (int k = 0; k < E4; ++k)
                        if (q0 + (size_t)k * TH < nq) {
                            const Quad x = ld_quad(v + 4 * (q0 + (size_t)k * TH));
                            s = x.x * f[k].x + s;
                            s = x.y * f[k].y + s;
                            s = x.z * f[k].z + s;
                            s = x.w * f[k].w + s;
                        }
                    t[q] = s;
                }
        }
        if (cnt > 8) multidot_group<16>(t, g, m, ws);
        else if (cnt > 4) multidot_group<8>(t, g, m, ws);
        else multidot_group<4>(t, g, m, ws);
    }
    __syncthreads();
    if (threadIdx.x < m) {
        const double *w = ws[threadIdx.x];
        const double s = (((w[0] + w[1]) + (w[2] + w[3])) + ((w[4] + w[5]) + (w[6] + w[7]))) +
                         (((w[8] + w[9]) + (w[10] + w[11])) + ((w[12] + w[13]) + (w[14] + w[15])));
        pout[(size_t)threadIdx.x * P + blockIdx.x] = s;
    }
    if (blockIdx.x == 0)   // the chunk slots past the grid
        for (int i = threadIdx.x; i < m * (P - (int)gridDim.x); i += TH)
            pout[(size_t)(i / (P - (int)gridDim.x)) * P + gridDim.x + i % (P - (int)gridDim.x)] = 0.0;
}

// ---- stage vectors k = sum_i c_i V_i + h F, FMA build: quads of entries ---------
// Each thread forms four consecutive entries (32-byte loads, four independent
// FMA chains in the basis order of stage_vec_kernel, so the same values), one
// quad per thread and no grid-stride remainder.
__device__ __forceinline__ void st_quad(double *p, const Quad &q)
{
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(q.x), "d"(q.y), "d"(q.z), "d"(q.w)
                 : "memory");
}

template <class T>
__global__ void __launch_bounds__(RT) stage_vec_quad_kernel(double *__restrict__ k, const double *__restrict__ F,
                                                            const T *__restrict__ V, size_t ldv, size_t nq,
                                                            int stage, const StepState *st)
{
    __shared__ double c[kMaxKrylov];
    const int m = st->meff;
    const double h = st->h;
    for (int i = threadIdx.x; i < m; i += blockDim.x) c[i] = st->cvec[stage][i];
    __syncthreads();
    const size_t q = (size_t)blockIdx.x * RT + threadIdx.x;
    if (q >= nq) return;
    Quad a{0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int i = 0; i < m; ++i) {
        const Quad v = ld_quad(V + (size_t)i * ldv + 4 * q);
        const double ci = c[i];
        a.x = a.x + ci * v.x;
        a.y = a.y + ci * v.y;
        a.z = a.z + ci * v.z;
        a.w = a.w + ci * v.w;
    }
    const Quad f = ld_quad(F + 4 * q);
    st_quad(k + 4 * q, Quad{a.x + h * f.x, a.y + h * f.y, a.z + h * f.z, a.w + h * f.w});
}

// ---- Gram-Schmidt by block passes (grids beyond the column kernel, batches) -----
// One vector a pass moves 32 B an entry (w in and out, the vector to subtract,
// the next one to project on) and ends with a grid-wide sum.  Four vectors a
// pass move 80 B per four (20 B a vector): for the block (v_{4b}, .., v_{4b+3})
// one pass gives alpha_q = <v_{4b+q}, w>, the coefficients are
// h_q = alpha_q - sum_{p<q} <v_q, v_p> h_p (forward substitution with the block's
// Gram entries: the product of the four modified Gram-Schmidt projections, as
// in the pairs of arnoldi_pair_kernel), and the next pass subtracts them while
// it projects on the next block.  A vector's Gram entries are formed in the pass
// that first projects on it (its own column), from values already in registers.
// The sums are finished by the CTA that arrives last, in a fixed order.
// Measured, 1024^2 (4.2 M entries): 60 us a pass of four vectors (FP64 9
// instructions an entry, 73 % busy), 56 us a pass of one before; the Gram-Schmidt
// of a ROK4 step with M = 20 there 13.2 -> 5.1 ms, of the batch of 64 20 -> 13 ms.
constexpr int kGsCtas = 3;   // CTAs per SM of the single-grid pass
struct GsPass {
    int j;        // column
    int b, nb;    // block to subtract, its vectors (0: none, the column's first pass)
    int b2, nn;   // block to project on, its vectors (0: form ||w||^2 instead)
    int next;     // another column follows: normalise
    __device__ __forceinline__ bool fresh() const { return nn > 1 && 4 * b2 + nn - 1 == j; }   // v_j's Gram entries too
};

__device__ __forceinline__ void gs_zero(double (&t)[16])
{
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = 0.0;
}

// one lane's 8 entries: t[q] += <v_q, w>, t[4 + q] += <v_q, v_j> (fresh), or t[0] += <w, w>.
// INT: <v_q, w> on the integer pipe (batches: the passes of the batch of 64
// 13.1 -> 12.0 ms; the single grid's, 59 us either way at 1024^2, is held by memory)
template <bool INT>
__device__ __forceinline__ void gs_lane(double *__restrict__ w, const double *__restrict__ V, size_t ldv, size_t e0,
                                        size_t n, const GsPass &ps, const StepState *st, double (&t)[16])
{
    double wv[EPL];
    load8(w, e0, n, wv);
    if (ps.nb > 0) {
        const double *vb = V + (size_t)(4 * ps.b) * ldv;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q < ps.nb) {
                double v[EPL];
                load8(vb + (size_t)q * ldv, e0, n, v);
                const double h = st->gs_h[q];
#pragma unroll
                for (int k = 0; k < EPL; ++k) wv[k] = wv[k] - h * v[k];
            }
        }
        store8(w, e0, n, wv);
    }
    if (ps.nn == 0) {
        t[0] += lane_dot(wv, wv);
        return;
    }
    const double *vn = V + (size_t)(4 * ps.b2) * ldv;
    idot::Limb wl[EPL];
    int ew = 0;
    if (INT) ew = lane_limbs(wv, wl);
    auto dot = [&](const double (&v)[EPL]) { return INT ? lane_idot(v, wl, ew, w, e0, n) : lane_dot(v, wv); };
    if (ps.fresh()) {
        double vj[EPL];
        load8(V + (size_t)ps.j * ldv, e0, n, vj);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q < ps.nn - 1) {
                double v[EPL];
                load8(vn + (size_t)q * ldv, e0, n, v);
                t[q] += dot(v);
                t[4 + q] += lane_dot(v, vj);
            } else if (q == ps.nn - 1) {
                t[q] += dot(vj);
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q < ps.nn) {
                double v[EPL];
                load8(vn + (size_t)q * ldv, e0, n, v);
                t[q] += dot(v);
            }
        }
    }
}

// the block's coefficients (or the norm) from its eight sums, by one thread
__device__ __forceinline__ void gs_finish(const GsPass &ps, const double (*tot)[8], StepState *st)
{
    if (ps.nn == 0) {
        if (!ps.next) return;
        // the norm and its reciprocal as the column kernel forms them
        const double hn2 = tot[0][0], rh = rsqrt(hn2), h0 = hn2 * rh, hn = fma(fma(-h0, h0, hn2), 0.5 * rh, h0);
        const double wnorm0 = sqrt(st->gs_ssq + hn2);   // ||J v_j|| (Pythagoras for the orthonormal basis)
        st->wnorm0 = wnorm0;
        if (!(hn > 1e-12 * wnorm0)) {
            st->active = 0;
            st->meff = ps.j + 1;
        } else {
            st->H[(ps.j + 1) * kMaxKrylov + ps.j] = hn;
            st->gs_rh = rh;
        }
        return;
    }
    if (ps.fresh())
        for (int q = 0; q < ps.nn - 1; ++q) st->bgram[ps.j][q] = tot[4 + q][0];
    double ssq = ps.nb == 0 ? 0.0 : st->gs_ssq;
    double h[4];
    for (int q = 0; q < ps.nn; ++q) {
        double a = tot[q][0];
        for (int k = 0; k < q; ++k) a = fma(-st->bgram[4 * ps.b2 + q][k], h[k], a);
        h[q] = a;
        ssq = fma(a, a, ssq);
        st->gs_h[q] = a;
        st->H[(4 * ps.b2 + q) * kMaxKrylov + ps.j] = a;
    }
    st->gs_ssq = ssq;
}

// The CTA's eight sums into part[q stride + id], q < 8; the last of the P
// arrivals adds them up (warp q the q-th: lanes stride over the partials, then
// the butterfly) and finishes the block.  ws: the warps' sums; flag: shared.
__device__ __forceinline__ void gs_reduce(double (&t)[16], const GsPass &ps, double *__restrict__ part, size_t stride,
                                          int id, int P, StepState *st, double (*ws)[8], int *flag)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nv = ps.nn == 0 ? 1 : (ps.fresh() ? 8 : 4);
    const double s = lane_treeR<8>(t, lane);
    const int q = lane_treeR_value<8>(lane);
    __syncthreads();
    if (lane < 8) ws[q][wid] = s;
    __syncthreads();
    if (threadIdx.x < nv) {
        __stcg(part + threadIdx.x * stride + id, warp8_tree(ws[threadIdx.x]));
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned before = atomicAdd(&st->gs_count, 1u);
        *flag = before + 1 == (unsigned)P;
        if (*flag) st->gs_count = 0;
        __threadfence();
    }
    __syncthreads();
    if (!*flag) return;
    if (wid < nv) {
        const double *p = part + wid * stride;
        double a = 0.0, b = 0.0;
        for (int i = lane; i < P; i += 64) {
            a += __ldcg(p + i);
            if (i + 32 < P) b += __ldcg(p + i + 32);
        }
        a = lane_tree(a + b);
        if (lane == 0) ws[wid][0] = a;
    }
    __syncthreads();
    if (threadIdx.x == 0) gs_finish(ps, ws, st);
}

// one grid: CTA b takes chunks b, b + G, ... and adds up its lanes' sums over them
__global__ void __launch_bounds__(RT) gs_pass_kernel(double *__restrict__ w, const double *__restrict__ V, size_t ldv,
                                                     size_t n, const GsPass ps, double *__restrict__ part, StepState *st)
{
    __shared__ double ws[8][8];
    __shared__ int flag;
    if (threadIdx.x == 0) flag = st->active;
    __syncthreads();
    if (flag == 0) return;
    double t[16];
    gs_zero(t);
    for (size_t c = blockIdx.x; c * RB < n; c += gridDim.x)
        gs_lane<false>(w, V, ldv, (c * RT + threadIdx.x) * EPL, n, ps, st, t);
    gs_reduce(t, ps, part, gridDim.x, blockIdx.x, gridDim.x, st, ws, &flag);
}

__global__ void __launch_bounds__(RT) gs_normalize_kernel(const double *__restrict__ w, double *__restrict__ v,
                                                          size_t n, const StepState *st)
{
    if (st->active == 0) return;
    const double rh = st->gs_rh;
    const size_t e0 = lane_e0();
    double x[EPL];
    load8(w, e0, n, x);
#pragma unroll
    for (int k = 0; k < EPL; ++k) x[k] = x[k] * rh;
    store8(v, e0, n, x);
}

static cudaError_t gs_column(double *w, double *V, size_t ldv, size_t n, int j, int next, double *part, StepState *st,
                             long long *launches, cudaStream_t s)
{
    const int chunks = reduction_blocks(n);
    const int sms = sm_count();
    if (sms <= 0) return cudaErrorUnknown;
    const int G = chunks < kGsCtas * sms ? chunks : kGsCtas * sms;
    const int blocks = (j + 4) / 4;
    for (int b = -1; b < blocks; ++b) {
        GsPass ps;
        ps.j = j;
        ps.b = b < 0 ? 0 : b;
        ps.nb = b < 0 ? 0 : (j + 1 - 4 * b < 4 ? j + 1 - 4 * b : 4);
        ps.b2 = b + 1;
        ps.nn = b + 1 < blocks ? (j + 1 - 4 * ps.b2 < 4 ? j + 1 - 4 * ps.b2 : 4) : 0;
        ps.next = next;
        gs_pass_kernel<<<G, RT, 0, s>>>(w, V, ldv, n, ps, part, st);
        ++*launches;
    }
    if (next) {
        gs_normalize_kernel<<<chunks, RT, 0, s>>>(w, V + (size_t)(j + 1) * ldv, n, st);
        ++*launches;
    }
    return cudaGetLastError();
}
#endif  // ROK_LINALG_FAST

// First basis vector: partials of ||(T)F1||^2 ...
template <class T>
__global__ void __launch_bounds__(RT) first_partials_kernel(const double *__restrict__ F, size_t n, T *partials)
{
    __shared__ T sh[10];
    const size_t e0 = lane_e0();
    double fd[EPL];
    load8(F, e0, n, fd);
    T x[EPL];
#pragma unroll
    for (int k = 0; k < EPL; ++k) {
        T t = (T)fd[k];
        x[k] = t * t;
    }
    T s = chunk_sum(x, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

// ... then beta = sqrt(tree), v_1 = (T)F1 * (1/beta); beta = 0 leaves an empty basis
template <class T>
__global__ void __launch_bounds__(RT) first_normalize_kernel(const double *__restrict__ F, T *__restrict__ V0,
                                                             size_t n, const T *partials, int P, StepState *st)
{
    __shared__ T sh[10];
    __shared__ int act;
    if (threadIdx.x == 0) act = st->active;
    __syncthreads();
    if (act == 0) return;
    const T beta = sqrt(tree_partials(partials, P, sh));
    if (!(beta > T(0))) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->active = 0;
            st->meff = 0;
        }
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) st->beta = (double)beta;
    const T r = T(1) / beta;
    const size_t e0 = lane_e0();
    double fd[EPL];
    load8(F, e0, n, fd);
    T x[EPL];
#pragma unroll
    for (int k = 0; k < EPL; ++k) x[k] = (T)fd[k] * r;
    store8(V0, e0, n, x);
}

#ifdef ROK_LINALG_FAST
// The instantiation of arnoldi_pair_kernel for e entries a thread: the smallest
// that holds them.  An FP64 instruction whose lanes are all predicated off still
// occupies the unit, so a loose fit costs as much as the entries it could hold
// (64 x 64 cells, 4 entries of 8: 6.8 us a pass, as 7 of 8 on 256 x 512).
struct PairKernel {
    int E;
    const void *fn;
    size_t smem;
};
template <int E>
PairKernel pair_kernel_of()
{
    return {E, (const void *)arnoldi_pair_kernel<E>, pair_stage_bytes<E>()};
}
static PairKernel pair_kernel(int e)
{
    if (e <= 1) return pair_kernel_of<1>();
    if (e <= 2) return pair_kernel_of<2>();
    if (e <= 3) return pair_kernel_of<3>();
    if (e <= 4) return pair_kernel_of<4>();
    if (e <= 5) return pair_kernel_of<5>();
    if (e <= 6) return pair_kernel_of<6>();
    if (e <= 7) return pair_kernel_of<7>();
    if (e <= 8) return pair_kernel_of<8>();
    if (e <= 10) return pair_kernel_of<10>();
    if (e <= 12) return pair_kernel_of<12>();
    if (e <= 14) return pair_kernel_of<14>();
    return pair_kernel_of<16>();
}
#endif

static int arnoldi_column_ctas(int sms)
{
    int dev = 0, coop = 0, p64 = 0, p32 = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p64, arnoldi_column_kernel<double>, RT, 0) != cudaSuccess)
        return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p32, arnoldi_column_kernel<float>, RT, 0) != cudaSuccess)
        return 0;
#ifdef ROK_LINALG_FAST
    int pc = 0, pe = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pc, cgs2_column_kernel, RT, 0) != cudaSuccess) return 0;
    if (pc < p32) p32 = pc;
    // the binary64 column runs as arnoldi_pair_kernel, kEvenThreads threads a CTA
    // and a dynamic staging buffer: its grid is ctas RT / kEvenThreads, which must
    // be co-resident too
    for (int E = 1; E <= kEvenPerThread; ++E) {
        const PairKernel k = pair_kernel(E);
        if (k.E != E) continue;
        if (cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem) != cudaSuccess) return 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pe, k.fn, kEvenThreads, k.smem) != cudaSuccess) return 0;
        if (pe * kEvenThreads < p64 * RT) p64 = pe * kEvenThreads / RT;
    }
#endif
    return (p64 < p32 ? p64 : p32) * sms;
}

static cudaError_t arnoldi_column(const double *w, void *V, int fp32, size_t ldv, size_t n, int j, int next, int P,
                                  double *partA, double *partB, unsigned *cnt, StepState *st, int ctas,
                                  cudaStream_t s)
{
    if (ctas <= 0) return cudaErrorNotSupported;
    const int G = P < ctas ? P : ctas;
    if ((P + G - 1) / G > kColChunks) return cudaErrorNotSupported;
    if (fp32) {
        float *Vf = static_cast<float *>(V);
        float *pa = reinterpret_cast<float *>(partA), *pb = reinterpret_cast<float *>(partB);
        double tol = 1e-5;
#ifdef ROK_LINALG_FAST
        // CGS2: partA holds 2 (kMaxKrylov + 1) G binary32 partials
        (void)pb;
        if (G > 32 * kCgsMaxCtasPerLane) return cudaErrorNotSupported;
        void *cargs[] = {&w, &Vf, &ldv, &n, &j, &next, &P, &pa, &cnt, &st, &tol};
        return cudaLaunchCooperativeKernel((const void *)cgs2_column_kernel, dim3(G), dim3(RT), cargs, 0, s);
#else
        void *args[] = {&w, &Vf, &ldv, &n, &j, &next, &P, &pa, &pb, &cnt, &st, &tol};
        return cudaLaunchCooperativeKernel((const void *)arnoldi_column_kernel<float>, dim3(G), dim3(RT), args, 0, s);
#endif
    }
    double *Vd = static_cast<double *>(V);
    double tol = 1e-12;
#ifdef ROK_LINALG_FAST
    // even split: Ge CTAs of kEvenThreads threads and L entries each; down to one
    // entry a thread, so that small vectors take many SMs, every CTA with at least
    // one entry.  16k entries (64 x 64 cells), 12 columns: 8 CTAs of 4 entries a
    // thread 352 us, 32 of 1 218 us; the projections 18 -> 6 us a launch
    const int Gmax = min(ctas * RT / kEvenThreads, kEvenMaxGrid);
    const size_t want = (n + kEvenThreads - 1) / kEvenThreads;
    int Ge = want < (size_t)Gmax ? (int)want : Gmax;
    auto range = [&] {
        const size_t l = (n + Ge - 1) / Ge;
        return l + (l & 1);
    };
    while (Ge > 1 && (size_t)(Ge - 1) * range() >= n) --Ge;
    size_t L = Ge > 0 ? range() : 0;
    if (Ge < 1 || L > (size_t)kEvenThreads * kEvenPerThread || Ge > kEvenMaxGrid) return cudaErrorNotSupported;
    // the bulk copies of the CTA ranges want 16-byte aligned starts and lengths
    if ((n & 1) || (ldv & 1) || ((uintptr_t)Vd & 15)) return cudaErrorNotSupported;
    double *partP = partA + 4 * (size_t)Ge;   // partA: the even passes' two sums and the next column's Gram partials
    void *eargs[] = {&w, &Vd, &ldv, &n, &j, &next, &L, &partA, &partP, &cnt, &st, &tol};
    const PairKernel k = pair_kernel((int)((L + kEvenThreads - 1) / kEvenThreads));
    return cudaLaunchCooperativeKernel(k.fn, dim3(Ge), dim3(kEvenThreads), eargs, k.smem, s);
#else
    void *args[] = {&w, &Vd, &ldv, &n, &j, &next, &P, &partA, &partB, &cnt, &st, &tol};
    return cudaLaunchCooperativeKernel((const void *)arnoldi_column_kernel<double>, dim3(G), dim3(RT), args, 0, s);
#endif
}

static cudaError_t first_vector(const double *F, void *V0, int fp32, size_t n, double *partials, int P,
                                StepState *st, cudaStream_t s)
{
    if (fp32) {
        float *pf = reinterpret_cast<float *>(partials);
        first_partials_kernel<float><<<P, RT, 0, s>>>(F, n, pf);
        first_normalize_kernel<float><<<P, RT, 0, s>>>(F, static_cast<float *>(V0), n, pf, P, st);
    } else {
        first_partials_kernel<double><<<P, RT, 0, s>>>(F, n, partials);
        first_normalize_kernel<double><<<P, RT, 0, s>>>(F, static_cast<double *>(V0), n, partials, P, st);
    }
    return cudaGetLastError();
}

constexpr int kLuThreads = 128;      // threads of the LU launch
constexpr int kSolveThreads = 1024;  // threads of the stage-solve launch (one warp per projection)

// |x| as an integer that orders like it, -1 for NaN: comparisons on the integer
// pipe (an FP64 instruction of one warp occupies its sub-partition's FP64 unit for 64
// cycles, and five butterfly levels of the pivot search compared twice each)
__device__ __forceinline__ long long magnitude_key(double x)
{
    const long long b = __double_as_longlong(x) & 0x7fffffffffffffffll;
    return b > 0x7ff0000000000000ll ? -1 : b;
}

#ifdef ROK_LINALG_FAST
// 1/x for |x| in [2^-991, 2^992): the hardware estimate and one third-order Newton step
__device__ __forceinline__ bool reciprocal_range(double x) { return ((unsigned)__double2hiint(x) >> 20 & 0x7ffu) - 32u <= 1982u; }
__device__ __forceinline__ double reciprocal(double x)
{
    double r0;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r0) : "d"(x));
    const double d = fma(-x, r0, 1.0);
    return fma(r0, fma(d, d, d), r0);
}
// a / d with rd = reciprocal(d): the product corrected by its remainder, which rounds as
// the division does
__device__ __forceinline__ double quotient(double a, double d, double rd)
{
    const double q = a * rd;
    return fma(fma(-q, d, a), rd, q);
}
#endif

// LU with partial pivoting of L = I - h g H (first largest |pivot|), row-major
// stride kMaxKrylov, by the whole CTA: warp 0 searches the pivot, then the row
// multipliers and the trailing update are spread over the threads.  Each entry
// sees the same operation sequence as a sequential elimination (one multiplier
// division per row, one update per step), so the strict build's factors are those
// of the plain loops.
// Bound by the latency of FP64 instructions (64 cycles each on one warp): integer
// comparisons in the pivot search and, in the FMA build, one reciprocal a step and three
// instructions a row instead of a division (42 -> 23 us at m = 20, 67 -> 37 us at m = 30),
// which pivots outside the reciprocal's range keep.
__device__ __forceinline__ void lu_body(StepState *st)
{
    // the factorisation runs in shared memory; the factors and the pivots are
    // written back at the end
    __shared__ double A[kMaxKrylov * kMaxKrylov];
    __shared__ int piv[kMaxKrylov];
    __shared__ int failed, pk;
    const int m = st->meff;
    const double hg = st->hg;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    if (tid == 0) failed = 0;
    for (int idx = tid; idx < m * m; idx += nt) {
        int i = idx / m, j = idx % m;
        A[i * kMaxKrylov + j] = (i == j ? 1.0 : 0.0) - hg * st->H[i * kMaxKrylov + j];
    }
    __syncthreads();
    for (int k = 0; k < m; ++k) {
        if (tid < 32) {
            long long best = -1;
            int bi = k;
            for (int i = k + lane; i < m; i += 32) {
                const long long a = magnitude_key(A[i * kMaxKrylov + k]);
                if (a > best) { best = a; bi = i; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
                int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (lane == 0) {
                piv[k] = bi;
                pk = bi;
            }
        }
        __syncthreads();
        const int bi = pk;
        if (bi != k)
            for (int j = tid; j < m; j += nt) {
                double t = A[k * kMaxKrylov + j];
                A[k * kMaxKrylov + j] = A[bi * kMaxKrylov + j];
                A[bi * kMaxKrylov + j] = t;
            }
        __syncthreads();
        const double d = A[k * kMaxKrylov + k];
        const long long dk = magnitude_key(d);
        if (dk <= 0 || dk == 0x7ff0000000000000ll) {   // zero, infinite or NaN; the same value in every thread
            if (tid == 0) {
                st->status |= kStatusSingular;
                failed = 1;
            }
            break;
        }
#ifdef ROK_LINALG_FAST
        if (reciprocal_range(d)) {
            const double rd = reciprocal(d);
            for (int i = k + 1 + tid; i < m; i += nt) A[i * kMaxKrylov + k] = quotient(A[i * kMaxKrylov + k], d, rd);
        } else
#endif
            for (int i = k + 1 + tid; i < m; i += nt) A[i * kMaxKrylov + k] = A[i * kMaxKrylov + k] / d;
        __syncthreads();
        const int w = m - k - 1;
        for (int idx = tid; idx < w * w; idx += nt) {
            const int i = k + 1 + idx / w, j = k + 1 + idx % w;
            A[i * kMaxKrylov + j] = A[i * kMaxKrylov + j] - A[i * kMaxKrylov + k] * A[k * kMaxKrylov + j];
        }
        __syncthreads();
    }
    __syncthreads();
    if (failed) return;
    for (int idx = tid; idx < m * m; idx += nt) {
        int i = idx / m, j = idx % m;
        st->LU[i * kMaxKrylov + j] = A[i * kMaxKrylov + j];
    }
    for (int k = tid; k < m; k += nt) st->piv[k] = piv[k];
}

__global__ void __launch_bounds__(kLuThreads) lu_kernel(StepState *st) { lu_body(st); }

struct GamRow {
    double g[4];
};

// stage i: phi = V^T F_i (tree of the CTA partials), rhs = h phi + h H acc with
// acc = sum_{j<i} gamma_ij lambda_j, lambda_i = LU solve, cvec_i = lambda_i - h phi.
// The partials of <V_i, F> are pin[i * istride + (0 .. P)].
__device__ __forceinline__ void stage_solve_body(int stage, const GamRow &gr, const double *pin, size_t istride,
                                                 int P, StepState *st)
{
    const int m = st->meff;
    const double h = st->h;
    __shared__ double phi[kMaxKrylov], acc[kMaxKrylov], x[kMaxKrylov];
    __shared__ double A[kMaxKrylov * kMaxKrylov];
    __shared__ int piv[kMaxKrylov];
    for (int i = threadIdx.x >> 5; i < m; i += blockDim.x >> 5) {
        double v = warp_tree_partials(pin + (size_t)i * istride, P);
        if ((threadIdx.x & 31) == 0) phi[i] = v;
    }
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double a = 0.0;
        for (int j = 0; j < stage; ++j) a = a + gr.g[j] * st->lam[j][i];
        acc[i] = a;
        piv[i] = st->piv[i];
    }
    // H beside the factors where both fit, so that its rows are not read from L2 one
    // entry after another (with the solve below, m = 12: 8.4 -> 6.8 us; m = 20 at 512^2: 19.8 -> 16.6)
    constexpr int HS = 32;
    __shared__ double Hs[HS * (HS + 1)];
    const bool small = m <= HS;
    for (int idx = threadIdx.x; idx < m * m; idx += blockDim.x) {
        int i = idx / m, j = idx % m;
        A[i * kMaxKrylov + j] = st->LU[i * kMaxKrylov + j];
        if (small) Hs[i * (HS + 1) + j] = st->H[i * kMaxKrylov + j];
    }
    __syncthreads();
    // rhs_i = h phi_i + h (H acc)_i, one row per thread, columns in order
    const double *Hm = small ? Hs : st->H;
    const int hstride = small ? HS + 1 : kMaxKrylov;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double t = 0.0;
        if (stage > 0)
            for (int j = 0; j < m; ++j) t = t + Hm[i * hstride + j] * acc[j];
        x[i] = h * phi[i] + h * t;
    }
    __syncthreads();
#ifdef ROK_LINALG_FAST
    // FMA build: warp 0 solves column by column, lane l holding rows l and l + 32
    // (other summation order than the row loops below)
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        if (lane == 0)
            for (int k = 0; k < m; ++k) {
                int p = piv[k];
                if (p != k) { double t = x[k]; x[k] = x[p]; x[p] = t; }
            }
        __syncwarp();
        const int i0 = lane, i1 = lane + 32;
        double r0 = i0 < m ? x[i0] : 0.0, r1 = i1 < m ? x[i1] : 0.0;
        if (small) {   // no rows beyond 32 (an FP64 instruction costs the same with no lane in it)
            for (int j = 0; j + 1 < m; ++j) {   // unit lower factor
                const double xj = __shfl_sync(0xffffffffu, r0, j);
                if (i0 > j && i0 < m) r0 = r0 - A[i0 * kMaxKrylov + j] * xj;
            }
            const double d0 = i0 < m ? 1.0 / A[i0 * kMaxKrylov + i0] : 0.0;
            for (int j = m - 1; j >= 0; --j) {   // upper factor
                if (i0 == j) r0 = r0 * d0;
                const double xj = __shfl_sync(0xffffffffu, r0, j);
                if (i0 < j) r0 = r0 - A[i0 * kMaxKrylov + j] * xj;
            }
        } else {
            for (int j = 0; j + 1 < m; ++j) {   // unit lower factor
                const double xj = __shfl_sync(0xffffffffu, j < 32 ? r0 : r1, j & 31);
                if (i0 > j && i0 < m) r0 = r0 - A[i0 * kMaxKrylov + j] * xj;
                if (i1 > j && i1 < m) r1 = r1 - A[i1 * kMaxKrylov + j] * xj;
            }
            const double d0 = i0 < m ? 1.0 / A[i0 * kMaxKrylov + i0] : 0.0;
            const double d1 = i1 < m ? 1.0 / A[i1 * kMaxKrylov + i1] : 0.0;
            for (int j = m - 1; j >= 0; --j) {   // upper factor
                if (i0 == j) r0 = r0 * d0;
                if (i1 == j) r1 = r1 * d1;
                const double xj = __shfl_sync(0xffffffffu, j < 32 ? r0 : r1, j & 31);
                if (i0 < j) r0 = r0 - A[i0 * kMaxKrylov + j] * xj;
                if (i1 < j) r1 = r1 - A[i1 * kMaxKrylov + j] * xj;
            }
        }
        if (i0 < m) x[i0] = r0;
        if (i1 < m) x[i1] = r1;
    }
#else
    if (threadIdx.x == 0) {
        for (int k = 0; k < m; ++k) {
            int p = piv[k];
            if (p != k) { double t = x[k]; x[k] = x[p]; x[p] = t; }
        }
        for (int i = 0; i < m; ++i) {
            double t = x[i];
            for (int j = 0; j < i; ++j) t = t - A[i * kMaxKrylov + j] * x[j];
            x[i] = t;
        }
        for (int i = m - 1; i >= 0; --i) {
            double t = x[i];
            for (int j = i + 1; j < m; ++j) t = t - A[i * kMaxKrylov + j] * x[j];
            x[i] = t / A[i * kMaxKrylov + i];
        }
    }
#endif
    __syncthreads();
    int bad = 0;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        st->lam[stage][i] = x[i];
        st->cvec[stage][i] = x[i] - h * phi[i];
        st->phi[i] = phi[i];
        st->phis[stage][i] = phi[i];
        bad |= !isfinite(x[i]);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) st->status |= kStatusNonfinite;
}

__global__ void __launch_bounds__(kSolveThreads) stage_solve_kernel(int stage, GamRow gr, const double *pin, int P, StepState *st)
{
    stage_solve_body(stage, gr, pin, (size_t)P, P, st);
}

// k = sum_{i<meff} cvec[stage][i] V_i + h F (basis order, binary64)
template <class T>
__global__ void __launch_bounds__(RT) stage_vec_kernel(double *__restrict__ k, const double *__restrict__ F,
                                                       const T *__restrict__ V, size_t ldv, size_t n, int stage,
                                                       const StepState *st)
{
    __shared__ double c[kMaxKrylov];
    const int m = st->meff;
    const double h = st->h;
    for (int i = threadIdx.x; i < m; i += blockDim.x) c[i] = st->cvec[stage][i];
    __syncthreads();
    for (size_t e = (size_t)blockIdx.x * RT + threadIdx.x; e < n; e += (size_t)gridDim.x * RT) {
        double a = 0.0;
        for (int i = 0; i < m; ++i) a = a + c[i] * (double)V[(size_t)i * ldv + e];
        k[e] = a + h * F[e];
    }
}

struct AxpyArgs {
    const double *v[8];
    double c[8];
};

// out = base + sum_q c_q v_q in order; skipped when a guard status is latched
__global__ void __launch_bounds__(RT) axpy_n_kernel(double *out, const double *base, AxpyArgs a, int count,
                                                    size_t n, const StepState *guard)
{
    if (guard && guard->status != 0) return;
    for (size_t e = (size_t)blockIdx.x * RT + threadIdx.x; e < n; e += (size_t)gridDim.x * RT) {
        double t = base ? base[e] : 0.0;
        for (int q = 0; q < count; ++q) t = t + a.c[q] * a.v[q][e];
        out[e] = t;
    }
}

__global__ void __launch_bounds__(RT) basis_combine_kernel(double *out, const double *base, const double *V,
                                                           size_t ldv, size_t n, int count, const double *gcoef,
                                                           const int *count_dev)
{
    __shared__ double c[kMaxKrylov + 1];
    if (count_dev && *count_dev < count) count = *count_dev;
    for (int i = threadIdx.x; i < count; i += blockDim.x) c[i] = gcoef[i];
    __syncthreads();
    for (size_t e = (size_t)blockIdx.x * RT + threadIdx.x; e < n; e += (size_t)gridDim.x * RT) {
        double a = 0.0;
        for (int i = 0; i < count; ++i) a = a + c[i] * V[(size_t)i * ldv + e];
        out[e] = base[e] + a;
    }
}

// eps = sqrt(u (1 + ||y||)) / ||v|| rounded to the nearest power of two (or as given)
__global__ void eps_kernel(const double *pin, int P, int v_unit, double eps_given, StepState *st)
{
    __shared__ double sh[10];
    const double yn = sqrt(tree_partials(pin, P, sh));
    const double vn = v_unit ? 1.0 : sqrt(tree_partials(pin + P, P, sh));
    if (threadIdx.x == 0) {
        double eps = eps_given;
        if (!(eps > 0.0)) {
            double x = sqrt(2.220446049250313e-16 * (1.0 + yn)) / vn;
            int e2;
            double mant = frexp(x, &e2);
            if (mant < sqrt(0.5)) e2 -= 1;
            eps = ldexp(1.0, e2);
        }
        st->eps = eps;
        st->inv_eps = 1.0 / eps;
        st->ynorm = yn;
    }
}

__global__ void sum_sqrt_kernel(const double *pin, int P, double *dst)
{
    __shared__ double sh[10];
    double s = tree_partials(pin, P, sh);
    if (threadIdx.x == 0) *dst = sqrt(s);
}

// ---- restarted GMRES(m) on the device (stage solves of the comparators) ----------
// The Arnoldi columns of a cycle are the Gram-Schmidt column kernels above
// applied to w = (I - h g J) v_j; these small kernels keep the least-squares
// problem min ||beta e_1 - H y|| (Givens rotations, as in Saad & Schultz) and the
// stop decision on the device, so the host reads the state once per cycle.

__global__ void __launch_bounds__(RT) gmres_start_kernel(const double *pin, int P, double tol, int m, StepState *st)
{
    __shared__ double sh[10];
    const double bn = sqrt(tree_partials(pin, P, sh));
    if (threadIdx.x == 0) {
        GmresState &g = st->gm;
        g.bnorm = bn;
        g.tol_abs = tol * bn;
        g.res = bn;
        g.m = m;
        g.k = 0;
        g.its = 0;
        g.live = 0;
        g.conv = bn == 0.0 ? 1 : 0;
        st->active = 0;
    }
}

__global__ void __launch_bounds__(RT) gmres_cycle_kernel(const double *pin, int P, StepState *st)
{
    __shared__ double sh[10];
    const double beta = sqrt(tree_partials(pin, P, sh));
    if (threadIdx.x == 0) {
        GmresState &g = st->gm;
        g.k = 0;
        if (g.conv || beta <= g.tol_abs) {
            g.conv = 1;
            g.live = 0;
            st->active = 0;
        } else {
            g.live = 1;
            g.res = beta;
            st->active = 1;
            g.g[0] = beta;
            for (int i = 1; i <= g.m; ++i) g.g[i] = 0.0;
            for (int j = 0; j < g.m; ++j) st->H[(j + 1) * kMaxKrylov + j] = 0.0;
        }
    }
}

// one thread: the rotations of column j (their count is the restart length at most)
__global__ void gmres_givens_kernel(int j, StepState *st)
{
    GmresState &g = st->gm;
    if (!g.live) return;
    const bool brk = st->active == 0;   // the Arnoldi column stopped at a breakdown
    double *H = st->H;
    constexpr int L = kMaxKrylov;
    for (int i = 0; i < j; ++i) {
        const double a = H[i * L + j], b = H[(i + 1) * L + j];
        H[i * L + j] = g.cs[i] * a + g.sn[i] * b;
        H[(i + 1) * L + j] = -g.sn[i] * a + g.cs[i] * b;
    }
    const double a = H[j * L + j], b = brk ? 0.0 : H[(j + 1) * L + j];
    const double r = hypot(a, b);
    const double cs = r > 0.0 ? a / r : 1.0, sn = r > 0.0 ? b / r : 0.0;
    g.cs[j] = cs;
    g.sn[j] = sn;
    H[j * L + j] = r;
    g.g[j + 1] = -sn * g.g[j];
    g.g[j] = cs * g.g[j];
    g.its += 1;
    g.k = j + 1;
    g.res = fabs(g.g[j + 1]);
    if (g.res <= g.tol_abs || brk) {
        g.conv = 1;
        g.live = 0;
        st->active = 0;
    } else if (j + 1 >= g.m) {
        g.live = 0;
        st->active = 0;
    }
}

// one thread: R y = g[0 .. k) by back substitution (R the rotated upper triangle of H)
__global__ void gmres_lsq_kernel(StepState *st)
{
    const GmresState &g = st->gm;
    constexpr int L = kMaxKrylov;
    const int k = g.k;
    for (int i = k - 1; i >= 0; --i) {
        double t = g.g[i];
        for (int q = i + 1; q < k; ++q) t -= st->H[i * L + q] * st->gcoef[q];
        st->gcoef[i] = t / st->H[i * L + i];
    }
}

// ---- batches of independent instances --------------------------------------------
// A flat batch vector is a sequence of 2048-entry chunks; chunk c belongs to
// instance k = chunk_inst[c] and covers entries inst[k].off + (c - chunk0) 2048
// + [0, 2048) of it, bounded by the instance length.  A CTA handles chunks
// blockIdx.x, blockIdx.x + gridDim.x, ... (the chunks-per-CTA setting only
// changes the grid); partials are stored per chunk, so instance k's partials
// are part[chunk0 .. chunk0 + P_k) and its sums are the same trees as for a
// single instance.  Instances whose Arnoldi flag is clear are skipped chunk by
// chunk (the skip is uniform within the CTA).

struct ChunkRef {
    int k;            // instance
    size_t off, n;    // instance's first entry and length
    size_t e0;        // this lane's first entry within the instance
    int chunk0, P;    // instance's first chunk and chunk count
};

__device__ __forceinline__ ChunkRef chunk_ref(const BSeg &sg, int c)
{
    ChunkRef r;
    r.k = sg.chunk_inst[c];
    const BatchInst &I = sg.inst[r.k];
    r.off = I.off;
    r.n = I.n;
    r.chunk0 = I.chunk0;
    r.P = I.nchunks;
    r.e0 = ((size_t)(c - r.chunk0) * RT + threadIdx.x) * EPL;
    return r;
}

// instance flag read once per CTA and chunk (uniform branch)
__device__ __forceinline__ bool chunk_active(const StepState *st, int *sh_flag)
{
    __syncthreads();
    if (threadIdx.x == 0) *sh_flag = st->active;
    __syncthreads();
    return *sh_flag != 0;
}

// part[c] = <a0, b0>, part[nchunks + c] = <a1, b1> (a1 nullable) over chunk c
__global__ void __launch_bounds__(RT) bdot2_kernel(const double *__restrict__ a0, const double *__restrict__ b0,
                                                   const double *__restrict__ a1, const double *__restrict__ b1,
                                                   double *__restrict__ part, const BSeg sg, int use_active)
{
    __shared__ double sh[10];
    __shared__ int flag;
    for (int c = blockIdx.x; c < sg.nchunks; c += gridDim.x) {
        const ChunkRef r = chunk_ref(sg, c);
        if (use_active && !chunk_active(sg.st + r.k, &flag)) continue;
        double x[EPL], y[EPL];
        load8(a0 + r.off, r.e0, r.n, x);
        load8(b0 + r.off, r.e0, r.n, y);
#pragma unroll
        for (int k = 0; k < EPL; ++k) x[k] = x[k] * y[k];
        double s0 = chunk_sum(x, sh);
        double s1 = 0.0;
        if (a1) {
            load8(a1 + r.off, r.e0, r.n, x);
            load8(b1 + r.off, r.e0, r.n, y);
#pragma unroll
            for (int k = 0; k < EPL; ++k) x[k] = x[k] * y[k];
            s1 = chunk_sum(x, sh);
        }
        if (threadIdx.x == 0) {
            part[c] = s0;
            part[sg.nchunks + c] = s1;
        }
    }
}

// one CTA per instance: eps = sqrt(u (1 + ||y||)) rounded to a power of two (unit v)
__global__ void beps_kernel(const double *part, const BSeg sg)
{
    __shared__ double sh[10];
    const BatchInst &I = sg.inst[blockIdx.x];
    StepState *st = sg.st + blockIdx.x;
    const double yn = sqrt(tree_partials(part + I.chunk0, I.nchunks, sh));
    if (threadIdx.x == 0) {
        double x = sqrt(2.220446049250313e-16 * (1.0 + yn)) / 1.0;
        int e2;
        double mant = frexp(x, &e2);
        if (mant < sqrt(0.5)) e2 -= 1;
        const double eps = ldexp(1.0, e2);
        st->eps = eps;
        st->inv_eps = 1.0 / eps;
        st->ynorm = yn;
    }
}

// v_1 = F1 * (1/beta), beta = sqrt(tree(part)); beta = 0 leaves an empty basis
__global__ void __launch_bounds__(RT) bfirst_normalize_kernel(const double *__restrict__ F, double *__restrict__ V0,
                                                              const double *part, const BSeg sg)
{
    __shared__ double sh[10];
    __shared__ int flag;
    for (int c = blockIdx.x; c < sg.nchunks; c += gridDim.x) {
        const ChunkRef r = chunk_ref(sg, c);
        StepState *st = sg.st + r.k;
        if (!chunk_active(st, &flag)) continue;
        const double beta = sqrt(tree_partials(part + r.chunk0, r.P, sh));
        if (!(beta > 0.0)) {
            if (c == r.chunk0 && threadIdx.x == 0) {
                st->active = 0;
                st->meff = 0;
            }
            continue;
        }
        if (c == r.chunk0 && threadIdx.x == 0) st->beta = beta;
        const double rb = 1.0 / beta;
        double x[EPL];
        load8(F + r.off, r.e0, r.n, x);
#pragma unroll
        for (int k = 0; k < EPL; ++k) x[k] = x[k] * rb;
        store8(V0 + r.off, r.e0, r.n, x);
    }
}

#ifndef ROK_LINALG_FAST
// MGS pass i of column j: h = tree(pin); H[i-1][j] = h; w -= h V_{i-1};
// pout[c] = <V_i, w> (i <= j) or <w, w> (i = j + 1); first pass also
// wnorm0 = sqrt(tree(pin + nchunks))
__global__ void __launch_bounds__(RT) bmgs_kernel(double *__restrict__ w, const double *__restrict__ V, size_t ldv,
                                                  int i, int j, const double *__restrict__ pin,
                                                  double *__restrict__ pout, const BSeg sg)
{
    __shared__ double sh[10];
    __shared__ int flag;
    const double *vprev = V + (size_t)(i - 1) * ldv;
    const double *vnext = i <= j ? V + (size_t)i * ldv : nullptr;
    for (int c = blockIdx.x; c < sg.nchunks; c += gridDim.x) {
        const ChunkRef r = chunk_ref(sg, c);
        StepState *st = sg.st + r.k;
        if (!chunk_active(st, &flag)) continue;
        double wv[EPL], vp[EPL], vn[EPL];
        load8(w + r.off, r.e0, r.n, wv);
        load8(vprev + r.off, r.e0, r.n, vp);
        if (vnext) load8(vnext + r.off, r.e0, r.n, vn);
        const double h = tree_partials(pin + r.chunk0, r.P, sh);
        if (i == 1) {
            const double wn2 = tree_partials(pin + sg.nchunks + r.chunk0, r.P, sh);
            if (c == r.chunk0 && threadIdx.x == 0) st->wnorm0 = sqrt(wn2);
        }
        if (c == r.chunk0 && threadIdx.x == 0) st->H[(i - 1) * kMaxKrylov + j] = h;
#pragma unroll
        for (int k = 0; k < EPL; ++k) wv[k] = wv[k] - h * vp[k];
        store8(w + r.off, r.e0, r.n, wv);
        const double s = chunk_sumv(vnext ? lane_dot(vn, wv) : lane_dot(wv, wv), sh);
        if (threadIdx.x == 0) pout[c] = s;
    }
}

// column >= 1: hn = sqrt(tree(pin)); breakdown when hn <= 1e-12 ||J v_j||;
// else H[column][column-1] = hn, V_column = w * (1/hn)
__global__ void __launch_bounds__(RT) bnormalize_kernel(const double *__restrict__ w, double *__restrict__ V,
                                                        size_t ldv, int column, const double *__restrict__ pin,
                                                        const BSeg sg)
{
    __shared__ double sh[10];
    __shared__ int flag;
    double *v = V + (size_t)column * ldv;
    for (int c = blockIdx.x; c < sg.nchunks; c += gridDim.x) {
        const ChunkRef r = chunk_ref(sg, c);
        StepState *st = sg.st + r.k;
        if (!chunk_active(st, &flag)) continue;
        const double hn = sqrt(tree_partials(pin + r.chunk0, r.P, sh));
        if (!(hn > 1e-12 * st->wnorm0)) {
            if (c == r.chunk0 && threadIdx.x == 0) {
                st->active = 0;
                st->meff = column;
            }
            continue;
        }
        if (c == r.chunk0 && threadIdx.x == 0) st->H[column * kMaxKrylov + column - 1] = hn;
        const double rh = 1.0 / hn;
        double x[EPL];
        load8(w + r.off, r.e0, r.n, x);
#pragma unroll
        for (int k = 0; k < EPL; ++k) x[k] = x[k] * rh;
        store8(v + r.off, r.e0, r.n, x);
    }
}

#else
// block passes of a batch: chunk c's partials, reduced by the CTA that finishes
// its instance last (the order of the sums does not depend on cpc)
__global__ void __launch_bounds__(RT, kGsCtas) bgs_pass_kernel(double *__restrict__ w, const double *__restrict__ V, size_t ldv,
                                                      const GsPass ps, double *__restrict__ part, const BSeg sg)
{
    __shared__ double ws[8][8];
    __shared__ int flag;
    for (int c = blockIdx.x; c < sg.nchunks; c += gridDim.x) {
        const ChunkRef r = chunk_ref(sg, c);
        StepState *st = sg.st + r.k;
        if (!chunk_active(st, &flag)) continue;
        double t[16];
        gs_zero(t);
        gs_lane<true>(w + r.off, V + r.off, ldv, r.e0, r.n, ps, st, t);
        gs_reduce(t, ps, part + r.chunk0, sg.nchunks, c - r.chunk0, r.P, st, ws, &flag);
    }
}

__global__ void __launch_bounds__(RT) bgs_normalize_kernel(const double *__restrict__ w, double *__restrict__ v,
                                                           const BSeg sg)
{
    __shared__ int flag;
    for (int c = blockIdx.x; c < sg.nchunks; c += gridDim.x) {
        const ChunkRef r = chunk_ref(sg, c);
        const StepState *st = sg.st + r.k;
        if (!chunk_active(st, &flag)) continue;
        const double rh = st->gs_rh;
        double x[EPL];
        load8(w + r.off, r.e0, r.n, x);
#pragma unroll
        for (int k = 0; k < EPL; ++k) x[k] = x[k] * rh;
        store8(v + r.off, r.e0, r.n, x);
    }
}
#endif

// pout[m * nchunks + c] = <V_m, F> over chunk c, m < meff of its instance
// (sums formed together as in multidot_kernel)
__global__ void __launch_bounds__(RT) bmultidot_kernel(const double *__restrict__ F, const double *__restrict__ V,
                                                       size_t ldv, double *__restrict__ pout, const BSeg sg)
{
    __shared__ double ws[kMaxKrylov][8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int c = blockIdx.x; c < sg.nchunks; c += gridDim.x) {
        const ChunkRef r = chunk_ref(sg, c);
        const int m = sg.st[r.k].meff;
        double f[EPL];
        load8(F + r.off, r.e0, r.n, f);
        __syncthreads();
        for (int g = 0; g < m; g += 16) {
            double t[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                t[q] = 0.0;
                if (g + q < m) {
                    double v[EPL];
                    load8(V + (size_t)(g + q) * ldv + r.off, r.e0, r.n, v);
                    t[q] = lane_dot(v, f);
                }
            }
            const double s = lane_tree16(t, lane);
            const int q = lane_tree16_value(lane);
            if (lane < 16 && g + q < m) ws[g + q][wid] = s;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += RT) pout[(size_t)i * sg.nchunks + c] = warp8_tree(ws[i]);
    }
}

// one CTA per instance: the projected stage solve
__global__ void __launch_bounds__(kSolveThreads) bstage_solve_kernel(int stage, GamRow gr, const double *pin, const BSeg sg)
{
    const BatchInst &I = sg.inst[blockIdx.x];
    stage_solve_body(stage, gr, pin + I.chunk0, (size_t)sg.nchunks, I.nchunks, sg.st + blockIdx.x);
}

// one warp per instance: LU of I - h gamma H
__global__ void __launch_bounds__(kLuThreads) blu_kernel(StepState *st) { lu_body(st + blockIdx.x); }

// k = sum_{m<meff} cvec[stage][m] V_m + h F over each chunk (instance coefficients)
__global__ void __launch_bounds__(RT) bstage_vec_kernel(double *__restrict__ kout, const double *__restrict__ F,
                                                        const double *__restrict__ V, size_t ldv, int stage,
                                                        const BSeg sg)
{
    __shared__ double cv[kMaxKrylov];
    for (int c = blockIdx.x; c < sg.nchunks; c += gridDim.x) {
        const ChunkRef r = chunk_ref(sg, c);
        const StepState *st = sg.st + r.k;
        const int m = st->meff;
        const double h = st->h;
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += RT) cv[i] = st->cvec[stage][i];
        __syncthreads();
        double a[EPL], f[EPL];
#pragma unroll
        for (int k = 0; k < EPL; ++k) a[k] = 0.0;
        for (int i = 0; i < m; ++i) {
            double v[EPL];
            load8(V + (size_t)i * ldv + r.off, r.e0, r.n, v);
#pragma unroll
            for (int k = 0; k < EPL; ++k) a[k] = a[k] + cv[i] * v[k];
        }
        load8(F + r.off, r.e0, r.n, f);
#pragma unroll
        for (int k = 0; k < EPL; ++k) a[k] = a[k] + h * f[k];
        store8(kout + r.off, r.e0, r.n, a);
    }
}

// y = y + sum_q b_q k_q (q = 0..3, in order), skipped for instances with a latched status
__global__ void __launch_bounds__(RT) bupdate_kernel(double *__restrict__ y, const double *__restrict__ k0,
                                                     const double *__restrict__ k1, const double *__restrict__ k2,
                                                     const double *__restrict__ k3, double b0, double b1, double b2,
                                                     double b3, const BSeg sg)
{
    __shared__ int flag;
    for (int c = blockIdx.x; c < sg.nchunks; c += gridDim.x) {
        const ChunkRef r = chunk_ref(sg, c);
        __syncthreads();
        if (threadIdx.x == 0) flag = sg.st[r.k].status;
        __syncthreads();
        if (flag != 0) continue;
        double t[EPL], v[EPL];
        load8(y + r.off, r.e0, r.n, t);
        load8(k0 + r.off, r.e0, r.n, v);
#pragma unroll
        for (int k = 0; k < EPL; ++k) t[k] = t[k] + b0 * v[k];
        load8(k1 + r.off, r.e0, r.n, v);
#pragma unroll
        for (int k = 0; k < EPL; ++k) t[k] = t[k] + b1 * v[k];
        load8(k2 + r.off, r.e0, r.n, v);
#pragma unroll
        for (int k = 0; k < EPL; ++k) t[k] = t[k] + b2 * v[k];
        load8(k3 + r.off, r.e0, r.n, v);
#pragma unroll
        for (int k = 0; k < EPL; ++k) t[k] = t[k] + b3 * v[k];
        store8(y + r.off, r.e0, r.n, t);
    }
}

static int bgrid(const BSeg &sg, int cpc) { return (sg.nchunks + cpc - 1) / cpc; }

static cudaError_t b_dot2(const double *a0, const double *b0, const double *a1, const double *b1, double *part,
                          const BSeg &sg, int use_active, int cpc, cudaStream_t s)
{
    bdot2_kernel<<<bgrid(sg, cpc), RT, 0, s>>>(a0, b0, a1, b1, part, sg, use_active);
    return cudaGetLastError();
}

static cudaError_t b_eps(const double *part, const BSeg &sg, int ninst, cudaStream_t s)
{
    beps_kernel<<<ninst, RT, 0, s>>>(part, sg);
    return cudaGetLastError();
}

static cudaError_t b_first_normalize(const double *F, double *V0, const double *part, const BSeg &sg, int cpc,
                                     cudaStream_t s)
{
    bfirst_normalize_kernel<<<bgrid(sg, cpc), RT, 0, s>>>(F, V0, part, sg);
    return cudaGetLastError();
}

#ifndef ROK_LINALG_FAST
static cudaError_t b_mgs(double *w, const double *V, size_t ldv, int i, int j, const double *pin, double *pout,
                         const BSeg &sg, int cpc, cudaStream_t s)
{
    bmgs_kernel<<<bgrid(sg, cpc), RT, 0, s>>>(w, V, ldv, i, j, pin, pout, sg);
    return cudaGetLastError();
}

static cudaError_t b_normalize(const double *w, double *V, size_t ldv, int column, const double *pin, const BSeg &sg,
                               int cpc, cudaStream_t s)
{
    bnormalize_kernel<<<bgrid(sg, cpc), RT, 0, s>>>(w, V, ldv, column, pin, sg);
    return cudaGetLastError();
}

#else
static cudaError_t b_gs_pass(double *w, const double *V, size_t ldv, int j, int b, int nb, int b2, int nn, int next,
                             double *part, const BSeg &sg, int cpc, cudaStream_t s)
{
    bgs_pass_kernel<<<bgrid(sg, cpc), RT, 0, s>>>(w, V, ldv, GsPass{j, b, nb, b2, nn, next}, part, sg);
    return cudaGetLastError();
}

static cudaError_t b_gs_normalize(const double *w, double *V, size_t ldv, int j, const BSeg &sg, int cpc, cudaStream_t s)
{
    bgs_normalize_kernel<<<bgrid(sg, cpc), RT, 0, s>>>(w, V + (size_t)(j + 1) * ldv, sg);
    return cudaGetLastError();
}
#endif

static cudaError_t b_multidot(const double *F, const double *V, size_t ldv, double *pout, const BSeg &sg, int cpc,
                              cudaStream_t s)
{
    bmultidot_kernel<<<bgrid(sg, cpc), RT, 0, s>>>(F, V, ldv, pout, sg);
    return cudaGetLastError();
}

static cudaError_t b_stage_solve(int stage, const double *gam_row, const double *pin, const BSeg &sg, int ninst,
                                 cudaStream_t s)
{
    GamRow gr;
    for (int j = 0; j < 4; ++j) gr.g[j] = gam_row[j];
    bstage_solve_kernel<<<ninst, kSolveThreads, 0, s>>>(stage, gr, pin, sg);
    return cudaGetLastError();
}

static cudaError_t b_lu(StepState *st, int ninst, cudaStream_t s)
{
    blu_kernel<<<ninst, kLuThreads, 0, s>>>(st);
    return cudaGetLastError();
}

static cudaError_t b_stage_vec(double *k, const double *F, const double *V, size_t ldv, int stage, const BSeg &sg,
                               int cpc, cudaStream_t s)
{
    bstage_vec_kernel<<<bgrid(sg, cpc), RT, 0, s>>>(k, F, V, ldv, stage, sg);
    return cudaGetLastError();
}

static cudaError_t b_update(double *y, const double *const *kv, const double *b, const BSeg &sg, int cpc,
                            cudaStream_t s)
{
    bupdate_kernel<<<bgrid(sg, cpc), RT, 0, s>>>(y, kv[0], kv[1], kv[2], kv[3], b[0], b[1], b[2], b[3], sg);
    return cudaGetLastError();
}

#ifdef ROK_LINALG_FAST
const BatchOps bops = {b_dot2,     b_eps,         b_first_normalize, b_gs_pass,   b_gs_normalize, nullptr, nullptr,
                       b_multidot, b_stage_solve, b_lu,              b_stage_vec, b_update};
#else
const BatchOps bops = {b_dot2,     b_eps,         b_first_normalize, nullptr,     nullptr, b_mgs, b_normalize,
                       b_multidot, b_stage_solve, b_lu,              b_stage_vec, b_update};
#endif

// ---- embedded error estimates ------------------------------------------------------
struct ErrArgs {
    const double *k[8];
    double d[8];
};

// partials[b] = sum over CTA b's entries of (e_i / sc_i)^2 with
// e_i = sum_q d_q k_q[i] (in order) and sc_i = atol + rtol max(|y_i|, |ynew_i|)
__global__ void __launch_bounds__(RT) err_kernel(const double *__restrict__ y, const double *__restrict__ ynew,
                                                 ErrArgs a, int count, double atol, double rtol, size_t n,
                                                 double *__restrict__ partials)
{
    __shared__ double sh[10];
    const size_t e0 = lane_e0();
    double x[EPL];
#pragma unroll
    for (int k = 0; k < EPL; ++k) {
        const size_t e = e0 + k;
        x[k] = 0.0;
        if (e < n) {
            double ev = 0.0;
            for (int q = 0; q < count; ++q) ev = ev + a.d[q] * a.k[q][e];
            const double sc = atol + rtol * fmax(fabs(y[e]), fabs(ynew[e]));
            const double r = ev / sc;
            x[k] = r * r;
        }
    }
    const double s = chunk_sum(x, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

// ---- launchers ----------------------------------------------------------------

inline int blocks_for(size_t n) { return (int)((n + RB - 1) / RB); }

static cudaError_t dot2(const double *a0, const double *b0, const double *a1, const double *b1, size_t n,
                        double *partials, int P, const int *active, cudaStream_t s)
{
    dot2_kernel<<<P, RT, 0, s>>>(a0, b0, a1, b1, n, partials, P, active);
    return cudaGetLastError();
}

static cudaError_t mgs(double *w, const double *vprev, const double *vnext, size_t n, const double *pin, int P,
                       double *hout, double *pout, bool first, StepState *st, cudaStream_t s)
{
    mgs_kernel<<<P, RT, 0, s>>>(w, vprev, vnext, n, pin, P, hout, pout, first ? 1 : 0, st);
    return cudaGetLastError();
}

#ifndef ROK_LINALG_FAST
static cudaError_t normalize(const double *w, double *v, size_t n, const double *pin, int P, double *hsub,
                             int column, StepState *st, cudaStream_t s)
{
    normalize_kernel<<<P, RT, 0, s>>>(w, v, n, pin, P, hsub, column, st);
    return cudaGetLastError();
}

#endif

static cudaError_t multidot(const double *F, const void *V, int fp32, size_t ldv, size_t n, double *pout, int P,
                            const StepState *st, cudaStream_t s)
{
#ifdef ROK_LINALG_FAST
    {   // even split, one CTA per SM (the strict build keeps the oracle's chunks)
        const int sms = sm_count();
        int G = sms > 0 && P > sms ? sms : P;
        auto range = [&] { return ((n + G - 1) / G + 3) & ~(size_t)3; };
        while (G > 1 && (size_t)(G - 1) * range() >= n) --G;   // every CTA has entries
        const size_t L = range();
        // loads of entry quads: lengths multiples of 4, aligned starts
        const uintptr_t va = fp32 ? 15 : 31;
        if (!fp32 && sms > 0 && L > (size_t)kEvenThreads * kEvenPerThread && !(n & 3) && !(ldv & 3) &&
            !((uintptr_t)F & 31) && !((uintptr_t)V & 31)) {
            multidot_long_kernel<8><<<G, kEvenThreads, 0, s>>>(F, static_cast<const double *>(V), ldv, n, L, pout, P, st);
            return cudaGetLastError();
        }
        if (sms > 0 && L <= (size_t)kEvenThreads * kEvenPerThread && !(n & 3) && !(ldv & 3) &&
            !((uintptr_t)F & 31) && !((uintptr_t)V & va)) {
            const bool e4 = L <= (size_t)kEvenThreads * 4, e8 = L <= (size_t)kEvenThreads * 8;
            if (fp32) {
                const float *Vf = static_cast<const float *>(V);
                if (e4) multidot_even_kernel<4, float><<<G, kEvenThreads, 0, s>>>(F, Vf, ldv, n, L, pout, P, st);
                else if (e8) multidot_even_kernel<8, float><<<G, kEvenThreads, 0, s>>>(F, Vf, ldv, n, L, pout, P, st);
                else multidot_even_kernel<16, float><<<G, kEvenThreads, 0, s>>>(F, Vf, ldv, n, L, pout, P, st);
            } else {
                const double *Vd = static_cast<const double *>(V);
                if (e4) multidot_even_kernel<4, double><<<G, kEvenThreads, 0, s>>>(F, Vd, ldv, n, L, pout, P, st);
                else if (e8) multidot_even_kernel<8, double><<<G, kEvenThreads, 0, s>>>(F, Vd, ldv, n, L, pout, P, st);
                else multidot_even_kernel<16, double><<<G, kEvenThreads, 0, s>>>(F, Vd, ldv, n, L, pout, P, st);
            }
            return cudaGetLastError();
        }
    }
#endif
    if (fp32) multidot_kernel<float><<<P, RT, 0, s>>>(F, static_cast<const float *>(V), ldv, n, pout, P, st);
    else multidot_kernel<double><<<P, RT, 0, s>>>(F, static_cast<const double *>(V), ldv, n, pout, P, st);
    return cudaGetLastError();
}

static cudaError_t stage_solve(int stage, const double *gam_row, const double *pin, int P, StepState *st,
                               cudaStream_t s)
{
    GamRow gr;
    for (int j = 0; j < 4; ++j) gr.g[j] = gam_row[j];
    stage_solve_kernel<<<1, kSolveThreads, 0, s>>>(stage, gr, pin, P, st);
    return cudaGetLastError();
}

static cudaError_t lu(StepState *st, cudaStream_t s)
{
    lu_kernel<<<1, kLuThreads, 0, s>>>(st);
    return cudaGetLastError();
}

static cudaError_t stage_vec(double *k, const double *F, const void *V, int fp32, size_t ldv, size_t n, int stage,
                             const StepState *st, int grid, cudaStream_t s)
{
#ifdef ROK_LINALG_FAST
    if (!(n & 3) && !(ldv & 3) && !((uintptr_t)F & 31) && !((uintptr_t)V & (fp32 ? 15 : 31)) &&
        !((uintptr_t)k & 31)) {
        const size_t nq = n / 4;
        const unsigned grid = (unsigned)((nq + RT - 1) / RT);
        if (fp32)
            stage_vec_quad_kernel<float><<<grid, RT, 0, s>>>(k, F, static_cast<const float *>(V), ldv, nq, stage, st);
        else
            stage_vec_quad_kernel<double><<<grid, RT, 0, s>>>(k, F, static_cast<const double *>(V), ldv, nq, stage, st);
        return cudaGetLastError();
    }
#endif
    if (fp32) stage_vec_kernel<float><<<grid, RT, 0, s>>>(k, F, static_cast<const float *>(V), ldv, n, stage, st);
    else stage_vec_kernel<double><<<grid, RT, 0, s>>>(k, F, static_cast<const double *>(V), ldv, n, stage, st);
    return cudaGetLastError();
}

static cudaError_t axpy_n(double *out, const double *base, const double *const *v, const double *c, int count,
                          size_t n, const StepState *guard, int grid, cudaStream_t s)
{
    if (count > 8) return cudaErrorInvalidValue;
    AxpyArgs a;
    for (int q = 0; q < 8; ++q) {
        a.v[q] = q < count ? v[q] : nullptr;
        a.c[q] = q < count ? c[q] : 0.0;
    }
    axpy_n_kernel<<<grid, RT, 0, s>>>(out, base, a, count, n, guard);
    return cudaGetLastError();
}

static cudaError_t basis_combine(double *out, const double *base, const double *V, size_t ldv, size_t n, int count,
                                 const double *gcoef, const int *count_dev, int grid, cudaStream_t s)
{
    basis_combine_kernel<<<grid, RT, 0, s>>>(out, base, V, ldv, n, count, gcoef, count_dev);
    return cudaGetLastError();
}

static cudaError_t gmres_start(const double *pin, int P, double tol, int m, StepState *st, cudaStream_t s)
{
    gmres_start_kernel<<<1, RT, 0, s>>>(pin, P, tol, m, st);
    return cudaGetLastError();
}

static cudaError_t gmres_cycle(const double *pin, int P, StepState *st, cudaStream_t s)
{
    gmres_cycle_kernel<<<1, RT, 0, s>>>(pin, P, st);
    return cudaGetLastError();
}

static cudaError_t gmres_givens(int j, StepState *st, cudaStream_t s)
{
    gmres_givens_kernel<<<1, 1, 0, s>>>(j, st);
    return cudaGetLastError();
}

static cudaError_t gmres_lsq(StepState *st, cudaStream_t s)
{
    gmres_lsq_kernel<<<1, 1, 0, s>>>(st);
    return cudaGetLastError();
}

static cudaError_t eps(const double *pin, int P, bool v_unit, double eps_given, StepState *st, cudaStream_t s)
{
    eps_kernel<<<1, RT, 0, s>>>(pin, P, v_unit ? 1 : 0, eps_given, st);
    return cudaGetLastError();
}

static cudaError_t sum_sqrt(const double *pin, int P, double *dst, cudaStream_t s)
{
    sum_sqrt_kernel<<<1, RT, 0, s>>>(pin, P, dst);
    return cudaGetLastError();
}

static cudaError_t err_sum(const double *y, const double *ynew, const double *const *kv, const double *d, int count,
                           double atol, double rtol, size_t n, double *partials, int P, cudaStream_t s)
{
    if (count > 8) return cudaErrorInvalidValue;
    ErrArgs a;
    for (int q = 0; q < 8; ++q) {
        a.k[q] = q < count ? kv[q] : nullptr;
        a.d[q] = q < count ? d[q] : 0.0;
    }
    err_kernel<<<P, RT, 0, s>>>(y, ynew, a, count, atol, rtol, n, partials);
    return cudaGetLastError();
}

#ifdef ROK_LINALG_FAST
#define ROK_GS_OPS mgs, nullptr
#else
#define ROK_GS_OPS mgs, normalize
static constexpr decltype(LinalgOps::gs_column) gs_column = nullptr;
#endif
const LinalgOps ops = {dot2,      ROK_GS_OPS,  multidot,       stage_solve,         lu,           stage_vec,
                       axpy_n,    basis_combine, eps,          sum_sqrt,            arnoldi_column, gs_column,
                       arnoldi_column_ctas, first_vector, err_sum, gmres_start,     gmres_cycle,  gmres_givens,
                       gmres_lsq};
#undef ROK_GS_OPS

#endif  // ROK_LINALG_DEVICE_ONLY

}  // namespace ROK_NS
}  // namespace rok
