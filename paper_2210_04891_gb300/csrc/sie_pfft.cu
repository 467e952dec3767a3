// pfft_matvec: the loop-space product of Eq. (FinalME) with the inductive part
// applied by the pre-corrected FFT (Sec. IV-A, IV-B of arXiv 2210.04891):
//
//   alpha = A^T x                     (Eq. CurT; Euler-tour subtree sums)
//   Q_g   = sum_T W(n,T) c_T          (Eq. Projection with the point currents
//                                      J_q = sum_k c_k (w_q/2)(r_q - v_k) folded in)
//   phi_g = H Q_g                     (Eq. FFTCal; zero-padded FFT convolution)
//   y_T   = Z_s G_T c_T + c_L (sum_n W(n,T)^T phi_n + sum_T' L_d(T,T') c_T')
//                                     (Eq. interpolation with I = B^T, Eq. Zb, Eq. Lb)
//   y     = A y_b                     (Eq. VolT; Euler-tour root-path sums)
//
// A^T x: the current of a twig equals minus the current its subtree receives
// through links (Kirchhoff's current law), a subtree sum = a difference of two
// prefix sums along the Euler tour.  A y: the voltage of a fundamental loop is
// its link's voltage plus psi(head) - psi(tail), psi(v) the sum of twig
// voltages on v's path to the root = a prefix sum of +-delta over the tour.
// Both are exact rewrites of the sparse products (no approximation).
//
// Projection, interpolation and near field are block-sparse x dense products
// with 3x3 real blocks and complex right-hand sides: every dense operand is
// stored with the right-hand sides innermost (c_T as [T][3][R], potentials as
// [n][3][R]), one warp reads a block once and applies it to a slab of up to
// 128 right-hand sides with coalesced loads.
#include <algorithm>
#include <cmath>
#include <complex>
#include <memory>
#include <type_traits>
#include <vector>

#include "sie_dd.cuh"
#include "sie_plan.h"

using namespace sie;

namespace {

constexpr double kMu0 = 4e-7 * M_PI;

template <typename V> __device__ __forceinline__ V shfl_up(V v, int d) {
    V o;
    o.x = __shfl_up_sync(0xffffffffu, v.x, d);
    o.y = __shfl_up_sync(0xffffffffu, v.y, d);
    return o;
}

// Elements of the loop/branch maps after the field computation: complex128 in
// the FP64 form, double-float float4 (sie_dd.cuh) in the mixed and double-float forms.
template <typename T> using TourE = typename std::conditional<std::is_same<T, double>::value, double2, float4>::type;
template <typename T> constexpr bool is_f32 = std::is_same<T, float>::value;
template <typename T> constexpr bool is_f64 = std::is_same<T, double>::value;
template <typename T> constexpr bool is_df = std::is_same<T, df>::value;

__device__ __forceinline__ double2 eadd(double2 a, double2 b) { return cadd(a, b); }
__device__ __forceinline__ float4 eadd(float4 a, float4 b) {
    return cdd(dd_add(cdd_re(a), cdd_re(b)), dd_add(cdd_im(a), cdd_im(b)));
}
__device__ __forceinline__ double2 eneg(double2 a) { return make_double2(-a.x, -a.y); }
__device__ __forceinline__ float4 eneg(float4 a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }
template <typename E> __device__ __forceinline__ E ezero();
template <> __device__ __forceinline__ double2 ezero<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float4 ezero<float4>() { return make_float4(0.f, 0.f, 0.f, 0.f); }
// conversions: FP64 value -> element; element -> FP64, FP32 or another element type
__device__ __forceinline__ void eset(double2 &e, double2 v) { e = v; }
__device__ __forceinline__ void eset(float4 &e, double2 v) { e = cdd(dd_split(v.x), dd_split(v.y)); }
__device__ __forceinline__ void eset(double2 &e, float4 v) {
    e = make_double2(double(v.x) + double(v.y), double(v.z) + double(v.w));
}
__device__ __forceinline__ void eset(float4 &e, float4 v) { e = v; }
__device__ __forceinline__ double2 to_c(double2 v, double2) { return v; }
__device__ __forceinline__ float2 to_c(double2 v, float2) { return make_float2(dd_split(v.x).hi, dd_split(v.y).hi); }
__device__ __forceinline__ float2 to_c(float4 e, float2) { return make_float2(e.x + e.y, e.z + e.w); }
__device__ __forceinline__ cdf to_c(double2 v, cdf) {
    const DD a = dd_split(v.x), b = dd_split(v.y);
    return cdf{df(a.hi, a.lo), df(b.hi, b.lo)};
}
__device__ __forceinline__ cdf to_c(float4 e, cdf) { return cdf{df(e.x, e.y), df(e.z, e.w)}; }
__device__ __forceinline__ float4 shfl_up(float4 v, int d) {
    v.x = __shfl_up_sync(0xffffffffu, v.x, d);
    v.y = __shfl_up_sync(0xffffffffu, v.y, d);
    v.z = __shfl_up_sync(0xffffffffu, v.z, d);
    v.w = __shfl_up_sync(0xffffffffu, v.w, d);
    return v;
}

// i = q n + r without a 64-bit division where 32 bits hold i (uniform branch)
__device__ __forceinline__ void divmod(int64_t i, int64_t n, int64_t &q, int64_t &r) {
    if ((uint64_t(i) | uint64_t(n)) >> 32) {
        q = i / n;
        r = i - q * n;
    } else {
        const uint32_t a = uint32_t(i) / uint32_t(n);
        q = a;
        r = uint32_t(i) - a * uint32_t(n);
    }
}

// ---- Prefix sums over the Euler tour, of values that are formed where they are
// summed (the current the links inject at a slot, Eq. CurT; the voltage step of
// a slot's twig, Eq. VolT).  A row (right-hand side) is cut into chunks of
// kTourChunk slots, one CTA of 1024 threads per (row, chunk), 4 slots per
// thread.  With more than one chunk a first pass (k_tour_part) forms each
// chunk's sums, and k_tour_sums starts each chunk from the chain of those before
// it.  The sums are associated as by one CTA walking the row chunk by chunk
// (per thread, per warp, over the warps, over the chunks), so the result does
// not depend on the split; what the split buys is R x chunks CTAs instead of R.
// Bound by latency (a chunk: one code, one value, two block scans of 16-byte
// elements).  Currents' sums with a kernel that wrote the values and one CTA per row that
// summed them: 64 us for 3 right-hand sides on 12k triangles (24k slots), 255 us
// for 128 on 40k (79k slots); here 28 and 220 us.
struct TourLinks {   // values of A^T: +x of links entering the slot's node, -x of links leaving it
    const double2 *__restrict__ x;
    int64_t nl;
    const int32_t *__restrict__ slot, *__restrict__ nl_ptr, *__restrict__ nl_loop;
    const int8_t *__restrict__ nl_sign;
};
template <typename V> struct TourTwigs {   // values of A: +-voltage of the twig above the slot's node
    const V *__restrict__ y_br;
    int64_t ldy;
    const int32_t *__restrict__ slot;
};
// Chunk's scan: v[k] inclusive within the thread, incl inclusive over the warp's
// threads, warp_tot inclusive over the warps; run the thread's total.
template <typename E>
__device__ __forceinline__ void chunk_scan(E (&v)[4], E &run, E &incl, E *warp_tot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    run = ezero<E>();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        run = eadd(run, v[k]);
        v[k] = run;
    }
    incl = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        E o = shfl_up(incl, d);
        if (lane >= d) incl = eadd(incl, o);
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        E w = warp_tot[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            E o = shfl_up(w, d);
            if (lane >= d) w = eadd(w, o);
        }
        warp_tot[lane] = w;
    }
    __syncthreads();
}
// codes of the thread's four slots from i0 on (padded to whole chunks), and their
// values: the four loads first, unconditioned by each other, then nodes of
// several links (few), then signs and conversions
template <typename S> __device__ __forceinline__ int4 chunk_codes(const S &src, int64_t i0) {
    return __ldg(reinterpret_cast<const int4 *>(src.slot + i0));
}
__device__ __forceinline__ double2 node_links(const TourLinks &s, const double2 *x, int32_t n) {
    double2 v = make_double2(0.0, 0.0);
#pragma unroll 8
    for (int32_t k = s.nl_ptr[n]; k < s.nl_ptr[n + 1]; ++k) {
        const double2 xv = x[s.nl_loop[k]];
        v = s.nl_sign[k] > 0 ? cadd(v, xv) : csub(v, xv);
    }
    return v;
}
template <typename E>
__device__ __forceinline__ void chunk_load(const TourLinks &s, int64_t r, int4 codes, E (&v)[4]) {
    const int32_t c[4] = {codes.x, codes.y, codes.z, codes.w};
    const double2 *x = s.x + r * s.nl;
    double2 d[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        d[k] = make_double2(0.0, 0.0);
        if (c[k] != 0 && c[k] < kManyLinks) d[k] = __ldg(x + (abs(c[k]) - 1));
    }
    if (max(max(c[0], c[1]), max(c[2], c[3])) >= kManyLinks) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (c[k] >= kManyLinks) d[k] = node_links(s, x, c[k] - kManyLinks);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (c[k] < 0) d[k] = make_double2(-d[k].x, -d[k].y);
        v[k] = ezero<E>();
        if (c[k] != 0) eset(v[k], d[k]);
    }
}
template <typename E>
__device__ __forceinline__ void chunk_load(const TourTwigs<E> &s, int64_t r, int4 codes, E (&v)[4]) {
    const int32_t c[4] = {codes.x, codes.y, codes.z, codes.w};
    const E *y = s.y_br + r * s.ldy;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = ezero<E>();
        if (c[k] != 0) v[k] = __ldg(y + (abs(c[k]) - 1));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (c[k] < 0) v[k] = eneg(v[k]);
}
// The three terms the last thread of a chunk adds to its carry, in order: the
// warps before its own, the threads before it in its warp, its own slots.
template <typename E, typename S>
__global__ void __launch_bounds__(1024) k_tour_part(const S src, int32_t nchunk, E *__restrict__ part) {
    __shared__ E warp_tot[32];
    const int64_t r = blockIdx.x / nchunk;
    const int32_t c = blockIdx.x - int32_t(r) * nchunk;
    E v[4], run, incl;
    chunk_load(src, r, chunk_codes(src, int64_t(c) * kTourChunk + 4 * int64_t(threadIdx.x)), v);
    chunk_scan(v, run, incl, warp_tot);
    if (threadIdx.x == 1023) {
        E *p = part + (r * nchunk + c) * kTourPart;
        p[0] = warp_tot[30];
        p[1] = eadd(incl, eneg(run));
        p[2] = run;
    }
}
template <typename E, typename S>
__global__ void __launch_bounds__(1024) k_tour_sums(const S src, int64_t n, int32_t nchunk,
                                                    const E *__restrict__ part, E *__restrict__ out) {
    __shared__ E warp_tot[32];
    __shared__ E carry_s;
    constexpr int STAGE = 96 * kTourPart;
    __shared__ E stage[STAGE];
    const int64_t r = blockIdx.x / nchunk;
    const int32_t c = blockIdx.x - int32_t(r) * nchunk;
    const int64_t i0 = int64_t(c) * kTourChunk + 4 * int64_t(threadIdx.x);
    E v[4], run, incl;
    chunk_load(src, r, chunk_codes(src, i0), v);
    // carry: the chain over the chunks before this one, by one thread from shared memory
    if (threadIdx.x == 0) carry_s = ezero<E>();
    for (int32_t b = 0; b < c * kTourPart; b += STAGE) {
        const int m = min(STAGE, c * kTourPart - b);
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += 1024) stage[i] = part[r * nchunk * kTourPart + b + i];
        __syncthreads();
        if (threadIdx.x == 0) {
            E s = carry_s;
            for (int i = 0; i < m; ++i) s = eadd(s, stage[i]);
            carry_s = s;
        }
    }
    chunk_scan(v, run, incl, warp_tot);   // its barriers also publish carry_s
    E off = carry_s;
    const int warp = threadIdx.x >> 5;
    if (warp > 0) off = eadd(off, warp_tot[warp - 1]);
    off = eadd(off, eadd(incl, eneg(run)));   // exclusive within the warp
    E *row = out + r * n;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (i0 + k < n) row[i0 + k] = eadd(v[k], off);
}

// The same sums by one CTA per row, chunk by chunk: with a row for every SM the
// split only reads the values twice.  The next chunk's values and the codes of
// the one after are in flight during the block scan.
template <typename E, typename S>
__global__ void __launch_bounds__(1024) k_tour_rows(const S src, int64_t n, E *__restrict__ out) {
    __shared__ E warp_tot[32];
    __shared__ E carry_s;
    const int64_t r = blockIdx.x, np = (n + kTourChunk - 1) / kTourChunk * kTourChunk;
    const int warp = threadIdx.x >> 5;
    E *row = out + r * n;
    E carry = ezero<E>();
    int64_t i0 = 4 * int64_t(threadIdx.x);
    E vn[4];
    chunk_load(src, r, chunk_codes(src, i0), vn);
    int4 codes = make_int4(0, 0, 0, 0);
    if (i0 + kTourChunk < np) codes = chunk_codes(src, i0 + kTourChunk);
    for (; i0 < np; i0 += kTourChunk) {
        E v[4], run, incl;
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = vn[k];
        chunk_load(src, r, codes, vn);
        codes = make_int4(0, 0, 0, 0);
        if (i0 + 2 * kTourChunk < np) codes = chunk_codes(src, i0 + 2 * kTourChunk);
        chunk_scan(v, run, incl, warp_tot);
        E off = carry;
        if (warp > 0) off = eadd(off, warp_tot[warp - 1]);
        off = eadd(off, eadd(incl, eneg(run)));   // exclusive within the warp
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i0 + k < n) row[i0 + k] = eadd(v[k], off);
        if (threadIdx.x == 1023) carry_s = eadd(off, run);
        __syncthreads();
        carry = carry_s;
    }
}

// Branch current (loop space) from its record: a link carries its loop current;
// a twig above node v carries -sigma * (subtree inflow), a difference of two
// prefix sums taken in the tour's arithmetic.
template <typename T, typename E>
__device__ __forceinline__ C<T> branch_current(int4 s, int64_t r, const double2 *__restrict__ x, int64_t nl,
                                               const E *__restrict__ P, int64_t nslots) {
    C<T> d;
    if (s.x >= 0) {
        d = to_c(x[r * nl + s.x], C<T>{});
    } else {
        const E *row = P + r * nslots;
        E S = row[s.y];
        if (s.z >= 0) S = eadd(S, eneg(row[s.z]));
        d = to_c(S, C<T>{});
    }
    return s.w < 0 ? mk<T>(-d.x, -d.y) : d;
}

// Local currents c_T[k] = s_k alpha_{b(T,k)}: one thread per (T, r) for the
// three local edges, written as cT [T][3][R] (right-hand sides innermost), or
// with SMALL (FP32) as float4 [T][2R] (components innermost, re and im columns).
template <typename T, bool SMALL>
__global__ void k_alpha_tri(const double2 *__restrict__ x, int64_t nl, const TourE<T> *__restrict__ P, int64_t nslots,
                            const int4 *__restrict__ tri_src, const int32_t *__restrict__ tb,
                            const int8_t *__restrict__ ts, int64_t nt, int32_t nrhs, int space, int64_t nb,
                            C<T> *__restrict__ cT) {
    int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= nt * nrhs) return;
    int64_t t, r;
    divmod(i, nrhs, t, r);
    C<T> c[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int64_t tk = t * 3 + k;
        c[k] = mk<T>(T(0), T(0));
        if (space == SIE_SPACE_LOOP) {
            const int4 s = __ldg(tri_src + tk);
            if (s.w) c[k] = branch_current<T>(s, r, x, nl, P, nslots);
        } else {
            const int32_t b = tb[tk];
            if (b >= 0) {
                c[k] = to_c(x[r * nb + b], C<T>{});
                if (ts[tk] < 0) { c[k].x = -c[k].x; c[k].y = -c[k].y; }
            }
        }
    }
    if constexpr (!SMALL) {
#pragma unroll
        for (int k = 0; k < 3; ++k) cT[(t * 3 + k) * nrhs + r] = c[k];
    }
    if constexpr (SMALL) {
        static_assert(is_f32<T>, "component-inner currents in FP32 only");
        float4 *o = reinterpret_cast<float4 *>(cT) + (t * nrhs + r) * 2;
        o[0] = make_float4(c[0].x, c[1].x, c[2].x, 0.f);
        o[1] = make_float4(c[0].y, c[1].y, c[2].y, 0.f);
    }
}

// V complex values at p (16-byte aligned when V = 2).
template <typename T, int V> __device__ __forceinline__ void ldv(const C<T> *p, C<T> (&v)[V]) {
    if constexpr (V == 2) {
        static_assert(is_f32<T>, "two complex per load only in FP32");
        const float4 u = __ldg(reinterpret_cast<const float4 *>(p));
        v[0] = make_float2(u.x, u.y);
        v[1] = make_float2(u.z, u.w);
    } else {
        v[0] = __ldg(p);
    }
}
template <typename T, int V> __device__ __forceinline__ void stv(C<T> *p, const C<T> (&v)[V]) {
    if constexpr (V == 2) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    } else {
        *p = v[0];
    }
}

// acc[a][j][v] += sum over the records e of row [e0, e1) of
//                 sum_b rec_e.b[3a+b] X[col_e][b][r],   r = rl + 32 V j + v.
// X is [rows][3][R] (right-hand sides innermost).  FULL: every r < R.
// UNR records in flight per warp (measured: 1 for the projection, 4 for the
// interpolation and the triangle gathers).
template <typename T, int V, int J, bool FULL, int UNR = 4>
__device__ __forceinline__ void gather_rows(const Rec<T> *__restrict__ rec, int64_t e0, int64_t e1,
                                            const C<T> *__restrict__ X, int32_t R, int32_t rl,
                                            C<T> (&acc)[3][J][V]) {
    const int64_t ld = 3 * int64_t(R);
#pragma unroll UNR
    for (int64_t e = e0; e < e1; ++e) {
        T b[9];
        const int64_t col = load_rec<T>(rec + e, b);
        const C<T> *x = X + col * ld;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int32_t r = rl + 32 * V * j;
            if (FULL || r < R) {
                C<T> x0[V], x1[V], x2[V];
                ldv<T, V>(x + r, x0);
                ldv<T, V>(x + R + r, x1);
                ldv<T, V>(x + 2 * R + r, x2);
#pragma unroll
                for (int v = 0; v < V; ++v)
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        acc[a][j][v].x += b[3 * a] * x0[v].x + b[3 * a + 1] * x1[v].x + b[3 * a + 2] * x2[v].x;
                        acc[a][j][v].y += b[3 * a] * x0[v].y + b[3 * a + 1] * x1[v].y + b[3 * a + 2] * x2[v].y;
                    }
            }
        }
    }
}

template <typename T, int V, int J> __device__ __forceinline__ void zero(C<T> (&acc)[3][J][V]) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
            for (int v = 0; v < V; ++v) acc[a][j][v] = mk<T>(T(0), T(0));
}

// Grid currents (Eq. Projection): Q_g[d][n] = sum_T sum_k W(n,T)[d][k] c_T[k]
// for a slab of 32 V J right-hand sides.  A block of 8 warps takes 8
// consecutive nodes, one per warp (lanes over right-hand sides); the block's
// results go through shared memory so that each of the 3 x slab grids gets an
// 8-node run per block.  Grid layout [3][R][Ng].
constexpr int kProjNodes = 8;
template <typename T, int V, int J> __host__ __device__ constexpr int proj_rows() { return 3 * 32 * V * J + 2; }
template <typename T, int V, int J> constexpr size_t proj_smem() {
    return size_t(kProjNodes) * proj_rows<T, V, J>() * sizeof(C<T>);
}

template <typename T, int V, int J>
__global__ void __launch_bounds__(256) k_project(const int64_t *__restrict__ ptr, const Rec<T> *__restrict__ rec,
                                                 const C<T> *__restrict__ cT, int64_t Ng, int32_t R,
                                                 C<T> *__restrict__ grid) {
    constexpr int SLAB = 32 * V * J;
    // row stride 3 SLAB + 2 (= 2 mod 16 complex): the 8-node reads below hit distinct banks
    constexpr int ROWS = proj_rows<T, V, J>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C<T> *sm = reinterpret_cast<C<T> *>(smem_raw);   // [kProjNodes][ROWS]
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n0 = int64_t(blockIdx.x) * kProjNodes, n = n0 + w;
    const int32_t rbase = int32_t(blockIdx.y) * SLAB;
    const int32_t rl = rbase + V * lane;
    C<T> acc[3][J][V];
    zero<T, V, J>(acc);
    if (n < Ng) {
        if (rbase + SLAB <= R) gather_rows<T, V, J, true, 1>(rec, ptr[n], ptr[n + 1], cT, R, rl, acc);
        else gather_rows<T, V, J, false, 1>(rec, ptr[n], ptr[n + 1], cT, R, rl, acc);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int j = 0; j < J; ++j) stv<T, V>(sm + w * ROWS + d * SLAB + V * lane + 32 * V * j, acc[d][j]);
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * SLAB * kProjNodes; i += blockDim.x) {
        const int row = i / kProjNodes, nd = i % kProjNodes;
        const int d = row / SLAB;
        const int32_t r = rbase + row % SLAB;
        const int64_t nn = n0 + nd;
        if (r < R && nn < Ng) grid[(int64_t(d) * R + r) * Ng + nn] = sm[nd * ROWS + row];
    }
}

// ---- FP64 and double-float gathers by real columns.  A block is real, so the
// complex dense operand [rows][3][R] is a real one of C = 2R columns and re and
// im never mix: a lane owns a column (or J of them, 32 apart) instead of a
// complex right-hand side.  Both forms are bound by their arithmetic pipe (FP64:
// 16 cycles per warp instruction and SM; double-float: 12 FP32 operations per
// term), so what counts is full lanes and few operations: terms are chained
// FMAs (three per record, column and component; a product sum added to the
// accumulator takes four).
// A row's sum is the sum, in order, of the partial sums of SEG equal runs of its
// records.  With few columns a warp takes several runs at once, one per group of
// C lanes, and several rows; the order of the sum, and so the result, does not
// depend on how many right-hand sides are in the call.
template <typename T> __device__ __forceinline__ T ld_col(const T *p) {
    if constexpr (is_df<T>) {
        const float2 u = __ldg(reinterpret_cast<const float2 *>(p));
        return df(u.x, u.y);
    } else {
        return __ldg(p);
    }
}
__device__ __forceinline__ void col_acc(double &acc, double b, double x) { acc = ::fma(b, x, acc); }
__device__ __forceinline__ void col_acc(df &acc, df b, df x) { df_acc(acc, b, x); }
__device__ __forceinline__ double col_sum(double a, double b) { return a + b; }
// unnormalised: exact two-sum of the high parts, its error and the low parts in the low part
__device__ __forceinline__ df col_sum(df a, df b) { return df_qadd(a, b); }
__device__ __forceinline__ double col_val(double a) { return a; }
__device__ __forceinline__ df col_val(df a) { return df_norm(a); }

// Lane of a row's team: G groups of C lanes, 32 / (G C) rows per warp while C <= 16
// (J = 1); above, one row, one group and J column sets.
template <int J, int G> struct ColLane {
    int row, rpw, g;   // row of the warp's rpw rows, group
    int32_t c[J];      // columns (lanes beyond the last column repeat a valid one)
    bool col[J], on;   // column exists; lane belongs to a row
    __device__ __forceinline__ ColLane(int32_t C, int32_t slab0, int lane) {
        static_assert(J == 1 || G == 1, "one column per lane in a group");
        if (J == 1 && C <= 16) {
            rpw = 32 / (G * C);
            row = lane / (G * C);
            g = (lane - row * G * C) / C;
            c[0] = lane - (row * G + g) * C;
            on = row < rpw;
            col[0] = on;
        } else {
            row = g = 0;
            rpw = 1;
            on = true;
#pragma unroll
            for (int j = 0; j < J; ++j) {
                col[j] = slab0 + lane + 32 * j < C;
                c[j] = col[j] ? slab0 + lane + 32 * j : slab0 + (lane & 1);
            }
        }
    }
};
// rows per warp of such a team
template <int J, int G> int cols_rpw(int32_t R) { return J == 1 && R <= 8 ? 32 / (G * 2 * R) : 1; }

// v[a][j] = sum over row [e0, e1) of sum_b rec.b[3a+b] X[col][b][c[j]], in the
// order described above, in the lanes of group 0.  Every lane of the warp calls.
template <typename T, int J, int G, int SEG, int UNR>
__device__ __forceinline__ void gather_cols(const Rec<T> *__restrict__ rec, int64_t e0, int64_t e1,
                                            const T *__restrict__ X, int32_t C, const ColLane<J, G> &l, int lane,
                                            T (&v)[3][J]) {
    constexpr int PER = SEG / G;      // runs per group
    static_assert(PER * G == SEG, "runs divide among the groups");
    const int64_t ld = 3 * int64_t(C);
    const int64_t len = e1 - e0;
    T part[G == 1 ? 1 : PER][3][J];   // G > 1: kept apart until the groups are joined
#pragma unroll(G == 1 ? 1 : PER)
    for (int q = 0; q < PER; ++q) {
        T acc[3][J];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int j = 0; j < J; ++j) acc[a][j] = T(0.0);
        const int s = l.g * PER + q;
        const int64_t b0 = e0 + len * s / SEG, b1 = e0 + len * (s + 1) / SEG;
#pragma unroll UNR
        for (int64_t e = b0; e < b1; ++e) {
            T b[9];
            const int64_t col = load_rec<T>(rec + e, b);
            const T *x = X + col * ld;
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const T x0 = ld_col(x + l.c[j]), x1 = ld_col(x + C + l.c[j]), x2 = ld_col(x + 2 * C + l.c[j]);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    col_acc(acc[a][j], b[3 * a], x0);
                    col_acc(acc[a][j], b[3 * a + 1], x1);
                    col_acc(acc[a][j], b[3 * a + 2], x2);
                }
            }
        }
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int j = 0; j < J; ++j) {
                if constexpr (G == 1) v[a][j] = q == 0 ? acc[a][j] : col_sum(v[a][j], acc[a][j]);
                else part[q][a][j] = acc[a][j];
            }
    }
    if constexpr (G > 1) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            v[a][0] = part[0][a][0];
#pragma unroll
            for (int q = 1; q < PER; ++q) v[a][0] = col_sum(v[a][0], part[q][a][0]);
        }
#pragma unroll 1
        for (int g = 1; g < G; ++g)
#pragma unroll
            for (int q = 0; q < PER; ++q)
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    v[a][0] = col_sum(v[a][0], shfl1(part[q][a][0], (lane + g * C) & 31));
    }
}

// Grid currents as k_project, by real columns: a warp takes its rpw nodes, a
// block 8 warps' worth, grid (node blocks, slabs of 32 J columns).  A node has
// some 20 records: four runs in FP64, which is bound by its pipe (bond wires, 48
// right-hand sides: 3.84 ms, 6.29 with a complex right-hand side per lane; bar, one:
// 16 us, 30 in one run), one in double-float, where starting a run shows (same
// sizes: 1.18 ms in one run, 1.70 in four, 1.51 with complex lanes).
template <typename T> constexpr int kProjSeg = is_f64<T> ? 4 : 1;
constexpr int kTriSeg = 8;   // runs per triangle (about 300 near, 60 grid records)
// shared pitch of a node, 2 x odd: the 8-node reads of the store hit distinct banks
template <typename T, int J> __host__ __device__ constexpr int proj_cols_pitch() { return 3 * 32 * J + 2; }
template <typename T, int J, int G>
__global__ void __launch_bounds__(256) k_project_cols(const int64_t *__restrict__ ptr, const Rec<T> *__restrict__ rec,
                                                      const T *__restrict__ cT, int64_t Ng, int32_t R,
                                                      C<T> *__restrict__ grid) {
    constexpr int SLAB = 32 * J, ROWS = proj_cols_pitch<T, J>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *sm = reinterpret_cast<T *>(smem_raw);   // [8 rpw nodes][pitch]
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t Cn = 2 * R, slab0 = int32_t(blockIdx.y) * SLAB;
    const ColLane<J, G> l(Cn, slab0, lane);
    const int nodes = kProjNodes * l.rpw;
    const int dstep = l.rpw > 1 ? Cn : SLAB, pitch = l.rpw > 1 ? 3 * Cn + 2 : ROWS;
    const int64_t n0 = int64_t(blockIdx.x) * nodes, n = n0 + w * l.rpw + l.row;
    T v[3][J];
    const bool act = l.on && n < Ng;
    gather_cols<T, J, G, kProjSeg<T>, 1>(rec, act ? ptr[n] : 0, act ? ptr[n + 1] : 0, cT, Cn, l, lane, v);
    if (l.on && l.g == 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int j = 0; j < J; ++j)
                if (l.col[j]) sm[(w * l.rpw + l.row) * pitch + a * dstep + (l.c[j] - slab0)] = col_val(v[a][j]);
    }
    __syncthreads();
    const int nr = min(SLAB, Cn - slab0) / 2;   // right-hand sides of the slab
    for (int i = threadIdx.x; i < 3 * nr * nodes; i += blockDim.x) {
        const int row = i / nodes, nd = i - row * nodes;
        const int d = row / nr, rl = row - d * nr;
        const int64_t nn = n0 + nd;
        if (nn < Ng)
            grid[(int64_t(d) * R + slab0 / 2 + rl) * Ng + nn] =
                *reinterpret_cast<const C<T> *>(sm + nd * pitch + d * dstep + 2 * rl);
    }
}

// ---- FP32 gathers of few right-hand sides (C = 2R <= 32 columns): a lane owns
// a real column of a row, up to 5 right-hand sides one output component of it
// (COMP), and a warp takes several rows, where the wider form gives a warp one
// row and leaves 32 - R lanes idle.  Each lane sums its row's records in order
// with the wider form's expression, so the result is the same bit for bit at
// every number of right-hand sides.
// With little arithmetic per record these kernels are bound by their loads: by
// latency on a small mesh (a row is a chain of record, then the operand it
// names: U records are in flight and the next U columns are fetched a chunk ahead,
// which leaves one round trip per chunk), by L1 wavefronts on a larger one (a
// warp's load takes one per row and 128 bytes, however few lanes it serves).
// Hence the operand's layout: the three components of a column are one 16-byte
// load (float4 [row][C]).
constexpr int kSmallWarps = 2;   // warps per block: a small mesh still reaches every SM

template <int U>   // COMP: output component a of column c
__device__ __forceinline__ void gather_row(const Rec<float> *__restrict__ rec, int64_t e0, int64_t e1,
                                           const float4 *__restrict__ X, int32_t C, int32_t c, int a,
                                           float (&acc)[1]) {
    const int n = int(e1 - e0);
    if (n <= 0) return;
    constexpr int W = sizeof(Rec<float>) / 4;   // words per record: b[9], column
    const float *v = rec[e0].b;
    X += c;
    int32_t cn[U];
#pragma unroll
    for (int u = 0; u < U; ++u) cn[u] = __float_as_int(__ldg(v + W * int64_t(min(u, n - 1)) + 9));
    for (int i = 0; i < n; i += U) {
        float b0[U], b1[U], b2[U];
        float4 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            x[u] = __ldg(X + int64_t(cn[u]) * C);
            const float *r = v + W * int64_t(min(i + u, n - 1)) + 3 * a;
            b0[u] = __ldg(r);
            b1[u] = __ldg(r + 1);
            b2[u] = __ldg(r + 2);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) cn[u] = __float_as_int(__ldg(v + W * int64_t(min(i + U + u, n - 1)) + 9));
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u < n) acc[0] += b0[u] * x[u].x + b1[u] * x[u].y + b2[u] * x[u].z;
    }
}
template <int U>   // all three components of column c
__device__ __forceinline__ void gather_row(const Rec<float> *__restrict__ rec, int64_t e0, int64_t e1,
                                           const float4 *__restrict__ X, int32_t C, int32_t c, int,
                                           float (&acc)[3]) {
    const int n = int(e1 - e0);
    if (n <= 0) return;
    const float4 *v = reinterpret_cast<const float4 *>(rec + e0);
    auto tail = [&](int i) {   // b[8] and the column
        return __ldg(reinterpret_cast<const float2 *>(v + 3 * int64_t(min(i, n - 1)) + 2));
    };
    X += c;
    float2 bn[U];
#pragma unroll
    for (int u = 0; u < U; ++u) bn[u] = tail(u);
    for (int i = 0; i < n; i += U) {
        float4 u0[U], u1[U], x[U];
        float b8[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            b8[u] = bn[u].x;
            x[u] = __ldg(X + int64_t(__float_as_int(bn[u].y)) * C);
            const float4 *r = v + 3 * int64_t(min(i + u, n - 1));
            u0[u] = __ldg(r);
            u1[u] = __ldg(r + 1);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) bn[u] = tail(i + U + u);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u < n) {
                acc[0] += u0[u].x * x[u].x + u0[u].y * x[u].y + u0[u].z * x[u].z;
                acc[1] += u0[u].w * x[u].x + u1[u].x * x[u].y + u1[u].y * x[u].z;
                acc[2] += u1[u].z * x[u].x + u1[u].w * x[u].y + b8[u] * x[u].z;
            }
    }
}
// lane of a warp of rpw rows: row, output component (0 without COMP) and column
template <bool COMP> struct SmallLane {
    int row, a;
    int32_t c;
    __device__ __forceinline__ SmallLane(int32_t C, int lane) {
        const int per = COMP ? 3 * C : C;
        row = lane / per;
        a = (lane - row * per) / C;
        c = lane - row * per - a * C;
    }
};

// Grid currents (k_project) of few right-hand sides: rpw nodes per warp.
template <bool COMP>
__global__ void __launch_bounds__(32 * kSmallWarps)
    k_project_small(const int64_t *__restrict__ ptr, const Rec<float> *__restrict__ rec, const float4 *__restrict__ cT,
                    int64_t Ng, int32_t R, int rpw, float2 *__restrict__ grid) {
    constexpr int NA = COMP ? 1 : 3;
    extern __shared__ __align__(16) float smf[];   // [nodes][pitch]
    const int w = threadIdx.x >> 5;
    const int32_t Cn = 2 * R;
    const SmallLane<COMP> l(Cn, threadIdx.x & 31);
    const int nodes = kSmallWarps * rpw, pitch = 3 * Cn + 2;
    const int64_t n0 = int64_t(blockIdx.x) * nodes, n = n0 + w * rpw + l.row;
    if (l.row < rpw) {
        float acc[NA] = {};
        if (n < Ng) gather_row<4>(rec, ptr[n], ptr[n + 1], cT, Cn, l.c, l.a, acc);
#pragma unroll
        for (int a = 0; a < NA; ++a) smf[(w * rpw + l.row) * pitch + (l.a + a) * Cn + l.c] = acc[a];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * R * nodes; i += blockDim.x) {
        const int q = i / nodes, nd = i - q * nodes;   // q = d R + r
        if (n0 + nd < Ng)
            grid[int64_t(q) * Ng + n0 + nd] = *reinterpret_cast<const float2 *>(smf + nd * pitch + 2 * q);
    }
}

// k_tri_gather of few right-hand sides (mixed form): re and im of a right-hand
// side sit in neighbouring lanes, each forming its half of Eq. Zb.
template <bool COMP>
__global__ void __launch_bounds__(32 * kSmallWarps)
    k_tri_small(const int64_t *__restrict__ near_ptr, const Rec<float> *__restrict__ near_rec,
                const int64_t *__restrict__ pt_ptr, const Rec<float> *__restrict__ pt_rec,
                const float4 *__restrict__ cT, const float4 *__restrict__ phiT, const double *__restrict__ gram,
                const int32_t *__restrict__ cond, const float2 *__restrict__ coef_dd, int ncond, int64_t nt,
                int32_t R, int rpw, float4 *__restrict__ y_tri) {
    constexpr int NA = COMP ? 1 : 3, U = COMP ? 8 : 6;
    const int64_t gw = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int32_t Cn = 2 * R;
    const SmallLane<COMP> l(Cn, lane);
    const bool act = l.row < rpw && gw * rpw + l.row < nt;
    const int64_t t = act ? gw * rpw + l.row : 0;
    float acc[NA] = {};
    if (act) {
        gather_row<U>(near_rec, near_ptr[t], near_ptr[t + 1], cT, Cn, l.c, l.a, acc);
        gather_row<U>(pt_rec, pt_ptr[t], pt_ptr[t + 1], phiT, Cn, l.c, l.a, acc);
    }
    const float4 x = cT[t * Cn + l.c];
    const int cd = cond[t], im = l.c & 1;
    const int32_t r = l.c >> 1;
    const float2 *cf = coef_dd + int64_t(r) * (2 * ncond + 1);
    const float2 zr = cf[2 * cd], zi = cf[2 * cd + 1], cl = cf[2 * ncond];
    const DD Zr{zr.x, zr.y}, Zi{zi.x, zi.y}, Cl{cl.x, cl.y};
#pragma unroll
    for (int a = 0; a < NA; ++a) {
        const int k = l.a + a;
        const double *gm = gram + 9 * t + 3 * k;
        const float G0 = float(__ldg(gm)), G1 = float(__ldg(gm + 1)), G2 = float(__ldg(gm + 2));
        const float g = G0 * x.x + G1 * x.y + G2 * x.z;
        const float go = shfl1(g, lane ^ 1), fo = shfl1(acc[a], lane ^ 1);
        // re = zr gr - zi gi - cl fi,  im = zr gi + zi gr + cl fr (the sums of dd_zb)
        const DD zg = dd_mul(Zi, go), cfo = dd_mul(Cl, DD{fo, 0.f});
        const DD y = dd_add(dd_add(dd_mul(Zr, g), im ? zg : dd_neg(zg)), im ? cfo : dd_neg(cfo));
        if (act) reinterpret_cast<float2 *>(y_tri + (int64_t(r) * nt + t) * 3 + k)[im] = make_float2(y.hi, y.lo);
    }
}

// Grid potentials as float4 [node][2R] (k_regroup for few right-hand sides): one
// thread per (right-hand side, node of a tile with stencil nodes).
__global__ void __launch_bounds__(256) k_regroup_small(const float2 *__restrict__ grid,
                                                       const int32_t *__restrict__ tiles, int64_t n_tiles, int64_t Ng,
                                                       int32_t R, float4 *__restrict__ phiT) {
    const int64_t w = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    if (w >= n_tiles * R) return;
    const int64_t r = w % R, n = int64_t(tiles[w / R]) * 32 + (threadIdx.x & 31);
    if (n >= Ng) return;
    float2 v[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) v[d] = grid[(int64_t(d) * R + r) * Ng + n];
    float4 *o = phiT + (n * R + r) * 2;
    o[0] = make_float4(v[0].x, v[1].x, v[2].x, 0.f);
    o[1] = make_float4(v[0].y, v[1].y, v[2].y, 0.f);
}

// Grid currents (Eq. Projection) of the mixed form by node chunks whose
// triangles' local currents are staged in shared memory: one CTA per (chunk,
// slab of kChunkRhs right-hand sides).  The rows c_T [T][3][R] of the chunk's
// triangles are read once per slab (coalesced 256-byte rows) instead of once
// per (node, triangle) record, which the direct form reads through L2 (a
// triangle has about 57 stencil nodes); each warp then takes one node at a
// time, lanes over right-hand sides, sums its records in order (the sums of
// k_project) from the staged rows named by the records' chunk-local indices,
// and groups of 8 nodes pass through shared memory so that each grid row
// [d][r] gets runs of consecutive nodes (a tile's z extent is 8).
constexpr int kPTRows = 3 * kChunkRhs + 2;   // staging pitch: the 8-node reads hit distinct banks
constexpr size_t kPTSmem = size_t(kChunkTri) * 3 * kChunkRhs * sizeof(float2) + size_t(8) * kPTRows * sizeof(float2);

__global__ void __launch_bounds__(256, 4)
    k_project_tiled(const int32_t *__restrict__ node_ptr, const int32_t *__restrict__ nodes,
                    const int32_t *__restrict__ tri_ptr, const int32_t *__restrict__ tri,
                    const int64_t *__restrict__ pn_ptr, const Rec<float> *__restrict__ rec,
                    const uint16_t *__restrict__ lcol, const float2 *__restrict__ cT, int64_t Ng, int32_t R,
                    float2 *__restrict__ grid) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *X = reinterpret_cast<float2 *>(smem_raw);   // [kChunkTri][3][kChunkRhs]
    float2 *O = X + kChunkTri * 3 * kChunkRhs;         // [8][kPTRows]
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t c = blockIdx.x;
    const int32_t r0 = int32_t(blockIdx.y) * kChunkRhs;
    const int32_t nr = min(kChunkRhs, R - r0);
    const int32_t t0 = tri_ptr[c], nT = tri_ptr[c + 1] - t0;
    // staging by asynchronous 8-byte copies, all in flight at once (lanes beyond
    // the slab's last right-hand side copy nothing and zero-fill)
    for (int i = w; i < 3 * nT; i += 8) {
        const int32_t t = tri[t0 + i / 3];
        const int l = i - 3 * (i / 3);
        const bool in = lane < nr;
        const float2 *src = cT + (int64_t(t) * 3 + l) * R + r0 + (in ? lane : 0);
        const uint32_t dst = uint32_t(__cvta_generic_to_shared(X + i * kChunkRhs + lane));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(in ? 8 : 0)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;\n cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const int32_t n0 = node_ptr[c], nN = node_ptr[c + 1] - n0;
    for (int32_t g = 0; g < nN; g += 8) {
        float2 acc[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) acc[d] = make_float2(0.f, 0.f);
        if (g + w < nN) {
            const int64_t n = nodes[n0 + g + w];
#pragma unroll 2
            for (int64_t e = pn_ptr[n]; e < pn_ptr[n + 1]; ++e) {
                float b[9];
                load_rec<float>(rec + e, b);
                const float2 *x = X + int(__ldg(lcol + e)) * (3 * kChunkRhs) + lane;
                const float2 x0 = x[0], x1 = x[kChunkRhs], x2 = x[2 * kChunkRhs];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    acc[a].x += b[3 * a] * x0.x + b[3 * a + 1] * x1.x + b[3 * a + 2] * x2.x;
                    acc[a].y += b[3 * a] * x0.y + b[3 * a + 1] * x1.y + b[3 * a + 2] * x2.y;
                }
            }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) O[w * kPTRows + d * kChunkRhs + lane] = acc[d];
        __syncthreads();
        for (int i = threadIdx.x; i < 3 * kChunkRhs * 8; i += 256) {
            const int row = i >> 3, nd = i & 7;
            const int d = row / kChunkRhs, r = row - d * kChunkRhs;
            if (r < nr && g + nd < nN)
                grid[(int64_t(d) * R + r0 + r) * Ng + nodes[n0 + g + nd]] = O[nd * kPTRows + row];
        }
        __syncthreads();
    }
}

// Grid potentials regrouped with the right-hand sides innermost:
// phiT[n][b] = grid[b][n], b = d R + r, for the 32-node tiles that hold a
// stencil node (no other node is interpolated from).
template <typename T>
__global__ void __launch_bounds__(256) k_regroup(const C<T> *__restrict__ grid, const int32_t *__restrict__ tiles,
                                                 int64_t Ng, int32_t B, C<T> *__restrict__ phiT) {
    __shared__ C<T> s[32][33];
    const int64_t n0 = int64_t(tiles[blockIdx.x]) * 32;
    const int32_t b0 = int32_t(blockIdx.y) * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
    for (int i = ty; i < 32; i += 8) {
        const int32_t b = b0 + i;
        const int64_t n = n0 + tx;
        if (b < B && n < Ng) s[i][tx] = grid[int64_t(b) * Ng + n];
    }
    __syncthreads();
#pragma unroll
    for (int i = ty; i < 32; i += 8) {
        const int64_t n = n0 + i;
        const int32_t b = b0 + tx;
        if (b < B && n < Ng) phiT[n * B + b] = s[tx][i];
    }
}

// y_T[k] = Z_s sum_l G_T[k][l] c_T[l] + j c_L f_T[k] (Eq. Zb) for the right-hand
// sides rl + 32 V j + v < R of a warp's slab, f_T = acc (FP64, or double-float
// from the FP32 field in the mixed form).
template <typename T, int V, int J>
__device__ __forceinline__ void tri_epilogue(const C<T> (&acc)[3][J][V], int64_t t, int32_t rl, int32_t R,
                                             const C<T> *__restrict__ cT, const double *__restrict__ gram,
                                             const int32_t *__restrict__ cond, const double *__restrict__ coef,
                                             const float2 *__restrict__ coef_dd, int ncond, int64_t nt,
                                             TourE<T> *__restrict__ y_tri) {
    const int cd = cond[t];
    if constexpr (is_f32<T>) {
        // mixed form: Gram term in FP32 like the field, Eq. Zb in double-float
        float G[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) G[i] = float(__ldg(gram + 9 * t + i));
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int32_t r = rl + 32 * V * j + v;
                if (r >= R) continue;
                const float2 *cf = coef_dd + int64_t(r) * (2 * ncond + 1);
                const float2 zr = cf[2 * cd], zi = cf[2 * cd + 1], cl = cf[2 * ncond];
                float2 c[3];
#pragma unroll
                for (int l = 0; l < 3; ++l) c[l] = cT[(t * 3 + l) * R + r];
                float4 *out = y_tri + (int64_t(r) * nt + t) * 3;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float gr = G[3 * k] * c[0].x + G[3 * k + 1] * c[1].x + G[3 * k + 2] * c[2].x;
                    const float gi = G[3 * k] * c[0].y + G[3 * k + 1] * c[1].y + G[3 * k + 2] * c[2].y;
                    out[k] = dd_zb(zr, zi, cl, gr, gi, DD{acc[k][j][v].x, 0.f}, DD{acc[k][j][v].y, 0.f});
                }
            }
    } else {
        double G[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) G[i] = __ldg(gram + 9 * t + i);
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int32_t r = rl + 32 * V * j + v;
                if (r >= R) continue;
                const double *cf = coef + int64_t(r) * (2 * ncond + 1);
                const double zr = cf[2 * cd], zi = cf[2 * cd + 1], cl = cf[2 * ncond];
                double2 c[3];
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    const C<T> u = cT[(t * 3 + l) * R + r];
                    c[l] = make_double2(double(u.x), double(u.y));
                }
                double2 *out = y_tri + (int64_t(r) * nt + t) * 3;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const double gr = G[3 * k] * c[0].x + G[3 * k + 1] * c[1].x + G[3 * k + 2] * c[2].x;
                    const double gi = G[3 * k] * c[0].y + G[3 * k + 1] * c[1].y + G[3 * k + 2] * c[2].y;
                    const double fr = double(acc[k][j][v].x), fi = double(acc[k][j][v].y);
                    // Z_s * gram + j c_L * f
                    out[k] = make_double2(zr * gr - zi * gi - cl * fi, zr * gi + zi * gr + cl * fr);
                }
            }
    }
}

// Per triangle T and right-hand side r:
//   f_T[k] = sum_{T' near T} sum_l L_d(T,T')[k][l] c_T'[l]          (Eq. Lb, pre-corrected)
//          + sum_n sum_d W(n,T)[d][k] phi_g[d][n]                   (interpolation, I = B^T)
//   y_T[k] = Z_s sum_l G_T[k][l] c_T[l] + j c_L f_T[k]             (Eq. Zb, FP64)
// One warp per (T, slab of 32 V J right-hand sides), lanes over right-hand
// sides; each block record is read once per slab.  y_tri layout [R][nt][3].
template <typename T, int V, int J>
__global__ void __launch_bounds__(256)
    k_tri_gather(const int64_t *__restrict__ near_ptr, const Rec<T> *__restrict__ near_rec,
                 const int64_t *__restrict__ pt_ptr, const Rec<T> *__restrict__ pt_rec, const C<T> *__restrict__ cT,
                 const C<T> *__restrict__ phiT, const double *__restrict__ gram, const int32_t *__restrict__ cond,
                 const double *__restrict__ coef, const float2 *__restrict__ coef_dd, int ncond, int64_t nt,
                 int32_t R, int32_t nslab, TourE<T> *__restrict__ y_tri) {
    constexpr int SLAB = 32 * V * J;
    const int64_t gw = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (gw >= nt * nslab) return;
    const int64_t t = gw / nslab;
    const int32_t rbase = int32_t(gw % nslab) * SLAB;
    const int32_t rl = rbase + V * lane;
    C<T> acc[3][J][V];
    zero<T, V, J>(acc);
    if (rbase + SLAB <= R) {
        gather_rows<T, V, J, true>(near_rec, near_ptr[t], near_ptr[t + 1], cT, R, rl, acc);
        gather_rows<T, V, J, true>(pt_rec, pt_ptr[t], pt_ptr[t + 1], phiT, R, rl, acc);
    } else {
        gather_rows<T, V, J, false>(near_rec, near_ptr[t], near_ptr[t + 1], cT, R, rl, acc);
        gather_rows<T, V, J, false>(pt_rec, pt_ptr[t], pt_ptr[t + 1], phiT, R, rl, acc);
    }
    tri_epilogue<T, V, J>(acc, t, rl, R, cT, gram, cond, coef, coef_dd, ncond, nt, y_tri);
}

// k_tri_gather by real columns (FP64 and double-float): a warp takes its rpw
// triangles and a slab of 32 J columns.  Column c = 2 r + p holds the real
// (p = 0) or imaginary (p = 1) part of right-hand side r, so the two halves of a
// complex product sit in neighbouring lanes: each lane forms its own half of
// Eq. Zb from its Gram term and its neighbour's.
// FP64 on the bond wires (40k triangles, 14.1M records), 48 right-hand sides:
// 20.3 ms, 96 % of the FP64 pipe (98 % in a capture on 20k triangles), against 38.6 ms with a complex right-hand side
// per lane (48 of 64 lanes, four operations per term); 20k triangles, 8
// right-hand sides: 1.71 against 9.06 ms; 1.5k triangles, one: 44 against 843 us.
// Double-float on the 40k triangles, 16: 2.37 against 3.65 ms.
template <typename T, int J, int G>
__global__ void __launch_bounds__(256)
    k_tri_cols(const int64_t *__restrict__ near_ptr, const Rec<T> *__restrict__ near_rec,
               const int64_t *__restrict__ pt_ptr, const Rec<T> *__restrict__ pt_rec, const T *__restrict__ cT,
               const T *__restrict__ phiT, const double *__restrict__ gram, const int32_t *__restrict__ cond,
               const double *__restrict__ coef, const float2 *__restrict__ coef_dd, int ncond, int64_t nt, int32_t R,
               int32_t nslab, TourE<T> *__restrict__ y_tri) {
    const int64_t gw = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int32_t Cn = 2 * R, slab0 = int32_t(gw % nslab) * 32 * J;
    const ColLane<J, G> l(Cn, slab0, lane);
    const int64_t t0 = gw / nslab * l.rpw;
    if (t0 >= nt) return;
    const bool act = l.on && t0 + l.row < nt;
    const int64_t t = act ? t0 + l.row : t0;
    T acc[3][J], far[3][J];
    gather_cols<T, J, G, kTriSeg, 2>(near_rec, near_ptr[t], near_ptr[t + 1], cT, Cn, l, lane, acc);
    gather_cols<T, J, G, kTriSeg, 2>(pt_rec, pt_ptr[t], pt_ptr[t + 1], phiT, Cn, l, lane, far);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int j = 0; j < J; ++j) acc[a][j] = col_sum(acc[a][j], far[a][j]);
    const int cd = cond[t];
    const int im = lane & 1;   // C is even and slabs start at multiples of 32: lane and column parity agree
    T gm[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const double v = __ldg(gram + 9 * t + i);
        if constexpr (is_df<T>) {
            const DD d = dd_from(v);
            gm[i] = df(d.hi, d.lo);
        } else {
            gm[i] = v;
        }
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const T *x = cT + t * 3 * Cn + l.c[j];
        const T x0 = ld_col(x), x1 = ld_col(x + Cn), x2 = ld_col(x + 2 * Cn);
        const int32_t r = l.c[j] >> 1;
        const bool out_on = act && l.g == 0 && l.col[j];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const T f = col_val(acc[k][j]);
            if constexpr (is_df<T>) {
                DD g = dd_mul(to_dd(gm[3 * k]), to_dd(x0));
                g = dd_add(g, dd_mul(to_dd(gm[3 * k + 1]), to_dd(x1)));
                g = dd_add(g, dd_mul(to_dd(gm[3 * k + 2]), to_dd(x2)));
                const df go = shfl1(df(g.hi, g.lo), lane ^ 1), fo = shfl1(f, lane ^ 1);
                if (out_on) {
                    const float2 *cf = coef_dd + int64_t(r) * (2 * ncond + 1);
                    const float2 zr = cf[2 * cd], zi = cf[2 * cd + 1], cl = cf[2 * ncond];
                    // re = zr gr - zi gi - cl fi,  im = zr gi + zi gr + cl fr
                    const DD o = dd_add(dd_mul(DD{zi.x, zi.y}, to_dd(go)), dd_mul(DD{cl.x, cl.y}, to_dd(fo)));
                    const DD y = dd_add(dd_mul(DD{zr.x, zr.y}, g), im ? o : dd_neg(o));
                    reinterpret_cast<float2 *>(y_tri + (int64_t(r) * nt + t) * 3 + k)[im] = make_float2(y.hi, y.lo);
                }
            } else {
                const double g = ::fma(gm[3 * k + 2], x2, ::fma(gm[3 * k + 1], x1, gm[3 * k] * x0));
                const double go = shfl1(g, lane ^ 1), fo = shfl1(f, lane ^ 1);
                if (out_on) {
                    const double *cf = coef + int64_t(r) * (2 * ncond + 1);
                    const double zr = cf[2 * cd], zi = cf[2 * cd + 1], cl = cf[2 * ncond];
                    const double o = ::fma(cl, fo, zi * go);
                    reinterpret_cast<double *>(y_tri + (int64_t(r) * nt + t) * 3 + k)[im] =
                        ::fma(zr, g, im ? o : -o);
                }
            }
        }
    }
}

// The lossy kernel (pfft_params.kernel = SIE_KERNEL_LOSSY): as k_tri_gather with
// complex near blocks that depend on the frequency,
//   f_T[k] = sum_{T' near T} sum_l L_d,k(w_r)(T,T')[k][l] c_T'[l]
//          + sum_n sum_d W(n,T)[d][k] phi_g[d][n],
// Ltab[rslot[r]] being the blocks [n_near][3][3] of right-hand side r's
// frequency.  One warp per (T, slab of 32 J right-hand sides), one right-hand
// side per lane and load; lanes of one frequency read the same block.
template <typename T, int J>
__global__ void __launch_bounds__(256)
    k_tri_gather_lossy(const int64_t *__restrict__ near_ptr, const int32_t *__restrict__ near_col,
                       const C<T> *const *__restrict__ Ltab, const int32_t *__restrict__ rslot,
                       const int64_t *__restrict__ pt_ptr, const Rec<T> *__restrict__ pt_rec,
                       const C<T> *__restrict__ cT, const C<T> *__restrict__ phiT, const double *__restrict__ gram,
                       const int32_t *__restrict__ cond, const double *__restrict__ coef,
                       const float2 *__restrict__ coef_dd, int ncond, int64_t nt, int32_t R, int32_t nslab,
                       TourE<T> *__restrict__ y_tri) {
    constexpr int SLAB = 32 * J;
    const int64_t gw = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (gw >= nt * nslab) return;
    const int64_t t = gw / nslab;
    const int32_t rl = int32_t(gw % nslab) * SLAB + lane;
    C<T> acc[3][J][1];
    zero<T, 1, J>(acc);
    const C<T> *L[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int32_t r = rl + 32 * j;
        L[j] = r < R ? Ltab[rslot[r]] : nullptr;
    }
    const int64_t ld = 3 * int64_t(R);
    for (int64_t e = near_ptr[t]; e < near_ptr[t + 1]; ++e) {
        const C<T> *x = cT + int64_t(near_col[e]) * ld;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int32_t r = rl + 32 * j;
            if (r >= R) continue;
            const C<T> x0 = x[r], x1 = x[R + r], x2 = x[2 * R + r];
            const C<T> *b = L[j] + 9 * e;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const C<T> b0 = b[3 * k], b1 = b[3 * k + 1], b2 = b[3 * k + 2];
                acc[k][j][0].x += b0.x * x0.x - b0.y * x0.y + b1.x * x1.x - b1.y * x1.y + b2.x * x2.x - b2.y * x2.y;
                acc[k][j][0].y += b0.x * x0.y + b0.y * x0.x + b1.x * x1.y + b1.y * x1.x + b2.x * x2.y + b2.y * x2.x;
            }
        }
    }
    gather_rows<T, 1, J, false>(pt_rec, pt_ptr[t], pt_ptr[t + 1], phiT, R, rl, acc);
    tri_epilogue<T, 1, J>(acc, t, rl, R, cT, gram, cond, coef, coef_dd, ncond, nt, y_tri);
}

// Interpolated far field alone (mixed form, where the near blocks run on the
// tensor cores): ffar[T][k][r] = sum_n sum_d W(n,T)[d][k] phi_g[d][n].
template <typename T, int V, int J>
__global__ void __launch_bounds__(256)
    k_far_gather(const int64_t *__restrict__ pt_ptr, const Rec<T> *__restrict__ pt_rec,
                 const C<T> *__restrict__ phiT, int64_t nt, int32_t R, int32_t nslab, C<T> *__restrict__ ffar) {
    constexpr int SLAB = 32 * V * J;
    const int64_t gw = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (gw >= nt * nslab) return;
    const int64_t t = gw / nslab;
    const int32_t rbase = int32_t(gw % nslab) * SLAB;
    const int32_t rl = rbase + V * lane;
    C<T> acc[3][J][V];
    zero<T, V, J>(acc);
    if (rbase + SLAB <= R) gather_rows<T, V, J, true>(pt_rec, pt_ptr[t], pt_ptr[t + 1], phiT, R, rl, acc);
    else gather_rows<T, V, J, false>(pt_rec, pt_ptr[t], pt_ptr[t + 1], phiT, R, rl, acc);
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int32_t r = rl + 32 * V * j;
        if (r < R)
#pragma unroll
            for (int k = 0; k < 3; ++k) stv<T, V>(ffar + (t * 3 + k) * R + r, acc[k][j]);
    }
}

// y_b = sum over the branch's two triangles of s * y_T[k]; EO is the output
// element (complex128 for a branch-space result).
template <typename E, typename EO>
__global__ void k_branch_out(const E *__restrict__ y_tri, const int32_t *__restrict__ br_tri,
                             const int8_t *__restrict__ br_local, int64_t nt, int64_t nb, int64_t ldy, int32_t nrhs,
                             EO *__restrict__ y) {
    int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= ldy * nrhs) return;
    int64_t r, b;
    divmod(i, ldy, r, b);
    E v = ezero<E>();
    if (b < nb) {
        const E a = y_tri[(r * nt + br_tri[2 * b]) * 3 + br_local[2 * b]];
        const E c = y_tri[(r * nt + br_tri[2 * b + 1]) * 3 + br_local[2 * b + 1]];
        v = eadd(a, eneg(c));
    }
    EO o;
    eset(o, v);
    y[i] = o;
}

// Loop voltage: its link's plus psi(head) - psi(tail), psi the prefix sums P.
template <typename E>
__global__ void k_loop_out(const E *__restrict__ y_br, int64_t ldy, const E *__restrict__ P, int64_t nslots,
                           const int4 *__restrict__ loop_dst, int64_t nl, int32_t nrhs, double2 *__restrict__ y) {
    int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= nl * nrhs) return;
    int64_t r, l;
    divmod(i, nl, r, l);
    const int4 d = __ldg(loop_dst + l);
    const E *row = P + r * nslots;
    E v = y_br[r * ldy + d.x];
    v = eadd(v, row[d.y]);
    v = eadd(v, eneg(row[d.z]));
    double2 o;
    eset(o, v);
    y[i] = o;
}

// Post-processing (Eq. CurT): current of every mesh branch, grid (branches, right-hand sides).
__global__ void k_branch_alpha(const double2 *__restrict__ x, int64_t nl, const double2 *__restrict__ P,
                               int64_t nslots, const int4 *__restrict__ branch_src, int64_t nb,
                               double2 *__restrict__ alpha) {
    const int64_t b = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const int64_t r = blockIdx.y;
    alpha[r * nb + b] = branch_current<double>(branch_src[b], r, x, nl, P, nslots);
}

// Post-processing: panel potential = root-path sum of the panel's node minus that
// of its conductor's reference node, grid (panels, right-hand sides).
__global__ void k_panel_phi(const double2 *__restrict__ P, int64_t nslots, const int32_t *__restrict__ slot,
                            const int32_t *__restrict__ ref, int64_t nt, double2 *__restrict__ phi) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    const int64_t r = blockIdx.y;
    const double2 *row = P + r * nslots;
    phi[r * nt + t] = csub(row[slot[t]], row[ref[t]]);
}

inline unsigned nblk(int64_t n, int t = 256) { return unsigned((n + t - 1) / t); }

}  // namespace

namespace sie {

// Grows the matvec scratch to hold nrhs right-hand sides in precision `prec`.
// Buffers only grow: a plan used in both precisions keeps FP64-sized buffers
// (the mixed form reads them as complex64) and the mixed form's far-field
// buffer, so alternating precisions (iterative refinement) never reallocates.
int scratch_reserve(pfft_plan *p, int32_t nrhs, int prec) {
    Scratch &s = p->scr;
    // complex values of the field steps: complex64 in the mixed form, 16 bytes
    // (complex128 or complex double-float) otherwise
    const bool mixed = prec == SIE_PREC_MIXED;
    const int want_cs = mixed ? int(sizeof(float2)) : int(sizeof(double2));
    if (s.cap_rhs >= nrhs && s.cs >= want_cs && (!mixed || s.ffar)) return SIE_OK;
    const int64_t R = std::max<int64_t>({int64_t(nrhs), int64_t(s.cap_rhs), 1});
    const size_t cs = size_t(std::max(want_cs, s.cs));
    const bool with_far = mixed || s.ffar != nullptr;
    for (void *a : {s.tour, s.part, s.grid, s.spec, s.phiT, s.y_tri, s.y_br, (void *)s.coef, s.cT, s.ffar})
        if (a) cudaFree(a);
    s = Scratch{};
    constexpr int kBufs = 10;
    // bytes per row of the right-hand-sides-inner operands, and of the float4
    // columns that few right-hand sides use instead
    const size_t row = std::max(size_t(R) * 3 * cs, size_t(std::min<int64_t>(R, kSmallRhs)) * 2 * sizeof(float4));
    const size_t sizes[kBufs] = {
        size_t(R) * 2 * p->nn * sizeof(double2),
        size_t(R) * 3 * p->Ng * cs,
        size_t(R) * 3 * p->Mx * (p->Ny + (p->large_plane ? p->My : 0)) * p->Nz * cs,
        row * p->Ng,
        size_t(R) * p->nt * 3 * sizeof(double2),
        size_t(R) * (p->nb + p->np) * sizeof(double2),
        size_t(R) * (2 * p->ncond + 1) * (sizeof(double) + sizeof(float2)),
        row * p->nt,
        with_far ? size_t(R) * p->nt * 3 * sizeof(float2) : 0,
        size_t(R) * ((2 * p->nn + kTourChunk - 1) / kTourChunk) * kTourPart * sizeof(double2)};
    void **dst[kBufs] = {&s.tour, &s.grid, &s.spec, &s.phiT, &s.y_tri, &s.y_br, (void **)&s.coef, &s.cT,
                         &s.ffar, &s.part};
    for (int i = 0; i < kBufs; ++i) {
        if (!sizes[i]) continue;
        cudaError_t e = plan_malloc(p, dst[i], sizes[i]);
        if (e != cudaSuccess) {
            for (int j = 0; j < i; ++j) if (*dst[j]) { cudaFree(*dst[j]); *dst[j] = nullptr; }
            set_error(std::string("scratch allocation failed: ") + cudaGetErrorString(e));
            s = Scratch{};
            return SIE_ERR_OOM;
        }
        s.bytes += sizes[i];
    }
    s.cap_rhs = int32_t(R);
    s.cs = int(cs);
    ++p->scr_gen;
    return SIE_OK;
}

// block records by precision: projection (rows = nodes), interpolation (rows = triangles), near field
template <typename T> const Rec<T> *rec_pn(const pfft_plan *p) {
    if constexpr (is_df<T>) return p->d_pn_recdf;
    else if constexpr (is_f64<T>) return p->d_pn_rec64;
    else return p->d_pn_rec32;
}
template <typename T> const Rec<T> *rec_pt(const pfft_plan *p) {
    if constexpr (is_df<T>) return p->d_pt_recdf;
    else if constexpr (is_f64<T>) return p->d_pt_rec64;
    else return p->d_pt_rec32;
}
template <typename T> const Rec<T> *rec_near(const pfft_plan *p) {
    if constexpr (is_df<T>) return p->d_near_recdf;
    else if constexpr (is_f64<T>) return p->d_near_rec64;
    else return p->d_near_rec32;
}

// Block-sparse stages by real columns (FP64, double-float): J column sets per
// lane, G groups of lanes per row.
template <typename T, int J, int G> struct Cols {
    static int project(pfft_plan *p, int32_t R, cudaStream_t st) {
        constexpr int GP = G < kProjSeg<T> ? G : kProjSeg<T>;
        const int rpw = cols_rpw<J, GP>(R), nodes = kProjNodes * rpw;
        const dim3 grid(unsigned((p->Ng + nodes - 1) / nodes), unsigned((2 * R + 32 * J - 1) / (32 * J)));
        const size_t smem = size_t(nodes) * (rpw > 1 ? 6 * R + 2 : proj_cols_pitch<T, J>()) * sizeof(T);
        k_project_cols<T, J, GP><<<grid, 32 * kProjNodes, smem, st>>>(p->d_pn_ptr, rec_pn<T>(p), (const T *)p->scr.cT,
                                                                  p->Ng, R, (C<T> *)p->scr.grid);
        SIE_LAUNCH_CHECK(p);
        return SIE_OK;
    }
    static int tri_gather(pfft_plan *p, int32_t R, cudaStream_t st) {
        const int32_t nslab = (2 * R + 32 * J - 1) / (32 * J);
        const int rpw = cols_rpw<J, G>(R);
        const int64_t warps = (p->nt + rpw - 1) / rpw * nslab;
        k_tri_cols<T, J, G><<<unsigned((warps * 32 + 255) / 256), 256, 0, st>>>(
            p->d_near_ptr, rec_near<T>(p), p->d_pt_ptr, rec_pt<T>(p), (const T *)p->scr.cT, (const T *)p->scr.phiT,
            p->d_gram, p->d_cond, p->scr.coef, coef_dd(p), p->ncond, p->nt, R, nslab, (TourE<T> *)p->scr.y_tri);
        SIE_LAUNCH_CHECK(p);
        return SIE_OK;
    }
};
// Column sets per lane above 16 right-hand sides.  FP64 takes one: its pipe needs
// 144 cycles per record and set, so reading a record once per set costs nothing
// (bond wires, 48 right-hand sides, near field: 20.2 ms with one, 20.4 with three).  In
// double-float a set's arithmetic (27 cycles) is of the order of the record's
// loads: three or two sets, whichever wastes fewer lanes (6.62, 8.31 and 5.93 ms
// with one, two and three sets, two having a quarter of its lanes idle there).
template <typename T> int col_sets(int32_t R) {
    const int sets = (2 * R + 31) / 32;
    if (is_f64<T> || sets == 1) return 1;
    return (sets + 2) / 3 * 3 <= (sets + 1) / 2 * 2 ? 3 : 2;
}
// Up to 8 right-hand sides the most groups that fit a warp.
#define SIE_COLS_DISPATCH(T, R, CALL)                                       \
    do {                                                                   \
        if ((R) <= 2) return Cols<T, 1, 8>::CALL;                          \
        if ((R) <= 4) return Cols<T, 1, 4>::CALL;                          \
        if ((R) <= 8) return Cols<T, 1, 2>::CALL;                          \
        if constexpr (is_df<T>) {                                          \
            if (col_sets<T>(R) == 2) return Cols<T, 2, 1>::CALL;           \
            if (col_sets<T>(R) == 3) return Cols<T, 3, 1>::CALL;           \
        }                                                                  \
        return Cols<T, 1, 1>::CALL;                                        \
    } while (0)

// Block-sparse stages for one slab shape: V complex per load, J loads per lane
// (mixed form; FP64 for the lossy kernel's gather).
template <typename T, int V, int J> struct Blocks {
    static constexpr int SLAB = 32 * V * J;
    static int project(pfft_plan *p, int32_t R, cudaStream_t st) {
        const dim3 grid(unsigned((p->Ng + kProjNodes - 1) / kProjNodes), unsigned((R + SLAB - 1) / SLAB));
        k_project<T, V, J><<<grid, 32 * kProjNodes, proj_smem<T, V, J>(), st>>>(
            p->d_pn_ptr, rec_pn<T>(p), (const C<T> *)p->scr.cT, p->Ng, R, (C<T> *)p->scr.grid);
        SIE_LAUNCH_CHECK(p);
        return SIE_OK;
    }
    static int far_gather(pfft_plan *p, int32_t R, cudaStream_t st) {
        const int32_t nslab = (R + SLAB - 1) / SLAB;
        const int64_t warps = p->nt * nslab;
        k_far_gather<T, V, J><<<unsigned((warps * 32 + 255) / 256), 256, 0, st>>>(
            p->d_pt_ptr, rec_pt<T>(p), (const C<T> *)p->scr.phiT, p->nt, R, nslab, (C<T> *)p->scr.ffar);
        SIE_LAUNCH_CHECK(p);
        return SIE_OK;
    }
    static int tri_gather_lossy(pfft_plan *p, int32_t R, cudaStream_t st) {
        static_assert(V == 1 && !is_df<T>, "one right-hand side per lane and load; FP64 or mixed");
        const int32_t nslab = (R + SLAB - 1) / SLAB;
        const int64_t warps = p->nt * nslab;
        const int prec = is_f64<T> ? SIE_PREC_FP64 : SIE_PREC_MIXED;
        k_tri_gather_lossy<T, J><<<unsigned((warps * 32 + 255) / 256), 256, 0, st>>>(
            p->d_near_ptr, p->d_near_col, reinterpret_cast<const C<T> *const *>(lossy_ltab(p, prec)),
            lossy_rslot(p), p->d_pt_ptr, rec_pt<T>(p), (const C<T> *)p->scr.cT, (const C<T> *)p->scr.phiT, p->d_gram,
            p->d_cond, p->scr.coef, coef_dd(p), p->ncond, p->nt, R, nslab, (TourE<T> *)p->scr.y_tri);
        SIE_LAUNCH_CHECK(p);
        return SIE_OK;
    }
    static int tri_gather(pfft_plan *p, int32_t R, cudaStream_t st) {
        const int32_t nslab = (R + SLAB - 1) / SLAB;
        const int64_t warps = p->nt * nslab;
        k_tri_gather<T, V, J><<<unsigned((warps * 32 + 255) / 256), 256, 0, st>>>(
            p->d_near_ptr, rec_near<T>(p), p->d_pt_ptr, rec_pt<T>(p), (const C<T> *)p->scr.cT, (const C<T> *)p->scr.phiT,
            p->d_gram, p->d_cond, p->scr.coef, coef_dd(p), p->ncond, p->nt, R, nslab, (TourE<T> *)p->scr.y_tri);
        SIE_LAUNCH_CHECK(p);
        return SIE_OK;
    }
};

// Slab shape per right-hand-side count: a warp serves one triangle (or node)
// and 32 V J right-hand sides, V complex per load (FP32: two per 16-byte load
// when R is even, so that rows of [.][3][R] start on 16-byte boundaries), J
// loads per lane; the smallest slab that covers R keeps every lane busy.
#define SIE_SLAB_DISPATCH(R, CALL)                                                        \
    do {                                                                                 \
        if ((R) <= 32) return Blocks<float, 1, 1>::CALL;                                  \
        if ((R) <= 64) return (R) % 2 == 0 ? Blocks<float, 2, 1>::CALL : Blocks<float, 1, 2>::CALL; \
        return (R) % 2 == 0 ? Blocks<float, 2, 2>::CALL : Blocks<float, 1, 4>::CALL;      \
    } while (0)
// The far-field gather keeps slabs at most 64 wide in FP32: its 128-wide form
// needs 80 registers a thread, which caps residency at 3 CTAs per SM for this
// latency-bound gather; two 64-wide slabs (61 registers) read each block record
// twice but keep 4 CTAs resident (measured: 0.77 -> 0.66 ms on the bond-wire
// step; the projection, whose block records dominate its loads, is faster 128
// wide).
#define SIE_SLAB_DISPATCH_NARROW(R, CALL)                                                 \
    do {                                                                                 \
        if ((R) > 32) return (R) % 2 == 0 ? Blocks<float, 2, 1>::CALL : Blocks<float, 1, 2>::CALL; \
        SIE_SLAB_DISPATCH(R, CALL);                                                       \
    } while (0)
// Few-column FP32 gathers: the static kernel with at most kSmallRhs right-hand
// sides, unless the tuning asks for a path that reads the [row][3][R] operands.
bool small_rhs(const pfft_plan *p, int32_t R) {
    return R <= kSmallRhs && p->params.kernel == SIE_KERNEL_STATIC && !(p->kt.near == 1 && R % 2 == 0) &&
           p->kt.proj_slab != kChunkRhs;
}
// A lane per output component (COMP) or per column of all three, and rows per warp.
// Small meshes are bound by latency: the component form has a third of the loads in a
// lane's chain and three times the warps; larger ones by load wavefronts, of which the
// column form takes fewer.  us of both at 1, 3 and 5 right-hand sides, component form
// first: near field, 4.7k triangles 41, 41, 47 and 63, 66, 68; 6.0k 51, 60, 65 and 79,
// 83, 86; 8.0k 63, 105, 113 and 92, 98, 101: the line is at 40 rows an SM.  Projection,
// 4.1k nodes 15, 16, 16 and 17, 17, 17; 8.2k 15, 17, 19 and 14, 15, 15: at 32.
// Several rows per warp, as many as fit (columns or components x rows <= 32), while
// 16 warps an SM remain; near field of one right-hand side with 8, 16 and 32 of them:
// 12.0k triangles 119, 111 and 216 us, 5.2k 57, 58 and 89.
constexpr int kCompTri = 40, kCompNodes = 32, kFillWarps = 16;
struct SmallShape {
    bool comp;
    int rpw;   // rows per warp
    int64_t blocks;
};
SmallShape small_shape(const pfft_plan *p, int64_t rows, int32_t R, int comp_rows) {
    SmallShape o;
    o.comp = R <= 5 && rows <= int64_t(comp_rows) * p->sms;
    const int64_t fit = 32 / ((o.comp ? 6 : 2) * R);
    o.rpw = int(std::max<int64_t>(1, std::min(fit, rows / (int64_t(kFillWarps) * p->sms))));
    o.blocks = (rows + kSmallWarps * o.rpw - 1) / (kSmallWarps * o.rpw);
    return o;
}
int project_small(pfft_plan *p, int32_t R, cudaStream_t st) {
    const SmallShape g = small_shape(p, p->Ng, R, kCompNodes);
    const size_t smem = size_t(kSmallWarps * g.rpw) * (6 * R + 2) * sizeof(float);
    const auto fn = g.comp ? k_project_small<true> : k_project_small<false>;
    fn<<<unsigned(g.blocks), 32 * kSmallWarps, smem, st>>>(p->d_pn_ptr, p->d_pn_rec32, (const float4 *)p->scr.cT,
                                                           p->Ng, R, g.rpw, (float2 *)p->scr.grid);
    SIE_LAUNCH_CHECK(p);
    return SIE_OK;
}
int tri_gather_small(pfft_plan *p, int32_t R, cudaStream_t st) {
    const SmallShape g = small_shape(p, p->nt, R, kCompTri);
    const auto fn = g.comp ? k_tri_small<true> : k_tri_small<false>;
    fn<<<unsigned(g.blocks), 32 * kSmallWarps, 0, st>>>(
        p->d_near_ptr, p->d_near_rec32, p->d_pt_ptr, p->d_pt_rec32, (const float4 *)p->scr.cT,
        (const float4 *)p->scr.phiT, p->d_gram, p->d_cond, coef_dd(p), p->ncond, p->nt, R, g.rpw,
        (float4 *)p->scr.y_tri);
    SIE_LAUNCH_CHECK(p);
    return SIE_OK;
}
template <typename T> int run_project(pfft_plan *p, int32_t R, cudaStream_t st) {
    if constexpr (is_f32<T>) {
        // mixed form: staged node chunks when asked for (pfft_plan_set_kernel_tuning,
        // the autotuner); the direct gather is the default (measured on the bond
        // wires at 128 right-hand sides: 0.68 ms direct against 1.28 ms staged, whose
        // 32-wide slabs read each block record four times as often)
        if (p->n_pchunk > 0 && p->kt.proj_slab == kChunkRhs) {
            if (p->n_pchunk > INT32_MAX) return fail(SIE_ERR_ARG, "projection: too many node chunks");
            if (int rc = set_smem((const void *)k_project_tiled, kPTSmem)) return rc;
            const dim3 grid(unsigned(p->n_pchunk), unsigned((R + kChunkRhs - 1) / kChunkRhs));
            k_project_tiled<<<grid, 256, kPTSmem, st>>>(p->d_pch_node_ptr, p->d_pch_nodes, p->d_pch_tri_ptr,
                                                        p->d_pch_tri, p->d_pn_ptr, p->d_pn_rec32, p->d_pn_lcol,
                                                        (const float2 *)p->scr.cT, p->Ng, R, (float2 *)p->scr.grid);
            SIE_LAUNCH_CHECK(p);
            return SIE_OK;
        }
        if (p->kt.proj_slab == 64) SIE_SLAB_DISPATCH_NARROW(R, project(p, R, st));
        SIE_SLAB_DISPATCH(R, project(p, R, st));
    } else {
        SIE_COLS_DISPATCH(T, R, project(p, R, st));
    }
}
int run_far_gather(pfft_plan *p, int32_t R, cudaStream_t st) {
    if (p->kt.far_slab == 128) SIE_SLAB_DISPATCH(R, far_gather(p, R, st));
    SIE_SLAB_DISPATCH_NARROW(R, far_gather(p, R, st));
}
template <typename T> int run_tri_gather(pfft_plan *p, int32_t R, cudaStream_t st) {
    if constexpr (is_f32<T>) SIE_SLAB_DISPATCH(R, tri_gather(p, R, st));
    else SIE_COLS_DISPATCH(T, R, tri_gather(p, R, st));
}
template <typename T> int run_tri_gather_lossy(pfft_plan *p, int32_t R, cudaStream_t st) {
    if (R <= 32) return Blocks<T, 1, 1>::tri_gather_lossy(p, R, st);
    if (R <= 64) return Blocks<T, 1, 2>::tri_gather_lossy(p, R, st);
    return Blocks<T, 1, 4>::tri_gather_lossy(p, R, st);
}

// from this many rows on one CTA per row (wires, 79k slots: 128 rows 220 us for the
// currents' sums against 343 split, 64 rows 208 against 190 split)
constexpr int32_t kTourRowsMin = 96;
// Prefix sums of src's values over the tour, for R right-hand sides, into tour [R][2 nn].
template <typename E, typename S> int tour_sums(pfft_plan *p, const S &src, E *tour, int32_t R, cudaStream_t st) {
    const int64_t n = 2 * p->nn, nchunk = (n + kTourChunk - 1) / kTourChunk;
    if (R * nchunk > INT32_MAX) return fail(SIE_ERR_ARG, "tour sums: too many right-hand sides");
    E *part = (E *)p->scr.part;
    if (nchunk > 1 && R >= kTourRowsMin) {
        k_tour_rows<E><<<unsigned(R), 1024, 0, st>>>(src, n, tour);
        SIE_LAUNCH_CHECK(p);
        return SIE_OK;
    }
    if (nchunk > 1) {
        k_tour_part<E><<<unsigned(R * nchunk), 1024, 0, st>>>(src, int32_t(nchunk), part);
        SIE_LAUNCH_CHECK(p);
    }
    k_tour_sums<E><<<unsigned(R * nchunk), 1024, 0, st>>>(src, n, int32_t(nchunk), part, tour);
    SIE_LAUNCH_CHECK(p);
    return SIE_OK;
}
TourLinks tour_links(const pfft_plan *p, const double2 *x) {
    return TourLinks{x, p->nl, p->d_slot_link, p->d_nl_ptr, p->d_nl_loop, p->d_nl_sign};
}

// Smallest right-hand-side count for the tensor-core near field (mixed form).
constexpr int32_t kNearMmaMinRhs = 96;

template <typename T>
int matvec_t(pfft_plan *p, const double2 *x, double2 *y, int32_t R, int space, cudaStream_t st) {
    Scratch &s = p->scr;
    const int64_t nslots = 2 * p->nn;
    const int64_t ldy = p->nb + p->np;
    using E = TourE<T>;
    E *tour = (E *)s.tour;
    E *y_tri = (E *)s.y_tri, *y_br = (E *)s.y_br;
    int rc = SIE_OK;
    std::unique_ptr<StageTimer> tm(new StageTimer(p, SIE_STAGE_LOOP_TO_BRANCH, st));
    if (space == SIE_SPACE_LOOP) {
        rc = tour_sums<E>(p, tour_links(p, x), tour, R, st);
        if (rc) return rc;
    }
    const bool small = is_f32<T> && small_rhs(p, R);
    auto alpha = k_alpha_tri<T, false>;
    if constexpr (is_f32<T>)
        if (small) alpha = k_alpha_tri<T, true>;
    alpha<<<nblk(p->nt * R), 256, 0, st>>>(x, p->nl, tour, nslots, p->d_tri_src, p->d_tb, p->d_ts, p->nt, R, space,
                                           p->nb, (C<T> *)s.cT);
    SIE_LAUNCH_CHECK(p);
    tm.reset(new StageTimer(p, SIE_STAGE_PROJECT, st));
    rc = small ? project_small(p, R, st) : run_project<T>(p, R, st);
    if (rc) return rc;
    tm.reset();
    const int prec = is_df<T> ? SIE_PREC_DF : is_f64<T> ? SIE_PREC_FP64 : SIE_PREC_MIXED;
    const bool lossy = !is_df<T> && p->params.kernel == SIE_KERNEL_LOSSY;
    rc = fft_conv(p, s.grid, s.spec, R, prec, st, lossy ? lossy_sel(p, prec) : nullptr, true);
    if (rc) return rc;
    tm.reset(new StageTimer(p, SIE_STAGE_INTERP, st));
    if (small) {
        k_regroup_small<<<nblk(p->n_tiles * R * 32), 256, 0, st>>>((const float2 *)s.grid, p->d_tiles, p->n_tiles,
                                                                   p->Ng, R, (float4 *)s.phiT);
        SIE_LAUNCH_CHECK(p);
    } else {
        const int32_t B = 3 * R;
        const dim3 grid(unsigned(p->n_tiles), unsigned((B + 31) / 32));
        k_regroup<T><<<grid, 256, 0, st>>>((const C<T> *)s.grid, p->d_tiles, p->Ng, B, (C<T> *)s.phiT);
        SIE_LAUNCH_CHECK(p);
    }
    // mixed form, R even and at least kNearMmaMinRhs: near blocks on the tensor
    // cores (their operand rows are 16-byte aligned only for even R; a 128-column
    // slab costs the same however few of its columns are used, so below about
    // three quarters of a slab the CUDA-core gather is faster); otherwise one
    // CUDA-core gather
    if constexpr (is_df<T>) {
        tm.reset(new StageTimer(p, SIE_STAGE_NEAR, st));
        rc = run_tri_gather<T>(p, R, st);       // near + interpolation + y_T in one gather
    } else if (lossy) {
        // complex near blocks per frequency: one CUDA-core gather (near + interpolation + y_T)
        tm.reset(new StageTimer(p, SIE_STAGE_NEAR, st));
        rc = run_tri_gather_lossy<T>(p, R, st);
    } else if (small) {
        tm.reset(new StageTimer(p, SIE_STAGE_NEAR, st));
        rc = tri_gather_small(p, R, st);        // near + interpolation + y_T in one gather
    } else if (is_f32<T> && R % 2 == 0 && p->kt.near != 2 && (R >= kNearMmaMinRhs || p->kt.near == 1)) {
        rc = run_far_gather(p, R, st);          // interpolation (step 3) on the CUDA cores
        if (rc) return rc;
        tm.reset(new StageTimer(p, SIE_STAGE_NEAR, st));
        rc = near_mma_launch(p, R, st);         // near blocks on the tensor cores + y_T
    } else {
        tm.reset(new StageTimer(p, SIE_STAGE_NEAR, st));
        rc = run_tri_gather<T>(p, R, st);       // near + interpolation + y_T in one gather
    }
    if (rc) return rc;
    tm.reset(new StageTimer(p, SIE_STAGE_BRANCH_TO_LOOP, st));
    if (space == SIE_SPACE_BRANCH) {
        k_branch_out<E, double2><<<nblk(p->nb * R), 256, 0, st>>>(y_tri, p->d_br_tri, p->d_br_local, p->nt, p->nb,
                                                                  p->nb, R, y);
        SIE_LAUNCH_CHECK(p);
        return SIE_OK;
    }
    k_branch_out<E, E><<<nblk(ldy * R), 256, 0, st>>>(y_tri, p->d_br_tri, p->d_br_local, p->nt, p->nb, ldy, R,
                                                        y_br);
    SIE_LAUNCH_CHECK(p);
    rc = tour_sums<E>(p, TourTwigs<E>{y_br, ldy, p->d_slot_twig}, tour, R, st);
    if (rc) return rc;
    k_loop_out<E><<<nblk(p->nl * R), 256, 0, st>>>(y_br, ldy, tour, nslots, p->d_loop_dst, p->nl, R, y);
    SIE_LAUNCH_CHECK(p);
    return SIE_OK;
}

float2 *coef_dd(const pfft_plan *p) {
    return reinterpret_cast<float2 *>(p->scr.coef + size_t(p->scr.cap_rhs) * (2 * p->ncond + 1));
}

std::complex<double> surface_impedance(const pfft_plan *p, int c, double w) {
    using cd = std::complex<double>;
    const double sig = p->sigma[c], t = p->t_eff.empty() ? 0.0 : p->t_eff[c];
    if (!(t > 0.0)) return cd(1.0, 1.0) * std::sqrt(w * kMu0 / (2.0 * sig));
    const cd gamma = cd(1.0, 1.0) * std::sqrt(w * kMu0 * sig / 2.0);
    const cd z = gamma * (t / 2.0);
    // z coth z: Taylor series for small |z|, else coth from exp(-2z) (Re z >= 0)
    cd zc;
    if (std::abs(z) < 1e-2) {
        const cd z2 = z * z;
        zc = 1.0 + z2 / 3.0 - z2 * z2 / 45.0;
    } else {
        const cd e = std::exp(-2.0 * z);
        zc = z * (1.0 + e) / (1.0 - e);
    }
    return 2.0 / (sig * t) * zc;
}

// Per right-hand side: Z_s of each conductor and c_L / j (Eq. ImpedanceOp, Eq. Zb),
// in FP64 and as double-float pairs.
int fill_coef(const pfft_plan *p, const double *omega, int32_t R, double *cf, float2 *cd) {
    const size_t n = size_t(R) * (2 * p->ncond + 1);
    for (int32_t r = 0; r < R; ++r) {
        const double w = omega[r];
        if (!(w >= 0.0) || !std::isfinite(w)) return fail(SIE_ERR_ARG, "pfft_matvec: omega must be finite and >= 0");
        for (int c = 0; c < p->ncond; ++c) {
            const std::complex<double> zs = surface_impedance(p, c, w);
            cf[r * (2 * p->ncond + 1) + 2 * c] = zs.real();
            cf[r * (2 * p->ncond + 1) + 2 * c + 1] = zs.imag();
        }
        cf[r * (2 * p->ncond + 1) + 2 * p->ncond] = w * kMu0 / (4.0 * M_PI);
    }
    for (size_t i = 0; i < n; ++i) {
        const float hi = float(cf[i]);
        cd[i] = make_float2(hi, float(cf[i] - double(hi)));
    }
    return SIE_OK;
}

int upload_coef(pfft_plan *p, const double *omega, int32_t R, cudaStream_t st) {
    const size_t n = size_t(R) * (2 * p->ncond + 1);
    std::vector<double> cf(n);
    std::vector<float2> cd(n);
    int rc = fill_coef(p, omega, R, cf.data(), cd.data());
    if (rc) return rc;
    SIE_CUDA(cudaMemcpyAsync(p->scr.coef, cf.data(), n * sizeof(double), cudaMemcpyHostToDevice, st));
    SIE_CUDA(cudaMemcpyAsync(coef_dd(p), cd.data(), n * sizeof(float2), cudaMemcpyHostToDevice, st));
    return SIE_OK;
}

int matvec_async(pfft_plan *p, const void *x, void *y, int32_t nrhs, const double *omega, int space, int prec,
                 cudaStream_t st) {
    int rc = scratch_reserve(p, nrhs, prec);
    if (rc) return rc;
    rc = upload_coef(p, omega, nrhs, st);
    if (rc) return rc;
    if (p->params.kernel == SIE_KERNEL_LOSSY && (rc = lossy_prepare(p, omega, nrhs, st))) return rc;
    if (prec == SIE_PREC_DF && (rc = df_prepare(p, st))) return rc;
    return matvec_launch(p, x, y, nrhs, space, prec, st);
}

int matvec_launch(pfft_plan *p, const void *x, void *y, int32_t nrhs, int space, int prec, cudaStream_t st) {
    if (prec == SIE_PREC_FP64)
        return matvec_t<double>(p, (const double2 *)x, (double2 *)y, nrhs, space, st);
    if (prec == SIE_PREC_DF) {
        if (!p->df_ready || p->params.kernel != SIE_KERNEL_STATIC)
            return fail(SIE_ERR_ARG, "double-float product: static kernel plans only, tables built first");
        return matvec_t<df>(p, (const double2 *)x, (double2 *)y, nrhs, space, st);
    }
    return matvec_t<float>(p, (const double2 *)x, (double2 *)y, nrhs, space, st);
}

}  // namespace sie

extern "C" int pfft_matvec(pfft_plan *p, const void *x, void *y, int32_t nrhs, const double *omega, int32_t space,
                           int32_t prec, void *cuda_stream) {
    if (!p || !x || !y || !omega) return fail(SIE_ERR_ARG, "pfft_matvec: NULL argument");
    if (nrhs < 1) return fail(SIE_ERR_ARG, "pfft_matvec: nrhs must be >= 1");
    if (space != SIE_SPACE_LOOP && space != SIE_SPACE_BRANCH) return fail(SIE_ERR_ARG, "pfft_matvec: bad space");
    if (prec != SIE_PREC_FP64 && prec != SIE_PREC_MIXED && prec != SIE_PREC_DF)
        return fail(SIE_ERR_ARG, "pfft_matvec: bad precision");
    if (prec == SIE_PREC_DF && p->params.kernel != SIE_KERNEL_STATIC)
        return fail(SIE_ERR_ARG, "pfft_matvec: the double-float product takes the static kernel only");
    const int64_t n = space == SIE_SPACE_LOOP ? p->nl : p->nb;
    const char *xb = (const char *)x, *yb = (const char *)y;
    const size_t bytes = size_t(nrhs) * n * sizeof(double2);
    if (xb < yb + bytes && yb < xb + bytes) return fail(SIE_ERR_ARG, "pfft_matvec: x and y overlap");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    (void)cudaGetLastError();   // clear a stale error left by earlier work in this thread
    int rc = sie::matvec_async(p, x, y, nrhs, omega, space, prec, st);
    if (rc) return rc;
    return sie::finish_call(p, st);
}

extern "C" int sie_postprocess(pfft_plan *p, const void *x, int32_t nrhs, const double *omega, int32_t prec,
                               void *i_branch, void *v_branch, void *phi, void *cuda_stream) {
    using namespace sie;
    if (!p || !x || nrhs < 1) return fail(SIE_ERR_ARG, "sie_postprocess: bad argument");
    if (prec != SIE_PREC_FP64 && prec != SIE_PREC_MIXED) return fail(SIE_ERR_ARG, "sie_postprocess: bad precision");
    if ((v_branch || phi) && !omega) return fail(SIE_ERR_ARG, "sie_postprocess: omega is needed for voltages");
    if (!i_branch && !v_branch && !phi) return SIE_OK;
    if (nrhs > 65535) return fail(SIE_ERR_ARG, "sie_postprocess: at most 65535 right-hand sides per call");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    (void)cudaGetLastError();
    const int64_t nb = p->nb, nt = p->nt, nslots = 2 * p->nn, R = nrhs;
    int rc = scratch_reserve(p, nrhs, prec);   // the size the product below uses: no later regrowth
    if (rc) return rc;
    // temporaries for outputs the caller did not ask for but later steps need
    double2 *alpha = static_cast<double2 *>(i_branch), *vb = static_cast<double2 *>(v_branch);
    double2 *tmp_a = nullptr, *tmp_v = nullptr;
    auto cleanup = [&]() {
        if (tmp_a) cudaFree(tmp_a);
        if (tmp_v) cudaFree(tmp_v);
    };
    if (!alpha) {
        if (plan_malloc(p, (void **)&tmp_a, size_t(R) * nb * sizeof(double2)) != cudaSuccess)
            return fail(SIE_ERR_OOM, "sie_postprocess: out of device memory");
        alpha = tmp_a;
    }
    if (phi && !vb) {
        if (plan_malloc(p, (void **)&tmp_v, size_t(R) * nb * sizeof(double2)) != cudaSuccess) {
            cleanup();
            return fail(SIE_ERR_OOM, "sie_postprocess: out of device memory");
        }
        vb = tmp_v;
    }
    double2 *tour = static_cast<double2 *>(p->scr.tour);
    const dim3 gb(nblk(nb), unsigned(R)), gt(nblk(nt), unsigned(R));
    // branch currents: alpha = A^T x through the tour prefix sums (FP64)
    rc = tour_sums<double2>(p, tour_links(p, static_cast<const double2 *>(x)), tour, nrhs, st);
    if (rc) { cleanup(); return rc; }
    k_branch_alpha<<<gb, 256, 0, st>>>(static_cast<const double2 *>(x), p->nl, tour, nslots, p->d_branch_src, nb,
                                       alpha);
    p->launches += 1;
    if (cudaGetLastError() != cudaSuccess) { cleanup(); return fail(SIE_ERR_CUDA, "sie_postprocess: launch failed"); }
    if (vb) {   // branch voltage drops: the branch-space product Z_b alpha
        rc = matvec_async(p, alpha, vb, nrhs, omega, SIE_SPACE_BRANCH, prec, st);
        if (rc) { cleanup(); return rc; }
    }
    if (phi) {   // potentials: root-path sums of the twig drops, minus the reference node's
        rc = tour_sums<double2>(p, TourTwigs<double2>{vb, nb, p->d_slot_twig}, tour, nrhs, st);
        if (rc) { cleanup(); return rc; }
        k_panel_phi<<<gt, 256, 0, st>>>(tour, nslots, p->d_panel_slot, p->d_panel_ref, nt,
                                        static_cast<double2 *>(phi));
        p->launches += 1;
        if (cudaGetLastError() != cudaSuccess) { cleanup(); return fail(SIE_ERR_CUDA, "sie_postprocess: launch failed"); }
    }
    const cudaError_t e = cudaStreamSynchronize(st);
    cleanup();
    if (e != cudaSuccess) return fail(SIE_ERR_CUDA, std::string("sie_postprocess: ") + cudaGetErrorString(e));
    return check_device_errors(p);
}
