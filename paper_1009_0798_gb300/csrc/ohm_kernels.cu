// ohm_kernels.cu -- sm_103a kernels of the implicit ohmic-dissipation step
// (T. Matsumoto 2011, Sec. 2).  One thread block works on one 8^3-cell block: it stages the
// block and a one-cell halo (faces and edges; corners are never read by the stencil) in
// shared memory, from the same-grid neighbour blocks or, where the grid has no neighbour,
// from the block's coarse-fine ghost slot.
//
// Face flux (Eqs. 4-6, 9-11), kept scaled as Phi = 2 h F:
//   Phi_a^b = (eta_lo + eta_hi) * (T/4 - N),  N = B_b(hi) - B_b(lo)                 (Eq. 9)
//   T = B_a(lo+e_b) + B_a(hi+e_b) - B_a(lo-e_b) - B_a(hi-e_b)                         (Eq. 10)
// and the flux divergence (Eq. 8) is sum_a (Phi_a(+) - Phi_a(-)) / (2 h^2).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cstdint>
#include <type_traits>
#include <utility>

#include "ohm_internal.h"

namespace ohm {

__device__ __forceinline__ int tix(int i, int j, int k) { return (k * TS + j) * TS + i; }

// Programmatic dependent launch.  The kernels of a step follow one another on one stream and many of
// them are short (a 64^3 step: 150 launches of 2-10 us), so each is launched while the one before it
// drains: its thread blocks come up, read the block tables (which never change) and wait for the
// grid before them to complete: 64^3 mixed step 1.67 -> 1.53 ms, three-level mixed step (64^3 base, 3 V-cycles)
// 2.50 -> 2.33, 128^3 float-float step 3.56 -> 3.43.  Every kernel launched through launch_pdl calls pdl_trigger() and,
// before it touches anything that another kernel writes and before any return, pdl_wait().  A load
// through a const __restrict__ parameter could be moved above the wait, so pdl_wait returns an opaque 0
// that goes into the block (or element) index from which the addresses of such loads are formed; the
// other loads follow a __syncthreads() in any case.
// (The opaque 0 also keeps the index out of the uniform registers, which costs the instruction-bound
// float32 stencils 2-6% on large grids: they have an instance without any of this, EARLY = false.)
template <bool EARLY = true>
__device__ __forceinline__ void pdl_trigger() {
    if constexpr (EARLY) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <bool EARLY = true>
__device__ __forceinline__ int pdl_wait() {
    int z = 0;
    if constexpr (EARLY) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("mov.b32 %0, 0;" : "=r"(z) : : "memory");
    }
    return z;
}
// Grids of more thread blocks are launched when the one before has drained: their own time hides the
// launch, and blocks that come up beside a running grid are spread unevenly over the SMs (28 boxes of
// 64^3: 13.7-13.9 ms per step launched early throughout, 13.4 with this bound).
constexpr unsigned PDL_GRID = 1024;
// Kernels that are captured into a graph are launched as before, too: a graph has short gaps of its own,
// and batches of 20 to 76 boxes of 16^3 lost 1-6% to the uneven placement.
static bool capturing(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    return s != nullptr && cudaStreamIsCapturing(s, &st) == cudaSuccess && st != cudaStreamCaptureStatusNone;
}
static bool pdl_small(unsigned grid) { return grid <= PDL_GRID; }
// As after <<< >>>, a refused launch also stays in the runtime's last error: every launcher ends in
// cudaGetLastError(), which returns and clears it (left there, the process's next check would report it
// from a call that succeeded).
template <typename... E, typename... A>
static cudaError_t launch_as(bool early, void (*k)(E...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = early && !capturing(s) ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, std::forward<A>(args)...);
}
template <typename... E, typename... A>
static cudaError_t launch_pdl(void (*k)(E...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A &&...args) {
    return launch_as(pdl_small(grid), k, grid, block, smem, s, std::forward<A>(args)...);
}
// kernels with an instance for each: the first for small grids, the second for large ones
template <typename... E, typename... A>
static cudaError_t launch_pdl2(void (*k)(E...), void (*kl)(E...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A &&...args) {
    return launch_as(pdl_small(grid), pdl_small(grid) ? k : kl, grid, block, smem, s, std::forward<A>(args)...);
}
// So are the kernels bound by the float64 pipe, whatever their size: the SM with the most thread blocks
// sets their time (half-refined float64 box: 6.5 ms per step, 7.2 launched early).
template <typename... E, typename... A>
static cudaError_t launch_full(void (*k)(E...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A &&...args) {
    return launch_as(false, k, grid, block, smem, s, std::forward<A>(args)...);
}

// batched inner iterations: block b belongs to an instance that is not iterated
__device__ __forceinline__ bool skip_block(const GridDev &g, int b) {
    return g.imask && !g.imask[g.inst_nblk ? b / g.inst_nblk : 0];
}

// ------------------------------------------------------------------ float-float arithmetic
// GB300 issues float64 at 1/58 of the float32 rate, so the outer residual of the mixed path
// runs on pairs of float32 values instead (Dekker 1971).  Every operation uses the explicitly
// rounded intrinsics, which the compiler never fuses into FMAs, so the error-free
// transformations stay exact:
//   two_sum (Knuth): s = fl(a + b) and the exact error of that addition;
//   fast_two_sum (Dekker): the same when |a| >= |b| (or a = 0), in three operations;
//   products: fl(a.hi b.hi) and its exact error from an FMA, plus the cross terms.
// Sums fold the trailing parts in before one renormalisation.  Their error is at most about
// 2^-47 (|a| + |b|): bounded against the operands, not the result, which is the measure the
// residual needs (its cancellation error is measured against |X|).
__device__ __forceinline__ dfloat df_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return dfloat(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
__device__ __forceinline__ dfloat df_fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return dfloat(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ dfloat operator+(dfloat a, dfloat b) {
    const dfloat s = df_two_sum(a.hi, b.hi);
    return df_fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ dfloat operator-(dfloat a) { return dfloat(-a.hi, -a.lo); }
__device__ __forceinline__ dfloat operator-(dfloat a, dfloat b) { return a + (-b); }
__device__ __forceinline__ dfloat operator*(dfloat a, dfloat b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return df_fast_two_sum(p, e);
}

// float64 -> float-float by bit manipulation (no float64 instruction): hi carries the sign,
// the exponent and the leading 24 significand bits (truncated), lo the remaining 29 bits
// rounded to 24, so hi + lo keeps about 48 of the 53 bits.  Magnitudes outside the normal
// float32 range give lo = 0 and a signed hi: NaN stays NaN, infinities and finite values of
// 2^128 and above become infinite, values below 2^-126 become zero.
__device__ __forceinline__ dfloat split_double(double x) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const unsigned int uh = (unsigned int)(u >> 32), ul = (unsigned int)u;
    const int e = (int)((uh >> 20) & 0x7ffu);  // biased float64 exponent
    const int fe = e - (1023 - 127);           // the same exponent biased for float32
    const unsigned int sgn = uh & 0x80000000u;
    if ((unsigned)(fe - 1) >= 254u) {
        const unsigned int nan = e == 0x7ff && ((uh & 0xfffffu) | ul) ? 0x400000u : 0u;
        return dfloat(__uint_as_float(fe >= 255 ? sgn | 0x7f800000u | nan : sgn));
    }
    const float hi = __uint_as_float(sgn | ((unsigned)fe << 23) | ((uh & 0xfffffu) << 3) | (ul >> 29));
    // lo = r 2^(e - 1075) for the 29 low significand bits r; where 2^(e - 1075) is below the
    // normal float32 range it is applied in two exact steps, 2^(e - 1075 + 64) and 2^-64
    const int k = e < 1075 - 126 ? 64 : 0;
    const float s1 = __uint_as_float((unsigned)(e - 1075 + k + 127) << 23);
    const float s2 = __uint_as_float((unsigned)(127 - k) << 23);
    const float lo = __fmul_rn(__fmul_rn(__uint2float_rn(ul & 0x1fffffffu), s1), s2);
    return dfloat(hi, sgn ? -lo : lo);
}

// Conversions used outside the float-float hot loop (flux registers, refluxing)
__device__ __forceinline__ double to_double(float v) { return (double)v; }
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(dfloat v) { return (double)v.hi + (double)v.lo; }
template <typename T>
__device__ __forceinline__ T from_double(double v) { return (T)v; }
template <>
__device__ __forceinline__ dfloat from_double<dfloat>(double v) {
    const float h = __double2float_rn(v);
    return dfloat(h, __double2float_rn(v - (double)h));
}
// staged tile value from a field value (float64 fields split for float-float tiles)
template <typename T, typename TS>
__device__ __forceinline__ T tile_val(TS v) {
    static_assert(sizeof(T) == sizeof(TS), "tile and field types differ in size");
    return v;
}
template <>
__device__ __forceinline__ dfloat tile_val<dfloat, double>(double v) { return split_double(v); }
// x / 4 (exact for every type)
__device__ __forceinline__ float quarter(float v) { return 0.25f * v; }
__device__ __forceinline__ double quarter(double v) { return 0.25 * v; }
__device__ __forceinline__ dfloat quarter(dfloat v) { return dfloat(0.25f * v.hi, 0.25f * v.lo); }
// leading value (the float32 or float64 approximation used for outputs and norms)
__device__ __forceinline__ float lead(float v) { return v; }
__device__ __forceinline__ double lead(double v) { return v; }
__device__ __forceinline__ float lead(dfloat v) { return v.hi; }
template <typename X>
struct Ident {
    using type = X;
};

// Shared-memory geometry of a staged 10^3 tile (block + 1-cell halo).  Rows along x are RS
// elements apart; PX is the row stride of the x-face flux array; tile x index ti sits at row
// offset OFF + ti.  float32 rows of 12 with OFF = 1 put the 8 interior cells of a row on an
// 8-byte boundary (staged as four 64-bit words); the compact tile (36 KB for the residual
// kernel) lets 4 thread blocks of 512 threads share an SM, which measured faster at 256^3
// (0.390 ms against 0.426 ms per residual + restriction) than rows padded to 24 floats, which
// avoid the 2-way bank conflicts of this layout but fit only 3 blocks per SM.  float64 kernels
// are bound by the float64 pipe and keep the compact stride.
template <typename T>
struct G10;
template <>
struct G10<float> {
    static constexpr int RS = 12, PX = 9, OFF = 1;
};
template <>
struct G10<double> {
    static constexpr int RS = 10, PX = 9, OFF = 0;
};
template <>
struct G10<dfloat> {
    static constexpr int RS = 10, PX = 9, OFF = 0;
};
// z-face planes are PZ apart: 72 for float32 (= 8 mod 32 banks, like the x- and y-face arrays
// and the tile planes, so a warp of 4 planes x 8 cells reads 32 distinct banks), 64 for float64
template <typename T>
struct Geo {
    static constexpr int RS = G10<T>::RS, PS = TS * RS, CS = TS * PS, PX = G10<T>::PX, OFF = G10<T>::OFF;
    static constexpr int PZ = sizeof(T) == 4 ? 72 : 64;
    static constexpr int PHI_X = 64 * PX;  // x faces per component
    static constexpr int PHI = 2 * PHI_X + 2 * 576 + 2 * 9 * PZ;
    __device__ static __forceinline__ int at(int i, int j, int k) { return k * PS + j * RS + i + OFF; }
    __device__ static __forceinline__ int xf(int fi, int j, int k) { return (k * 8 + j) * PX + fi; }
    __device__ static __forceinline__ int zf(int i, int j, int fk) { return fk * PZ + j * 8 + i; }
};

// 8 consecutive values of a block row (16-byte aligned in global memory) as vector loads
template <typename T>
struct Row8 {
    T v[8];
};
__device__ __forceinline__ Row8<float> load_row8(const float *__restrict__ p) {
    Row8<float> r;
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    const float4 b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    r.v[0] = a.x; r.v[1] = a.y; r.v[2] = a.z; r.v[3] = a.w;
    r.v[4] = b.x; r.v[5] = b.y; r.v[6] = b.z; r.v[7] = b.w;
    return r;
}
__device__ __forceinline__ Row8<double> load_row8(const double *__restrict__ p) {
    Row8<double> r;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const double2 a = __ldg(reinterpret_cast<const double2 *>(p) + q);
        r.v[2 * q] = a.x;
        r.v[2 * q + 1] = a.y;
    }
    return r;
}

// Row-wise staging of a block and a halo of width HW (tile edge S = 8 + 2 HW; rows along x
// RS elements apart, planes S*RS, components S*S*RS), NC components of field F, from the 27
// neighbour ids in shared memory (snb, -1 = absent).  One task per (component, tile row):
// the 8 interior values of the row come from one block as vector loads, the HW halo cells at
// each end from the x-neighbours of that block.  Rows or cells of an absent neighbour come
// from `ghost` ([NC][10^3] compact, HW = 1 only) or are zero.  Values at the corners of the
// box are never read by the stencil and may be left stale.
template <typename T, typename TS>
__device__ __forceinline__ void store_row8(T *dst, const Row8<TS> &row, bool aligned16, bool aligned8 = false) {
    if constexpr (sizeof(T) == 4) {
        if (aligned16) {
            float4 *d4 = reinterpret_cast<float4 *>(dst);
            d4[0] = make_float4((float)row.v[0], (float)row.v[1], (float)row.v[2], (float)row.v[3]);
            d4[1] = make_float4((float)row.v[4], (float)row.v[5], (float)row.v[6], (float)row.v[7]);
            return;
        }
        if (aligned8) {
            float2 *d2 = reinterpret_cast<float2 *>(dst);
#pragma unroll
            for (int q = 0; q < 4; q++) d2[q] = make_float2((float)row.v[2 * q], (float)row.v[2 * q + 1]);
            return;
        }
    }
#pragma unroll
    for (int q = 0; q < 8; q++) dst[q] = tile_val<T, TS>(row.v[q]);
}

// TS is the field's element type (T, or float64 for float-float tiles)
template <typename T, int NC, int HW, int RS, int OFF = 0, typename TS = T>
__device__ __forceinline__ void stage_rows(T *__restrict__ tile, const TS *__restrict__ F, const int *__restrict__ snb,
                                           const typename Ident<TS>::type *__restrict__ ghost) {
    constexpr int S = 8 + 2 * HW, S2 = S * S;
    constexpr bool A16 = sizeof(T) == 4 && (OFF + HW) % 4 == 0 && RS % 4 == 0;
    constexpr bool A8 = sizeof(T) == 4 && (OFF + HW) % 2 == 0 && RS % 2 == 0;
    for (int task = threadIdx.x; task < NC * S2; task += blockDim.x) {
        const int c = task / S2, rr = task - c * S2;
        const int tj = rr % S, tk = rr / S;
        const int lj = tj - HW, lk = tk - HW;
        const int dj = lj < 0 ? -1 : (lj > 7 ? 1 : 0), dk = lk < 0 ? -1 : (lk > 7 ? 1 : 0);
        const int sj = lj - 8 * dj, sk = lk - 8 * dk;
        T *dst = tile + c * (S2 * RS) + rr * RS + OFF;
        const TS *gh = ghost ? ghost + c * T3 + rr * S : nullptr;
        const int dcent = (dk + 1) * 9 + (dj + 1) * 3;
        const int src = snb[dcent + 1];
        if (src >= 0) {
            const Row8<TS> row = load_row8(F + ((size_t)src * NC + c) * B3 + (sk * 8 + sj) * 8);
            store_row8(dst + HW, row, A16, A8);
        } else {
#pragma unroll
            for (int q = 0; q < 8; q++) dst[HW + q] = gh ? tile_val<T, TS>(gh[HW + q]) : T(0);
        }
        const int slo = snb[dcent], shi = snb[dcent + 2];
        if constexpr (sizeof(T) == 4 && HW == 2 && OFF % 2 == 0 && RS % 2 == 0) {
          if (slo >= 0 && shi >= 0) {
            // two-cell halos as 8-byte words (cells 6,7 of the x- neighbour, 0,1 of the x+ one)
            const float2 lo = __ldg(reinterpret_cast<const float2 *>(F + ((size_t)slo * NC + c) * B3 + (sk * 8 + sj) * 8 + 6));
            const float2 hi = __ldg(reinterpret_cast<const float2 *>(F + ((size_t)shi * NC + c) * B3 + (sk * 8 + sj) * 8));
            *reinterpret_cast<float2 *>(dst) = lo;
            *reinterpret_cast<float2 *>(dst + HW + 8) = hi;
            continue;
          }
        }
#pragma unroll
        for (int h = 0; h < HW; h++) {
            // low end: cells 8-HW+h of the x- neighbour; high end: cells h of the x+ neighbour
            dst[h] = slo >= 0 ? tile_val<T, TS>(F[((size_t)slo * NC + c) * B3 + (sk * 8 + sj) * 8 + 8 - HW + h])
                              : (gh ? tile_val<T, TS>(gh[h]) : T(0));
            dst[HW + 8 + h] = shi >= 0 ? tile_val<T, TS>(F[((size_t)shi * NC + c) * B3 + (sk * 8 + sj) * 8 + h])
                                       : (gh ? tile_val<T, TS>(gh[HW + 8 + h]) : T(0));
        }
    }
}

// neighbour ids of block b into shared memory (call before stage_rows, then __syncthreads)
__device__ __forceinline__ void stage_nbr(int *snb, const int *__restrict__ nbr, int b) {
    if (threadIdx.x < 27) snb[threadIdx.x] = __ldg(nbr + b * 27 + threadIdx.x);
}

// Phi = 2hF for the face between tile cells p (low) and p + sa, axis a (Eqs. 4-6, 9-11).
// The two flux components are the axes other than a in ascending order, with tile strides
// s1 and s2; components of the tile are cs elements apart.
template <typename T>
__device__ __forceinline__ void face_phi_s(const T *__restrict__ tB, const T *__restrict__ tE, int p, int a, int sa,
                                           int s1, int s2, int cs, T &phi1, T &phi2) {
    const int b1 = a == 0 ? 1 : 0, b2 = a == 2 ? 1 : 2;
    const T es = tE[p] + tE[p + sa];
    const T *Ba = tB + a * cs;
    const T *B1 = tB + b1 * cs;
    const T *B2 = tB + b2 * cs;
    T n1 = B1[p + sa] - B1[p];
    T t1 = (Ba[p + sa + s1] + Ba[p + s1]) - (Ba[p + sa - s1] + Ba[p - s1]);
    phi1 = es * (quarter(t1) - n1);
    T n2 = B2[p + sa] - B2[p];
    T t2 = (Ba[p + sa + s2] + Ba[p + s2]) - (Ba[p + sa - s2] + Ba[p - s2]);
    phi2 = es * (quarter(t2) - n2);
}

// Faces of a 10^3 tile along axis a from the low tile cell p, in the geometry of T
template <typename T>
__device__ __forceinline__ void face10(const T *__restrict__ tB, const T *__restrict__ tE, int p, int a, T &p1, T &p2) {
    using G = Geo<T>;
    if (a == 0)
        face_phi_s(tB, tE, p, 0, 1, G::RS, G::PS, G::CS, p1, p2);
    else if (a == 1)
        face_phi_s(tB, tE, p, 1, G::RS, 1, G::PS, G::CS, p1, p2);
    else
        face_phi_s(tB, tE, p, 2, G::PS, 1, G::RS, G::CS, p1, p2);
}

// Offsets of the six flux arrays: x faces [2 comps][64 rows][PX] (index xf), y faces
// [2][8][9][8] ((k*9+fj)*8+i), z faces [2][9][PZ] (index zf).
template <typename T>
__device__ __forceinline__ int phi_base(int ax, int comp) {
    using G = Geo<T>;
    return ax == 0 ? comp * G::PHI_X : (ax == 1 ? 2 * G::PHI_X + comp * 576 : 2 * G::PHI_X + 2 * 576 + comp * 9 * G::PZ);
}

// Cell of thread t in the 512-thread stencil kernels.  float32: a warp takes one row index j of
// 4 consecutive planes (i fastest), whose tile and face-array offsets fall on 32 distinct banks
// for the compact strides above; float64 keeps i + 8 j + 64 k.
template <typename T>
__device__ __forceinline__ void cell_of_thread(int t, int &i, int &j, int &k) {
    if (sizeof(T) == 4) {
        i = t & 7;
        k = ((t >> 3) & 3) + 4 * (t >> 8);
        j = (t >> 5) & 7;
    } else {
        i = t & 7;
        j = (t >> 3) & 7;
        k = t >> 6;
    }
}

// All 1728 face fluxes of a staged block (512 threads): thread (i,j,k) computes the low x, y
// and z faces of its cell, then threads 0..191 compute the 3 x 64 faces of the high planes.
template <typename T>
__device__ __forceinline__ void all_faces_512(const T *__restrict__ tB, const T *__restrict__ tE, T *__restrict__ phi) {
    using G = Geo<T>;
    const int t = threadIdx.x;
    int i, j, k;
    cell_of_thread<T>(t, i, j, k);
    const int p = G::at(i + 1, j + 1, k + 1);
    T p1, p2;
    face10(tB, tE, p - 1, 0, p1, p2);
    phi[G::xf(i, j, k)] = p1;
    phi[G::PHI_X + G::xf(i, j, k)] = p2;
    face10(tB, tE, p - G::RS, 1, p1, p2);
    phi[phi_base<T>(1, 0) + (k * 9 + j) * 8 + i] = p1;
    phi[phi_base<T>(1, 1) + (k * 9 + j) * 8 + i] = p2;
    face10(tB, tE, p - G::PS, 2, p1, p2);
    phi[phi_base<T>(2, 0) + G::zf(i, j, k)] = p1;
    phi[phi_base<T>(2, 1) + G::zf(i, j, k)] = p2;
    if (t < 192) {
        const int ax = t >> 6, u = t & 7, v = (t >> 3) & 7;
        if (ax == 0) {  // x = 8 plane: (j, k) = (u, v)
            face10(tB, tE, G::at(8, u + 1, v + 1), 0, p1, p2);
            phi[G::xf(8, u, v)] = p1;
            phi[G::PHI_X + G::xf(8, u, v)] = p2;
        } else if (ax == 1) {  // y = 8 plane: (i, k) = (u, v)
            face10(tB, tE, G::at(u + 1, 8, v + 1), 1, p1, p2);
            phi[phi_base<T>(1, 0) + (v * 9 + 8) * 8 + u] = p1;
            phi[phi_base<T>(1, 1) + (v * 9 + 8) * 8 + u] = p2;
        } else {  // z = 8 plane: (i, j) = (u, v)
            face10(tB, tE, G::at(u + 1, v + 1, 8), 2, p1, p2);
            phi[phi_base<T>(2, 0) + G::zf(u, v, 8)] = p1;
            phi[phi_base<T>(2, 1) + G::zf(u, v, 8)] = p2;
        }
    }
}

// sum_a (Phi_a(+) - Phi_a(-)) at cell (i,j,k) for the three components
template <typename T>
__device__ __forceinline__ void cell_div(const T *__restrict__ phi, int i, int j, int k, T &dx, T &dy, T &dz) {
    using G = Geo<T>;
    const T *px0 = phi, *px1 = phi + G::PHI_X;                                // x faces: comps y, z
    const T *py0 = phi + phi_base<T>(1, 0), *py1 = phi + phi_base<T>(1, 1);  // y faces: comps x, z
    const T *pz0 = phi + phi_base<T>(2, 0), *pz1 = phi + phi_base<T>(2, 1);  // z faces: comps x, y
    const int xl = G::xf(i, j, k), yl = (k * 9 + j) * 8 + i, zl = G::zf(i, j, k);
    dx = (py0[yl + 8] - py0[yl]) + (pz0[zl + G::PZ] - pz0[zl]);
    dy = (px0[xl + 1] - px0[xl]) + (pz1[zl + G::PZ] - pz1[zl]);
    dz = (px1[xl + 1] - px1[xl]) + (py1[yl + 8] - py1[yl]);
}

// index in the flux arrays of the boundary-plane face (u, v) of side s = 2a + hi, where
// (u, v) run over the two axes other than a in ascending order
template <typename T>
__device__ __forceinline__ int plane_face(int a, int hi, int comp, int u, int v) {
    using G = Geo<T>;
    if (a == 0) return phi_base<T>(0, comp) + G::xf(hi ? 8 : 0, u, v);
    if (a == 1) return phi_base<T>(1, comp) + (v * 9 + (hi ? 8 : 0)) * 8 + u;
    return phi_base<T>(2, comp) + G::zf(u, v, hi ? 8 : 0);
}

// Block-wide sum / max in a fixed order (deterministic); the result is valid in thread 0.
template <typename T>
__device__ __forceinline__ T block_sum(T v, T *red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    T s = 0;
    if (w == 0) {
        s = threadIdx.x < nw ? red[threadIdx.x] : T(0);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    return s;
}

template <typename T>
__device__ __forceinline__ T block_max(T v, T *red) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    T s = 0;
    if (w == 0) {
        s = threadIdx.x < nw ? red[threadIdx.x] : T(0);
        for (int o = 16; o > 0; o >>= 1) s = fmax(s, __shfl_xor_sync(0xffffffffu, s, o));
    }
    return s;
}

// ------------------------------------------------------------------ composite operator
// Computed in TC: float-float (dfloat, from float64 fields) for the outer residual and the source of
// OHM_MIXED_FF, float32 for the inner residual of mixed precision (float64: k_composite_d below);
// refluxed fluxes travel through float64 registers.
template <typename TC>
struct CompTypes {
    using In = TC;   // element type of X, eta and the ghosts
    using Acc = TC;  // norm accumulation
    static constexpr int minb = sizeof(TC) == 4 ? 4 : 1;
};
template <>
struct CompTypes<dfloat> {
    using In = double;
    using Acc = float;
    static constexpr int minb = 3;
};

template <typename TC, typename TO, bool NORMS, typename YT = TC, bool EARLY = false>
__global__ void __launch_bounds__(512, CompTypes<TC>::minb)
    k_composite(GridDev g, const typename CompTypes<TC>::In *__restrict__ X, const YT *__restrict__ Y,
                const typename CompTypes<TC>::In *__restrict__ eta, const typename CompTypes<TC>::In *__restrict__ Gx,
                const typename CompTypes<TC>::In *__restrict__ Geta, TC a, TC coef, TC d, TO *__restrict__ out,
                TO *__restrict__ out2, double *__restrict__ reg, const int *__restrict__ rsrc_tab,
                double *__restrict__ partials, double vol, TC *__restrict__ outS, TC coef2, double inv2h, double twoh, bool ymx) {
    using G = Geo<TC>;
    using TA = typename CompTypes<TC>::Acc;
    using TM = typename std::conditional<sizeof(TO) == 4, float, TA>::type;  // max |out| from the output copy
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TC *tB = reinterpret_cast<TC *>(smem_raw);
    TC *tE = tB + 3 * G::CS;
    TC *phi = tE + G::CS;
    __shared__ int snb[27];
    const int b0 = blockIdx.x;
    pdl_trigger<EARLY>();
    if (!EARLY && skip_block(g, b0)) return;  // (masked blocks return before they load anything)
    stage_nbr(snb, g.nbr, b0);
    const int slot = g.gslot ? g.gslot[b0] : -1;
    const int b = b0 + pdl_wait<EARLY>();
    if (EARLY && skip_block(g, b)) return;
    if (g.covered && g.covered[b]) {
        if (NORMS && threadIdx.x < 3) partials[b * 3 + threadIdx.x] = 0.0;
        return;
    }
    __syncthreads();
    stage_rows<TC, 3, 1, G::RS, G::OFF>(tB, X, snb, slot >= 0 && Gx ? Gx + (size_t)slot * 3 * T3 : nullptr);
    stage_rows<TC, 1, 1, G::RS, G::OFF>(tE, eta, snb, slot >= 0 && Geta ? Geta + (size_t)slot * T3 : nullptr);
    __syncthreads();
    all_faces_512(tB, tE, phi);
    __syncthreads();
    // flux registers: faces with no same-level neighbour publish F = Phi / (2h) (inv2h = 1 / (2h)
    // and twoh = 2h come from the host: a float64 division here would cost the float32 kernels
    // dearly on a GPU with few float64 units)
    if (g.freg) {
        for (int s = 0; s < 6; s++) {
            int slotr = g.freg[b * 6 + s];
            if (slotr < 0) continue;
            int ax = s >> 1, hi = s & 1;
            for (int q = threadIdx.x; q < 128; q += blockDim.x) {
                int comp = q >> 6, uv = q & 63;
                reg[(size_t)slotr * 128 + q] = to_double(phi[plane_face<TC>(ax, hi, comp, uv & 7, uv >> 3)]) * inv2h;
            }
        }
    }
    // refluxing: faces next to a covered block take 2h * (mean of the four fine fluxes)
    if (g.rsrc) {
        for (int s = 0; s < 6; s++) {
            int src = g.rsrc[b * 6 + s];
            if (src < 0) continue;
            int ax = s >> 1, hi = s & 1;
            for (int q = threadIdx.x; q < 128; q += blockDim.x) {
                int comp = q >> 6, u = q & 7, v = (q >> 3) & 7;
                int fslot = rsrc_tab[src * 4 + (v >> 2) * 2 + (u >> 2)];
                const double *R = reg + (size_t)fslot * 128 + comp * 64;
                int fu = 2 * (u & 3), fv = 2 * (v & 3);
                double m = 0.25 * ((R[fv * 8 + fu] + R[fv * 8 + fu + 1]) + (R[(fv + 1) * 8 + fu] + R[(fv + 1) * 8 + fu + 1]));
                phi[plane_face<TC>(ax, hi, comp, u, v)] = from_double<TC>(m * twoh);
            }
        }
        __syncthreads();  // refluxed faces before the divergence (g.rsrc is uniform: legal)
    }
    int i, j, k;
    cell_of_thread<TC>(threadIdx.x, i, j, k);
    const int cell = (k * 8 + j) * 8 + i;
    TC dv[3];
    cell_div(phi, i, j, k, dv[0], dv[1], dv[2]);
    TA sr = 0, ss = 0;
    TM mx = 0;
    const int p = G::at(i + 1, j + 1, k + 1);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        size_t id = ((size_t)b * 3 + c) * B3 + cell;
        TC y = Y ? tile_val<TC, YT>(Y[id]) : TC(0);
        // ymx: a = -1, d = 1 (a residual), one operation less per component
        TC o = ymx ? (y - tB[c * G::CS + p]) + coef * dv[c] : a * tB[c * G::CS + p] + coef * dv[c] + d * y;
        if (sizeof(TC) == 8 && outS) {  // o is the source; the residual of X against it is coef2 divF(X)
            outS[id] = o;
            y = o;
            o = coef2 * dv[c];
        }
        const TA ol = lead(o);
        const TO oo = (TO)ol;
        out[id] = oo;
        if (out2) out2[id] = oo;
        if constexpr (NORMS) {
            const TA yl = lead(y);
            sr += ol * ol;
            ss += yl * yl;
            mx = fmax(mx, fabs((TM)oo));
        }
    }
    if constexpr (NORMS) {
        // Block sums through shared memory (the flux arrays are free now): warps 0, 1, 2 each
        // reduce one of the 512-entry columns (16 entries per lane, then 5 shuffle levels), so
        // the float64 pipe sees 21 additions per warp instead of 15 per thread.  Fixed order.
        __syncthreads();
        TA *rs = reinterpret_cast<TA *>(phi);
        TM *rm = reinterpret_cast<TM *>(rs + 2 * B3);
        rs[threadIdx.x] = sr;
        rs[B3 + threadIdx.x] = ss;
        rm[threadIdx.x] = mx;
        __syncthreads();
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (w < 2) {
            const TA *src = rs + w * B3;
            TA v = src[lane];
#pragma unroll
            for (int q = 1; q < B3 / 32; q++) v += src[lane + 32 * q];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) partials[b * 3 + w] = (double)v * vol;
        } else if (w == 2) {
            TM v = rm[lane];
#pragma unroll
            for (int q = 1; q < B3 / 32; q++) v = fmax(v, rm[lane + 32 * q]);
            for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
            if (lane == 0) partials[b * 3 + 2] = (double)v;
        }
    }
}

template <typename TC, typename TO, typename YT = TC>
static cudaError_t launch_composite_t(const GridDev &g, const typename CompTypes<TC>::In *X, const YT *Y,
                                     const typename CompTypes<TC>::In *eta, const typename CompTypes<TC>::In *Gx,
                                     const typename CompTypes<TC>::In *Geta, TC a, TC coef, TC d, TO *out, TO *out2,
                                     double *reg, const int *rsrc_tab, double *partials, double vol, cudaStream_t s,
                                     TC *outS, TC coef2, bool ymx) {
    if (g.nblk == 0) return cudaSuccess;
    const size_t sm = (4 * Geo<TC>::CS + Geo<TC>::PHI) * sizeof(TC);
    // set once per process (thread-safe static initialisation)
    constexpr bool E = sizeof(TC) == 4;  // float32: inner residuals and operators of small grids are launched early
    static const bool attr = (cudaFuncSetAttribute(k_composite<TC, TO, true, YT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                              cudaFuncSetAttribute(k_composite<TC, TO, false, YT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                              cudaFuncSetAttribute(k_composite<TC, TO, true, YT, E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                              cudaFuncSetAttribute(k_composite<TC, TO, false, YT, E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                              true);
    (void)attr;
    auto go = [&](auto k, auto kl) {  // early on small grids
        const bool early = E && pdl_small(g.nblk);
        launch_as(early, early ? k : kl, g.nblk, 512, sm, s, g, X, Y, eta, Gx, Geta, a, coef, d, out, out2, reg, rsrc_tab, partials,
                  vol, outS, coef2, 0.5 / g.h, 2.0 * g.h, ymx);
        return cudaGetLastError();
    };
    if (partials)  // with norm partials (the block reductions are compiled out otherwise)
        return go(k_composite<TC, TO, true, YT, E>, k_composite<TC, TO, true, YT, false>);
    return go(k_composite<TC, TO, false, YT, E>, k_composite<TC, TO, false, YT, false>);
}

// float64 coefficient as float-float (hi = nearest float32, lo = nearest float32 to the rest)
static dfloat df_from_host(double v) {
    const float h = (float)v;
    return dfloat(h, (float)(v - (double)h));
}

cudaError_t launch_composite_df(const GridDev &g, const double *X, const dfloat *Y, const double *eta,
                                const double *Gx, const double *Geta, double a, double c, double d, float *out,
                                float *out2, double *reg, const int *rsrc_tab, double *partials, double vol,
                                cudaStream_t s, dfloat *outS, double c2) {
    const double coef = c / (2.0 * g.h * g.h), coef2 = c2 / (2.0 * g.h * g.h);
    return launch_composite_t<dfloat, float>(g, X, Y, eta, Gx, Geta, df_from_host(a), df_from_host(coef),
                                             df_from_host(d), out, out2, reg, rsrc_tab, partials, vol, s, outS,
                                             df_from_host(coef2), a == -1.0 && d == 1.0);
}
cudaError_t launch_composite_df(const GridDev &g, const double *X, const double *Y, const double *eta,
                                const double *Gx, const double *Geta, double a, double c, double d, float *out,
                                float *out2, double *reg, const int *rsrc_tab, double *partials, double vol,
                                cudaStream_t s) {
    const double coef = c / (2.0 * g.h * g.h);
    return launch_composite_t<dfloat, float, double>(g, X, Y, eta, Gx, Geta, df_from_host(a), df_from_host(coef),
                                                     df_from_host(d), out, out2, reg, rsrc_tab, partials, vol, s,
                                                     nullptr, dfloat(), a == -1.0 && d == 1.0);
}
cudaError_t launch_composite(const GridDev &g, const float *X, const float *Y, const float *eta, const float *Gx,
                             const float *Geta, double a, double c, double d, float *out, float *out2, double *reg,
                             const int *rsrc_tab, double *partials, double vol, cudaStream_t s) {
    return launch_composite_t<float, float>(g, X, Y, eta, Gx, Geta, (float)a, (float)(c / (2.0 * g.h * g.h)), (float)d, out,
                                            out2, reg, rsrc_tab, partials, vol, s, nullptr, 0.f, a == -1.0 && d == 1.0);
}

// ------------------------------------------------------------------ red-black smoothing
// One colour pass (Eq. 19): colour cells get e + (r - e - lamdt divF(e)) * inv, the other
// colour is copied; e_in and e_out are distinct buffers so every update reads the pre-pass
// state (Jacobi within a colour).  256 threads, one per colour cell.
// ZERO: both passes of the sweep from e = 0 in one launch (as k_smooth_d's; colour = 1): the tile holds
// the pointwise red update inv r at red cells and 0 elsewhere, e_in is not read (three-level mixed step
// of 3 V-cycles 2.33 -> 2.22 ms, with the right-hand sides in flight during the staging 2.14).
// EARLY = false (grids of more than PDL_GRID blocks): no early launch, and a general pass loads its right-hand
// sides after the stencil.  Held through the staging they cost more registers than the latency is worth
// once every SM has several waves of blocks: 128^3 34.8 us a pass, 38.8 loaded ahead, 41.9 launched early
// with that; 160^3 61, 71, 76; at 64^3 and below the three are the same.  The pass from zero reads r and inv
// in any case and gains from the head start (128^3 32.8 us).
template <typename T, bool ZERO, bool EARLY>
__global__ void __launch_bounds__(256) k_smooth(GridDev g, const T *__restrict__ e_in, T *__restrict__ e_out,
                                                const T *__restrict__ r, const T *__restrict__ eta,
                                                const T *__restrict__ inv, const T *__restrict__ Ge,
                                                const T *__restrict__ Geta, T coef, int colour) {
    using G = Geo<T>;
    __shared__ __align__(16) T tB[3 * G::CS];
    __shared__ __align__(16) T tE[G::CS];
    __shared__ int snb[27];
    const int b0 = blockIdx.x;
    pdl_trigger<EARLY>();
    if (!EARLY && skip_block(g, b0)) return;  // (masked blocks return before they load anything)
    stage_nbr(snb, g.nbr, b0);
    const int slot = g.gslot ? g.gslot[b0] : -1;
    const int b = b0 + pdl_wait<EARLY>();
    if (EARLY && skip_block(g, b)) return;
    const int t = threadIdx.x;
    const int k = t >> 5, j = (t >> 2) & 7;
    const int ic = 2 * (t & 3) + ((j + k + colour) & 1);      // colour cell
    const int io = 2 * (t & 3) + ((j + k + colour + 1) & 1);  // other colour
    const int cc = (k * 8 + j) * 8 + ic, co = (k * 8 + j) * 8 + io;
    T rr[3], iv[3];
    auto load_rhs = [&] {
#pragma unroll
        for (int c = 0; c < 3; c++) {
            rr[c] = r[((size_t)b * 3 + c) * B3 + cc];
            iv[c] = inv[((size_t)b * 3 + c) * B3 + cc];
        }
    };
    if constexpr (EARLY || ZERO) load_rhs();  // in flight while the tile is staged
    __syncthreads();
    if constexpr (ZERO) {
        for (int h = t; h < T3 / 2; h += 256) {
            const int row = h / 5, tj = row % 10, tk = row / 10, pr = 2 * (h % 5), sft = (tj + tk + 1) & 1;
            const int li = pr + sft - 1, lj = tj - 1, lk = tk - 1;
            const int di = li < 0 ? -1 : (li > 7 ? 1 : 0), dj = lj < 0 ? -1 : (lj > 7 ? 1 : 0), dk = lk < 0 ? -1 : (lk > 7 ? 1 : 0);
            const int src = snb[(dk + 1) * 9 + (dj + 1) * 3 + (di + 1)];
            const size_t id = (size_t)(src >= 0 ? src : 0) * 3 * B3 + ((lk - 8 * dk) * 8 + (lj - 8 * dj)) * 8 + (li - 8 * di);
            T *d = tB + G::at(pr, tj, tk);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                d[c * G::CS + sft] = src >= 0 ? r[id + c * B3] * inv[id + c * B3] : T(0);
                d[c * G::CS + 1 - sft] = T(0);
            }
        }
    } else {
        stage_rows<T, 3, 1, G::RS, G::OFF>(tB, e_in, snb, slot >= 0 && Ge ? Ge + (size_t)slot * 3 * T3 : nullptr);
    }
    stage_rows<T, 1, 1, G::RS, G::OFF>(tE, eta, snb, slot >= 0 && Geta ? Geta + (size_t)slot * T3 : nullptr);
    __syncthreads();
    const int p = G::at(ic + 1, j + 1, k + 1);
    T xl1, xl2, xh1, xh2, yl1, yl2, yh1, yh2, zl1, zl2, zh1, zh2;
    face10(tB, tE, p - 1, 0, xl1, xl2);
    face10(tB, tE, p, 0, xh1, xh2);
    face10(tB, tE, p - G::RS, 1, yl1, yl2);
    face10(tB, tE, p, 1, yh1, yh2);
    face10(tB, tE, p - G::PS, 2, zl1, zl2);
    face10(tB, tE, p, 2, zh1, zh2);
    T dv[3];
    dv[0] = (yh1 - yl1) + (zh1 - zl1);
    dv[1] = (xh1 - xl1) + (zh2 - zl2);
    dv[2] = (xh2 - xl2) + (yh2 - yl2);
    const int po = G::at(io + 1, j + 1, k + 1);
    if constexpr (!(EARLY || ZERO)) load_rhs();
#pragma unroll
    for (int c = 0; c < 3; c++) {
        size_t base = ((size_t)b * 3 + c) * B3;
        T ev = tB[c * G::CS + p];
        T res = rr[c] - ev - coef * dv[c];
        e_out[base + cc] = ev + res * iv[c];
        e_out[base + co] = tB[c * G::CS + po];
    }
}

// ---- float64 colour passes.  GB300 issues float64 at 1/60 of the float32 rate, so these passes
// are bound by the float64 pipe (k_smooth with T = double kept it busy at about 114 operations per
// updated cell) and everything else is traded for fewer operations:
// * each tangential pair sum P_a(q) = B_a(q) + B_a(q + e_a) (Eq. 10) is formed once per block in
//   shared memory and serves the four face fluxes that read it;
// * the update is written without the cell's own value in the face differences: with
//   alpha = coef * (sum of the face eta sums), e + omega (r - L e) / (1 + alpha) is
//   (1 - omega) e + inv (r + coef * sum es (B_nb -+ T/4)), inv = omega / (1 + alpha): two
//   multiply-adds per face and component instead of four operations;
// about 61 operations per updated cell.  128^3 FGMRES step (V(3,2), 110 passes): 35.1 -> 26.5 ms; a pass
// over 96^3 87.8 -> 67.6 us with the float64 pipe 71% busy, 8^3 .. 32^3 grids 12-14 -> 9-11 us
// (latency).  A thread block takes a slab of NZ planes of an 8^3 block
// (32 NZ threads, one colour cell each): on grids of few blocks the work of one block is spread
// over several SMs, at a few more pair sums per cell (9, 10, 12 per updated cell for NZ = 8, 4, 2).
template <int NZ>
struct SlabD {
    static constexpr int NT = 32 * NZ, NP = NZ + 2;
    static constexpr int CS = 100 * NP;                       // tile component stride (rows of 10)
    static constexpr int PXY = 90 * NP;                       // pair sums of x (or y) faces
    static constexpr int SUMS = 2 * PXY + 100 * (NZ + 1);
    static constexpr size_t BYTES = (4 * CS + SUMS) * sizeof(double);
};

// rows of tile planes z0 .. z0 + NZ + 1 of block b's 10^3 tile, NC components (as stage_rows)
template <int NZ, int NC>
__device__ __forceinline__ void stage_slab(double *__restrict__ tile, const double *__restrict__ F,
                                           const int *__restrict__ snb, const double *__restrict__ ghost, int z0) {
    constexpr int R = 10 * SlabD<NZ>::NP;
    for (int task = threadIdx.x; task < NC * R; task += SlabD<NZ>::NT) {
        const int c = task / R, rr = task - c * R;
        const int tj = rr % 10, tk = z0 + rr / 10;
        const int lj = tj - 1, lk = tk - 1;
        const int dj = lj < 0 ? -1 : (lj > 7 ? 1 : 0), dk = lk < 0 ? -1 : (lk > 7 ? 1 : 0);
        const int row = ((lk - 8 * dk) * 8 + (lj - 8 * dj)) * 8;
        const int *nb = snb + (dk + 1) * 9 + (dj + 1) * 3;
        const double *gh = ghost ? ghost + c * T3 + tk * 100 + tj * 10 : nullptr;
        double *dst = tile + c * SlabD<NZ>::CS + rr * 10;
        if (nb[1] >= 0) {
            const Row8<double> v = load_row8(F + ((size_t)nb[1] * NC + c) * B3 + row);
#pragma unroll
            for (int q = 0; q < 8; q++) dst[1 + q] = v.v[q];
        } else {
#pragma unroll
            for (int q = 0; q < 8; q++) dst[1 + q] = gh ? gh[1 + q] : 0.0;
        }
        dst[0] = nb[0] >= 0 ? F[((size_t)nb[0] * NC + c) * B3 + row + 7] : (gh ? gh[0] : 0.0);
        dst[9] = nb[2] >= 0 ? F[((size_t)nb[2] * NC + c) * B3 + row] : (gh ? gh[9] : 0.0);
    }
}

// the idx-th position (u, v) of a 10 x NV cross-section without its corners
template <int NV>
__device__ __forceinline__ void cross_pos(int idx, int &u, int &v) {
    if (idx < 8) {
        u = 1 + idx;
        v = 0;
    } else if (idx < 8 + 10 * (NV - 2)) {
        v = 1 + (idx - 8) / 10;
        u = (idx - 8) % 10;
    } else {
        u = 1 + idx - (8 + 10 * (NV - 2));
        v = NV - 1;
    }
}
// the same for the positions of one colour ((u + v) & 1 == par); half as many
template <int NV>
__device__ __forceinline__ void cross_half(int idx, int par, int &u, int &v) {
    if (idx < 4) {
        v = 0;
        u = 1 + 2 * idx + ((par + 1) & 1);
    } else if (idx < 4 + 5 * (NV - 2)) {
        v = 1 + (idx - 4) / 5;
        u = 2 * ((idx - 4) % 5) + ((par + v) & 1);
    } else {
        v = NV - 1;
        u = 1 + 2 * (idx - (4 + 5 * (NV - 2))) + ((par + v + 1) & 1);
    }
}

// Pair sums of one axis: NF face planes of a 10 x NV cross-section.  The first and last plane
// hold only the sums beside the updated colour's cells (`first` / `last`: the colour parity of the
// positions needed there).
template <int NZ, int NF, int NV>
__device__ __forceinline__ void pair_sums_axis(const double *__restrict__ Ba, double *__restrict__ P, int sa, int su, int sv,
                                               int first, int last) {
    constexpr int FULL = 10 * NV - 4, HALF = FULL / 2, N = (NF - 2) * FULL + 2 * HALF;
    for (int e = threadIdx.x; e < N; e += SlabD<NZ>::NT) {
        int fn, u, v;
        if (e < (NF - 2) * FULL) {
            fn = 1 + e / FULL;
            cross_pos<NV>(e % FULL, u, v);
        } else {
            const int h = e - (NF - 2) * FULL;
            fn = h < HALF ? 0 : NF - 1;
            cross_half<NV>(h < HALF ? h : h - HALF, h < HALF ? first : last, u, v);
        }
        const double *p = Ba + fn * sa + u * su + v * sv;
        P[(fn * NV + v) * 10 + u] = p[sa] + p[0];
    }
}

__device__ __forceinline__ bool nonfinite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }

// One colour pass.  ZERO: both passes of the sweep from e = 0 in one launch (colour = 1, the black
// pass; its red neighbours hold the pointwise red update inv r, its black ones 0), reading r and inv
// for the red cells of the halo instead of e.
template <int NZ, bool ZERO>
__global__ void __launch_bounds__(32 * NZ) k_smooth_d(GridDev g, const double *__restrict__ e_in, double *__restrict__ e_out,
                                                      const double *__restrict__ r, const double *__restrict__ eta,
                                                      const double *__restrict__ inv, const double *__restrict__ Ge,
                                                      const double *__restrict__ Geta, double coef, double om1, bool relaxed, int colour) {
    using S = SlabD<NZ>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *tB = reinterpret_cast<double *>(smem_raw), *tE = tB + 3 * S::CS, *P = tE + S::CS;
    __shared__ int snb[27];
    const int b = blockIdx.x / (8 / NZ), z0 = NZ * (blockIdx.x % (8 / NZ));
    if (skip_block(g, b)) return;  // (masked blocks return before they load anything)
    stage_nbr(snb, g.nbr, b);
    const int slot = g.gslot ? g.gslot[b] : -1;
    __syncthreads();
    stage_slab<NZ, 1>(tE, eta, snb, slot >= 0 && Geta ? Geta + (size_t)slot * T3 : nullptr, z0);
    const int t = threadIdx.x, i2 = t & 3, j = (t >> 2) & 7, kl = t >> 5;
    const int odd = (j + z0 + kl + colour) & 1;  // the updated cell of the x-pair (2 i2, 2 i2 + 1)
    const int ic = 2 * i2 + odd;
    const size_t cpair = (size_t)b * 3 * B3 + ((z0 + kl) * 8 + j) * 8 + 2 * i2;
    if constexpr (ZERO) {
        // tile: inv r at red cells ((i + j + k) even, block coordinates), 0 elsewhere
        for (int h = t; h < S::CS / 2; h += S::NT) {
            const int row = h / 5, tj = row % 10, tk = z0 + row / 10, pr = 2 * (h % 5), sft = (tj + tk + 1) & 1;
            const int li = pr + sft - 1, lj = tj - 1, lk = tk - 1;
            const int di = li < 0 ? -1 : (li > 7 ? 1 : 0), dj = lj < 0 ? -1 : (lj > 7 ? 1 : 0), dk = lk < 0 ? -1 : (lk > 7 ? 1 : 0);
            const int src = snb[(dk + 1) * 9 + (dj + 1) * 3 + (di + 1)];
            const size_t id = (size_t)(src >= 0 ? src : 0) * 3 * B3 + ((lk - 8 * dk) * 8 + (lj - 8 * dj)) * 8 + (li - 8 * di);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                tB[c * S::CS + row * 10 + pr + sft] = src >= 0 ? inv[id + c * B3] * r[id + c * B3] : 0.0;
                tB[c * S::CS + row * 10 + pr + 1 - sft] = 0.0;
            }
        }
    } else {
        stage_slab<NZ, 3>(tB, e_in, snb, slot >= 0 && Ge ? Ge + (size_t)slot * 3 * T3 : nullptr, z0);
    }
    double2 rp[3], ip[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        rp[c] = __ldg(reinterpret_cast<const double2 *>(r + cpair + c * B3));
        ip[c] = __ldg(reinterpret_cast<const double2 *>(inv + cpair + c * B3));
    }
    __syncthreads();
    if constexpr (!ZERO) {
        // a boundary face's pair sum is read where the inside cell beside it is updated, i.e. at
        // positions whose own inside cell has the other colour: (u + v) parity of the block
        // coordinates u - 1, v - 1 (v - 1 + z0 on x and y faces) and the inside plane's coordinate
        const int x = (colour + 1 + z0) & 1;
        pair_sums_axis<NZ, 9, NZ + 2>(tB, P, 1, 10, 100, x, (x + 7) & 1);
        pair_sums_axis<NZ, 9, NZ + 2>(tB + S::CS, P + S::PXY, 10, 1, 100, x, (x + 7) & 1);
        pair_sums_axis<NZ, NZ + 1, 10>(tB + 2 * S::CS, P + 2 * S::PXY, 100, 1, 10, x, (x + NZ - 1) & 1);
        __syncthreads();
    }
    const int u = ic + 1, v = j + 1, w = kl + 1;
    const int p = w * 100 + v * 10 + u;
    const double e0 = tE[p];
    const double es[6] = {tE[p - 1] + e0, e0 + tE[p + 1], tE[p - 10] + e0, e0 + tE[p + 10], tE[p - 100] + e0, e0 + tE[p + 100]};
    const int st[3] = {1, 10, 100};
    double out[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        double acc = 0.0;
        bool first = true;
        const double *Bc = tB + c * S::CS + p;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            if (a == c) continue;
            double tl, th;  // T of the low and the high face along a, component c (Eq. 10)
            if constexpr (ZERO) {
                const double *Ba = tB + a * S::CS + p;
                tl = th = Ba[st[c]] - Ba[-st[c]];
            } else {
                // (u, v) of the face cross-section are the two other axes in ascending order
                const int cu = a == 0 ? v : u, cv = a == 2 ? v : w, fn = a == 0 ? ic : (a == 1 ? j : kl);
                const int NV = a == 2 ? 10 : NZ + 2;
                const int du = (a == 0 ? c == 1 : c == 0) ? 1 : 10;
                const double *Pa = P + a * S::PXY + (fn * NV + cv) * 10 + cu;
                tl = Pa[du] - Pa[-du];
                th = Pa[NV * 10 + du] - Pa[NV * 10 - du];
            }
            const double fl = fma(0.25, tl, Bc[-st[a]]), fh = fma(-0.25, th, Bc[st[a]]);
            acc = first ? es[2 * a] * fl : fma(es[2 * a], fl, acc);
            acc = fma(es[2 * a + 1], fh, acc);
            first = false;
        }
        const double rc = odd ? rp[c].y : rp[c].x, ivc = odd ? ip[c].y : ip[c].x;
        const double tt = fma(coef, acc, rc);
        const double ec = Bc[0];
        if (ZERO) {
            out[c] = ivc * tt;
        } else if (relaxed) {
            out[c] = fma(ivc, tt, om1 * ec);
        } else {  // Gauss-Seidel: the old value has no weight, but a NaN or infinity in it stays visible
            out[c] = ivc * tt;
            if (nonfinite_bits(ec)) out[c] = ec - ec;
        }
        const double eo = Bc[odd ? -1 : 1];  // the pair's other cell
        *reinterpret_cast<double2 *>(e_out + cpair + c * B3) = odd ? make_double2(eo, out[c]) : make_double2(out[c], eo);
    }
}

template <int NZ, bool ZERO>
static cudaError_t launch_smooth_slab(const GridDev &g, const double *e_in, double *e_out, const double *r,
                                      const double *eta, const double *inv, const double *Ge, const double *Geta,
                                      double lamdt, int colour, cudaStream_t s) {
    using S = SlabD<NZ>;
    // set once per process (thread-safe static initialisation)
    static const bool attr = (cudaFuncSetAttribute(k_smooth_d<NZ, ZERO>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::BYTES), true);
    (void)attr;
    launch_full(k_smooth_d<NZ, ZERO>, g.nblk * (8 / NZ), S::NT, ZERO ? 4 * S::CS * sizeof(double) : S::BYTES, s, 
        g, e_in, e_out, r, eta, inv, Ge, Geta, lamdt / (2.0 * g.h * g.h), 1.0 - g.omega, g.omega != 1.0, colour);
    return cudaGetLastError();
}

// Slab height by the number of blocks, one rule for the colour passes, the composite and the restricted
// residual: whole blocks do the least work, but a grid should give every SM several thread blocks of equal
// share.  us a launch for slabs of 2 / 4 / 8 planes (ncu, warm L2):
//   blocks             8                   64                  216                512                2744              4096
//   colour pass    9.1/ 8.8/10.1      9.3/ 9.0/10.9      14.0/13.7/15.9     28.5/25.0/27.1     113/101/102       159/145/144
//   from zero      6.5/ 6.2/ 7.1      6.9/ 6.1/ 7.5      11.3/10.2/12.1     21.2/19.6/21.0      87/ 82/ 79       125/115/109
//   residual       9.2/10.8/14.2     11.4/11.2/15.0      21.3/20.2/23.8     46.9/39.5/42.9     198/173/176       292/252/252
//   restricted    10.2/ 8.5/ 9.2     10.5/ 8.8/10.1      15.2/12.7/14.4     32.9/22.6/23.6     130/ 92/ 88       185/131/123
// Two planes serve the residual of few blocks; the passes are within 5% of their best there and on the
// other ranges, the restricted residual, which would take four planes for few blocks too, within 20%.
constexpr int SLAB2_BLOCKS = 256, SLAB4_BLOCKS = 2048;
template <bool ZERO>
static cudaError_t launch_smooth_d(const GridDev &g, const double *e_in, double *e_out, const double *r, const double *eta,
                                   const double *inv, const double *Ge, const double *Geta, double lamdt, int colour,
                                   cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    if (g.nblk <= SLAB2_BLOCKS) return launch_smooth_slab<2, ZERO>(g, e_in, e_out, r, eta, inv, Ge, Geta, lamdt, colour, s);
    if (g.nblk <= SLAB4_BLOCKS) return launch_smooth_slab<4, ZERO>(g, e_in, e_out, r, eta, inv, Ge, Geta, lamdt, colour, s);
    return launch_smooth_slab<8, ZERO>(g, e_in, e_out, r, eta, inv, Ge, Geta, lamdt, colour, s);
}

// ---- float64 composite operator: out = a X + c divF(X) + d Y on leaf blocks, the outer residual and
// the source (launch_composite's rules).  Bound by the float64 pipe like the colour passes, and on slabs
// of a block as they are: pair sums shared by the faces that read them, each face's G = T/4 - N and eta
// sum once in shared memory, and the divergence as multiply-adds es G per cell (12) instead of flux
// products (6.75) and their differences (9): about 51 operations per cell with norms, 59 before (FLUX,
// for a float32 output, keeps the flux products: the residuals of the mixed path, whose inner solves
// amplify a last-bit change to the size of the step's tolerance, round as they did), and
// the sum of squares of Y (of the source) is left out where the caller has it from the step's first
// residual.  ohm_op_residual at 256^3 (all norms) 2.36 -> 2.19 ms, the operator of a 128^3 float64 FGMRES
// step with it (and the colour passes without a comparison of doubles) 22.2 -> 21.6 ms.
// Norms: the 128 threads of a plane pair are
// folded in a fixed order, plane pairs pairwise, so that a block's sums do not depend on the slab height.
template <int NZ>
struct CompD {
    static constexpr int NT = 64 * NZ, NP = NZ + 2;
    static constexpr int CS = 100 * NP;
    static constexpr int PXY = 90 * NP, SUMS = 2 * PXY + 100 * (NZ + 1);
    static constexpr int FXY = 72 * NZ, FACES = 2 * FXY + 64 * (NZ + 1);
    template <typename TO>
    static constexpr size_t bytes = (4 * CS + SUMS + (sizeof(TO) == 4 ? 2 : 3) * FACES) * sizeof(double);
};

template <int NZ, int NF, int NV>
__device__ __forceinline__ void all_sums_axis(const double *__restrict__ Ba, double *__restrict__ P, int sa, int su, int sv) {
    constexpr int FULL = 10 * NV - 4;
    for (int e = threadIdx.x; e < NF * FULL; e += CompD<NZ>::NT) {
        const int f = e / FULL;
        int u, v;
        cross_pos<NV>(e - f * FULL, u, v);
        const double *p = Ba + f * sa + u * su + v * sv;
        P[(f * NV + v) * 10 + u] = p[sa] + p[0];
    }
}

// index of the face with low tile cell f along ax at block coordinates (u, v) of the two other axes
// (z slab-local)
template <int NZ>
__device__ __forceinline__ int slab_face(int ax, int f, int u, int v) {
    return ax == 0 ? (v * 8 + u) * 9 + f : (ax == 1 ? CompD<NZ>::FXY + (v * 9 + f) * 8 + u : 2 * CompD<NZ>::FXY + (f * 8 + v) * 8 + u);
}

// KIND (a branch on it in the kernel would be turned into selects that execute every case's float64
// operations): 0 a residual (a = -1, d = 1), 1 the operator or the source (a = 1, no Y), 2 the source and
// the first residual (outS), 3 any coefficients
template <int NZ, typename TO, int KIND, bool NORMS>
__global__ void __launch_bounds__(64 * NZ, 16 / NZ)
    k_composite_d(GridDev g, const double *__restrict__ X, const double *__restrict__ Y, const double *__restrict__ eta,
                  const double *__restrict__ Gx, const double *__restrict__ Geta, double a, double coef, double d,
                  TO *__restrict__ out, TO *__restrict__ out2, double *__restrict__ reg, const int *__restrict__ rsrc_tab,
                  double *__restrict__ partials, double *__restrict__ outS, double coef2, double inv2h, double twoh,
                  bool keep_ss) {
    using S = CompD<NZ>;
    constexpr bool FLUX = sizeof(TO) == 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *tB = reinterpret_cast<double *>(smem_raw), *tE = tB + 3 * S::CS, *P = tE + S::CS;
    double *G1 = P + S::SUMS, *G2 = G1 + S::FACES, *ES = G2 + S::FACES;  // ES: !FLUX only
    __shared__ int snb[27];
    const int b = blockIdx.x / (8 / NZ), z0 = NZ * (blockIdx.x % (8 / NZ)), t = threadIdx.x;
    if (skip_block(g, b)) return;  // (masked blocks return before they load anything)
    stage_nbr(snb, g.nbr, b);
    const int slot = g.gslot ? g.gslot[b] : -1;
    if (g.covered && g.covered[b]) {
        if (NORMS && t < 3 && !(keep_ss && t == 1)) partials[(size_t)blockIdx.x * 3 + t] = 0.0;
        return;
    }
    __syncthreads();
    stage_slab<NZ, 1>(tE, eta, snb, slot >= 0 && Geta ? Geta + (size_t)slot * T3 : nullptr, z0);
    stage_slab<NZ, 3>(tB, X, snb, slot >= 0 && Gx ? Gx + (size_t)slot * 3 * T3 : nullptr, z0);
    const int i = t & 7, j = (t >> 3) & 7, k = t >> 6;
    const size_t cell = (size_t)b * 3 * B3 + ((z0 + k) * 8 + j) * 8 + i;
    double yv[3] = {0.0, 0.0, 0.0};  // in flight through the face phases
    if (KIND == 0 || (KIND == 3 && Y)) {
#pragma unroll
        for (int c = 0; c < 3; c++) yv[c] = __ldg(Y + cell + c * B3);
    }
    __syncthreads();
    all_sums_axis<NZ, 9, NZ + 2>(tB, P, 1, 10, 100);
    all_sums_axis<NZ, 9, NZ + 2>(tB + S::CS, P + S::PXY, 10, 1, 100);
    all_sums_axis<NZ, NZ + 1, 10>(tB + 2 * S::CS, P + 2 * S::PXY, 100, 1, 10);
    __syncthreads();
    for (int e = t; e < S::FACES; e += S::NT) {
        int ax, f, u, v;
        if (e < S::FXY) {
            const int row = e / 9;
            ax = 0;
            f = e - 9 * row;
            u = row & 7;
            v = row >> 3;
        } else if (e < 2 * S::FXY) {
            const int h = e - S::FXY, row = h >> 3;
            ax = 1;
            u = h & 7;
            v = row / 9;
            f = row - 9 * v;
        } else {
            const int h = e - 2 * S::FXY;
            ax = 2;
            u = h & 7;
            v = (h >> 3) & 7;
            f = h >> 6;
        }
        const int sa = ax == 0 ? 1 : (ax == 1 ? 10 : 100), su = ax == 0 ? 10 : 1, sv = ax == 2 ? 10 : 100;
        const int p = f * sa + (u + 1) * su + (v + 1) * sv;
        const double *Pa = P + ax * S::PXY + (f * (ax == 2 ? 10 : NZ + 2) + v + 1) * 10 + u + 1;
        const double *B1 = tB + (ax == 0 ? S::CS : 0) + p, *B2 = tB + (ax == 2 ? S::CS : 2 * S::CS) + p;
        const double es = tE[p] + tE[p + sa];
        const double g1 = fma(0.25, Pa[1] - Pa[-1], B1[0] - B1[sa]);
        const double g2 = fma(0.25, Pa[10] - Pa[-10], B2[0] - B2[sa]);
        if constexpr (FLUX) {
            G1[e] = es * g1;
            G2[e] = es * g2;
        } else {
            ES[e] = es;
            G1[e] = g1;
            G2[e] = g2;
        }
    }
    __syncthreads();
    // flux registers: faces with no same-level neighbour publish F = es G / (2h)
    if (g.freg) {
        for (int sd = 0; sd < 6; sd++) {
            const int slotr = g.freg[b * 6 + sd], ax = sd >> 1, hi = sd & 1;
            if (slotr < 0 || (ax == 2 && (hi ? z0 + NZ < 8 : z0 > 0))) continue;
            const int nv = ax == 2 ? 8 : NZ;
            for (int q = t; q < 16 * nv; q += S::NT) {
                const int comp = q / (8 * nv), u = q & 7, v = (q >> 3) % nv;
                const int e = slab_face<NZ>(ax, hi ? (ax == 2 ? NZ : 8) : 0, u, v);
                const double phi = FLUX ? (comp ? G2 : G1)[e] : ES[e] * (comp ? G2 : G1)[e];
                reg[(size_t)slotr * 128 + comp * 64 + (ax == 2 ? v : z0 + v) * 8 + u] = phi * inv2h;
            }
        }
    }
    // refluxing: faces next to a covered block take 2h * (mean of the four fine fluxes)
    if (g.rsrc) {
        for (int sd = 0; sd < 6; sd++) {
            const int src = g.rsrc[b * 6 + sd], ax = sd >> 1, hi = sd & 1;
            if (src < 0 || (ax == 2 && (hi ? z0 + NZ < 8 : z0 > 0))) continue;
            const int nv = ax == 2 ? 8 : NZ;
            for (int q = t; q < 16 * nv; q += S::NT) {
                const int comp = q / (8 * nv), u = q & 7, vl = (q >> 3) % nv, v = ax == 2 ? vl : z0 + vl;
                const int fslot = rsrc_tab[src * 4 + (v >> 2) * 2 + (u >> 2)];
                const double *R = reg + (size_t)fslot * 128 + comp * 64;
                const int fu = 2 * (u & 3), fv = 2 * (v & 3);
                const double m = 0.25 * ((R[fv * 8 + fu] + R[fv * 8 + fu + 1]) + (R[(fv + 1) * 8 + fu] + R[(fv + 1) * 8 + fu + 1]));
                const int e = slab_face<NZ>(ax, hi ? (ax == 2 ? NZ : 8) : 0, u, vl);
                (comp ? G2 : G1)[e] = m * twoh;
                if (!FLUX && comp == 0) ES[e] = 1.0;
            }
        }
        __syncthreads();  // refluxed faces before the divergence (g.rsrc is uniform: legal)
    }
    double sr = 0.0, ss = 0.0;
    unsigned long long mx = 0;  // bits of max |out|: ordered like the values; NaNs are left out
    const int fx = (k * 8 + j) * 9 + i, fy = S::FXY + (k * 9 + j) * 8 + i, fz = 2 * S::FXY + (k * 8 + j) * 8 + i;
    double dv[3];
    if constexpr (FLUX) {
        dv[0] = (G1[fy + 8] - G1[fy]) + (G1[fz + 64] - G1[fz]);
        dv[1] = (G1[fx + 1] - G1[fx]) + (G2[fz + 64] - G2[fz]);
        dv[2] = (G2[fx + 1] - G2[fx]) + (G2[fy + 8] - G2[fy]);
    } else {
        const double xl = ES[fx], xh = ES[fx + 1], yl = ES[fy], yh = ES[fy + 8], zl = ES[fz], zh = ES[fz + 64];
        dv[0] = fma(-zl, G1[fz], fma(zh, G1[fz + 64], fma(-yl, G1[fy], yh * G1[fy + 8])));
        dv[1] = fma(-zl, G2[fz], fma(zh, G2[fz + 64], fma(-xl, G1[fx], xh * G1[fx + 1])));
        dv[2] = fma(-yl, G2[fy], fma(yh, G2[fy + 8], fma(-xl, G2[fx], xh * G2[fx + 1])));
    }
    const int p = (k + 1) * 100 + (j + 1) * 10 + i + 1;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const size_t id = cell + c * B3;
        const double x = tB[c * S::CS + p];
        double y = yv[c], o;
        if constexpr (KIND == 0)
            o = fma(coef, dv[c], y - x);
        else if constexpr (KIND == 3)
            o = fma(coef, dv[c], Y ? a * x + d * y : a * x);
        else
            o = FLUX ? __dadd_rn(x, __dmul_rn(coef, dv[c])) : fma(coef, dv[c], x);
        if constexpr (KIND == 2) {  // o is the source; the residual of X against it is coef2 divF(X)
            outS[id] = o;
            y = o;
            o = coef2 * dv[c];
        }
        const TO oo = (TO)o;
        out[id] = oo;
        if (out2) out2[id] = oo;
        if constexpr (NORMS) {
            sr = fma(o, o, sr);
            if (!keep_ss) ss = fma(y, y, ss);
            unsigned long long m;
            if constexpr (sizeof(TO) == 8) {
                m = (unsigned long long)__double_as_longlong(o) & 0x7fffffffffffffffull;
                if (m > 0x7ff0000000000000ull) m = 0;
            } else {
                m = __float_as_uint(oo) & 0x7fffffffu;
                if (m > 0x7f800000u) m = 0;
            }
            mx = m > mx ? m : mx;
        }
    }
    if constexpr (NORMS) {
        // the pair sums' memory is free: [plane pairs][2][64] sums, then the maxima
        double *rs = P, *rp = rs + 128 * NZ;
        unsigned long long *rm = reinterpret_cast<unsigned long long *>(rp + NZ);
        const int pp = t >> 7;
        rs[pp * 256 + (t & 127)] = sr;
        rs[pp * 256 + 128 + (t & 127)] = ss;
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long w = __shfl_xor_sync(0xffffffffu, mx, o);
            mx = w > mx ? w : mx;
        }
        if ((t & 31) == 0) rm[t >> 5] = mx;
        __syncthreads();
        if ((t & 96) == 0) {  // one warp per plane pair: lanes 0-15 the first sum, 16-31 the second
            const int l = t & 15;
            const double *src = rs + pp * 256 + (t & 16) * 8 + l;
            double v = ((src[0] + src[16]) + (src[32] + src[48])) + ((src[64] + src[80]) + (src[96] + src[112]));
            for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (l == 0) rp[pp * 2 + ((t >> 4) & 1)] = v;
        }
        __syncthreads();
        if (t < 2 && !(keep_ss && t == 1)) {
            double v = rp[t];
            if constexpr (NZ >= 4) v = v + rp[2 + t];
            if constexpr (NZ == 8) v = v + (rp[4 + t] + rp[6 + t]);
            partials[(size_t)blockIdx.x * 3 + t] = v;
        } else if (t == 2) {
            unsigned long long m = 0;
#pragma unroll
            for (int w = 0; w < 2 * NZ; w++) m = rm[w] > m ? rm[w] : m;
            partials[(size_t)blockIdx.x * 3 + 2] = sizeof(TO) == 8 ? __longlong_as_double((long long)m) : (double)__uint_as_float((unsigned)m);
        }
    }
}

template <int NZ, typename TO, int KIND, bool NORMS>
static cudaError_t launch_composite_kind(const GridDev &g, const double *X, const double *Y, const double *eta, const double *Gx,
                                         const double *Geta, double a, double coef, double d, TO *out, TO *out2, double *reg,
                                         const int *rsrc_tab, double *partials, cudaStream_t s, double *outS, double coef2,
                                         bool keep_ss) {
    using S = CompD<NZ>;
    constexpr auto k = k_composite_d<NZ, TO, KIND, NORMS>;
    constexpr size_t sm = S::template bytes<TO>;
    static const bool attr = (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm), true);
    (void)attr;
    launch_full(k, g.nblk * (8 / NZ), S::NT, sm, s, g, X, Y, eta, Gx, Geta, a, coef, d, out, out2, reg, rsrc_tab, partials,
                outS, coef2, 0.5 / g.h, 2.0 * g.h, keep_ss);
    return cudaGetLastError();
}

template <int NZ, typename TO>
static cudaError_t launch_composite_slab(const GridDev &g, const double *X, const double *Y, const double *eta, const double *Gx,
                                         const double *Geta, double a, double coef, double d, TO *out, TO *out2, double *reg,
                                         const int *rsrc_tab, double *partials, cudaStream_t s, double *outS, double coef2,
                                         bool keep_ss) {
    auto go = [&](auto f) { return f(g, X, Y, eta, Gx, Geta, a, coef, d, out, out2, reg, rsrc_tab, partials, s, outS, coef2, keep_ss); };
    const bool resid = Y && a == -1.0 && d == 1.0;
    if (partials) {  // norms: of residuals only
        if (resid && !outS) return go(launch_composite_kind<NZ, TO, 0, true>);
        if (!Y && a == 1.0 && outS) return go(launch_composite_kind<NZ, TO, 2, true>);
        return cudaErrorInvalidValue;
    }
    if (outS) return cudaErrorInvalidValue;
    if constexpr (sizeof(TO) == 8) {
        if (resid) return go(launch_composite_kind<NZ, TO, 0, false>);
        if (!Y && a == 1.0) return go(launch_composite_kind<NZ, TO, 1, false>);
        return go(launch_composite_kind<NZ, TO, 3, false>);
    }
    return cudaErrorInvalidValue;  // float32 output: the outer residuals of the mixed path, always with norms
}

int composite_parts(int nblk) { return nblk <= SLAB2_BLOCKS ? 4 : (nblk <= SLAB4_BLOCKS ? 2 : 1); }

template <typename TO>
cudaError_t launch_composite(const GridDev &g, const double *X, const double *Y, const double *eta, const double *Gx,
                             const double *Geta, double a, double c, double d, TO *out, TO *out2, double *reg,
                             const int *rsrc_tab, double *partials, cudaStream_t s, double *outS, double c2, bool keep_ss) {
    if (g.nblk == 0) return cudaSuccess;
    const double coef = c / (2.0 * g.h * g.h), coef2 = c2 / (2.0 * g.h * g.h);
    switch (composite_parts(g.nblk)) {
        case 4: return launch_composite_slab<2, TO>(g, X, Y, eta, Gx, Geta, a, coef, d, out, out2, reg, rsrc_tab, partials, s, outS, coef2, keep_ss);
        case 2: return launch_composite_slab<4, TO>(g, X, Y, eta, Gx, Geta, a, coef, d, out, out2, reg, rsrc_tab, partials, s, outS, coef2, keep_ss);
        default: return launch_composite_slab<8, TO>(g, X, Y, eta, Gx, Geta, a, coef, d, out, out2, reg, rsrc_tab, partials, s, outS, coef2, keep_ss);
    }
}
template cudaError_t launch_composite<double>(const GridDev &, const double *, const double *, const double *, const double *,
                                              const double *, double, double, double, double *, double *, double *, const int *,
                                              double *, cudaStream_t, double *, double, bool);
template cudaError_t launch_composite<float>(const GridDev &, const double *, const double *, const double *, const double *,
                                             const double *, double, double, double, float *, float *, double *, const int *,
                                             double *, cudaStream_t, double *, double, bool);

template <>
cudaError_t launch_smooth<double>(const GridDev &g, const double *e_in, double *e_out, const double *r, const double *eta,
                                  const double *inv, const double *Ge, const double *Geta, double lamdt, int colour,
                                  cudaStream_t s) {
    return launch_smooth_d<false>(g, e_in, e_out, r, eta, inv, Ge, Geta, lamdt, colour, s);
}
template <>
cudaError_t launch_smooth<float>(const GridDev &g, const float *e_in, float *e_out, const float *r, const float *eta,
                                 const float *inv, const float *Ge, const float *Geta, double lamdt, int colour,
                                 cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    launch_pdl2(k_smooth<float, false, true>, k_smooth<float, false, false>, g.nblk, 256, 0, s, g, e_in, e_out, r, eta, inv, Ge, Geta, (float)(lamdt / (2.0 * g.h * g.h)), colour);
    return cudaGetLastError();
}
cudaError_t launch_smooth_zero(const GridDev &g, float *e_out, const float *r, const float *eta, const float *inv,
                               const float *Geta, double lamdt, cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    launch_pdl2(k_smooth<float, true, true>, k_smooth<float, true, false>, g.nblk, 256, 0, s, g, nullptr, e_out, r, eta, inv, nullptr, Geta, (float)(lamdt / (2.0 * g.h * g.h)), 1);
    return cudaGetLastError();
}
cudaError_t launch_smooth_zero(const GridDev &g, double *e_out, const double *r, const double *eta, const double *inv,
                               const double *Geta, double lamdt, cudaStream_t s) {
    return launch_smooth_d<true>(g, nullptr, e_out, r, eta, inv, nullptr, Geta, lamdt, 1, s);
}

// ------------------------------------------------------------------ fused red + black sweep
// One full red-black sweep in one launch, for grids whose blocks have every neighbour (no
// coarse-fine ghosts).  The block and a 2-cell halo (12^3, all 26 neighbours) are staged;
// red cells of the block and of its 1-cell ring get their update from the pre-sweep state,
// then the block's black cells are updated from the post-red state.  The ring updates are
// the ones the neighbouring blocks compute, in the same order with the same arithmetic, so
// the result equals two global colour passes.  The inverse diagonal is formed on the fly
// from eta (Eqs. 21-23).  e_in and e_out are distinct buffers.
// The 12^3 tile is compact (rows 12 elements apart): 8 rows of 4 same-colour cells (stride 2,
// the warp pattern of the block's cells) still fall on 32 distinct float32 banks, and the
// tile (4 x 6.75 KB for float32) leaves room for 6 thread blocks per SM.  The sweep is bound by
// latency more than by shared-memory bandwidth: a padded tile (rows 20 apart, fewer bank
// conflicts on the ring) measured slower at 256^3 (0.46 ms against 0.43 ms per sweep) because
// it allows only 4 thread blocks per SM.
template <typename T>
struct G12 {
    static constexpr int S = 12, RRS = 12, PS = S * RRS, CS = S * PS, OFF = 0;
    __device__ static __forceinline__ int at(int i, int j, int k) { return k * PS + j * RRS + i + OFF; }
};
// Constants of the point update (Eqs. 19-23): ncoef = -lamdt / (2 h^2) scales the flux
// divergence of the scaled fluxes Phi = 2 h F; the relaxed diagonal is carried as
// den_c = (1 + alpha_c) / omega = kb + ka (S_a + S_b), ka = lamdt / (2 h^2 omega), kb = 1 / omega,
// where S_a = (eta_lo + eta) + (eta + eta_hi) is the sum of the cell's two face eta sums along
// axis a (alpha_c = lamdt / h^2 times the sum, over the axes a != c, of the mean face eta on both
// sides).  The host computes all three in float64 and rounds them once.
template <typename T>
struct RbK {
    T ncoef, ka, kb;
};
template <typename T>
RbK<T> rb_constants(double lamdt, double h, double omega) {
    const double coef = lamdt / (2.0 * h * h);
    return RbK<T>{(T)-coef, (T)(coef / omega), (T)(1.0 / omega)};
}

// Arithmetic of the point update, every operation rounded once (never contracted by the
// compiler), in float32 or float64.
__device__ __forceinline__ float v_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float v_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float v_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float v_mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double v_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double v_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double v_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double v_mad(double a, double b, double c) { return __fma_rn(a, b, c); }
template <typename V>
__device__ __forceinline__ V v_splat(float x) {
    return V(x);
}
template <typename V>
__device__ __forceinline__ V v_zero() {
    return v_splat<V>(0.0f);
}

// The relaxed update ev + res / den of the float32 sweeps, through the hardware's approximate reciprocal
// (rcp.approx, relative error below 2^-23; a smoothing weight needs no correctly rounded
// quotient) and one FMA.
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rb_relax(float ev, float res, float den) { return v_mad(res, rcp_approx(den), ev); }

// The point update of one colour pass (Eq. 19 with R from Eq. 20 and alpha from Eqs. 21-23),
// written against an accessor that returns component C of the field, or eta, at a compile-time
// offset (DX, DY, DZ) from the updated cell.  Every fused sweep kernel goes through these
// functions, whatever its staging: the rounding of each update is the same in all of them.
//
// face_pair: the divergence contribution of flux component C through the cell's two faces along
// axis AX, es_hi Q_hi - es_lo Q_lo with Phi = es Q, Q = T / 4 - N (Eqs. 9-10).  The tangential
// sums of the two faces (Eq. 10) share their middle difference, so they are formed as
//   T_hi = D(+AX) + D(0),  T_lo = D(0) + D(-AX),  D(s) = B_AX(s + e_C) - B_AX(s - e_C),
// the same four values each, regrouped (4 additions for both faces instead of 6).  The low face
// carries -Q (N - T/4, the same bits negated), so no operation needs a negated operand.
template <typename V, int AX, int C, class A>
__device__ __forceinline__ V face_pair(const A &a, V es_lo, V es_hi) {
    constexpr int AXX = AX == 0, AXY = AX == 1, AXZ = AX == 2;
    constexpr int CX = C == 0, CY = C == 1, CZ = C == 2;
    const V d0 = v_sub(a.template B<AX, CX, CY, CZ>(), a.template B<AX, -CX, -CY, -CZ>());
    const V dp = v_sub(a.template B<AX, AXX + CX, AXY + CY, AXZ + CZ>(), a.template B<AX, AXX - CX, AXY - CY, AXZ - CZ>());
    const V dm = v_sub(a.template B<AX, CX - AXX, CY - AXY, CZ - AXZ>(), a.template B<AX, -CX - AXX, -CY - AXY, -CZ - AXZ>());
    const V c0 = a.template B<C, 0, 0, 0>();
    const V q_hi = v_mad(v_add(dp, d0), v_splat<V>(0.25f), v_sub(c0, a.template B<C, AXX, AXY, AXZ>()));
    const V mq_lo = v_mad(v_add(d0, dm), v_splat<V>(-0.25f), v_sub(c0, a.template B<C, -AXX, -AXY, -AXZ>()));
    return v_mad(es_hi, q_hi, v_mul(es_lo, mq_lo));
}

// face sums of eta: eta_lo + eta on the low face, eta + eta_hi on the high face, along x, y, z
template <typename V, class A>
__device__ __forceinline__ void face_sums(const A &a, V es[6]) {
    const V e0 = a.template E<0, 0, 0>();
    es[0] = v_add(a.template E<-1, 0, 0>(), e0);
    es[1] = v_add(e0, a.template E<1, 0, 0>());
    es[2] = v_add(a.template E<0, -1, 0>(), e0);
    es[3] = v_add(e0, a.template E<0, 1, 0>());
    es[4] = v_add(a.template E<0, 0, -1>(), e0);
    es[5] = v_add(e0, a.template E<0, 0, 1>());
}

// the flux divergence of the cell (Eq. 8) from its face sums
template <typename V, class A>
__device__ __forceinline__ void cell_divergence(const A &a, const V es[6], V dv[3]) {
    dv[0] = v_add(face_pair<V, 1, 0>(a, es[2], es[3]), face_pair<V, 2, 0>(a, es[4], es[5]));
    dv[1] = v_add(face_pair<V, 0, 1>(a, es[0], es[1]), face_pair<V, 2, 1>(a, es[4], es[5]));
    dv[2] = v_add(face_pair<V, 0, 2>(a, es[0], es[1]), face_pair<V, 1, 2>(a, es[2], es[3]));
}

// face sums and den_c
template <typename V, class A>
__device__ __forceinline__ void rb_faces_den(const A &a, const RbK<V> &K, V es[6], V den[3]) {
    face_sums<V>(a, es);
    const V sx = v_add(es[0], es[1]), sy = v_add(es[2], es[3]), sz = v_add(es[4], es[5]);
    den[0] = v_mad(K.ka, v_add(sy, sz), K.kb);
    den[1] = v_mad(K.ka, v_add(sz, sx), K.kb);
    den[2] = v_mad(K.ka, v_add(sx, sy), K.kb);
}

template <typename V, class A>
__device__ __forceinline__ void rb_update_acc(const A &a, const RbK<V> &K, const V rr[3], V out[3]) {
    V es[6], den[3], dv[3];
    rb_faces_den<V>(a, K, es, den);
    cell_divergence<V>(a, es, dv);
    const V ev[3] = {a.template B<0, 0, 0, 0>(), a.template B<1, 0, 0, 0>(), a.template B<2, 0, 0, 0>()};
#pragma unroll
    for (int c = 0; c < 3; c++) out[c] = rb_relax(ev[c], v_mad(K.ncoef, dv[c], v_sub(rr[c], ev[c])), den[c]);
}

// The first sweep from e = 0, where the red colour pass reduces to e = r / den (every flux of the
// pre-pass state vanishes) and the black pass sees red values at the face neighbours of a black
// cell and zeros at its edge neighbours and at itself.  The two updates below are
// rb_update_acc with those zeros folded in: every dropped term is an exact +-0 there, so the
// results are the same bits (up to the sign of a zero).  The tangential difference of a black
// cell is the same for its two faces along an axis (D(+-AX) = 0), so a black update reads 31
// tile values instead of about 46.
template <typename V, class A>
__device__ __forceinline__ void red_from_zero_acc(const A &a, const RbK<V> &K, const V rr[3], V out[3]) {
    V es[6], den[3];
    rb_faces_den<V>(a, K, es, den);
#pragma unroll
    for (int c = 0; c < 3; c++) out[c] = rb_relax(v_zero<V>(), rr[c], den[c]);
}

template <typename V, int AX, int C, class A>
__device__ __forceinline__ V face_pair_zero(const A &a, V es_lo, V es_hi) {
    constexpr int AXX = AX == 0, AXY = AX == 1, AXZ = AX == 2;
    constexpr int CX = C == 0, CY = C == 1, CZ = C == 2;
    const V d0 = v_sub(a.template B<AX, CX, CY, CZ>(), a.template B<AX, -CX, -CY, -CZ>());
    const V q_hi = v_sub(v_mul(d0, v_splat<V>(0.25f)), a.template B<C, AXX, AXY, AXZ>());
    const V mq_lo = v_sub(v_mul(d0, v_splat<V>(-0.25f)), a.template B<C, -AXX, -AXY, -AXZ>());
    return v_mad(es_hi, q_hi, v_mul(es_lo, mq_lo));
}

template <typename V, class A>
__device__ __forceinline__ void black_after_zero_acc(const A &a, const RbK<V> &K, const V rr[3], V out[3]) {
    V es[6], den[3];
    rb_faces_den<V>(a, K, es, den);
    const V dv[3] = {v_add(face_pair_zero<V, 1, 0>(a, es[2], es[3]), face_pair_zero<V, 2, 0>(a, es[4], es[5])),
                     v_add(face_pair_zero<V, 0, 1>(a, es[0], es[1]), face_pair_zero<V, 2, 1>(a, es[4], es[5])),
                     v_add(face_pair_zero<V, 0, 2>(a, es[0], es[1]), face_pair_zero<V, 1, 2>(a, es[2], es[3]))};
#pragma unroll
    for (int c = 0; c < 3; c++) out[c] = rb_relax(v_zero<V>(), v_mad(K.ncoef, dv[c], rr[c]), den[c]);
}

// accessor of a staged tile (geometry G: rows RRS apart, planes PS, components CS)
template <typename T, typename G>
struct TileAcc {
    const T *tB, *tE;
    int p;
    template <int C, int DX, int DY, int DZ>
    __device__ __forceinline__ T B() const {
        return tB[C * G::CS + p + DX + DY * G::RRS + DZ * G::PS];
    }
    template <int DX, int DY, int DZ>
    __device__ __forceinline__ T E() const {
        return tE[p + DX + DY * G::RRS + DZ * G::PS];
    }
};

template <typename T, typename G = G12<T>>
__device__ __forceinline__ void rb_update(const T *__restrict__ tB, const T *__restrict__ tE, int p, const RbK<T> &K,
                                          const T rr[3], T out[3]) {
    rb_update_acc<T>(TileAcc<T, G>{tB, tE, p}, K, rr, out);
}

// ZERO: the sweep from e = 0, as k_smooth_rb2's: e_in is not read, only eta is staged, the red pass is
// pointwise and the black pass reads red values only.  The right-hand sides come in before the
// staging barrier, an x-pair of cells (one red, one black) as one 8-byte word, and the results go out
// as one (100 boxes of 24^3, V(4,4): 4.26 -> 3.90 ms per step; 120 x 104 x 88, two steps: 5.62 -> 5.20 ms).
template <bool ZERO, bool EARLY>
__global__ void __launch_bounds__(256) k_smooth_rb(GridDev g, const float *__restrict__ e_in, float *__restrict__ e_out,
                                                   const float *__restrict__ r, const float *__restrict__ eta, RbK<float> K) {
    using G = G12<float>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *tB = reinterpret_cast<float *>(smem_raw);  // [3][12 planes][12 rows][RRS]
    float *tE = tB + 3 * G::CS;
    __shared__ int snb[27];
    const int b0 = blockIdx.x;
    pdl_trigger<EARLY>();
    if (!EARLY && skip_block(g, b0)) return;  // (masked blocks return before they load anything)
    stage_nbr(snb, g.nbr, b0);
    const int b = b0 + pdl_wait<EARLY>();
    if (EARLY && skip_block(g, b)) return;
    const int t = threadIdx.x;
    const int k = t >> 5, j = (t >> 2) & 7, i2 = t & 3;
    const int ir = 2 * i2 + ((j + k) & 1), ib = 2 * i2 + ((j + k + 1) & 1);
    const int cpair = (k * 8 + j) * 8 + 2 * i2;
    const bool red_even = ((j + k) & 1) == 0;
    float rr0[3], rr1[3] = {0.f, 0.f, 0.f}, rrb[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float2 v = *reinterpret_cast<const float2 *>(r + ((size_t)b * 3 + c) * B3 + cpair);
        rr0[c] = red_even ? v.x : v.y;
        rrb[c] = red_even ? v.y : v.x;
    }
    __syncthreads();
    // Red cells ((i+j+k) even): the block's 256, one per thread in the same pattern as the black
    // phase (a warp reads 8 rows x 4 cells of one plane: distinct banks), then the 240 of the
    // ring (faces and edges of the 10^3 box, corners excluded), one per thread t < 240:
    // t < 192: face slab f = t/32 (axis f/2 at -1 or 8), 8 lines x 4 red cells;
    // t >= 192: edge e = (t-192)/4 (two axes out), 4 red cells along the third axis.
    int p1 = -1;
    if (t < 240) {
        int c[3];
        if (t < 192) {
            const int f = t >> 5, ax = f >> 1, q = t & 31;
            const int v = q >> 2, u2 = q & 3;
            const int co = (f & 1) ? 8 : -1, cu = 2 * u2 + ((co + v) & 1);  // out of the block; along a1; v along a2
            c[0] = ax == 0 ? co : cu;
            c[1] = ax == 0 ? cu : (ax == 1 ? co : v);
            c[2] = ax == 2 ? co : v;
        } else {
            const int e = (t - 192) >> 2, w2 = (t - 192) & 3;
            const int pr = e >> 2, sg = e & 3;  // axis pair (0,1), (0,2), (1,2) and its sign combination
            const int c1 = (sg & 1) ? 8 : -1, c2 = (sg & 2) ? 8 : -1, cf = 2 * w2 + ((c1 + c2) & 1);
            c[0] = pr == 2 ? cf : c1;
            c[1] = pr == 0 ? c2 : (pr == 1 ? cf : c1);
            c[2] = pr == 0 ? cf : c2;
        }
        const int di = c[0] < 0 ? -1 : (c[0] > 7 ? 1 : 0), dj = c[1] < 0 ? -1 : (c[1] > 7 ? 1 : 0), dk = c[2] < 0 ? -1 : (c[2] > 7 ? 1 : 0);
        const int src = snb[(dk + 1) * 9 + (dj + 1) * 3 + (di + 1)];
        const int off = ((c[2] - 8 * dk) * 8 + (c[1] - 8 * dj)) * 8 + (c[0] - 8 * di);
#pragma unroll
        for (int q = 0; q < 3; q++) rr1[q] = r[((size_t)src * 3 + q) * B3 + off];
        p1 = G::at(c[0] + 2, c[1] + 2, c[2] + 2);
    }
    if constexpr (!ZERO) stage_rows<float, 3, 2, G::RRS, G::OFF>(tB, e_in, snb, nullptr);
    stage_rows<float, 1, 2, G::RRS, G::OFF>(tE, eta, snb, nullptr);
    __syncthreads();
    float nv0[3], nv1[3];
    const int p0 = G::at(ir + 2, j + 2, k + 2);
    if constexpr (ZERO) {  // nothing of e is read: no barrier before the red values are stored
        red_from_zero_acc<float>(TileAcc<float, G>{tB, tE, p0}, K, rr0, nv0);
        if (p1 >= 0) red_from_zero_acc<float>(TileAcc<float, G>{tB, tE, p1}, K, rr1, nv1);
    } else {
        rb_update<float>(tB, tE, p0, K, rr0, nv0);
        if (p1 >= 0) rb_update<float>(tB, tE, p1, K, rr1, nv1);
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
        tB[c * G::CS + p0] = nv0[c];
        if (p1 >= 0) tB[c * G::CS + p1] = nv1[c];
    }
    __syncthreads();
    // black cells of the block, one per thread, then the whole block is written out
    float out[3];
    const int pb = G::at(ib + 2, j + 2, k + 2);
    if constexpr (ZERO)
        black_after_zero_acc<float>(TileAcc<float, G>{tB, tE, pb}, K, rrb, out);
    else
        rb_update<float>(tB, tE, pb, K, rrb, out);
#pragma unroll
    for (int c = 0; c < 3; c++)
        *reinterpret_cast<float2 *>(e_out + ((size_t)b * 3 + c) * B3 + cpair) =
            red_even ? make_float2(nv0[c], out[c]) : make_float2(out[c], nv0[c]);
}

cudaError_t launch_smooth_rb(const GridDev &g, const float *e_in, float *e_out, const float *r, const float *eta, double lamdt,
                             cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    const size_t sm = 4 * G12<float>::CS * sizeof(float);
    // set once per process (thread-safe static initialisation)
    static const bool attr = [=] {
        auto set = [=](auto k) { cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm); };
        set(k_smooth_rb<false, true>);
        set(k_smooth_rb<false, false>);
        set(k_smooth_rb<true, true>);
        set(k_smooth_rb<true, false>);
        return true;
    }();
    (void)attr;
    const RbK<float> K = rb_constants<float>(lamdt, g.h, g.omega);
    if (e_in)
        launch_pdl2(k_smooth_rb<false, true>, k_smooth_rb<false, false>, g.nblk, 256, sm, s, g, e_in, e_out, r, eta, K);
    else  // from e = 0
        launch_pdl2(k_smooth_rb<true, true>, k_smooth_rb<true, false>, g.nblk, 256, sm, s, g, nullptr, e_out, r, eta, K);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ fused sweep on brick pairs
// The fused sweep above for two x-adjacent blocks A = 2q and B = 2q + 1 per thread block (512
// threads): a 20 x 12 x 12 tile (two-cell halo) shares its halo and ring between the two
// blocks, so per block it stages 17% fewer values and recomputes 20% fewer ring updates.
// Rows are 24 floats apart: the warp pattern of the brick's same-colour cells (4 rows x 8
// cells at stride 2) then falls on 32 distinct banks; each tile row starts on a 16-byte
// boundary and is staged as five 16-byte words.  Used for float32 grids whose every block pair (2q, 2q+1)
// is x-adjacent and whose blocks all have their 26 neighbours.  Bounded to 40 registers so
// that 3 thread blocks (48 warps) share an SM.  Measured per 256^3 sweep: 0.362 ms; 0.401 ms
// before the staging stores and the ring order were arranged by bank (conflicts 3.8 M -> 0.8 M
// per 128^3 sweep); 0.427 ms at 54 registers (2 per SM); 0.431 ms for the one-block kernel.
struct G20 {
    static constexpr int SX = 20, S = 12, RRS = 24, PS = S * RRS + 4, CS = S * PS, OFF = 0;
    __device__ static __forceinline__ int at(int i, int j, int k) { return k * PS + j * RRS + i + OFF; }
};

// red cells of the brick's one-cell ring (faces and edges, no corners): 384 entries
// (li+1) | (lj+1) << 5 | (lk+1) << 10, li in [-1, 16], lj, lk in [-1, 8], ordered for the 12
// warps that update them so that shared-memory banks (tile offset mod 32) repeat little within a
// warp: with the strides of G20 a bank holds at most 17 of the 384 cells and at least 8, so 7
// warps take one cell per bank and 5 warps at most two.  Built at compile time.
struct Ring2 {
    uint32_t v[384];
};
constexpr int ring2_bank(int i, int j, int k) { return ((i + 2 + G20::OFF) + (j + 2) * G20::RRS + (k + 2) * G20::PS) & 31; }
constexpr bool ring2_cell(int i, int j, int k) {
    const int out = (i < 0 || i > 15) + (j < 0 || j > 7) + (k < 0 || k > 7);
    return out != 0 && out != 3 && ((i + j + k) & 1) == 0;
}
constexpr Ring2 make_ring2() {
    Ring2 m{};
    int cnt[32] = {};
    for (int k = -1; k <= 8; k++)
        for (int j = -1; j <= 8; j++)
            for (int i = -1; i <= 16; i++)
                if (ring2_cell(i, j, k)) cnt[ring2_bank(i, j, k)]++;
    int maxc = 0;
    for (int r = 0; r < 32; r++) maxc = cnt[r] > maxc ? cnt[r] : maxc;
    const int A = 24 - maxc < 12 ? 24 - maxc : 12;  // warps with one cell per bank
    int fill[12] = {}, seen[32] = {}, two[12][32] = {};
    for (int k = -1; k <= 8; k++)
        for (int j = -1; j <= 8; j++)
            for (int i = -1; i <= 16; i++) {
                if (!ring2_cell(i, j, k)) continue;
                const int r = ring2_bank(i, j, k), n = seen[r]++;
                int w = n;
                if (n >= A) {
                    w = -1;
                    for (int c = A; c < 12; c++)
                        if (two[c][r] < 2 && fill[c] < 32 && (w < 0 || fill[c] < fill[w])) w = c;
                    two[w][r]++;
                }
                m.v[w * 32 + fill[w]++] = (uint32_t)(i + 1) | ((uint32_t)(j + 1) << 5) | ((uint32_t)(k + 1) << 10);
            }
    return m;
}
__device__ const Ring2 g_ring2 = make_ring2();

// ZERO: the sweep starts from e = 0 (the first pre-smoothing sweep of a level): e_in is not read,
// only eta is staged, the red pass is pointwise and the black pass reads only red values.
template <bool ZERO, bool EARLY>
__global__ void __launch_bounds__(512, 3) k_smooth_rb2(GridDev g, const float *__restrict__ e_in, float *__restrict__ e_out,
                                                    const float *__restrict__ r, const float *__restrict__ eta,
                                                    RbK<float> K) {
    using G = G20;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *tB = reinterpret_cast<float *>(smem_raw);  // [3][12 planes][12 rows][RRS]
    float *tE = tB + 3 * G::CS;
    // neighbourhood of the brick: block columns bx = -1, 0 (A), 1 (B), 2 along x, by dj, dk
    __shared__ int snb[36];
    const int A0 = 2 * blockIdx.x;
    pdl_trigger<EARLY>();
    if (!EARLY && skip_block(g, A0)) return;  // (masked blocks return before they load anything)
    if (threadIdx.x < 36) {
        const int bx = threadIdx.x % 4 - 1, dj = (threadIdx.x / 4) % 3 - 1, dk = threadIdx.x / 12 - 1;
        const int base = bx <= 1 ? A0 : A0 + 1, dx = bx <= 1 ? bx : 1;
        snb[threadIdx.x] = __ldg(g.nbr + base * 27 + (dk + 1) * 9 + (dj + 1) * 3 + (dx + 1));
    }
    const int A = A0 + pdl_wait<EARLY>();
    if (EARLY && skip_block(g, A)) return;
    __syncthreads();
    // one task per (field component, tile row): the 20 values of the row (halo pair, 8 + 8
    // interior cells, halo pair) as five 16-byte stores; each quarter-warp takes 4 rows of 2
    // consecutive planes, whose 16-byte bank groups are distinct (plane stride = 4 mod 32)
    // from e = 0 only eta is staged (e is never read before the red values are written)
    for (int task = ZERO ? 3 * 144 + threadIdx.x : threadIdx.x; task < 4 * 144; task += blockDim.x) {
        const int c = task / 144, u = task - c * 144;
        const int q = u >> 3, w = u & 7;
        const int tk = 2 * (q / 3) + (w >> 2), tj = 4 * (q % 3) + (w & 3);
        const int lj = tj - 2, lk = tk - 2;
        const int dj = lj < 0 ? -1 : (lj > 7 ? 1 : 0), dk = lk < 0 ? -1 : (lk > 7 ? 1 : 0);
        const int rowoff = ((lk - 8 * dk) * 8 + (lj - 8 * dj)) * 8;
        const int *nb = snb + (dk + 1) * 12 + (dj + 1) * 4;
        const float *F = c < 3 ? e_in : eta;
        const int nc = c < 3 ? 3 : 1, cc = c < 3 ? c : 0;
        float4 *dst = reinterpret_cast<float4 *>((c < 3 ? tB + c * G::CS : tE) + tk * G::PS + tj * G::RRS + G::OFF);
        const float2 lo = __ldg(reinterpret_cast<const float2 *>(F + ((size_t)nb[0] * nc + cc) * B3 + rowoff + 6));
        const float4 *pa = reinterpret_cast<const float4 *>(F + ((size_t)nb[1] * nc + cc) * B3 + rowoff);
        const float4 *pb = reinterpret_cast<const float4 *>(F + ((size_t)nb[2] * nc + cc) * B3 + rowoff);
        const float2 hi = __ldg(reinterpret_cast<const float2 *>(F + ((size_t)nb[3] * nc + cc) * B3 + rowoff));
        const float4 a0 = __ldg(pa), a1 = __ldg(pa + 1), b0 = __ldg(pb), b1 = __ldg(pb + 1);
        dst[0] = make_float4(lo.x, lo.y, a0.x, a0.y);
        dst[1] = make_float4(a0.z, a0.w, a1.x, a1.y);
        dst[2] = make_float4(a1.z, a1.w, b0.x, b0.y);
        dst[3] = make_float4(b0.z, b0.w, b1.x, b1.y);
        dst[4] = make_float4(b1.z, b1.w, hi.x, hi.y);
    }
    const int t = threadIdx.x;
    const int k = t >> 6, j = (t >> 3) & 7, i2 = t & 7;
    const int ir = 2 * i2 + ((j + k) & 1), ib = 2 * i2 + ((j + k + 1) & 1);  // both in block A (i2 < 4) or B
    const int own = A + (i2 >> 2);
    // the red and the black cell of a thread are the x-pair (2 i2, 2 i2 + 1) of a block row:
    // their right-hand sides come in, and their results go out, as one 8-byte word each
    const int cpair = (k * 8 + j) * 8 + ((2 * i2) & 7);
    const bool red_even = ((j + k) & 1) == 0;
    float rr0[3], rr1[3] = {0.f, 0.f, 0.f}, rrb[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float2 v = *reinterpret_cast<const float2 *>(r + ((size_t)own * 3 + c) * B3 + cpair);
        rr0[c] = red_even ? v.x : v.y;
        rrb[c] = red_even ? v.y : v.x;
    }
    int p1 = -1;
    if (t < 384) {
        const uint32_t code = __ldg(&g_ring2.v[t]);
        const int li = (int)(code & 31u) - 1, lj = (int)((code >> 5) & 31u) - 1, lk = (int)((code >> 10) & 31u) - 1;
        const int bx = li < 0 ? -1 : (li > 15 ? 2 : (li >> 3));
        const int dj = lj < 0 ? -1 : (lj > 7 ? 1 : 0), dk = lk < 0 ? -1 : (lk > 7 ? 1 : 0);
        const int src = snb[(dk + 1) * 12 + (dj + 1) * 4 + (bx + 1)];
        const int off = ((lk - 8 * dk) * 8 + (lj - 8 * dj)) * 8 + (li - 8 * bx);
#pragma unroll
        for (int c = 0; c < 3; c++) rr1[c] = r[((size_t)src * 3 + c) * B3 + off];
        p1 = G::at(li + 2, lj + 2, lk + 2);
    }
    __syncthreads();
    // red: the brick's 512 (one per thread), then the 384 of its ring, from the pre-sweep state
    float nv0[3], nv1[3];
    const int p0 = G::at(ir + 2, j + 2, k + 2);
    if constexpr (ZERO) {  // nothing of e is read: no barrier before the red values are stored
        red_from_zero_acc<float>(TileAcc<float, G>{tB, tE, p0}, K, rr0, nv0);
        if (p1 >= 0) red_from_zero_acc<float>(TileAcc<float, G>{tB, tE, p1}, K, rr1, nv1);
    } else {
        rb_update<float, G>(tB, tE, p0, K, rr0, nv0);
        if (p1 >= 0) rb_update<float, G>(tB, tE, p1, K, rr1, nv1);
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
        tB[c * G::CS + p0] = nv0[c];
        if (p1 >= 0) tB[c * G::CS + p1] = nv1[c];
    }
    __syncthreads();
    // black cells of the brick from the post-red state, then both blocks are written out
    float out[3];
    if constexpr (ZERO)  // black cells read only red neighbours (their black neighbours are 0)
        black_after_zero_acc<float>(TileAcc<float, G>{tB, tE, G::at(ib + 2, j + 2, k + 2)}, K, rrb, out);
    else
        rb_update<float, G>(tB, tE, G::at(ib + 2, j + 2, k + 2), K, rrb, out);
#pragma unroll
    for (int c = 0; c < 3; c++)
        *reinterpret_cast<float2 *>(e_out + ((size_t)own * 3 + c) * B3 + cpair) =
            red_even ? make_float2(nv0[c], out[c]) : make_float2(out[c], nv0[c]);
}

cudaError_t launch_smooth_rb2(const GridDev &g, const float *e_in, float *e_out, const float *r, const float *eta,
                              double lamdt, cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    const size_t sm = 4 * G20::CS * sizeof(float);
    static const bool attr = (cudaFuncSetAttribute(k_smooth_rb2<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                              cudaFuncSetAttribute(k_smooth_rb2<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                              cudaFuncSetAttribute(k_smooth_rb2<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                              cudaFuncSetAttribute(k_smooth_rb2<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                              true);
    (void)attr;
    const RbK<float> K = rb_constants<float>(lamdt, g.h, g.omega);
    if (e_in)
        launch_pdl2(k_smooth_rb2<false, true>, k_smooth_rb2<false, false>, g.nblk / 2, 512, sm, s, g, e_in, e_out, r, eta, K);
    else  // from e = 0
        launch_pdl2(k_smooth_rb2<true, true>, k_smooth_rb2<true, false>, g.nblk / 2, 512, sm, s, g, nullptr, e_out, r, eta, K);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ residual on brick pairs
// The float32 operator and residual of the inner solve on the same x-adjacent block pairs as
// the pair sweep (512 threads, one thread block per pair), with the flux divergence formed per
// cell by the sweep's face_pair (Eqs. 8-10) instead of through face-flux arrays: no flux
// arrays, one barrier, a 18 x 10 x 10 tile (one-cell halo; rows staged as 16-byte words with
// the block interiors 16-byte aligned at OFF = 3).  Modes:
//   APPLY:    out = X + kc divF(X)                    (L X, the Krylov operator)
//   residual: out = (Y - X) + kc divF(X), kc = -lamdt / (2 h^2)   (Eq. 20)
// and RESTRICT: the residual's octet means written into the coarser grid (Sec. 2.2), for grids
// whose children sit in Morton octets (block b's parent is b / 8, its octant b % 8).  A warp
// takes 8 cells of a row x 2 rows x 2 planes of one block: every 2^3 octet is in one warp (sums
// by three shuffles), and with rows 24 and planes 240 floats apart (240 = 16 mod 32) its
// shared-memory reads at one offset fall on 32 distinct banks.
struct G18 {
    static constexpr int S = 10, RRS = 24, PS = S * RRS, CS = S * PS, OFF = 3;
    __device__ static __forceinline__ int at(int i, int j, int k) { return k * PS + j * RRS + i + OFF; }
};

// Contribution of a cell's face along AX to the flux divergence of component C, for the face on
// side so (+-1 cell along AX, as a tile offset) with qs = +-1/4: es Q on the high side, -es Q on
// the low one -- the terms of face_pair for that face alone, in the same operations.
template <int AX, int C>
__device__ __forceinline__ float octet_face(const float *__restrict__ tB, int p, int so, float qs, float es) {
    constexpr int SC = C == 0 ? 1 : (C == 1 ? G18::RRS : G18::PS);
    const float *BA = tB + AX * G18::CS + p, *BC = tB + C * G18::CS + p;
    const float d0 = v_sub(BA[SC], BA[-SC]);
    const float dn = v_sub(BA[so + SC], BA[so - SC]);
    return v_mul(es, v_mad(v_add(dn, d0), qs, v_sub(BC[0], BC[so])));
}

// NV >= 0 (APPLY only): also the FGMRES products of the output w with the NV vectors of V and
// with itself, <w, v_i> and <w, w>, each weighted by wt (h^3 for the cells of a single-level
// grid) and folded per block pair in a fixed order into part[i][pair] (column-major, so that
// the column sums read contiguous rows).
// OCT (residual + restriction with no fine output): the restriction needs only the octet sums
// of the flux divergence, and in the conservative form (Eq. 8) every flux through a face inside
// an octet enters its two cells with opposite signs, so the sum over the octet is the net flux
// through the octet's 24 outer faces.  Each cell of an octet sits at one of its corners and
// owns exactly one outer face per axis (the high face where its coordinate is odd, the low one
// where it is even); it computes those three faces instead of its six, and the octet sum of
// (Y - X) + kc divF(X) is formed as before.  Equal to the full form in exact arithmetic (the
// internal fluxes cancel); about 40% fewer operations and 30% fewer tile reads per cell.
template <bool APPLY, bool RESTRICT, int NV = -1, bool OCT = false, bool EARLY = false>
__global__ void __launch_bounds__(512, NV >= 0 ? 3 : 4)
    k_pair_op(GridDev g, const float *__restrict__ X, const float *__restrict__ Y, const float *__restrict__ eta, float kc,
              float *__restrict__ out, float *__restrict__ coarse, VecSet V, double wt,
              double *__restrict__ part) {
    using G = G18;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *tB = reinterpret_cast<float *>(smem_raw);  // [3][10 planes][10 rows][RRS]
    float *tE = tB + 3 * G::CS;
    __shared__ int snb[36];
    const int A0 = 2 * blockIdx.x;
    pdl_trigger<EARLY>();
    if (!EARLY && skip_block(g, A0)) return;  // (masked blocks return before they load anything)
    if (threadIdx.x < 36) {
        const int bx = threadIdx.x % 4 - 1, dj = (threadIdx.x / 4) % 3 - 1, dk = threadIdx.x / 12 - 1;
        const int base = bx <= 1 ? A0 : A0 + 1, dx = bx <= 1 ? bx : 1;
        snb[threadIdx.x] = __ldg(g.nbr + base * 27 + (dk + 1) * 9 + (dj + 1) * 3 + (dx + 1));
    }
    const int A = A0 + pdl_wait<EARLY>();
    if (EARLY && skip_block(g, A)) return;
    __syncthreads();
    // one task per (field component, tile row): 1 + 8 + 8 + 1 values, the interiors as 16-byte words
    if (threadIdx.x < 400) {
        const int c = threadIdx.x / 100, u = threadIdx.x - c * 100;
        const int tk = u / 10, tj = u - 10 * tk;
        const int lj = tj - 1, lk = tk - 1;
        const int dj = lj < 0 ? -1 : (lj > 7 ? 1 : 0), dk = lk < 0 ? -1 : (lk > 7 ? 1 : 0);
        const int rowoff = ((lk - 8 * dk) * 8 + (lj - 8 * dj)) * 8;
        const int *nb = snb + (dk + 1) * 12 + (dj + 1) * 4;
        const float *F = c < 3 ? X : eta;
        const int nc = c < 3 ? 3 : 1, cc = c < 3 ? c : 0;
        float *row = (c < 3 ? tB + c * G::CS : tE) + tk * G::PS + tj * G::RRS + G::OFF;
        const float lo = __ldg(F + ((size_t)nb[0] * nc + cc) * B3 + rowoff + 7);
        const float4 *pa = reinterpret_cast<const float4 *>(F + ((size_t)nb[1] * nc + cc) * B3 + rowoff);
        const float4 *pb = reinterpret_cast<const float4 *>(F + ((size_t)nb[2] * nc + cc) * B3 + rowoff);
        const float hi = __ldg(F + ((size_t)nb[3] * nc + cc) * B3 + rowoff);
        const float4 a0 = __ldg(pa), a1 = __ldg(pa + 1), b0 = __ldg(pb), b1 = __ldg(pb + 1);
        row[0] = lo;
        float4 *r4 = reinterpret_cast<float4 *>(row + 1);
        r4[0] = a0;
        r4[1] = a1;
        r4[2] = b0;
        r4[3] = b1;
        row[17] = hi;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int x = lane & 7, y = 2 * (w & 3) + ((lane >> 3) & 1), z = 2 * ((w >> 2) & 3) + (lane >> 4);
    const int cell = (z * 8 + y) * 8 + x;
    constexpr int ND = NV >= 0 ? NV + 1 : 1;
    float dots[ND];
#pragma unroll
    for (int i = 0; i < ND; i++) dots[i] = 0.f;
#pragma unroll
    for (int h = 0; h < 2; h++) {  // the same cell of block A, then of block B
        const int b = A + h;
        const TileAcc<float, G> acc{tB, tE, G::at(1 + 8 * h + x, 1 + y, 1 + z)};
        float dv[3];
        if constexpr (OCT) {
            const int p = acc.p, ox = (x & 1) ? 1 : -1, oy = (y & 1) ? G::RRS : -G::RRS, oz = (z & 1) ? G::PS : -G::PS;
            const float qx = (x & 1) ? 0.25f : -0.25f, qy = (y & 1) ? 0.25f : -0.25f, qz = (z & 1) ? 0.25f : -0.25f;
            const float e0 = tE[p];
            const float esx = v_add(e0, tE[p + ox]), esy = v_add(e0, tE[p + oy]), esz = v_add(e0, tE[p + oz]);
            dv[0] = v_add(octet_face<1, 0>(tB, p, oy, qy, esy), octet_face<2, 0>(tB, p, oz, qz, esz));
            dv[1] = v_add(octet_face<0, 1>(tB, p, ox, qx, esx), octet_face<2, 1>(tB, p, oz, qz, esz));
            dv[2] = v_add(octet_face<0, 2>(tB, p, ox, qx, esx), octet_face<1, 2>(tB, p, oy, qy, esy));
        } else {
            float es[6];
            face_sums<float>(acc, es);
            cell_divergence<float>(acc, es, dv);
        }
        const float ev[3] = {acc.template B<0, 0, 0, 0>(), acc.template B<1, 0, 0, 0>(), acc.template B<2, 0, 0, 0>()};
        float o[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const size_t id = ((size_t)b * 3 + c) * B3 + cell;
            o[c] = v_mad(kc, dv[c], APPLY ? ev[c] : v_sub(Y[id], ev[c]));
            if (!OCT && out) out[id] = o[c];
            if constexpr (NV >= 0) {
#pragma unroll
                for (int i = 0; i < NV; i++) dots[i] = fmaf(o[c], V.v[i][id], dots[i]);
                dots[NV] = fmaf(o[c], o[c], dots[NV]);
            }
        }
        if constexpr (RESTRICT) {
            const int oct = b & 7, pb = b >> 3;
            const int cx = 4 * (oct & 1) + (x >> 1), cy = 4 * ((oct >> 1) & 1) + (y >> 1), cz = 4 * (oct >> 2) + (z >> 1);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                float sum = v_add(o[c], __shfl_xor_sync(0xffffffffu, o[c], 1));
                sum = v_add(sum, __shfl_xor_sync(0xffffffffu, sum, 8));
                sum = v_add(sum, __shfl_xor_sync(0xffffffffu, sum, 16));
                if ((lane & 0x19) == 0) coarse[((size_t)pb * 3 + c) * B3 + (cz * 8 + cy) * 8 + cx] = v_mul(sum, 0.125f);
            }
        }
    }
    if constexpr (NV >= 0) {  // warp sums, then the 16 warps in order (the tile is free by now)
        __syncthreads();
        double *sred = reinterpret_cast<double *>(smem_raw);  // [16][NV + 1]
#pragma unroll
        for (int i = 0; i <= NV; i++) {
            float v = dots[i];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) sred[w * (NV + 1) + i] = (double)v;
        }
        __syncthreads();
        if (threadIdx.x <= NV) {
            double a = 0.0;
            for (int q = 0; q < 16; q++) a += sred[q * (NV + 1) + threadIdx.x];
            part[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = a * wt;
        }
    }
}

cudaError_t launch_pair_op(const GridDev &g, const float *X, const float *Y, const float *eta, double kc, bool apply,
                           float *out, float *coarse, cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    const size_t sm = 4 * G18::CS * sizeof(float);
    static const bool attr = [=] {
        auto set = [=](auto k) { cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm); };
        set(k_pair_op<true, false>);
        set(k_pair_op<false, false>);
        set(k_pair_op<false, true>);
        set(k_pair_op<false, true, -1, true>);
        set(k_pair_op<true, false, -1, false, true>);
        set(k_pair_op<false, false, -1, false, true>);
        set(k_pair_op<false, true, -1, false, true>);
        set(k_pair_op<false, true, -1, true, true>);
        return true;
    }();
    (void)attr;
    if (apply)
        launch_pdl2(k_pair_op<true, false, -1, false, true>, k_pair_op<true, false>, g.nblk / 2, 512, sm, s, g, X, nullptr, eta, (float)kc, out, nullptr, VecSet(), 0.0, (double *)nullptr);
    else if (coarse && !out)  // only the octet means: outer faces of each octet
        launch_pdl2(k_pair_op<false, true, -1, true, true>, k_pair_op<false, true, -1, true>, g.nblk / 2, 512, sm, s, g, X, Y, eta, (float)kc, nullptr, coarse, VecSet(), 0.0, (double *)nullptr);
    else if (coarse)
        launch_pdl2(k_pair_op<false, true, -1, false, true>, k_pair_op<false, true>, g.nblk / 2, 512, sm, s, g, X, Y, eta, (float)kc, out, coarse, VecSet(), 0.0, (double *)nullptr);
    else
        launch_pdl2(k_pair_op<false, false, -1, false, true>, k_pair_op<false, false>, g.nblk / 2, 512, sm, s, g, X, Y, eta, (float)kc, out, nullptr, VecSet(), 0.0, (double *)nullptr);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ FGMRES scalars
// One thread per instance: the steps of FGMRES(m) (Saad 1993) that the single-problem solver
// takes on the host, in the same order and float64 arithmetic, for every instance of a batch.
__global__ void __launch_bounds__(128) k_fg(FgState f, int op, int j) {
    pdl_trigger();
    pdl_wait();
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= f.K) return;
    constexpr int KC = KMAX + 1;
    const double *d = f.dots + (size_t)q * KC;
    float *c = f.coef + (size_t)q * KC;
    double *H = f.Hm + (size_t)q * KC * KMAX, *cs = f.cs + (size_t)q * KMAX, *sn = f.sn + (size_t)q * KMAX;
    double *g = f.g + (size_t)q * KC;
    auto h = [&](int i, int k) -> double & { return H[i * KMAX + k]; };
    auto clear = [&](float scale) {
        for (int i = 0; i < KMAX; i++) c[i] = 0.f;
        c[KMAX] = scale;
    };
    auto act = [&](int step) {
        if (q == 0) f.any_need2[step & 1] = 0;
        const uint8_t a = f.arn[q] && f.cycles[q] < f.max_outer;
        f.act[q] = a;
        f.imask[q] = a;
        f.cycles[q] += a;
    };
    switch (op) {
        case FG_START: {  // v_0 = rhs / beta0 for the instances that iterate
            const double b = sqrt(fmax(d[0], 0.0));
            f.beta0[q] = f.beta[q] = f.brest[q] = b;
            f.live[q] = f.run[q] && b > 0 && isfinite(b);
            clear(f.live[q] ? (float)(1.0 / b) : 1.f);
            break;
        }
        case FG_CYCLE: {  // a restart cycle begins: g = beta e_0
            f.arn[q] = f.live[q];
            f.jend[q] = 0;
            for (int i = 0; i < KC; i++) g[i] = 0.0;
            g[0] = f.beta[q];
            break;
        }
        case FG_ACT: {  // instances that take Arnoldi step j (their V-cycle is counted)
            act(j);
            break;
        }
        case FG_ORTHO: {  // h_ij = <w, v_i>; one-pass normalisation unless cancellation is large
            clear(1.f);
            f.need2[q] = 0;
            if (!f.act[q]) break;
            double proj = 0.0;
            for (int i = 0; i <= j; i++) {
                h(i, j) = d[i];
                c[i] = (float)d[i];
                proj += d[i] * d[i];
            }
            const double ww = d[j + 1];
            if (ww - proj > 0.01 * ww) {
                f.hn[q] = sqrt(ww - proj);
                c[KMAX] = (float)(1.0 / f.hn[q]);
            } else {
                f.need2[q] = 1;
                atomicOr(f.any_need2 + (j & 1), 1);  // the norm pass after orthogonalising runs
            }
            break;
        }
        // the rest of step j's scalars in one launch: the norm measured after orthogonalising, where the
        // one pass was refused, the Givens update, and the instances that take step j + 1 (the vector
        // update that the measured norm scales follows; its gate is step j's flag)
        case FG_STEP: {
            clear(1.f);
            if (f.act[q]) {
                if (f.need2[q]) {
                    f.hn[q] = sqrt(fmax(d[0], 0.0));
                    if (f.hn[q] > 0) c[KMAX] = (float)(1.0 / f.hn[q]);
                }
                const double hnq = f.hn[q];
                h(j + 1, j) = hnq;
                for (int i = 0; i < j; i++) {
                    const double t = cs[i] * h(i, j) + sn[i] * h(i + 1, j);
                    h(i + 1, j) = -sn[i] * h(i, j) + cs[i] * h(i + 1, j);
                    h(i, j) = t;
                }
                const double den = hypot(h(j, j), h(j + 1, j));
                cs[j] = den > 0 ? h(j, j) / den : 1.0;
                sn[j] = den > 0 ? h(j + 1, j) / den : 0.0;
                h(j, j) = den;
                h(j + 1, j) = 0.0;
                g[j + 1] = -sn[j] * g[j];
                g[j] = cs[j] * g[j];
                f.jend[q] = j + 1;
                if (fabs(g[j + 1]) <= f.target[q] * f.beta0[q] || !(hnq > 0)) {
                    f.arn[q] = 0;
                    f.live[q] = 0;  // converged (or breakdown): no restart
                }
            }
            if (j + 1 < f.m) act(j + 1);
            break;
        }
        case FG_SOLVE: {  // x += sum y_i z_i with R y = g
            clear(1.f);
            const int je = f.jend[q];
            double y[KMAX];
            for (int i = je - 1; i >= 0; i--) {
                double t = g[i];
                for (int k = i + 1; k < je; k++) t -= h(i, k) * y[k];
                y[i] = h(i, i) != 0 ? t / h(i, i) : 0.0;
            }
            for (int i = 0; i < je; i++) c[i] = (float)(-y[i]);
            break;
        }
        case FG_RESTART_MASK: {  // restart where the instance is live and may take more cycles
            if (f.live[q] && (f.cycles[q] >= f.max_outer || f.jend[q] == 0)) f.live[q] = 0;
            f.imask[q] = f.live[q];
            break;
        }
        case FG_RESTART: {  // stop at the target, on breakdown, or when the cycle gained < 2x
            clear(1.f);
            if (!f.live[q]) break;
            const double b = sqrt(fmax(d[0], 0.0));
            f.beta[q] = b;
            if (b <= f.target[q] * f.beta0[q] || !(b > 0) || b > 0.5 * f.brest[q]) {
                f.live[q] = 0;
                break;
            }
            f.brest[q] = b;
            c[KMAX] = (float)(1.0 / b);
            break;
        }
    }
}

cudaError_t launch_fg(const FgState &f, FgOp op, int j, cudaStream_t s) {
    if (f.K == 0) return cudaSuccess;
    launch_pdl(k_fg, (f.K + 127) / 128, 128, 0, s, f, (int)op, j);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ inverse diagonal
// inv_c = omega / (1 + alpha_c), alpha_c = lamdt/h^2 sum_{a != c} (eta_{-1/2} + eta_{+1/2})
// with face eta the mean of the two cells (Eqs. 11, 21-23).
template <typename T>
__global__ void __launch_bounds__(512) k_invdiag(GridDev g, const T *__restrict__ eta, const T *__restrict__ Geta,
                                                 double lh2, T *__restrict__ inv) {
    using G = Geo<T>;
    __shared__ __align__(16) T tE[G::CS];
    __shared__ int snb[27];
    const int b = blockIdx.x;
    if (skip_block(g, b)) return;
    const int slot = g.gslot ? g.gslot[b] : -1;
    stage_nbr(snb, g.nbr, b);
    __syncthreads();
    stage_rows<T, 1, 1, G::RS, G::OFF>(tE, eta, snb, slot >= 0 && Geta ? Geta + (size_t)slot * T3 : nullptr);
    __syncthreads();
    // computed in T: the inverse diagonal only scales smoother updates
    const int t = threadIdx.x, i = t & 7, j = (t >> 3) & 7, k = t >> 6;
    const int p = G::at(i + 1, j + 1, k + 1);
    const T e0 = tE[p], h = T(0.5), l = (T)lh2;
    const T sa[3] = {h * (e0 + tE[p + 1]) + h * (e0 + tE[p - 1]), h * (e0 + tE[p + G::RS]) + h * (e0 + tE[p - G::RS]),
                     h * (e0 + tE[p + G::PS]) + h * (e0 + tE[p - G::PS])};
#pragma unroll
    for (int c = 0; c < 3; c++) {
        T al = T(0);
        for (int ax = 0; ax < 3; ax++)
            if (ax != c) al += l * sa[ax];
        inv[((size_t)b * 3 + c) * B3 + t] = (T)g.omega / (T(1) + al);
    }
}

template <typename T>
cudaError_t launch_invdiag(const GridDev &g, const T *eta, const T *Geta, double lamdt, T *inv, cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    k_invdiag<T><<<g.nblk, 512, 0, s>>>(g, eta, Geta, lamdt / (g.h * g.h), inv);
    return cudaGetLastError();
}
template cudaError_t launch_invdiag<double>(const GridDev &, const double *, const double *, double, double *, cudaStream_t);
template cudaError_t launch_invdiag<float>(const GridDev &, const float *, const float *, double, float *, cudaStream_t);

// Offset of block b's instance in a lexicographic grid of ld cells and ncomp components
// (batched hierarchies stack one such grid per instance)
__device__ __forceinline__ size_t lex_inst_offset(const GridDev &g, int b, int ncomp, int3 ld) {
    return g.inst_nblk ? (size_t)(b / g.inst_nblk) * ncomp * ((size_t)ld.x * ld.y * ld.z) : 0;
}

__device__ __forceinline__ bool inst_masked(const GridDev &g, const uint8_t *imask, int b) {
    return imask && !imask[g.inst_nblk ? b / g.inst_nblk : 0];
}

// ------------------------------------------------------------------ residual + restriction
template <typename T, bool EARLY>
__global__ void __launch_bounds__(512, sizeof(T) == 4 ? 4 : 1) k_resid_restrict(GridDev g, const T *__restrict__ e, const T *__restrict__ r,
                                                        const T *__restrict__ eta, const T *__restrict__ Ge,
                                                        const T *__restrict__ Geta, T coef, T *__restrict__ t_out,
                                                        T *__restrict__ coarse, T *__restrict__ lex, int3 ld) {
    using G = Geo<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *tB = reinterpret_cast<T *>(smem_raw);
    T *tE = tB + 3 * G::CS;
    T *phi = tE + G::CS;
    T *tt = phi + G::PHI;
    __shared__ int snb[27];
    const int b0 = blockIdx.x;
    pdl_trigger<EARLY>();
    if (!EARLY && skip_block(g, b0)) return;  // (masked blocks return before they load anything)
    stage_nbr(snb, g.nbr, b0);
    const int slot = g.gslot ? g.gslot[b0] : -1;
    const int b = b0 + pdl_wait<EARLY>();
    if (EARLY && skip_block(g, b)) return;
    __syncthreads();
    stage_rows<T, 3, 1, G::RS, G::OFF>(tB, e, snb, slot >= 0 && Ge ? Ge + (size_t)slot * 3 * T3 : nullptr);
    stage_rows<T, 1, 1, G::RS, G::OFF>(tE, eta, snb, slot >= 0 && Geta ? Geta + (size_t)slot * T3 : nullptr);
    __syncthreads();
    all_faces_512(tB, tE, phi);
    __syncthreads();
    {
        int i, j, k;
        cell_of_thread<T>(threadIdx.x, i, j, k);
        const int cell = (k * 8 + j) * 8 + i;
        T dv[3];
        cell_div(phi, i, j, k, dv[0], dv[1], dv[2]);
        const int p = G::at(i + 1, j + 1, k + 1);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            size_t id = ((size_t)b * 3 + c) * B3 + cell;
            T v = r[id] - tB[c * G::CS + p] - coef * dv[c];
            tt[c * B3 + cell] = v;
            if (t_out) t_out[id] = v;
        }
    }
    __syncthreads();
    if ((coarse || lex) && threadIdx.x < 192) {
        const int c = threadIdx.x >> 6, q = threadIdx.x & 63;
        const int ci = q & 3, cj = (q >> 2) & 3, ck = q >> 4;
        const T *src = tt + c * B3;
        T s = 0;
        for (int dk = 0; dk < 2; dk++)
            for (int dj = 0; dj < 2; dj++)
                for (int di = 0; di < 2; di++) s += src[((2 * ck + dk) * 8 + 2 * cj + dj) * 8 + 2 * ci + di];
        s = s / T(8);
        if (coarse) {
            const int pb = g.parent[b], o = g.octant[b];
            const int x = 4 * (o & 1) + ci, y = 4 * ((o >> 1) & 1) + cj, z = 4 * (o >> 2) + ck;
            coarse[((size_t)pb * 3 + c) * B3 + (z * 8 + y) * 8 + x] = s;
        } else {
            const int x = 4 * g.origin[b * 3 + 0] + ci, y = 4 * g.origin[b * 3 + 1] + cj, z = 4 * g.origin[b * 3 + 2] + ck;
            T *lx = lex + lex_inst_offset(g, b, 3, ld);
            lx[(((size_t)c * ld.z + z) * ld.y + y) * ld.x + x] = s;
        }
    }
}

// float64 residual and its restriction without the fine residual.  Bound by the float64 pipe: the
// octet sums of the flux divergence need only the fluxes through the octets' outer faces
// (k_pair_op's octet form), every one of which bounds two octets, so a thread takes one side of an
// octet (2 x 2 faces) and forms sum es (T/4 - N) over it for both flux components, from pair sums as
// in k_smooth_d, once for the two octets it separates: about 27 operations per cell instead of 66.
// Slabs of NZ planes as there.  t = r - e + kc divF summed over an octet and divided by 8 goes to the
// coarser grid.
template <int NZ>
struct OctD {
    static constexpr int NT = 32 * NZ, NP = NZ + 2, NZO = NZ / 2;
    static constexpr int CS = 100 * NP;
    static constexpr int PXY = 50 * NP;                        // 5 face planes of 10 NP sums
    static constexpr int SUMS = 2 * PXY + 100 * (NZO + 1);
    static constexpr int SXY = 5 * 4 * NZO, SZ = (NZO + 1) * 16, SIDES = 2 * SXY + SZ;
    static constexpr size_t BYTES = (4 * CS + SUMS + 2 * SIDES) * sizeof(double);
};

template <int NZ, int NF, int NV>
__device__ __forceinline__ void octet_sums_axis(const double *__restrict__ Ba, double *__restrict__ P, int sa, int su, int sv) {
    constexpr int FULL = 10 * NV - 4;
    for (int e = threadIdx.x; e < NF * FULL; e += OctD<NZ>::NT) {
        const int f = e / FULL;
        int u, v;
        cross_pos<NV>(e - f * FULL, u, v);
        const double *p = Ba + 2 * f * sa + u * su + v * sv;
        P[(f * NV + v) * 10 + u] = p[sa] + p[0];
    }
}

template <int NZ>
__global__ void __launch_bounds__(32 * NZ) k_resid_restrict_d(GridDev g, const double *__restrict__ e, const double *__restrict__ r,
                                                              const double *__restrict__ eta, const double *__restrict__ Ge,
                                                              const double *__restrict__ Geta, double kc, double *__restrict__ coarse,
                                                              double *__restrict__ lex, int3 ld) {
    using S = OctD<NZ>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *tB = reinterpret_cast<double *>(smem_raw), *tE = tB + 3 * S::CS, *P = tE + S::CS, *side = P + S::SUMS;
    __shared__ int snb[27];
    const int b = blockIdx.x / (8 / NZ), z0 = NZ * (blockIdx.x % (8 / NZ));
    if (skip_block(g, b)) return;  // (masked blocks return before they load anything)
    stage_nbr(snb, g.nbr, b);
    const int slot = g.gslot ? g.gslot[b] : -1, t = threadIdx.x;
    __syncthreads();
    stage_slab<NZ, 1>(tE, eta, snb, slot >= 0 && Geta ? Geta + (size_t)slot * T3 : nullptr, z0);
    stage_slab<NZ, 3>(tB, e, snb, slot >= 0 && Ge ? Ge + (size_t)slot * 3 * T3 : nullptr, z0);
    __syncthreads();
    octet_sums_axis<NZ, 5, NZ + 2>(tB, P, 1, 10, 100);
    octet_sums_axis<NZ, 5, NZ + 2>(tB + S::CS, P + S::PXY, 10, 1, 100);
    octet_sums_axis<NZ, S::NZO + 1, 10>(tB + 2 * S::CS, P + 2 * S::PXY, 100, 1, 10);
    __syncthreads();
    // sides: face plane f (tile cell 2f and the next along the axis), octet (m, n) of the cross-section
    for (int q = t; q < S::SIDES; q += S::NT) {
        const int ax = q < S::SXY ? 0 : (q < 2 * S::SXY ? 1 : 2);
        const int h = q - ax * S::SXY;
        const int per = ax == 2 ? 16 : 4 * S::NZO, f = h / per, m = (h - f * per) & 3, n = (h - f * per) >> 2;
        const int sa = ax == 0 ? 1 : (ax == 1 ? 10 : 100), su = ax == 0 ? 10 : 1, sv = ax == 2 ? 10 : 100;
        const int NV = ax == 2 ? 10 : NZ + 2;
        const double *B1 = tB + (ax == 0 ? 1 : 0) * S::CS, *B2 = tB + (ax == 2 ? 1 : 2) * S::CS;
        double s1 = 0.0, s2 = 0.0;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int u = 2 * m + 1 + (k & 1), v = 2 * n + 1 + (k >> 1), p = 2 * f * sa + u * su + v * sv;
            const double *Pa = P + ax * S::PXY + (f * NV + v) * 10 + u;
            const double es = tE[p] + tE[p + sa];
            const double g1 = fma(0.25, Pa[1] - Pa[-1], B1[p] - B1[p + sa]);
            const double g2 = fma(0.25, Pa[10] - Pa[-10], B2[p] - B2[p + sa]);
            s1 = k ? fma(es, g1, s1) : es * g1;
            s2 = k ? fma(es, g2, s2) : es * g2;
        }
        side[q] = s1;
        side[S::SIDES + q] = s2;
    }
    __syncthreads();
    // one thread per octet and component
    for (int q = t; q < 48 * S::NZO; q += S::NT) {
        const int c = q / (16 * S::NZO), w = q - c * (16 * S::NZO), ci = w & 3, cj = (w >> 2) & 3, ck = w >> 4;
        // the two axes of the component's fluxes: its own flux component index on them
        auto net = [&](int ax) {
            const int comp = ax == 0 ? (c == 1 ? 0 : 1) : (ax == 1 ? (c == 0 ? 0 : 1) : c);
            const int m = ax == 0 ? cj : ci, n = ax == 2 ? cj : ck, f = ax == 0 ? ci : (ax == 1 ? cj : ck);
            const int per = ax == 2 ? 16 : 4 * S::NZO;
            const double *sd = side + comp * S::SIDES + ax * S::SXY + f * per + n * 4 + m;
            return sd[per] - sd[0];
        };
        const double div = c == 0 ? net(1) + net(2) : (c == 1 ? net(0) + net(2) : net(0) + net(1));
        double sum = 0.0;
        const double *tc = tB + c * S::CS;
        const double *rc = r + ((size_t)b * 3 + c) * B3;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int x = 2 * ci + (k & 1), y = 2 * cj + ((k >> 1) & 1), z = 2 * ck + (k >> 2);
            const double d = rc[((z0 + z) * 8 + y) * 8 + x] - tc[(z + 1) * 100 + (y + 1) * 10 + x + 1];
            sum = k ? sum + d : d;
        }
        const double v = 0.125 * fma(kc, div, sum);
        const int cz = (z0 >> 1) + ck;
        if (coarse) {
            const int pb = g.parent[b], o = g.octant[b];
            const int x = 4 * (o & 1) + ci, y = 4 * ((o >> 1) & 1) + cj, z = 4 * (o >> 2) + cz;
            coarse[((size_t)pb * 3 + c) * B3 + (z * 8 + y) * 8 + x] = v;
        } else {
            const int x = 4 * g.origin[b * 3 + 0] + ci, y = 4 * g.origin[b * 3 + 1] + cj, z = 4 * g.origin[b * 3 + 2] + cz;
            double *lx = lex + lex_inst_offset(g, b, 3, ld);
            lx[(((size_t)c * ld.z + z) * ld.y + y) * ld.x + x] = v;
        }
    }
}

template <int NZ>
static cudaError_t launch_resid_restrict_slab(const GridDev &g, const double *e, const double *r, const double *eta,
                                              const double *Ge, const double *Geta, double kc, double *coarse, double *lex,
                                              int3 ld, cudaStream_t s) {
    using S = OctD<NZ>;
    static const bool attr = (cudaFuncSetAttribute(k_resid_restrict_d<NZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::BYTES), true);
    (void)attr;
    launch_full(k_resid_restrict_d<NZ>, g.nblk * (8 / NZ), S::NT, S::BYTES, s, g, e, r, eta, Ge, Geta, kc, coarse, lex, ld);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_resid_restrict(const GridDev &g, const T *e, const T *r, const T *eta, const T *Ge, const T *Geta,
                                  double lamdt, T *t_out, T *coarse, T *lex, const int *ldims, cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    const size_t sm = (4 * Geo<T>::CS + Geo<T>::PHI + 3 * B3) * sizeof(T);
    // set once per process (thread-safe static initialisation)
    constexpr bool E = sizeof(T) == 4;
    static const bool attr = (cudaFuncSetAttribute(k_resid_restrict<T, E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                              cudaFuncSetAttribute(k_resid_restrict<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm), true);
    (void)attr;
    int3 ld = make_int3(ldims ? ldims[0] : 0, ldims ? ldims[1] : 0, ldims ? ldims[2] : 0);
    if constexpr (std::is_same<T, double>::value) {
        if (!t_out && (coarse || lex)) {  // slab height as for the colour passes
            const double kc = -lamdt / (2.0 * g.h * g.h);
            if (g.nblk <= SLAB2_BLOCKS) return launch_resid_restrict_slab<2>(g, e, r, eta, Ge, Geta, kc, coarse, lex, ld, s);
            if (g.nblk <= SLAB4_BLOCKS) return launch_resid_restrict_slab<4>(g, e, r, eta, Ge, Geta, kc, coarse, lex, ld, s);
            return launch_resid_restrict_slab<8>(g, e, r, eta, Ge, Geta, kc, coarse, lex, ld, s);
        }
    }
    launch_pdl2(k_resid_restrict<T, E>, k_resid_restrict<T, false>, g.nblk, 512, sm, s, g, e, r, eta, Ge, Geta, (T)(lamdt / (2.0 * g.h * g.h)), t_out, coarse,
                                                lex, ld);
    return cudaGetLastError();
}
template cudaError_t launch_resid_restrict<double>(const GridDev &, const double *, const double *, const double *,
                                                   const double *, const double *, double, double *, double *, double *,
                                                   const int *, cudaStream_t);
template cudaError_t launch_resid_restrict<float>(const GridDev &, const float *, const float *, const float *,
                                                  const float *, const float *, double, float *, float *, float *,
                                                  const int *, cudaStream_t);

// ------------------------------------------------------------------ plain restriction
template <typename T>
__global__ void __launch_bounds__(512) k_restrict(GridDev g, const T *__restrict__ fine, int ncomp,
                                                  T *__restrict__ coarse, T *__restrict__ lex, int3 ld) {
    const int b = blockIdx.x;
    for (int q = threadIdx.x; q < 64 * ncomp; q += blockDim.x) {
        const int c = q >> 6, cq = q & 63;
        const int ci = cq & 3, cj = (cq >> 2) & 3, ck = cq >> 4;
        const T *src = fine + ((size_t)b * ncomp + c) * B3;
        T s = 0;
        for (int dk = 0; dk < 2; dk++)
            for (int dj = 0; dj < 2; dj++)
                for (int di = 0; di < 2; di++) s += src[((2 * ck + dk) * 8 + 2 * cj + dj) * 8 + 2 * ci + di];
        s = s / T(8);
        if (coarse) {
            const int pb = g.parent[b], o = g.octant[b];
            const int x = 4 * (o & 1) + ci, y = 4 * ((o >> 1) & 1) + cj, z = 4 * (o >> 2) + ck;
            coarse[((size_t)pb * ncomp + c) * B3 + (z * 8 + y) * 8 + x] = s;
        } else {
            const int x = 4 * g.origin[b * 3 + 0] + ci, y = 4 * g.origin[b * 3 + 1] + cj, z = 4 * g.origin[b * 3 + 2] + ck;
            T *lx = lex + lex_inst_offset(g, b, ncomp, ld);
            lx[(((size_t)c * ld.z + z) * ld.y + y) * ld.x + x] = s;
        }
    }
}

template <typename T>
cudaError_t launch_restrict(const GridDev &g, const T *fine, int ncomp, T *coarse, T *lex, const int *ldims,
                            cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    int3 ld = make_int3(ldims ? ldims[0] : 0, ldims ? ldims[1] : 0, ldims ? ldims[2] : 0);
    k_restrict<T><<<g.nblk, 256, 0, s>>>(g, fine, ncomp, coarse, lex, ld);
    return cudaGetLastError();
}
template cudaError_t launch_restrict<double>(const GridDev &, const double *, int, double *, double *, const int *, cudaStream_t);
template cudaError_t launch_restrict<float>(const GridDev &, const float *, int, float *, float *, const int *, cudaStream_t);

// ------------------------------------------------------------------ prolongation
// fine += trilinear interpolation (weights 3/4, 1/4 per axis) of the coarser grid, read
// through a 6^3 window around the block's footprint in its parent (blocked) or with
// periodic wrap (lexicographic coarse grid).
template <typename T, bool EARLY>
__global__ void __launch_bounds__(512) k_prolong_add(GridDev g, GridDev gc, const T *__restrict__ coarse,
                                                     const T *__restrict__ lex, int3 ld, T *__restrict__ fine,
                                                     int *__restrict__ err) {
    __shared__ T win[3 * 216];
    pdl_trigger<EARLY>();
    const int b = blockIdx.x + pdl_wait<EARLY>();
    if (skip_block(g, b)) return;
    const int o = lex ? 0 : g.octant[b];
    const int pb = lex ? 0 : g.parent[b];
    for (int q = threadIdx.x; q < 216; q += blockDim.x) {
        const int wx = q % 6, wy = (q / 6) % 6, wz = q / 36;
        if (lex) {
            int x = 4 * g.origin[b * 3 + 0] - 1 + wx, y = 4 * g.origin[b * 3 + 1] - 1 + wy, z = 4 * g.origin[b * 3 + 2] - 1 + wz;
            x = (x + ld.x) % ld.x; y = (y + ld.y) % ld.y; z = (z + ld.z) % ld.z;
            const T *lx = lex + lex_inst_offset(g, b, 3, ld);
            for (int c = 0; c < 3; c++) win[c * 216 + q] = lx[(((size_t)c * ld.z + z) * ld.y + y) * ld.x + x];
        } else {
            int cx = 4 * (o & 1) - 1 + wx, cy = 4 * ((o >> 1) & 1) - 1 + wy, cz = 4 * (o >> 2) - 1 + wz;
            int dx = cx < 0 ? -1 : (cx > 7 ? 1 : 0), dy = cy < 0 ? -1 : (cy > 7 ? 1 : 0), dz = cz < 0 ? -1 : (cz > 7 ? 1 : 0);
            int src = gc.nbr[pb * 27 + (dz + 1) * 9 + (dy + 1) * 3 + (dx + 1)];
            if (src < 0) {
                if (err) *err = 1;
                for (int c = 0; c < 3; c++) win[c * 216 + q] = T(0);
            } else {
                int lx = cx - 8 * dx, ly = cy - 8 * dy, lz = cz - 8 * dz;
                for (int c = 0; c < 3; c++) win[c * 216 + q] = coarse[((size_t)src * 3 + c) * B3 + (lz * 8 + ly) * 8 + lx];
            }
        }
    }
    __syncthreads();
    const int t = threadIdx.x, i = t & 7, j = (t >> 3) & 7, k = t >> 6;
    const int wi = (i >> 1) + 1, wj = (j >> 1) + 1, wk = (k >> 1) + 1;
    const int si = (i & 1) ? 1 : -1, sj = (j & 1) ? 1 : -1, sk = (k & 1) ? 1 : -1;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const T *w = win + c * 216;
        T v = 0;
        for (int ak = 0; ak < 2; ak++)
            for (int aj = 0; aj < 2; aj++)
                for (int ai = 0; ai < 2; ai++) {
                    T wt = (ai ? T(0.25) : T(0.75)) * (aj ? T(0.25) : T(0.75)) * (ak ? T(0.25) : T(0.75));
                    v += wt * w[((wk + ak * sk) * 6 + (wj + aj * sj)) * 6 + (wi + ai * si)];
                }
        fine[((size_t)b * 3 + c) * B3 + t] += v;
    }
}

// float64 prolongation.  Bound by the float64 pipe (8 multiply-adds per value above), so the
// interpolation is separable: along x over the window's 6 x 6 rows, along y over 6 planes, along z
// into the cells, each intermediate value formed once in shared memory: 12 operations per cell
// instead of 27, and a thread block per fine block also where one coarse block's 8 children fill the
// grid.  128^3: 134 us with the one-pass form on coarse blocks, one coarse block alone 36 us.
__global__ void __launch_bounds__(256) k_prolong_add_d(GridDev g, GridDev gc, const double *__restrict__ coarse,
                                                       const double *__restrict__ lex, int3 ld, double *__restrict__ fine,
                                                       int *__restrict__ err) {
    __shared__ double win[3 * 216], wx8[3 * 288], wy8[3 * 384];  // [6][6][6], [6][6][8], [6][8][8] per component
    const int b = blockIdx.x;
    if (skip_block(g, b)) return;
    const int o = lex ? 0 : g.octant[b];
    const int pb = lex ? 0 : g.parent[b];
    const int t = threadIdx.x;
    for (int q = t; q < 216; q += 256) {
        const int wx = q % 6, wy = (q / 6) % 6, wz = q / 36;
        if (lex) {
            int x = 4 * g.origin[b * 3 + 0] - 1 + wx, y = 4 * g.origin[b * 3 + 1] - 1 + wy, z = 4 * g.origin[b * 3 + 2] - 1 + wz;
            x = (x + ld.x) % ld.x; y = (y + ld.y) % ld.y; z = (z + ld.z) % ld.z;
            const double *lx = lex + lex_inst_offset(g, b, 3, ld);
            for (int c = 0; c < 3; c++) win[c * 216 + q] = lx[(((size_t)c * ld.z + z) * ld.y + y) * ld.x + x];
        } else {
            const int cx = 4 * (o & 1) - 1 + wx, cy = 4 * ((o >> 1) & 1) - 1 + wy, cz = 4 * (o >> 2) - 1 + wz;
            const int dx = cx < 0 ? -1 : (cx > 7 ? 1 : 0), dy = cy < 0 ? -1 : (cy > 7 ? 1 : 0), dz = cz < 0 ? -1 : (cz > 7 ? 1 : 0);
            const int src = gc.nbr[pb * 27 + (dz + 1) * 9 + (dy + 1) * 3 + (dx + 1)];
            if (src < 0) {
                if (err) *err = 1;
                for (int c = 0; c < 3; c++) win[c * 216 + q] = 0.0;
            } else {
                const int lx = cx - 8 * dx, ly = cy - 8 * dy, lz = cz - 8 * dz;
                for (int c = 0; c < 3; c++) win[c * 216 + q] = coarse[((size_t)src * 3 + c) * B3 + (lz * 8 + ly) * 8 + lx];
            }
        }
    }
    double old[2][3];  // the fine values come in while the window is interpolated
#pragma unroll
    for (int h = 0; h < 2; h++)
#pragma unroll
        for (int c = 0; c < 3; c++) old[h][c] = fine[((size_t)b * 3 + c) * B3 + t + 256 * h];
    __syncthreads();
    // fine cells 2w - 2 and 2w - 1 from window cell w = 1 .. 4 and its neighbours: (3 f0 + f-)/4, (3 f0 + f+)/4
    for (int q = t; q < 3 * 144; q += 256) {
        const int row = q >> 2, w = (q & 3) + 1;  // row: component and (z, y) of the window
        const double *p = win + row * 6 + w;
        const double m = 0.75 * p[0];
        wx8[row * 8 + 2 * w - 2] = fma(0.25, p[-1], m);
        wx8[row * 8 + 2 * w - 1] = fma(0.25, p[1], m);
    }
    __syncthreads();
    for (int q = t; q < 3 * 6 * 32; q += 256) {
        const int x = q & 7, w = ((q >> 3) & 3) + 1, cz = q >> 5;  // cz: component and z of the window
        const double *p = wx8 + (cz * 6 + w) * 8 + x;
        const double m = 0.75 * p[0];
        wy8[(cz * 8 + 2 * w - 2) * 8 + x] = fma(0.25, p[-8], m);
        wy8[(cz * 8 + 2 * w - 1) * 8 + x] = fma(0.25, p[8], m);
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int q = t + 256 * h, k = q >> 6, w = (k >> 1) + 1, sz = (k & 1) ? 64 : -64;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double *p = wy8 + (c * 6 + w) * 64 + (q & 63);
            fine[((size_t)b * 3 + c) * B3 + q] = fma(0.25, p[sz], fma(0.75, p[0], old[h][c]));
        }
    }
}

template <typename T>
cudaError_t launch_prolong_add(const GridDev &g, const GridDev *gc, const T *coarse, const T *lex, const int *ldims,
                               T *fine, int *err, cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    int3 ld = make_int3(ldims ? ldims[0] : 0, ldims ? ldims[1] : 0, ldims ? ldims[2] : 0);
    GridDev c = gc ? *gc : GridDev();
    if constexpr (std::is_same<T, double>::value)
        launch_full(k_prolong_add_d, g.nblk, 256, 0, s, g, c, coarse, lex, ld, fine, err);
    else
        launch_pdl2(k_prolong_add<T, true>, k_prolong_add<T, false>, g.nblk, 512, 0, s, g, c, coarse, lex, ld, fine, err);
    return cudaGetLastError();
}
template cudaError_t launch_prolong_add<double>(const GridDev &, const GridDev *, const double *, const double *,
                                                const int *, double *, int *, cudaStream_t);
template cudaError_t launch_prolong_add<float>(const GridDev &, const GridDev *, const float *, const float *,
                                               const int *, float *, int *, cudaStream_t);

// Prolongation for a coarse grid whose blocks' 8 children are the fine blocks 8c .. 8c+7 in
// octant order (Morton-ordered complete grids): one thread block per coarse block stages the
// coarse block and its 1-cell halo once (10^3, as the stencil kernels do) and adds the
// trilinear interpolant (3/4, 1/4 per axis, the weights of k_prolong_add) to all 4096 cells of
// the 8 children, one child block per pass of its 512 threads.
template <typename T, bool EARLY>
__global__ void __launch_bounds__(512) k_prolong_add8(GridDev gc, const T *__restrict__ coarse, T *__restrict__ fine) {
    using G = Geo<T>;
    __shared__ __align__(16) T tC[3 * G::CS];
    __shared__ int snb[27];
    const int c0 = blockIdx.x;
    pdl_trigger<EARLY>();
    if (!EARLY && skip_block(gc, c0)) return;  // (masked blocks return before they load anything)
    stage_nbr(snb, gc.nbr, c0);
    const int c = c0 + pdl_wait<EARLY>();
    if (EARLY && skip_block(gc, c)) return;
    __syncthreads();
    stage_rows<T, 3, 1, G::RS, G::OFF>(tC, coarse, snb, nullptr);
    __syncthreads();
    const int t = threadIdx.x, lx = t & 7, ly = (t >> 3) & 7, lz = t >> 6;
    for (int o = 0; o < 8; o++) {
        const int fx = lx + 8 * (o & 1), fy = ly + 8 * ((o >> 1) & 1), fz = lz + 8 * (o >> 2);
        const int cx = fx >> 1, cy = fy >> 1, cz = fz >> 1;
        const int sx = (fx & 1) ? 1 : -1, sy = (fy & 1) ? 1 : -1, sz = (fz & 1) ? 1 : -1;
        const int p = G::at(cx + 1, cy + 1, cz + 1);
        const size_t fb = ((size_t)(8 * c + o) * 3) * B3 + t;
#pragma unroll
        for (int comp = 0; comp < 3; comp++) {
            const T *w = tC + comp * G::CS;
            T v = 0;
            for (int ak = 0; ak < 2; ak++)
                for (int aj = 0; aj < 2; aj++)
                    for (int ai = 0; ai < 2; ai++) {
                        const T wt = (ai ? T(0.25) : T(0.75)) * (aj ? T(0.25) : T(0.75)) * (ak ? T(0.25) : T(0.75));
                        v += wt * w[p + ak * sz * G::PS + aj * sy * G::RS + ai * sx];
                    }
            fine[fb + (size_t)comp * B3] += v;
        }
    }
}

template <typename T>
cudaError_t launch_prolong_add8(const GridDev &gc, const T *coarse, T *fine, cudaStream_t s) {
    if (gc.nblk == 0) return cudaSuccess;
    launch_pdl2(k_prolong_add8<T, true>, k_prolong_add8<T, false>, gc.nblk, 512, 0, s, gc, coarse, fine);
    return cudaGetLastError();
}
template cudaError_t launch_prolong_add8<float>(const GridDev &, const float *, float *, cudaStream_t);

// ------------------------------------------------------------------ coarse-fine ghosts
// Ghost slot of a level-l block: the halo cells without a same-level neighbour get the tri-quadratic
// interpolant of the parent's 3x3x3 coarse neighbourhood at the child's centre (offset s h_c/4 per
// axis):
//   f0 + sum_d [s_d (f+ - f-)/8 + (f+ - 2 f0 + f-)/32] + sum_{d<e} s_d s_e (cross diff)/64.
// The coarse window is [4o-2, 4o+6) per axis in parent-local cells.  The interpolation is float64 and
// bound by that pipe, so only the faces and edges that a stencil reads from the slot are filled (the
// others lie in a same-level neighbour), and a thread takes one coarse cell and component: its
// differences serve the 4 fine ghosts of a face (2 of an edge), 8 operations per ghost instead of
// about 45.  One launch over the 296 slots of the third nested-sphere level (base 64^3): 74 -> 11 us;
// the three-level mixed step 3.98 -> 2.50 ms.
template <typename TS_, typename TD>
__global__ void __launch_bounds__(512) k_ghost_fill(GridDev g, GridDev gc, const TS_ *__restrict__ coarse, int ncomp,
                                                    TD *__restrict__ ghost, int *__restrict__ err) {
    __shared__ double win[3 * 512];
    __shared__ uint8_t side[144], unit[144];  // the units to fill: direction (0-5 faces, 6-17 edges) and coarse cell
    __shared__ int nunit;
    const int sl = blockIdx.x;
    const int b = g.slot_block[sl];
    pdl_trigger();
    const int o = g.octant[b], pb = g.parent[b] + pdl_wait();
    if (skip_block(g, b)) return;
    const int ox = 4 * (o & 1), oy = 4 * ((o >> 1) & 1), oz = 4 * (o >> 2);
    if (threadIdx.x < 32) {
        // direction l: face 2 axis + high, or edge 6 + 4 (free axis) + signs of the two others (ascending)
        const int l = threadIdx.x;
        int d[3] = {0, 0, 0};
        if (l < 6) {
            d[l >> 1] = (l & 1) ? 1 : -1;
        } else if (l < 18) {
            const int f = (l - 6) >> 2, a1 = f == 0 ? 1 : 0, a2 = f == 2 ? 1 : 2;
            d[a1] = (l - 6) & 1 ? 1 : -1;
            d[a2] = (l - 6) & 2 ? 1 : -1;
        }
        const int units = l < 18 && g.nbr[b * 27 + (d[2] + 1) * 9 + (d[1] + 1) * 3 + d[0] + 1] < 0 ? (l < 6 ? 16 : 4) : 0;
        int at = units;
        for (int k = 1; k < 32; k <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, at, k);
            if (l >= k) at += v;
        }
        for (int k = 0; k < units; k++) {
            side[at - units + k] = (uint8_t)l;
            unit[at - units + k] = (uint8_t)k;
        }
        if (l == 31) nunit = at;
    }
    for (int q = threadIdx.x; q < 512; q += blockDim.x) {
        const int wx = q & 7, wy = (q >> 3) & 7, wz = q >> 6;
        int cx = ox - 2 + wx, cy = oy - 2 + wy, cz = oz - 2 + wz;
        int dx = cx < 0 ? -1 : (cx > 7 ? 1 : 0), dy = cy < 0 ? -1 : (cy > 7 ? 1 : 0), dz = cz < 0 ? -1 : (cz > 7 ? 1 : 0);
        int src = gc.nbr[pb * 27 + (dz + 1) * 9 + (dy + 1) * 3 + (dx + 1)];
        if (src < 0) {
            if (err) *err = 1;
            for (int c = 0; c < ncomp; c++) win[c * 512 + q] = 0.0;
        } else {
            int lx = cx - 8 * dx, ly = cy - 8 * dy, lz = cz - 8 * dz;
            for (int c = 0; c < ncomp; c++)
                win[c * 512 + q] = (double)coarse[((size_t)src * ncomp + c) * B3 + (lz * 8 + ly) * 8 + lx];
        }
    }
    __syncthreads();
    const int nu = nunit;
    for (int idx = threadIdx.x; idx < nu * ncomp; idx += blockDim.x) {
        const int c = idx / nu, l = side[idx - c * nu], k = unit[idx - c * nu];
        // axes: n1 (and, on an edge, n2) point out of the block, the others run along it
        const bool face = l < 6;
        int n1, n2, f1, f2, s1, s2 = 0;  // s1, s2: the out-of-block side, 1 = high
        if (face) {
            n1 = l >> 1;
            s1 = l & 1;
            f1 = n1 == 0 ? 1 : 0;
            f2 = n1 == 2 ? 1 : 2;
            n2 = f2;
        } else {
            f1 = (l - 6) >> 2;
            n1 = f1 == 0 ? 1 : 0;
            n2 = f1 == 2 ? 1 : 2;
            s1 = (l - 6) & 1;
            s2 = ((l - 6) >> 1) & 1;
            f2 = n2;
        }
        auto wst = [](int ax) { return ax == 0 ? 1 : (ax == 1 ? 8 : 64); };    // window stride
        auto tst = [](int ax) { return ax == 0 ? 1 : (ax == 1 ? TS : TS * TS); };  // slot stride
        const int wn = wst(n1), wf = wst(f1), w2 = wst(f2);
        const int w0 = wn * (s1 ? 6 : 1) + wf * ((k & 3) + 2) + w2 * (face ? (k >> 2) + 2 : (s2 ? 6 : 1));
        const double *W = win + c * 512 + w0;
        const double f0 = W[0];
        const double p1 = W[wn], m1 = W[-wn], p2 = W[wf], m2 = W[-wf], p3 = W[w2], m3 = W[-w2];
        const double v0 = fma(1.0 / 32, fma(-6.0, f0, ((p1 + m1) + (p2 + m2)) + (p3 + m3)), f0);
        const double g1 = p1 - m1, g2 = p2 - m2, g3 = p3 - m3;
        const double x12 = (W[wn + wf] - W[wn - wf]) - (W[-wn + wf] - W[-wn - wf]);
        const double x13 = (W[wn + w2] - W[wn - w2]) - (W[-wn + w2] - W[-wn - w2]);
        const double x23 = (W[wf + w2] - W[wf - w2]) - (W[-wf + w2] - W[-wf - w2]);
        const double e8 = s1 ? -0.125 : 0.125, e64 = s1 ? -1.0 / 64 : 1.0 / 64;  // the ghost is the near child
        TD *dst = ghost + ((size_t)sl * ncomp + c) * T3 + tst(n1) * (s1 ? 9 : 0) + tst(f1) * (2 * (k & 3) + 1);
        if (face) {
            dst += tst(f2) * (2 * (k >> 2) + 1);
            const double base = fma(e8, g1, v0), x = x23 * (1.0 / 64);
            const double a2 = fma(e64, x12, 0.125 * g2), a3 = fma(e64, x13, 0.125 * g3);
            const double bp = base + x, bm = base - x, sp = a2 + a3, sm = a2 - a3;
            const int t1 = tst(f1), t2 = tst(f2);
            dst[0] = (TD)(bp - sp);
            dst[t1] = (TD)(bm + sm);
            dst[t2] = (TD)(bm - sm);
            dst[t1 + t2] = (TD)(bp + sp);
        } else {
            dst += tst(n2) * (s2 ? 9 : 0);
            const double u8 = s2 ? -0.125 : 0.125, u64 = s2 ? -1.0 / 64 : 1.0 / 64;
            const double base = fma(s2 ? -e64 : e64, x13, fma(u8, g3, fma(e8, g1, v0)));
            const double a2 = fma(u64, x23, fma(e64, x12, 0.125 * g2));
            dst[0] = (TD)(base - a2);
            dst[tst(f1)] = (TD)(base + a2);
        }
    }
}

template <typename TS_, typename TD>
cudaError_t launch_ghost_fill(const GridDev &g, const GridDev &gc, const TS_ *coarse, int ncomp, TD *ghost, int *err,
                              cudaStream_t s) {
    if (g.nslot == 0) return cudaSuccess;
    launch_pdl(k_ghost_fill<TS_, TD>, g.nslot, 512, 0, s, g, gc, coarse, ncomp, ghost + (size_t)g.slot0 * ncomp * T3, err);
    return cudaGetLastError();
}
template cudaError_t launch_ghost_fill<double, double>(const GridDev &, const GridDev &, const double *, int, double *,
                                                       int *, cudaStream_t);
template cudaError_t launch_ghost_fill<float, float>(const GridDev &, const GridDev &, const float *, int, float *,
                                                     int *, cudaStream_t);

// ------------------------------------------------------------------ sync down, update
template <typename T>
__global__ void __launch_bounds__(512) k_sync_down(GridDev gc, T *__restrict__ Bc, const T *__restrict__ Bf) {
    pdl_trigger();
    const int b = blockIdx.x + pdl_wait();
    if (!gc.covered[b] || skip_block(gc, b)) return;
    const int t = threadIdx.x, i = t & 7, j = (t >> 3) & 7, k = t >> 6;
    const int oc = (i >> 2) | ((j >> 2) << 1) | ((k >> 2) << 2);
    const int ch = gc.child[b * 8 + oc];
    const int fi = 2 * (i & 3), fj = 2 * (j & 3), fk = 2 * (k & 3);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const T *src = Bf + ((size_t)ch * 3 + c) * B3;
        T s = 0;
        for (int dk = 0; dk < 2; dk++)
            for (int dj = 0; dj < 2; dj++)
                for (int di = 0; di < 2; di++) s += src[((fk + dk) * 8 + fj + dj) * 8 + fi + di];
        Bc[((size_t)b * 3 + c) * B3 + t] = s / T(8);
    }
}

template <typename T>
cudaError_t launch_sync_down(const GridDev &gc, T *Bc, const T *Bf, cudaStream_t s) {
    if (gc.nblk == 0) return cudaSuccess;
    launch_pdl(k_sync_down<T>, gc.nblk, 512, 0, s, gc, Bc, Bf);
    return cudaGetLastError();
}
template cudaError_t launch_sync_down<double>(const GridDev &, double *, const double *, cudaStream_t);
template cudaError_t launch_sync_down<float>(const GridDev &, float *, const float *, cudaStream_t);

// x += y on leaf blocks (inner correction accumulation)
template <typename T>
__global__ void __launch_bounds__(512) k_axpy_leaf(GridDev g, T *__restrict__ x, const T *__restrict__ y,
                                                   const uint8_t *__restrict__ imask) {
    pdl_trigger();
    const int b = blockIdx.x + pdl_wait();
    if ((g.covered && g.covered[b]) || inst_masked(g, imask, b)) return;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        size_t id = ((size_t)b * 3 + c) * B3 + threadIdx.x;
        x[id] += y[id];
    }
}

template <typename T>
cudaError_t launch_axpy_leaf(const GridDev &g, T *x, const T *y, const uint8_t *imask, cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    launch_pdl(k_axpy_leaf<T>, g.nblk, 512, 0, s, g, x, y, imask);
    return cudaGetLastError();
}
template cudaError_t launch_axpy_leaf<float>(const GridDev &, float *, const float *, const uint8_t *, cudaStream_t);
template cudaError_t launch_axpy_leaf<double>(const GridDev &, double *, const double *, const uint8_t *, cudaStream_t);

template <typename T>
__global__ void __launch_bounds__(512) k_update(GridDev g, double *__restrict__ B, const T *__restrict__ e,
                                                const uint8_t *__restrict__ imask) {
    pdl_trigger();
    const int b = blockIdx.x + pdl_wait();
    if ((g.covered && g.covered[b]) || inst_masked(g, imask, b)) return;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        size_t id = ((size_t)b * 3 + c) * B3 + threadIdx.x;
        B[id] += (double)e[id];
    }
}

template <typename T>
cudaError_t launch_update(const GridDev &g, double *B, const T *e, const uint8_t *imask, cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    launch_pdl(k_update<T>, g.nblk, 512, 0, s, g, B, e, imask);
    return cudaGetLastError();
}
template cudaError_t launch_update<double>(const GridDev &, double *, const double *, const uint8_t *, cudaStream_t);
template cudaError_t launch_update<float>(const GridDev &, double *, const float *, const uint8_t *, cudaStream_t);

__global__ void __launch_bounds__(512) k_zero_covered(GridDev g, double *__restrict__ x) {
    const int b = blockIdx.x;
    if (!(g.covered && g.covered[b])) return;
    for (int c = 0; c < 3; c++) x[((size_t)b * 3 + c) * B3 + threadIdx.x] = 0.0;
}

cudaError_t launch_zero_covered(const GridDev &g, double *x, cudaStream_t s) {
    if (g.nblk == 0 || !g.covered) return cudaSuccess;
    k_zero_covered<<<g.nblk, 512, 0, s>>>(g, x);
    return cudaGetLastError();
}

// Deterministic reduction of per-block partials {sum R^2 dV, sum S^2 dV, max |R|}: every
// thread block folds a fixed contiguous chunk in a fixed order, and the last block to finish
// (atomic ticket) folds the per-chunk results in chunk order.
constexpr int NRED = 128;

// block i of level l: its entries added pairwise (as the kernel that wrote them adds the ones it
// holds), times the level's scale
__device__ __forceinline__ void norm_add(const double *__restrict__ part, const PartRanges &R, int l, int i, double &a, double &b,
                                         double &m) {
    const int ns = R.parts[l];
    const double *p = part + ((size_t)R.base[l] + (size_t)(i - R.off[l]) * ns) * 3;
    double x = p[0], y = p[1], z = p[2];
    if (ns == 2) {
        x = x + p[3];
        y = y + p[4];
        z = fmax(z, p[5]);
    } else if (ns == 4) {
        x = (x + p[3]) + (p[6] + p[9]);
        y = (y + p[4]) + (p[7] + p[10]);
        z = fmax(fmax(z, p[5]), fmax(p[8], p[11]));
    }
    a = fma(x, R.vol[l], a);
    b = fma(y, R.vol[l], b);
    m = fmax(m, z);
}

// sums of a and b and maximum of m over the thread block in a fixed order, valid in thread 0
__device__ __forceinline__ void block_norms(double &a, double &b, double &m, double (*red)[3]) {
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        red[w][0] = a;
        red[w][1] = b;
        red[w][2] = m;
    }
    __syncthreads();
    if (w == 0) {
        a = threadIdx.x < nw ? red[threadIdx.x][0] : 0.0;
        b = threadIdx.x < nw ? red[threadIdx.x][1] : 0.0;
        m = threadIdx.x < nw ? red[threadIdx.x][2] : 0.0;
        for (int o = 4; o > 0; o >>= 1) {  // 8 warps
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
            m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        }
    }
}

__global__ void __launch_bounds__(256) k_norm_reduce(const double *__restrict__ part, PartRanges R, int n, double *__restrict__ chunk,
                                                     unsigned int *__restrict__ ticket, double *__restrict__ out,
                                                     double *__restrict__ host_out, const int *__restrict__ err) {
    __shared__ double red[8][3];
    __shared__ bool last;
    pdl_trigger();
    const int z = pdl_wait();
    const int per = (n + gridDim.x - 1) / gridDim.x;
    const int lo = blockIdx.x * per + z, hi = min(n, lo + per);
    double a = 0.0, b = 0.0, m = 0.0;
    int l = 0;
    for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        while (l + 1 < R.nlev && i >= R.off[l + 1]) l++;
        norm_add(part, R, l, i, a, b, m);
    }
    block_norms(a, b, m, red);
    if (gridDim.x > 1) {
        if (threadIdx.x == 0) {
            chunk[blockIdx.x * 3 + 0] = a;
            chunk[blockIdx.x * 3 + 1] = b;
            chunk[blockIdx.x * 3 + 2] = m;
            __threadfence();
            last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        a = b = m = 0.0;
        for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
            a += __ldcg(chunk + i * 3 + 0);
            b += __ldcg(chunk + i * 3 + 1);
            m = fmax(m, __ldcg(chunk + i * 3 + 2));
        }
        block_norms(a, b, m, red);
    }
    if (threadIdx.x == 0) {
        out[0] = a;
        out[1] = b;
        out[2] = m;
        if (host_out) {  // pinned host memory mapped into the device: no copy needed to read them
            host_out[0] = a;
            host_out[1] = b;
            host_out[2] = m;
            reinterpret_cast<volatile int *>(host_out + 4)[0] = err ? err[z] : 0;
        }
        *ticket = 0u;
    }
}

// scratch: NRED * 3 doubles followed by one unsigned ticket (zero on first use)
cudaError_t launch_norm_reduce(const double *partials, const PartRanges &R, int nblocks, double *scratch, double *out,
                               cudaStream_t s, double *host_out, const int *err) {
    int grid = nblocks < NRED * 64 ? (nblocks + 63) / 64 : NRED;
    if (nblocks <= 512) grid = 1;  // one thread block, no second stage
    launch_pdl(k_norm_reduce, grid, 256, 0, s, partials, R, nblocks, scratch, (unsigned int *)(scratch + 3 * NRED), out, host_out, err);
    return cudaGetLastError();
}

// One thread block per instance; its level ranges are folded in level order, each range in a
// fixed thread-strided order, so the result does not depend on the other instances.
__global__ void __launch_bounds__(256) k_norm_inst(const double *__restrict__ part, PartRanges R, double *__restrict__ out) {
    __shared__ double red[8][3];
    pdl_trigger();
    const int q = blockIdx.x + pdl_wait();
    double a = 0.0, b = 0.0, m = 0.0;
    for (int l = 0; l < R.nlev; l++) {
        const int lo = R.off[l] + q * R.n[l], hi = lo + R.n[l];
        for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) norm_add(part, R, l, i, a, b, m);
    }
    block_norms(a, b, m, red);
    if (threadIdx.x == 0) {
        out[q * 4 + 0] = a;
        out[q * 4 + 1] = b;
        out[q * 4 + 2] = m;
        out[q * 4 + 3] = 0.0;
    }
}

cudaError_t launch_norm_inst(const double *partials, const PartRanges &R, int ninst, double *out, cudaStream_t s) {
    if (ninst <= 0) return cudaSuccess;
    launch_pdl(k_norm_inst, ninst, 256, 0, s, partials, R, out);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(512) k_scale_blocks(const double *__restrict__ src, double *__restrict__ dst,
                                                      const double *__restrict__ scale) {
    const size_t id = (size_t)blockIdx.x * B3 + threadIdx.x;
    dst[id] = src[id] * scale[blockIdx.x];
}

cudaError_t launch_scale_blocks(const double *src, double *dst, const double *scale, int nblk, cudaStream_t s) {
    if (nblk <= 0) return cudaSuccess;
    k_scale_blocks<<<nblk, 512, 0, s>>>(src, dst, scale);
    return cudaGetLastError();
}

template <typename TS_, typename TD>
__global__ void k_convert(const TS_ *__restrict__ src, TD *__restrict__ dst, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        dst[i] = (TD)src[i];
}

template <typename TS_, typename TD>
cudaError_t launch_convert(const TS_ *src, TD *dst, size_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    int grid = (int)((n + 255) / 256);
    if (grid > 152 * 32) grid = 152 * 32;
    k_convert<TS_, TD><<<grid, 256, 0, s>>>(src, dst, n);
    return cudaGetLastError();
}
template cudaError_t launch_convert<double, float>(const double *, float *, size_t, cudaStream_t);
template cudaError_t launch_convert<double, double>(const double *, double *, size_t, cudaStream_t);

// ------------------------------------------------------------------ Krylov vector kernels
// Vectors are block fields [nblk][3][512]; inner products are volume weighted over leaf
// blocks (weight w_b = h^3, 0 for covered blocks), the norm of the convergence tests.
// The number of vectors NV is a template parameter (one instantiation per count, chosen at
// launch), so a thread holds exactly NV + 1 partial sums: with a run-time count the compiler
// kept the 13 sums of the largest case, which cost occupancy (76 registers).
// One warp per 8^3 block: each lane forms 12 float4 products per column in float32, the warp
// reduces them by shuffles and lane 0 weights the sum in float64.
template <int NV>
__device__ __forceinline__ void warp_block_dots(const float *__restrict__ w, const VecSet &V, int b, int lane,
                                                double wt, double out[NV + 1]) {
    float f[NV + 1];
#pragma unroll
    for (int i = 0; i <= NV; i++) f[i] = 0.f;
    if (wt != 0.0) {
        const float4 *w4 = reinterpret_cast<const float4 *>(w + (size_t)b * 1536);
#pragma unroll 1
        for (int s = 0; s < 12; s++) {
            const float4 x = w4[lane + 32 * s];
            f[NV] += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
#pragma unroll
            for (int i = 0; i < NV; i++) {
                const float4 v = reinterpret_cast<const float4 *>(V.v[i] + (size_t)b * 1536)[lane + 32 * s];
                f[i] += x.x * v.x + x.y * v.y + x.z * v.z + x.w * v.w;
            }
        }
    }
#pragma unroll
    for (int i = 0; i <= NV; i++) {
        float v = f[i];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        out[i] = (double)v * wt;
    }
}

// the 8 warps of a thread block are folded in warp order into part[blockIdx][col]
template <int NV>
__global__ void __launch_bounds__(256) k_mdot(const float *__restrict__ w, VecSet V, const double *__restrict__ wb,
                                              int nblk, double *__restrict__ part, const int *__restrict__ gate) {
    pdl_trigger();
    const int z = pdl_wait();
    if (gate && !gate[z]) return;
    __shared__ double sred[8][NV + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.x * 8 + warp + z;
    double d[NV + 1];
    warp_block_dots<NV>(w, V, b < nblk ? b : 0, lane, b < nblk ? wb[b] : 0.0, d);
    if (lane == 0)
        for (int i = 0; i <= NV; i++) sred[warp][i] = d[i];
    __syncthreads();
    if (threadIdx.x <= NV) {
        double a = 0.0;
        for (int q = 0; q < 8; q++) a += sred[q][threadIdx.x];
        part[(size_t)blockIdx.x * (NV + 1) + threadIdx.x] = a;
    }
}

// column sums of part[nrow][ncol] in a fixed order (one thread block per column)
__global__ void __launch_bounds__(256) k_colsum(const double *__restrict__ part, int nrow, int ncol, double *__restrict__ out,
                                                const int *__restrict__ gate, double *__restrict__ host_out) {
    pdl_trigger();
    const int z = pdl_wait();
    if (gate && !gate[z]) return;
    __shared__ double red[32];
    const int c = blockIdx.x + z;
    double a = 0.0;
    for (int b = threadIdx.x; b < nrow; b += blockDim.x) a += part[(size_t)b * ncol + c];
    double s = block_sum(a, red);
    if (threadIdx.x == 0) {
        out[c] = s;
        if (host_out) host_out[c] = s;  // mapped pinned host memory
    }
}

// dst = (src - sum_i c_i v_i) * scale (dst may equal src; src null reads as 0); float4 over n/4 groups
template <int NV>
__global__ void __launch_bounds__(256) k_maxpy(float4 *dst, const float4 *src, VecSet V, float scale, size_t n4) {
    pdl_trigger();
    pdl_wait();
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n4; q += (size_t)gridDim.x * blockDim.x) {
        float4 x = src ? src[q] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < NV; i++) {
            const float4 v = reinterpret_cast<const float4 *>(V.v[i])[q];
            const float c = V.c[i];
            x.x -= c * v.x;
            x.y -= c * v.y;
            x.z -= c * v.z;
            x.w -= c * v.w;
        }
        x.x *= scale;
        x.y *= scale;
        x.z *= scale;
        x.w *= scale;
        dst[q] = x;
    }
}

// one instantiation per vector count 0 .. KMAX
#define OHM_NV_SWITCH(k, CALL)   \
    switch (k) {                 \
        case 0: CALL(0); break;  \
        case 1: CALL(1); break;  \
        case 2: CALL(2); break;  \
        case 3: CALL(3); break;  \
        case 4: CALL(4); break;  \
        case 5: CALL(5); break;  \
        case 6: CALL(6); break;  \
        case 7: CALL(7); break;  \
        case 8: CALL(8); break;  \
        case 9: CALL(9); break;  \
        case 10: CALL(10); break; \
        case 11: CALL(11); break; \
        default: CALL(12); break; \
    }

cudaError_t launch_mdot(const float *w, const VecSet &V, const double *wb, int nblk, double *part, double *out,
                        cudaStream_t s, const int *gate, double *host_out) {
    const int grid = (nblk + 7) / 8;
#define OHM_MDOT(N) launch_pdl(k_mdot<N>, grid, 256, 0, s, w, V, wb, nblk, part, gate)
    OHM_NV_SWITCH(V.k, OHM_MDOT)
#undef OHM_MDOT
    launch_pdl(k_colsum, V.k + 1, 256, 0, s, part, grid, V.k + 1, out, gate, host_out);
    return cudaGetLastError();
}

// float64 Krylov vectors: one warp per block for the products (double2 loads, float64 sums), a
// grid-stride loop for the updates
template <int NV>
__global__ void __launch_bounds__(256) k_mdot_d(const double *__restrict__ w, VecSetD V, const double *__restrict__ wb,
                                                int nblk, double *__restrict__ part) {
    pdl_trigger();
    const int z = pdl_wait();
    __shared__ double sred[8][NV + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.x * 8 + warp + z;
    double f[NV + 1];
#pragma unroll
    for (int i = 0; i <= NV; i++) f[i] = 0.0;
    const double wt = b < nblk ? wb[b] : 0.0;
    if (wt != 0.0) {
        const double2 *w2 = reinterpret_cast<const double2 *>(w + (size_t)b * 1536);
#pragma unroll 1
        for (int q = lane; q < 768; q += 32) {
            const double2 x = w2[q];
            f[NV] = fma(x.x, x.x, fma(x.y, x.y, f[NV]));
#pragma unroll
            for (int i = 0; i < NV; i++) {
                const double2 v = reinterpret_cast<const double2 *>(V.v[i] + (size_t)b * 1536)[q];
                f[i] = fma(x.x, v.x, fma(x.y, v.y, f[i]));
            }
        }
    }
#pragma unroll
    for (int i = 0; i <= NV; i++) {
        double v = f[i];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) sred[warp][i] = v * wt;
    }
    __syncthreads();
    if (threadIdx.x <= NV) {
        double a = 0.0;
        for (int q = 0; q < 8; q++) a += sred[q][threadIdx.x];
        part[(size_t)blockIdx.x * (NV + 1) + threadIdx.x] = a;
    }
}

template <int NV>
__global__ void __launch_bounds__(256) k_maxpy_d(double2 *dst, const double2 *src, VecSetD V, double scale, size_t n2) {
    pdl_trigger();
    pdl_wait();
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n2; q += (size_t)gridDim.x * blockDim.x) {
        double2 x = src ? src[q] : make_double2(0.0, 0.0);
#pragma unroll
        for (int i = 0; i < NV; i++) {
            const double2 v = reinterpret_cast<const double2 *>(V.v[i])[q];
            x.x = fma(-V.c[i], v.x, x.x);
            x.y = fma(-V.c[i], v.y, x.y);
        }
        x.x *= scale;
        x.y *= scale;
        dst[q] = x;
    }
}

cudaError_t launch_mdot(const double *w, const VecSetD &V, const double *wb, int nblk, double *part, double *out,
                        cudaStream_t s, double *host_out) {
    const int grid = (nblk + 7) / 8;
#define OHM_MDOTD(N) launch_pdl(k_mdot_d<N>, grid, 256, 0, s, w, V, wb, nblk, part)
    OHM_NV_SWITCH(V.k, OHM_MDOTD)
#undef OHM_MDOTD
    launch_pdl(k_colsum, V.k + 1, 256, 0, s, part, grid, V.k + 1, out, nullptr, host_out);
    return cudaGetLastError();
}

cudaError_t launch_maxpy(double *dst, const double *src, const VecSetD &V, double scale, size_t n, cudaStream_t s) {
    const size_t n2 = n / 2;
    const int grid = (int)std::min<size_t>((n2 + 255) / 256, 152 * 16);
    double2 *d2 = reinterpret_cast<double2 *>(dst);
    const double2 *s2 = reinterpret_cast<const double2 *>(src);
#define OHM_MAXPYD(N) launch_pdl(k_maxpy_d<N>, grid, 256, 0, s, d2, s2, V, scale, n2)
    OHM_NV_SWITCH(V.k, OHM_MAXPYD)
#undef OHM_MAXPYD
    return cudaGetLastError();
}

// column sums of part[ncol][nrow] (column-major) in a fixed order, one thread block per column
__global__ void __launch_bounds__(1024) k_colsum_cm(const double *__restrict__ part, int nrow, double *__restrict__ out,
                                                    double *__restrict__ host_out) {
    pdl_trigger();
    const int z = pdl_wait();
    __shared__ double red[32];
    const double *col = part + (size_t)(blockIdx.x + z) * nrow;
    double a = 0.0;
    for (int b = threadIdx.x; b < nrow; b += blockDim.x) a += col[b];
    const double s = block_sum(a, red);
    if (threadIdx.x == 0) {
        out[blockIdx.x] = s;
        if (host_out) host_out[blockIdx.x] = s;  // mapped pinned host memory
    }
}

// w = L z on block pairs (the float32 operator of the inner solve) together with <w, v_i> and
// <w, w> of the FGMRES Arnoldi step: one pass instead of the operator and the multi-dot
cudaError_t launch_pair_apply_dots(const GridDev &g, const float *X, const float *eta, double kc, float *w,
                                   const VecSet &V, double wt, double *part, double *out, double *host_out,
                                   cudaStream_t s) {
    if (g.nblk == 0) return cudaSuccess;
    const size_t sm = 4 * G18::CS * sizeof(float);
    const int npair = g.nblk / 2;
#define OHM_PAIRDOT(N)                                                                                          \
    {                                                                                                          \
        static const bool attr_ =                                                                              \
            (cudaFuncSetAttribute(k_pair_op<true, false, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm), \
             true);                                                                                            \
        (void)attr_;                                                                                           \
        launch_full(k_pair_op<true, false, N>, npair, 512, sm, s, g, X, nullptr, eta, (float)kc, w, nullptr, V, wt, part);  \
    }
    OHM_NV_SWITCH(V.k, OHM_PAIRDOT)
#undef OHM_PAIRDOT
    launch_pdl(k_colsum_cm, V.k + 1, 1024, 0, s, part, npair, out, host_out);
    return cudaGetLastError();
}

cudaError_t launch_maxpy(float *dst, const float *src, const VecSet &V, float scale, size_t n, cudaStream_t s) {
    const size_t n4 = n / 4;  // fields are whole 8^3 blocks: n is a multiple of 1536
    const int grid = (int)std::min<size_t>((n4 + 255) / 256, 152 * 16);
    float4 *d4 = reinterpret_cast<float4 *>(dst);
    const float4 *s4 = reinterpret_cast<const float4 *>(src);
#define OHM_MAXPY(N) launch_pdl(k_maxpy<N>, grid, 256, 0, s, d4, s4, V, scale, n4)
    OHM_NV_SWITCH(V.k, OHM_MAXPY)
#undef OHM_MAXPY
    return cudaGetLastError();
}


// Per-instance Krylov vector kernels of batched hierarchies.  Block partials: one warp per
// block writes its weighted products (no folding across blocks, so no sum mixes instances).
template <int NV>
__global__ void __launch_bounds__(256) k_mdot_blocks(const float *__restrict__ w, VecSet V, const double *__restrict__ wb,
                                                     int nblk, double *__restrict__ part, const int *__restrict__ gate) {
    pdl_trigger();
    const int z = pdl_wait();
    if (gate && !gate[z]) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.x * 8 + warp + z;
    if (b >= nblk) return;
    double d[NV + 1];
    warp_block_dots<NV>(w, V, b, lane, wb[b], d);
    if (lane == 0)
        for (int i = 0; i <= NV; i++) part[(size_t)b * (NV + 1) + i] = d[i];
}

// out[q][c] = sum of part[b][c] over instance q's blocks of every level, in a fixed order
__global__ void __launch_bounds__(256) k_colsum_inst(const double *__restrict__ part, InstRanges R, int ncol,
                                                     double *__restrict__ out, const int *__restrict__ gate) {
    pdl_trigger();
    const int z = pdl_wait();
    if (gate && !gate[z]) return;
    __shared__ double red[32];
    const int q = blockIdx.x + z;
    for (int c = 0; c < ncol; c++) {
        double a = 0.0;
        for (int l = 0; l < R.nlev; l++) {
            const int lo = R.off[l] + q * R.n[l], hi = lo + R.n[l];
            for (int b = lo + threadIdx.x; b < hi; b += blockDim.x) a += part[(size_t)b * ncol + c];
        }
        const double sum = block_sum(a, red);
        if (threadIdx.x == 0) out[(size_t)q * (KMAX + 1) + c] = sum;
    }
}

cudaError_t launch_mdot_inst(const float *w, const VecSet &V, const double *wb, int nblk, const InstRanges &R, int ninst,
                             double *part, double *out, cudaStream_t s, const int *gate) {
#define OHM_MDOTB(N) launch_pdl(k_mdot_blocks<N>, (nblk + 7) / 8, 256, 0, s, w, V, wb, nblk, part, gate)
    OHM_NV_SWITCH(V.k, OHM_MDOTB)
#undef OHM_MDOTB
    launch_pdl(k_colsum_inst, ninst, 256, 0, s, part, R, V.k + 1, out, gate);
    return cudaGetLastError();
}

// dst = (src - sum_i c[q][i] v_i) * c[q][KMAX] with q the instance of the element's block;
// terms whose coefficient is 0 are skipped (their vectors may hold anything for that instance)
template <int NV>
__global__ void __launch_bounds__(256) k_maxpy_inst(float4 *dst, const float4 *src, VecSet V,
                                                    const float *__restrict__ coef, const int *__restrict__ binst,
                                                    size_t n4, const int *__restrict__ gate) {
    pdl_trigger();
    const int z = pdl_wait();
    if (gate && !gate[z]) return;
    for (size_t e = z + blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n4; e += (size_t)gridDim.x * blockDim.x) {
        const float *cq = coef + (size_t)binst[e / 384] * (KMAX + 1);
        float4 x = src[e];
#pragma unroll
        for (int i = 0; i < NV; i++) {
            const float c = cq[i];
            if (c != 0.f) {
                const float4 v = reinterpret_cast<const float4 *>(V.v[i])[e];
                x.x -= c * v.x;
                x.y -= c * v.y;
                x.z -= c * v.z;
                x.w -= c * v.w;
            }
        }
        const float sc = cq[KMAX];
        x.x *= sc;
        x.y *= sc;
        x.z *= sc;
        x.w *= sc;
        dst[e] = x;
    }
}

cudaError_t launch_maxpy_inst(float *dst, const float *src, const VecSet &V, const float *coef, const int *binst,
                              size_t n, cudaStream_t s, const int *gate) {
    const size_t n4 = n / 4;
    const int grid = (int)std::min<size_t>((n4 + 255) / 256, 152 * 16);
    float4 *d4 = reinterpret_cast<float4 *>(dst);
    const float4 *s4 = reinterpret_cast<const float4 *>(src);
#define OHM_MAXPYI(N) launch_pdl(k_maxpy_inst<N>, grid, 256, 0, s, d4, s4, V, coef, binst, n4, gate)
    OHM_NV_SWITCH(V.k, OHM_MAXPYI)
#undef OHM_MAXPYI
    return cudaGetLastError();
}

// ------------------------------------------------------------------ coarsest grids
// Lexicographic periodic grids below the last blocked grid.  Face flux and divergence as above, with
// periodic wrap.
template <typename T>
struct LexGrid {
    int nx, ny, nz;
    __device__ __forceinline__ int wrap(int v, int n) const { return v < 0 ? v + n : (v >= n ? v - n : v); }
    __device__ __forceinline__ size_t id(int c, int x, int y, int z) const {
        return (((size_t)c * nz + wrap(z, nz)) * ny + wrap(y, ny)) * nx + wrap(x, nx);
    }
};

template <typename T>
__device__ __forceinline__ void lex_face(const LexGrid<T> &G, const T *B, const T *E, int x, int y, int z, int a,
                                         T &phi1, T &phi2) {
    int o[3] = {0, 0, 0};
    o[a] = 1;
    const int b1 = a == 0 ? 1 : 0, b2 = a == 2 ? 1 : 2;
    T es = E[G.id(0, x, y, z)] + E[G.id(0, x + o[0], y + o[1], z + o[2])];
    T ph[2];
    const int bb[2] = {b1, b2};
    for (int q = 0; q < 2; q++) {
        int b = bb[q];
        int e[3] = {0, 0, 0};
        e[b] = 1;
        T n = B[G.id(b, x + o[0], y + o[1], z + o[2])] - B[G.id(b, x, y, z)];
        T tr = (B[G.id(a, x + o[0] + e[0], y + o[1] + e[1], z + o[2] + e[2])] + B[G.id(a, x + e[0], y + e[1], z + e[2])]) -
               (B[G.id(a, x + o[0] - e[0], y + o[1] - e[1], z + o[2] - e[2])] + B[G.id(a, x - e[0], y - e[1], z - e[2])]);
        ph[q] = es * (T(0.25) * tr - n);
    }
    phi1 = ph[0];
    phi2 = ph[1];
}

template <typename T>
__device__ __forceinline__ void lex_div(const LexGrid<T> &G, const T *B, const T *E, int x, int y, int z, T dv[3]) {
    T xl1, xl2, xh1, xh2, yl1, yl2, yh1, yh2, zl1, zl2, zh1, zh2;
    lex_face(G, B, E, x - 1, y, z, 0, xl1, xl2);
    lex_face(G, B, E, x, y, z, 0, xh1, xh2);
    lex_face(G, B, E, x, y - 1, z, 1, yl1, yl2);
    lex_face(G, B, E, x, y, z, 1, yh1, yh2);
    lex_face(G, B, E, x, y, z - 1, 2, zl1, zl2);
    lex_face(G, B, E, x, y, z, 2, zh1, zh2);
    dv[0] = (yh1 - yl1) + (zh1 - zl1);
    dv[1] = (xh1 - xl1) + (zh2 - zl2);
    dv[2] = (xh2 - xl2) + (yh2 - yl2);
}

// The V-cycle over the coarsest grids in one launch: a cluster of CS thread blocks per instance.
// A grid of more than tail_divide cells is divided over the cluster in z-planes: every block keeps the
// grid's arrays at full size in its own shared memory but holds only its planes and the ones beside
// them, and writes its new values into the neighbours' copies through distributed shared memory, so
// that every read of a pass is a local one and a pass costs two cluster barriers.  Smaller grids are
// stepped by every block for itself, without any exchange, and the coarsest one with its stencil
// coefficients in registers.  What bounds these grids is latency and one SM's arithmetic (float64
// above all: 1.7 operations per clock and SM, a quarter of that for one warp scheduler), not bytes.
// Measured against one thread block per instance (which float32 had in shared memory, float64 in
// global memory): float32 16^3 .. 2^3, V(1,0), 2 coarsest sweeps, 46 -> 29 us; float64 below 32^3, V(2,2), 16
// coarsest sweeps, 470 -> 140 us (with the launches for 16^3 and 8^3 that it takes in); steps: 32^3
// float64 4.63 -> 2.35 ms, half-refined box 10.2 -> 7.9, 64^3 mixed 1.75 -> 1.63.
template <typename T>
struct LexAcc {
    const T *fB, *fE;
    int n;                    // cells of the grid (component stride)
    int xo[3], yo[3], zo[3];  // offsets of the cells at -1, 0, +1 along x, y, z (wrapped)
    template <int C, int DX, int DY, int DZ>
    __device__ __forceinline__ T B() const {
        return fB[C * n + zo[DZ + 1] + yo[DY + 1] + xo[DX + 1]];
    }
    template <int DX, int DY, int DZ>
    __device__ __forceinline__ T E() const {
        return fE[zo[DZ + 1] + yo[DY + 1] + xo[DX + 1]];
    }
};

struct LexDims {
    int nx, ny, nz;
    int lx, ly;  // log2 of nx, ny when every extent is a power of two (p2)
    bool p2;
    __device__ __forceinline__ int n() const { return nx * ny * nz; }
    __device__ __forceinline__ int id(int x, int y, int z) const { return (z * ny + y) * nx + x; }
    __device__ __forceinline__ void cell(int q, int &x, int &y, int &z) const {
        if (p2) {
            x = q & (nx - 1);
            y = (q >> lx) & (ny - 1);
            z = q >> (lx + ly);
        } else {
            const int t = q / nx;
            x = q - t * nx;
            z = t / ny;
            y = t - z * ny;
        }
    }
    // the slots of a colour's cells: (nx + 1) / 2 per row; x may come out as nx on odd extents (no cell)
    __host__ __device__ __forceinline__ int slots() const { return ((nx + 1) >> 1) * ny * nz; }
    __device__ __forceinline__ void colour_cell(int i, int colour, int &x, int &y, int &z) const {
        int h;
        if (p2 && nx > 1) {
            h = i & ((nx >> 1) - 1);
            y = (i >> (lx - 1)) & (ny - 1);
            z = i >> (lx - 1 + ly);
        } else {
            const int hx = (nx + 1) >> 1, t = i / hx;
            h = i - t * hx;
            z = t / ny;
            y = t - z * ny;
        }
        x = 2 * h + ((y + z + colour) & 1);
    }
    template <typename T>
    __device__ __forceinline__ LexAcc<T> acc(const T *B, const T *E, int x, int y, int z) const {
        LexAcc<T> a;
        a.fB = B;
        a.fE = E;
        a.n = n();
        const int pl = nx * ny;
        a.xo[0] = x > 0 ? x - 1 : nx - 1;
        a.xo[1] = x;
        a.xo[2] = x + 1 < nx ? x + 1 : 0;
        a.yo[0] = (y > 0 ? y - 1 : ny - 1) * nx;
        a.yo[1] = y * nx;
        a.yo[2] = (y + 1 < ny ? y + 1 : 0) * nx;
        a.zo[0] = (z > 0 ? z - 1 : nz - 1) * pl;
        a.zo[1] = z * pl;
        a.zo[2] = (z + 1 < nz ? z + 1 : 0) * pl;
        return a;
    }
};

constexpr int TAIL_LUT = 64;                  // blocks of the blocked grids of a tail, all together
constexpr size_t TAIL_SMEM_MAX = 220 * 1024;
// Grids of more cells are divided over the cluster: a pass over fewer takes one block less than the barriers
// of the division.  us of the whole solver with the line at 8 / 64 / 512 / 4096 cells, one instance.  float64, V(2,2), 16
// coarsest sweeps: from 8^3 91 / 70 / 98 / 98, from 12^3 228 / 105 / 111 / 261, from 16^3 146 / 125 / 158 / 522, from
// 10^3 (on 5^3, 125 cells) 185 / 185 / 154 / 230.  float32, V(1,1), 4 coarsest sweeps: from 8^3 37 / 31 / 24 / 24, from 12^3 48 / 41 /
// 36 / 40, from 16^3 49 / 43 / 39 / 57, from 20^3 68 / 68 / 60 / 60.
template <typename T>
constexpr int tail_divide() {
    return sizeof(T) == 8 ? 64 : 512;
}
// Threads: 512, and 1024 for an instance on one thread block in float32 whose first grid is large enough
// for 32 warps.  Two blocks of 512 share an SM there, so that a batch of up to 304 small instances
// (e.g. 200 boxes of 16^3) is one wave.  us with 512 / 1024 threads, V(1,1), 4 coarsest sweeps: 8^3 and below 24 / 26 for 100
// instances, 28 / 49 for 200; from 12^3 53 / 51 and 59 / 88; from 16^3 74 / 69 and 135 / 124; from 20^3 123 / 106 for 100.
constexpr int TAIL_WIDE_CELLS = 1024;
// coarsest grids of at most this many cells per colour keep their coefficients in registers (six
// threads per cell: components x the two axes of each)
constexpr int TAIL_REG_SLOTS = 18;

template <typename T>
struct TailP {  // no default member initialisers: the kernel keeps a __shared__ copy
    int n;
    T om1;                        // 1 - omega
    // The axes of the arrays in shared memory: axis k is the grids' axis axes[k], component k the field's
    // component axes[k] (the operator is the same under a relabelling of both), so that the planes that
    // the cluster divides lie along the longest extent.  float32 keeps the order (its sums would round
    // otherwise, and the mixed path's results move by up to the step's tolerance).
    int axes[3];
    int gx[MAX_SMALL], gy[MAX_SMALL];  // cells of the grid along its own x and y
    LexDims d[MAX_SMALL];
    int oe[MAX_SMALL], oE[MAX_SMALL], orr[MAX_SMALL], oi[MAX_SMALL];  // element offsets in shared memory: e[3n],
                                  // eta[n], r (first grid, divided: the own cells by colour, else [3n]) and, in
                                  // float64, the own cells' inverse diagonals by colour
    bool own;                     // the own cells' values are kept (else read from global memory in each pass)
    int ot;                       // new values of one pass
    int hz[MAX_SMALL];            // divided grids: planes per block (1, or even where the grid is restricted)
    int lut[MAX_SMALL], nbx[MAX_SMALL], nby[MAX_SMALL], nblk[MAX_SMALL];  // blocked grids: table offset, blocks
    bool divided[MAX_SMALL], blocked[MAX_SMALL];
    RbK<T> K[MAX_SMALL];
    const T *inv[MAX_SMALL], *eta[MAX_SMALL];
    const int *origin[MAX_SMALL];
    const T *r0;
    T *e0;
    const uint8_t *imask;
};

template <int CS>
__device__ __forceinline__ void tail_sync(bool cluster) {
    if (CS > 1 && cluster)
        cooperative_groups::this_cluster().sync();
    else
        __syncthreads();
}
template <int CS>
__device__ __forceinline__ int tail_rank() {
    return CS > 1 ? (int)cooperative_groups::this_cluster().block_rank() : 0;
}

// stores v at element offset o of the shared memory of every block of the cluster (or only here)
template <int CS, typename T>
__device__ __forceinline__ void tail_store_all(T *sh, int o, T v, bool cluster) {
    if (CS > 1 && cluster) {
        auto cl = cooperative_groups::this_cluster();
#pragma unroll
        for (int k = 0; k < CS; k++) cl.map_shared_rank(sh, k)[o] = v;
    } else {
        sh[o] = v;
    }
}

// stores the three components of a cell of plane z of grid s (offsets o, o + n, o + 2 n) here and in
// the blocks that read that plane: the owners of the planes within `reach` of it (1 where blocks own
// whole octets, 2 where a block owns one plane and reads its octet's other one)
template <int CS, typename T>
__device__ __forceinline__ void tail_store_cell(const TailP<T> &P, T *sh, int s, int z, int o, int n, const T v[3], int rank) {
#pragma unroll
    for (int c = 0; c < 3; c++) sh[o + c * n] = v[c];
    if (CS > 1 && P.divided[s]) {
        auto cl = cooperative_groups::this_cluster();
        const int hz = P.hz[s], nz = P.d[s].nz, reach = hz == 1 ? 2 : 1;
        int last = rank;
        for (int dz = -reach; dz <= reach; dz++) {
            int zz = z + dz;
            zz = zz < 0 ? zz + nz : (zz >= nz ? zz - nz : zz);
            const int k = zz / hz;
            if (k == rank || k == last) continue;
            last = k;
            T *rem = cl.map_shared_rank(sh, k);
#pragma unroll
            for (int c = 0; c < 3; c++) rem[o + c * n] = v[c];
        }
    }
}

// index in global memory of cell (u, v, w) of grid s (axes of shared memory): component stride cst for
// ncomp components
template <typename T>
__device__ __forceinline__ size_t tail_gidx(const TailP<T> &P, const int *lut, int s, int u, int v, int w, int ncomp, int &cst) {
    int x = u, y = v, z = w;
    if constexpr (sizeof(T) == 8) {
        x = P.axes[0] == 0 ? u : (P.axes[1] == 0 ? v : w);
        y = P.axes[0] == 1 ? u : (P.axes[1] == 1 ? v : w);
        z = P.axes[0] == 2 ? u : (P.axes[1] == 2 ? v : w);
    }
    if (P.blocked[s]) {
        const int b = lut[P.lut[s] + ((z >> 3) * P.nby[s] + (y >> 3)) * P.nbx[s] + (x >> 3)];
        cst = B3;
        return (size_t)b * ncomp * B3 + ((z & 7) * 8 + (y & 7)) * 8 + (x & 7);
    }
    cst = P.d[s].n();
    if constexpr (sizeof(T) == 4) return P.d[s].id(x, y, z);
    return ((size_t)z * P.gy[s] + y) * P.gx[s] + x;
}
// the field's component of component c in shared memory
template <typename T>
__device__ __forceinline__ int tail_comp(const TailP<T> &P, int c) {
    return sizeof(T) == 8 ? P.axes[c] : c;
}

// the planes of grid s that this block owns
template <int CS, typename T>
__device__ __forceinline__ void tail_planes(const TailP<T> &P, int s, int rank, int &z0, int &z1) {
    const int nz = P.d[s].nz;
    if (CS > 1 && P.divided[s]) {
        z0 = min(nz, rank * P.hz[s]);
        z1 = min(nz, z0 + P.hz[s]);
    } else {
        z0 = 0;
        z1 = nz;
    }
}

// the off-diagonal part of -2 h^2 divF of component C through its two faces along AX in float64, added
// to acc: es_lo (B_lo + T_lo / 4) + es_hi (B_hi - T_hi / 4) (k_smooth_d's form, the tangential
// differences formed per cell)
template <int AX, int C, class A>
__device__ __forceinline__ double offdiag_pair(const A &a, double acc) {
    constexpr int AXX = AX == 0, AXY = AX == 1, AXZ = AX == 2;
    constexpr int CX = C == 0, CY = C == 1, CZ = C == 2;
    const double e0 = a.template E<0, 0, 0>();
    const double d0 = a.template B<AX, CX, CY, CZ>() - a.template B<AX, -CX, -CY, -CZ>();
    const double dp = a.template B<AX, AXX + CX, AXY + CY, AXZ + CZ>() - a.template B<AX, AXX - CX, AXY - CY, AXZ - CZ>();
    const double dm = a.template B<AX, CX - AXX, CY - AXY, CZ - AXZ>() - a.template B<AX, -CX - AXX, -CY - AXY, -CZ - AXZ>();
    acc = fma(a.template E<-AXX, -AXY, -AXZ>() + e0, fma(0.25, d0 + dm, a.template B<C, -AXX, -AXY, -AXZ>()), acc);
    return fma(a.template E<AXX, AXY, AXZ>() + e0, fma(-0.25, dp + d0, a.template B<C, AXX, AXY, AXZ>()), acc);
}
// new value of component C of a cell in float64; zero: e = 0 everywhere (only r matters)
template <int C, class A>
__device__ __forceinline__ double tail_update_d(const A &a, double coef, double om1, double r, double inv, bool zero) {
    constexpr int A1 = C == 0 ? 1 : 0, A2 = C == 2 ? 1 : 2;
    const double acc = zero ? 0.0 : offdiag_pair<A2, C>(a, offdiag_pair<A1, C>(a, 0.0));
    return fma(inv, fma(coef, acc, r), om1 * a.template B<C, 0, 0, 0>());
}
// new values of a cell in float32 (the point update of the fused sweeps)
__device__ __forceinline__ void tail_update_f(const LexAcc<float> &a, const RbK<float> &K, const float rr[3], bool zero, float out[3]) {
    float es[6], den[3], dv[3] = {0.f, 0.f, 0.f};
    rb_faces_den<float>(a, K, es, den);
    if (!zero) cell_divergence<float>(a, es, dv);
    const float ev[3] = {a.template B<0, 0, 0, 0>(), a.template B<1, 0, 0, 0>(), a.template B<2, 0, 0, 0>()};
#pragma unroll
    for (int c = 0; c < 3; c++) out[c] = v_add(ev[c], rb_relax(0.f, v_mad(K.ncoef, dv[c], v_sub(rr[c], ev[c])), den[c]));
}

// one colour pass of grid s (Jacobi within the colour: every new value is formed before any is stored).
// float64 takes a thread per cell and component: its arithmetic is spread over the four schedulers of
// the SM, each of which has a quarter of the float64 rate.
template <typename T, int CS, int NT>
__device__ __forceinline__ void tail_colour(const TailP<T> &P, T *sh, const int *lut, size_t inst3, int s, int colour, bool zero) {
    const LexDims D = P.d[s];
    const int n = D.n(), row = D.slots() / D.nz, rank = tail_rank<CS>();
    const bool dv = P.divided[s];
    int z0, z1;
    tail_planes<CS>(P, s, rank, z0, z1);
    const int lo = z0 * row, own = (z1 - z0) * row;
    const T *e = sh + P.oe[s], *E = sh + P.oE[s];
    T *t = sh + P.ot;
    constexpr int NC = sizeof(T) == 8 ? 3 : 1;
    for (int i = threadIdx.x; i < NC * own; i += NT) {
        const int cc = NC == 1 ? 0 : i / own, il = i - cc * own;
        int x, y, z;
        D.colour_cell(lo + il, colour, x, y, z);
        if (x >= D.nx) continue;
        const int q = D.id(x, y, z), o = 3 * colour * own + il;
        size_t id = 0;
        int cst = 0;
        if (!P.own) id = inst3 * n + tail_gidx(P, lut, s, x, y, z, 3, cst);
        auto rhs = [&](int c) { return s > 0 || (P.own && !dv) ? sh[P.orr[s] + c * n + q] : (P.own ? sh[P.orr[0] + o + c * own] : P.r0[id + (size_t)tail_comp(P, c) * cst]); };
        const LexAcc<T> acc = D.acc(e, E, x, y, z);
        if constexpr (sizeof(T) == 8) {
            const double rv = rhs(cc), iv = P.own ? sh[P.oi[s] + o + cc * own] : P.inv[s][id + (size_t)tail_comp(P, cc) * cst];
            const double coef = -P.K[s].ncoef;
            t[cc * own + il] = cc == 0 ? tail_update_d<0>(acc, coef, P.om1, rv, iv, zero)
                                       : (cc == 1 ? tail_update_d<1>(acc, coef, P.om1, rv, iv, zero)
                                                  : tail_update_d<2>(acc, coef, P.om1, rv, iv, zero));
        } else {
            const T rr[3] = {rhs(0), rhs(1), rhs(2)};
            T out[3];
            tail_update_f(acc, P.K[s], rr, zero, out);
#pragma unroll
            for (int c = 0; c < 3; c++) t[c * own + il] = out[c];
        }
    }
    tail_sync<CS>(dv);
    for (int il = threadIdx.x; il < own; il += NT) {
        int x, y, z;
        D.colour_cell(lo + il, colour, x, y, z);
        if (x >= D.nx) continue;
        const T v[3] = {t[il], t[own + il], t[2 * own + il]};
        tail_store_cell<CS>(P, sh, s, z, P.oe[s] + D.id(x, y, z), n, v, rank);
    }
    tail_sync<CS>(dv);
}

template <typename T, int CS, int NT>
__device__ __forceinline__ void tail_sweeps(const TailP<T> &P, T *sh, const int *lut, size_t inst3, int s, int nsweep, bool zero) {
    for (int k = 0; k < nsweep; k++) {
        tail_colour<T, CS, NT>(P, sh, lut, inst3, s, 0, zero && k == 0);
        tail_colour<T, CS, NT>(P, sh, lut, inst3, s, 1, false);
    }
}

// float64 sweeps of a coarsest grid of at most TAIL_REG_SLOTS cells per colour: a colour update is linear
// in e with fixed coefficients, e_c <- (1 - omega) e_c + inv r + sum_k w_k e_k over 16 neighbour values
// (8 through each axis' two faces), so a thread keeps the 8 weights and offsets of one (cell,
// component, axis) for each colour in registers and a pass is 8 multiply-adds, one exchange between
// the two lanes of a component and one barrier pair (warp-wide when 32 threads hold the grid: 2^3).
__device__ __forceinline__ void tail_coarsest(const TailP<double> &P, double *sh, const int *lut, size_t inst3, int s, int nsweep) {
    const LexDims D = P.d[s];
    const int n = D.n(), slots = D.slots(), nthr = 6 * slots;
    double *e = sh + P.oe[s];
    const double *E = sh + P.oE[s];
    const bool one_warp = nthr <= 32;
    if (threadIdx.x < (one_warp ? 32 : 128)) {
        double w[2][8], base[2];
        int off[2][8], oc[2];
        const int half = threadIdx.x & 1, c = (threadIdx.x >> 1) % 3, il = threadIdx.x / 6;
        const int ax = c == 0 ? 1 + half : (c == 1 ? 2 * half : half);
#pragma unroll
        for (int colour = 0; colour < 2; colour++) {
            int x = 0, y = 0, z = 0;
            if (il < slots) D.colour_cell(il, colour, x, y, z);
            const bool live = il < slots && x < D.nx;
            if (!live) x = y = z = 0;
            const int q = D.id(x, y, z);
            const LexAcc<double> a = D.acc(e, E, x, y, z);
            // offsets of the cells at +-1 along ax, along c and along both
            auto at = [&](int da, int dc) {
                int dx = 1 + (ax == 0 ? da : 0) + (c == 0 ? dc : 0), dy = 1 + (ax == 1 ? da : 0) + (c == 1 ? dc : 0),
                    dz = 1 + (ax == 2 ? da : 0) + (c == 2 ? dc : 0);
                const int px = dx == 0 ? a.xo[0] : (dx == 1 ? a.xo[1] : a.xo[2]);
                const int py = dy == 0 ? a.yo[0] : (dy == 1 ? a.yo[1] : a.yo[2]);
                const int pz = dz == 0 ? a.zo[0] : (dz == 1 ? a.zo[1] : a.zo[2]);
                return px + py + pz;
            };
            const double es_lo = E[q] + E[at(-1, 0)], es_hi = E[q] + E[at(1, 0)];
            int cst;
            const size_t id = inst3 * n + tail_gidx(P, lut, s, x, y, z, 3, cst) + (size_t)tail_comp(P, c) * cst;
            const double rv = s == 0 ? P.r0[id] : sh[P.orr[s] + c * n + q];
            const double inv = P.inv[s][id];
            const double k_lo = -P.K[s].ncoef * es_lo * inv, k_hi = -P.K[s].ncoef * es_hi * inv;
            const double m_lo = 0.25 * k_lo, m_hi = 0.25 * k_hi, m_0 = m_lo - m_hi;
            w[colour][0] = k_lo; off[colour][0] = c * n + at(-1, 0);
            w[colour][1] = k_hi; off[colour][1] = c * n + at(1, 0);
            w[colour][2] = m_0; off[colour][2] = ax * n + at(0, 1);
            w[colour][3] = -m_0; off[colour][3] = ax * n + at(0, -1);
            w[colour][4] = m_lo; off[colour][4] = ax * n + at(-1, 1);
            w[colour][5] = -m_lo; off[colour][5] = ax * n + at(-1, -1);
            w[colour][6] = -m_hi; off[colour][6] = ax * n + at(1, 1);
            w[colour][7] = m_hi; off[colour][7] = ax * n + at(1, -1);
            base[colour] = inv * rv;
            oc[colour] = live ? c * n + q : -1;
        }
        for (int k = 0; k < nsweep; k++) {
#pragma unroll
            for (int colour = 0; colour < 2; colour++) {
                double v = half == 0 && oc[colour] >= 0 ? P.om1 * e[oc[colour]] + base[colour] : 0.0, u = 0.0;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    v += w[colour][j] * e[off[colour][j]];
                    u += w[colour][4 + j] * e[off[colour][4 + j]];
                }
                v += u;
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                if (one_warp)
                    __syncwarp();
                else
                    asm volatile("bar.sync 1, 128;" ::: "memory");  // the four warps of this branch
                if (half == 0 && oc[colour] >= 0) e[oc[colour]] = v;
                if (one_warp)
                    __syncwarp();
                else
                    asm volatile("bar.sync 1, 128;" ::: "memory");
            }
        }
    }
    __syncthreads();
}

// Contribution of one outer face of an octet's cell (octet_face's terms): along axis a at offset os
// from the cell at o0, component strides and the +-1 offsets of component c in the cell's own plane
// (p, m) and in the face neighbour's (ps, ms); qs = +-1/4
template <typename T>
__device__ __forceinline__ T tail_face(const T *Ba, const T *Bc, int o0, int os, int p, int m, int ps, int ms, T qs, T es) {
    const T d0 = v_sub(Ba[p], Ba[m]), dn = v_sub(Ba[ps], Ba[ms]);
    return v_mul(es, v_mad(v_add(dn, d0), qs, v_sub(Bc[o0], Bc[os])));
}

template <typename T, int CS, int NT>
__global__ void __launch_bounds__(NT, CS == 1 && sizeof(T) == 4 && NT == 512 ? 2 : 1) k_tail(const __grid_constant__ TailP<T> P_arg, int nu1, int nu2, int nc) {
    const int inst = blockIdx.x / CS;
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *sh = reinterpret_cast<T *>(smem_raw);
    __shared__ TailP<T> P;  // indexed by grid below: kernel parameters are only read at fixed indices
    __shared__ int lut[TAIL_LUT];
    static_assert(sizeof(TailP<T>) % sizeof(int) == 0, "copied as ints");
    for (int q = threadIdx.x; q < (int)(sizeof(TailP<T>) / sizeof(int)); q += NT)
        reinterpret_cast<int *>(&P)[q] = reinterpret_cast<const int *>(&P_arg)[q];
    __syncthreads();
    bool any = false;
    for (int s = 0; s < P.n; s++) {
        if (!P.blocked[s]) continue;
        any = true;
        for (int b = threadIdx.x; b < P.nblk[s]; b += NT) {
            const int *o = P.origin[s] + 3 * b;
            lut[P.lut[s] + (o[2] * P.nby[s] + o[1]) * P.nbx[s] + o[0]] = b;
        }
    }
    pdl_wait();
    if (P.imask && !P.imask[inst]) return;  // the whole cluster
    if (any) __syncthreads();
    const int rank = tail_rank<CS>();
    // eta of every grid (divided ones: the planes read here), e = 0 on the first; the own cells' r
    // (first grid) and inverse diagonals (float64)
    for (int s = 0; s < P.n; s++) {
        const LexDims D = P.d[s];
        const int n = D.n(), pl = D.nx * D.ny;
        const T *eta = P.eta[s] + (size_t)inst * n;
        int z0, z1;
        tail_planes<CS>(P, s, rank, z0, z1);
        const bool part = CS > 1 && P.divided[s] && z1 - z0 + 4 < D.nz;
        const int za = part ? z0 - 2 : 0, np = z0 < z1 ? (part ? z1 - z0 + 4 : D.nz) : 0;
        const bool same = sizeof(T) == 4 || (P.axes[0] == 0 && P.axes[1] == 1);  // the order of the grid's axes
        if (!part && !P.blocked[s] && same) {
            for (int q = threadIdx.x; q < np * pl; q += NT) sh[P.oE[s] + q] = eta[q];
        } else
#pragma unroll 4
        for (int q = threadIdx.x; q < np * pl; q += NT) {
            int x, y, z, cst;
            D.cell(q, x, y, z);
            z += za;
            z = z < 0 ? z + D.nz : (z >= D.nz ? z - D.nz : z);
            sh[P.oE[s] + D.id(x, y, z)] = eta[tail_gidx(P, lut, s, x, y, z, 1, cst)];
        }
        if (s == 0)
            for (int q = threadIdx.x; q < 3 * n; q += NT) sh[P.oe[0] + q] = T(0);
        if (!P.own || (s > 0 && sizeof(T) == 4)) continue;
        const bool full = s == 0 && !P.divided[0];  // r as it lies
        if (full && !P.blocked[0] && same) {
            const T *r0 = P.r0 + (size_t)inst * 3 * n;
            for (int q = threadIdx.x; q < 3 * n; q += NT) sh[P.orr[0] + q] = r0[q];
            if (sizeof(T) == 4) continue;
        }
        const int row = D.slots() / D.nz, lo = z0 * row, own = (z1 - z0) * row;
        for (int colour = 0; colour < 2; colour++)
#pragma unroll 2
            for (int i = threadIdx.x; i < own; i += NT) {
                int x, y, z, cst;
                D.colour_cell(lo + i, colour, x, y, z);
                if (x >= D.nx) continue;
                const size_t id = (size_t)inst * 3 * n + tail_gidx(P, lut, s, x, y, z, 3, cst);
                const int o = 3 * colour * own + i;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    if (s == 0 && !full) sh[P.orr[0] + o + c * own] = P.r0[id + (size_t)tail_comp(P, c) * cst];
                    if (full && (P.blocked[0] || !same)) sh[P.orr[0] + c * n + D.id(x, y, z)] = P.r0[id + (size_t)tail_comp(P, c) * cst];
                    if (sizeof(T) == 8) sh[P.oi[s] + o + c * own] = P.inv[s][id + (size_t)tail_comp(P, c) * cst];
                }
            }
    }
    tail_sync<CS>(true);  // every block of the cluster runs before its shared memory is written
    const size_t inst3 = 3 * (size_t)inst;
    int s = 0;
    for (; s < P.n - 1; s++) {
        tail_sweeps<T, CS, NT>(P, sh, lut, inst3, s, nu1, true);
        // residual and its restriction, 8 lanes per coarse cell: in float64 each with the three outer
        // faces of its child (k_pair_op's octet form: the fluxes between the children cancel in their
        // sum).  A block takes the coarse cells of its planes, or half of a coarse plane where it owns
        // one fine plane.
        const LexDims D = P.d[s], C = P.d[s + 1];
        const int n = D.n(), ncs = C.n(), cpl = C.nx * C.ny;
        const bool dv = P.divided[s];
        const T *e = sh + P.oe[s], *E = sh + P.oE[s];
        for (int q = threadIdx.x; q < 3 * ncs; q += NT) sh[P.oe[s + 1] + q] = T(0);
        int z0, z1, lo, hi;
        tail_planes<CS>(P, s, rank, z0, z1);
        if (z1 - z0 == 1) {
            const int mid = (z0 >> 1) * cpl + cpl / 2;
            lo = (z0 & 1) ? mid : (z0 >> 1) * cpl;
            hi = (z0 & 1) ? ((z0 >> 1) + 1) * cpl : mid;
        } else {
            lo = (z0 >> 1) * cpl;
            hi = (z1 >> 1) * cpl;
        }
        for (int w0 = 8 * lo + (threadIdx.x & ~31); w0 < 8 * hi; w0 += NT) {
            const int w = min(w0 + (int)(threadIdx.x & 31), 8 * hi - 1);  // the tail lanes repeat the last child
            const int cq = w >> 3, ch = w & 7;
            int x, y, z, cst;
            C.cell(cq, x, y, z);
            x = 2 * x + (ch & 1);
            y = 2 * y + ((ch >> 1) & 1);
            z = 2 * z + (ch >> 2);
            const int q = D.id(x, y, z);
            const LexAcc<T> a = D.acc(e, E, x, y, z);
            T o[3];
            if constexpr (sizeof(T) == 8) {
                const int X = a.xo[1], Y = a.yo[1], Z = a.zo[1];
                const int xs = (x & 1) ? a.xo[2] : a.xo[0], ys = (y & 1) ? a.yo[2] : a.yo[0], zs = (z & 1) ? a.zo[2] : a.zo[0];
                const T qx = (x & 1) ? T(0.25) : T(-0.25), qy = (y & 1) ? T(0.25) : T(-0.25), qz = (z & 1) ? T(0.25) : T(-0.25);
                const T eta0 = E[q];
                const T esx = v_add(eta0, E[Z + Y + xs]), esy = v_add(eta0, E[Z + ys + X]), esz = v_add(eta0, E[zs + Y + X]);
                const T *Bx = e, *By = e + n, *Bz = e + 2 * n;
                o[0] = v_add(tail_face(By, Bx, q, Z + ys + X, Z + Y + a.xo[2], Z + Y + a.xo[0], Z + ys + a.xo[2], Z + ys + a.xo[0], qy, esy),
                             tail_face(Bz, Bx, q, zs + Y + X, Z + Y + a.xo[2], Z + Y + a.xo[0], zs + Y + a.xo[2], zs + Y + a.xo[0], qz, esz));
                o[1] = v_add(tail_face(Bx, By, q, Z + Y + xs, Z + a.yo[2] + X, Z + a.yo[0] + X, Z + a.yo[2] + xs, Z + a.yo[0] + xs, qx, esx),
                             tail_face(Bz, By, q, zs + Y + X, Z + a.yo[2] + X, Z + a.yo[0] + X, zs + a.yo[2] + X, zs + a.yo[0] + X, qz, esz));
                o[2] = v_add(tail_face(Bx, Bz, q, Z + Y + xs, a.zo[2] + Y + X, a.zo[0] + Y + X, a.zo[2] + Y + xs, a.zo[0] + Y + xs, qx, esx),
                             tail_face(By, Bz, q, Z + ys + X, a.zo[2] + Y + X, a.zo[0] + Y + X, a.zo[2] + ys + X, a.zo[0] + ys + X, qy, esy));
            } else {
                T es[6];
                face_sums<T>(a, es);
                cell_divergence<T>(a, es, o);
            }
            size_t id = 0;
            if (s == 0) id = inst3 * n + tail_gidx(P, lut, 0, x, y, z, 3, cst);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const T rv = s == 0 && (dv || !P.own) ? P.r0[id + (size_t)tail_comp(P, c) * cst] : sh[P.orr[s] + c * n + q];
                T v = v_mad(P.K[s].ncoef, o[c], v_sub(rv, e[c * n + q]));
                if constexpr (sizeof(T) == 8) {
                    v = v_add(v, __shfl_xor_sync(0xffffffffu, v, 1));
                    v = v_add(v, __shfl_xor_sync(0xffffffffu, v, 2));
                    v = v_add(v, __shfl_xor_sync(0xffffffffu, v, 4));
                } else {  // the children in memory order
                    const T t = v;
                    v = __shfl_sync(0xffffffffu, t, threadIdx.x & 24);
#pragma unroll
                    for (int k = 1; k < 8; k++) v = v_add(v, __shfl_sync(0xffffffffu, t, (threadIdx.x & 24) + k));
                }
                if (ch == c) tail_store_all<CS>(sh, P.orr[s + 1] + c * ncs + cq, v_mul(v, T(0.125)), dv);
            }
        }
        tail_sync<CS>(dv);
    }
    bool done = false;
    if constexpr (sizeof(T) == 8) {
        if (!P.divided[s] && P.d[s].slots() <= TAIL_REG_SLOTS) {
            tail_coarsest(P, sh, lut, inst3, s, nc);
            done = true;
        }
    }
    if (!done) tail_sweeps<T, CS, NT>(P, sh, lut, inst3, s, nc, true);
    for (s = P.n - 2; s >= 0; s--) {
        const LexDims D = P.d[s], C = P.d[s + 1];
        const int n = D.n(), ncs = C.n(), pl = D.nx * D.ny;
        int z0, z1;
        if (CS > 1 && P.divided[s + 1]) {  // every block reads the coarse correction: hand out the own planes
            const int cpl = C.nx * C.ny;
            tail_planes<CS>(P, s + 1, rank, z0, z1);
            for (int i = threadIdx.x; i < 3 * (z1 - z0) * cpl; i += NT) {
                const int c = i / ((z1 - z0) * cpl), o = P.oe[s + 1] + c * ncs + z0 * cpl + i - c * (z1 - z0) * cpl;
                tail_store_all<CS>(sh, o, sh[o], true);
            }
            tail_sync<CS>(true);
        }
        const T *ec = sh + P.oe[s + 1];
        tail_planes<CS>(P, s, rank, z0, z1);
        for (int i = threadIdx.x; i < (z1 - z0) * pl; i += NT) {  // trilinear prolongation (weights 3/4, 1/4)
            int x, y, z;
            D.cell(z0 * pl + i, x, y, z);
            const int px = x >> 1, py = y >> 1, pz = z >> 1;
            int nx = px + ((x & 1) ? 1 : -1), ny = py + ((y & 1) ? 1 : -1), nz = pz + ((z & 1) ? 1 : -1);  // periodic wrap
            nx = nx < 0 ? nx + C.nx : (nx >= C.nx ? nx - C.nx : nx);
            ny = ny < 0 ? ny + C.ny : (ny >= C.ny ? ny - C.ny : ny);
            nz = nz < 0 ? nz + C.nz : (nz >= C.nz ? nz - C.nz : nz);
            T v[3] = {T(0), T(0), T(0)};
#pragma unroll
            for (int ak = 0; ak < 2; ak++)
#pragma unroll
                for (int aj = 0; aj < 2; aj++)
#pragma unroll
                    for (int ai = 0; ai < 2; ai++) {
                        const T wt = (ai ? T(0.25) : T(0.75)) * (aj ? T(0.25) : T(0.75)) * (ak ? T(0.25) : T(0.75));
                        const int o = C.id(ai ? nx : px, aj ? ny : py, ak ? nz : pz);
#pragma unroll
                        for (int c = 0; c < 3; c++) v[c] = v_mad(wt, ec[c * ncs + o], v[c]);
                    }
            const int o = P.oe[s] + z0 * pl + i;
#pragma unroll
            for (int c = 0; c < 3; c++) v[c] = v_add(sh[o + c * n], v[c]);
            tail_store_cell<CS>(P, sh, s, z, o, n, v, rank);  // no other block reads this cell in the pass
        }
        tail_sync<CS>(P.divided[s]);
        tail_sweeps<T, CS, NT>(P, sh, lut, inst3, s, nu2, false);
    }
    // e of the first grid: the own planes (all of them where one block has the instance)
    const LexDims D = P.d[0];
    const int n = D.n(), pl = D.nx * D.ny;
    int z0, z1;
    tail_planes<CS>(P, 0, rank, z0, z1);
    for (int q = z0 * pl + threadIdx.x; q < z1 * pl; q += NT) {
        int x, y, z, cst;
        D.cell(q, x, y, z);
        const size_t id = inst3 * n + tail_gidx(P, lut, 0, x, y, z, 3, cst);
#pragma unroll
        for (int c = 0; c < 3; c++) P.e0[id + (size_t)tail_comp(P, c) * cst] = sh[P.oe[0] + c * n + q];
    }
}

static int ilog2_exact(int v) {
    int l = 0;
    while ((1 << l) < v) l++;
    return (1 << l) == v ? l : -1;
}

// the solver's table and shared-memory bytes; false when the grids do not fit
template <typename T>
static bool tail_plan(const SmallDev<T> &sm, double lamdt, int cs, bool own, TailP<T> &P, size_t &bytes) {
    P.n = sm.n;
    P.own = own;
    P.om1 = (T)(1.0 - sm.omega);
    P.imask = sm.imask;
    // the longest extent last (ties and float32: the grids' own order)
    int last = 2;
    if (sizeof(T) == 8 && sm.n > 0)
        for (int ax = 1; ax >= 0; ax--)
            if (sm.dims[0][ax] > sm.dims[0][last]) last = ax;
    P.axes[2] = last;
    P.axes[0] = last == 0 ? 1 : 0;
    P.axes[1] = last == 2 ? 1 : 2;
    P.r0 = sm.r[0];
    P.e0 = sm.e[0];
    size_t off = 0, tmax = 0;
    int lut = 0;
    auto take = [&](size_t n) {
        const size_t o = off;
        off = (off + n + 3) & ~(size_t)3;
        return (int)o;
    };
    for (int s = 0; s < sm.n; s++) {
        const int e0 = sm.dims[s][P.axes[0]], e1 = sm.dims[s][P.axes[1]], e2 = sm.dims[s][P.axes[2]];
        const int lx = ilog2_exact(e0), ly = ilog2_exact(e1), lz = ilog2_exact(e2);
        const LexDims d{e0, e1, e2, lx, ly, lx >= 0 && ly >= 0 && lz >= 0};
        P.gx[s] = sm.dims[s][0];
        P.gy[s] = sm.dims[s][1];
        const size_t n = (size_t)d.nx * d.ny * d.nz;
        if (n > 16384) return false;
        P.d[s] = d;
        P.divided[s] = cs > 1 && n > (size_t)tail_divide<T>();
        // planes per block: one, or an even number (whole octets) where the grid is restricted
        P.hz[s] = P.divided[s] ? (d.nz + cs - 1) / cs : d.nz;
        if (P.divided[s] && P.hz[s] > 1) P.hz[s] += P.hz[s] & 1;
        const size_t per = (size_t)(d.slots() / d.nz) * P.hz[s];
        P.oe[s] = take(3 * n);
        P.oE[s] = take(n);
        P.orr[s] = take(s > 0 || (own && !P.divided[s]) ? 3 * n : (own ? 6 * per : 0));
        P.oi[s] = sizeof(T) == 8 && own ? take(6 * per) : 0;
        tmax = std::max(tmax, 3 * per);
        P.K[s] = rb_constants<T>(lamdt, sm.h[s], sm.omega);
        P.inv[s] = sm.inv[s];
        P.eta[s] = sm.eta[s];
        P.blocked[s] = sm.origin[s] != nullptr;
        P.origin[s] = sm.origin[s];
        P.lut[s] = lut;
        P.nbx[s] = sm.dims[s][0] / BS;
        P.nby[s] = sm.dims[s][1] / BS;
        P.nblk[s] = P.blocked[s] ? (int)(n / B3) : 0;
        lut += P.nblk[s];
    }
    P.ot = take(tmax);
    bytes = off * sizeof(T);
    return bytes <= TAIL_SMEM_MAX && lut <= TAIL_LUT;
}

// decided for one thread block per instance, so that an instance takes the same grids (and gives the
// same bits) alone and in any batch
template <typename T>
bool tail_fits(const SmallDev<T> &sm) {
    TailP<T> P;
    size_t bytes = 0;
    return sm.n > 0 && tail_plan(sm, 1.0, 1, false, P, bytes);
}
template bool tail_fits<double>(const SmallDev<double> &);
template bool tail_fits<float>(const SmallDev<float> &);

template <typename T, int CS, int NT>
static void tail_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute at[2], int ninst, size_t bytes, cudaStream_t s) {
    static const bool attr = (cudaFuncSetAttribute(k_tail<T, CS, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TAIL_SMEM_MAX),
                              CS > 8 ? cudaFuncSetAttribute(k_tail<T, CS, NT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : cudaSuccess,
                              true);
    (void)attr;
    cfg = {};
    cfg.gridDim = dim3((unsigned)(ninst * CS));
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = CS;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CS > 1 ? 2 : 1;
    if (sizeof(T) == 8 || capturing(s)) {  // as launch_full
        cfg.attrs = at + 1;
        cfg.numAttrs = CS > 1 ? 1 : 0;
    }
}

template <typename T, int CS, int NT = 512>
static cudaError_t launch_tail_cs(const TailP<T> &P, int ninst, size_t bytes, int nu_pre, int nu_post, int n_coarse,
                                  cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[2];
    tail_config<T, CS, NT>(cfg, at, ninst, bytes, s);
    cudaLaunchKernelEx(&cfg, k_tail<T, CS, NT>, P, nu_pre, nu_post, n_coarse);
    return cudaGetLastError();
}

// clusters of CS of the solver's blocks that the device holds at once (asked once, for the largest shared memory)
template <typename T, int CS>
static int tail_resident() {
    static const int n = [] {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at[2];
        tail_config<T, CS, 512>(cfg, at, 1, TAIL_SMEM_MAX, nullptr);
        int k = 0;
        if (cudaOccupancyMaxActiveClusters(&k, k_tail<T, CS, 512>, &cfg) == cudaSuccess) return k;
        cudaGetLastError();
        return 0;
    }();
    return n;
}

// Cluster size: the largest of which all instances run at once.  float64 goes up to 16 (the largest the
// hardware forms, beyond the portable 8): its passes are bound by the SMs' float64 units.  A cluster
// lies within one GPC, so fewer fit than the SMs would hold: on GB300 7 of 16 thread blocks, 15 of 8, 36 of
// 4, 76 of 2.  One instance more takes a second wave: 16^3 and below, V(2,2), 16 coarsest sweeps in float64
// 125 us on clusters of 16 (8 instances 247), 154 of 8 (16 instances 298), 207 of 4 (37: 399), 329 of 2
// (77: 641), 537 on one block each; V(1,1), 4 coarsest sweeps in float32 39 of 8 (16: 72), 50 of 4 (37: 96), 70 of 2
// (77: 119), 69 on one.
template <typename T>
static int tail_cluster(int ninst) {
    if constexpr (sizeof(T) == 8) {
        if (ninst <= tail_resident<T, 16>()) return 16;
    }
    if (ninst <= tail_resident<T, 8>()) return 8;
    if (ninst <= tail_resident<T, 4>()) return 4;
    return ninst <= tail_resident<T, 2>() ? 2 : 1;
}

template <typename T>
cudaError_t launch_tail(const SmallDev<T> &sm, double lamdt, int nu_pre, int nu_post, int n_coarse, cudaStream_t s) {
    if (sm.n == 0) return cudaSuccess;
    TailP<T> P;
    size_t bytes = 0;
    // (a first grid that is not divided has nothing for a cluster to do)
    const bool divide = (int64_t)sm.dims[0][0] * sm.dims[0][1] * sm.dims[0][2] > tail_divide<T>();
    const int cs = divide ? tail_cluster<T>(sm.ninst) : 1;
    if (!tail_plan(sm, lamdt, cs, true, P, bytes) && !tail_plan(sm, lamdt, cs, false, P, bytes))
        return cudaErrorInvalidValue;  // callers ask tail_fits first
    if constexpr (sizeof(T) == 8) {
        if (cs == 16) return launch_tail_cs<T, 16>(P, sm.ninst, bytes, nu_pre, nu_post, n_coarse, s);
    }
    switch (cs) {
        case 8: return launch_tail_cs<T, 8>(P, sm.ninst, bytes, nu_pre, nu_post, n_coarse, s);
        case 4: return launch_tail_cs<T, 4>(P, sm.ninst, bytes, nu_pre, nu_post, n_coarse, s);
        case 2: return launch_tail_cs<T, 2>(P, sm.ninst, bytes, nu_pre, nu_post, n_coarse, s);
        default: break;
    }
    if constexpr (sizeof(T) == 4) {
        if (P.d[0].slots() > TAIL_WIDE_CELLS / 2) return launch_tail_cs<T, 1, 1024>(P, sm.ninst, bytes, nu_pre, nu_post, n_coarse, s);
    }
    return launch_tail_cs<T, 1>(P, sm.ninst, bytes, nu_pre, nu_post, n_coarse, s);
}
template cudaError_t launch_tail<double>(const SmallDev<double> &, double, int, int, int, cudaStream_t);
template cudaError_t launch_tail<float>(const SmallDev<float> &, double, int, int, int, cudaStream_t);

// Lexicographic grids too large for the cluster solver, stepped by grid-wide launches over
// all instances (thread per instance and cell), one kernel per
// colour pass (e_in -> e_out, the other colour copied), per residual, per restriction and per
// prolongation.
template <typename T>
__device__ __forceinline__ bool lex_cell(const SmallDev<T> &sm, int s, size_t tid, int &q, int &cell) {
    const int n = sm.dims[s][0] * sm.dims[s][1] * sm.dims[s][2];
    if (tid >= (size_t)sm.ninst * n) return false;
    q = (int)(tid / n);
    cell = (int)(tid - (size_t)q * n);
    return !(sm.imask && !sm.imask[q]);
}

template <typename T>
__global__ void __launch_bounds__(256) k_lex_pass(SmallDev<T> sm, int s, double lamdt, int colour, int to_t) {
    pdl_trigger();
    pdl_wait();
    int q, cell;
    if (!lex_cell(sm, s, blockIdx.x * (size_t)blockDim.x + threadIdx.x, q, cell)) return;
    const LexGrid<T> G{sm.dims[s][0], sm.dims[s][1], sm.dims[s][2]};
    const int n = G.nx * G.ny * G.nz;
    const size_t o3 = (size_t)q * 3 * n;
    const T *src = (to_t ? sm.e[s] : sm.t[s]) + o3;
    T *dst = (to_t ? sm.t[s] : sm.e[s]) + o3;
    const int x = cell % G.nx, y = (cell / G.nx) % G.ny, z = cell / (G.nx * G.ny);
    if (((x + y + z) & 1) != colour) {
        for (int c = 0; c < 3; c++) dst[(size_t)c * n + cell] = src[(size_t)c * n + cell];
        return;
    }
    const T coef = (T)(lamdt / (2.0 * sm.h[s] * sm.h[s]));
    const T *r = sm.r[s] + o3, *inv = sm.inv[s] + o3, *E = sm.eta[s] + (size_t)q * n;
    T dv[3];
    lex_div(G, src, E, x, y, z, dv);
    for (int c = 0; c < 3; c++) {
        const size_t id = (size_t)c * n + cell;
        const T d = (r[id] - src[id] - coef * dv[c]) * inv[id];
        dst[id] = src[id] + d;
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_lex_resid(SmallDev<T> sm, int s, double lamdt) {
    pdl_trigger();
    pdl_wait();
    int q, cell;
    if (!lex_cell(sm, s, blockIdx.x * (size_t)blockDim.x + threadIdx.x, q, cell)) return;
    const LexGrid<T> G{sm.dims[s][0], sm.dims[s][1], sm.dims[s][2]};
    const int n = G.nx * G.ny * G.nz;
    const size_t o3 = (size_t)q * 3 * n;
    const T coef = (T)(lamdt / (2.0 * sm.h[s] * sm.h[s]));
    const T *e = sm.e[s] + o3, *r = sm.r[s] + o3, *E = sm.eta[s] + (size_t)q * n;
    T *t = sm.t[s] + o3;
    const int x = cell % G.nx, y = (cell / G.nx) % G.ny, z = cell / (G.nx * G.ny);
    T dv[3];
    lex_div(G, e, E, x, y, z, dv);
    for (int c = 0; c < 3; c++) {
        const size_t id = (size_t)c * n + cell;
        t[id] = r[id] - e[id] - coef * dv[c];
    }
}

// r of grid s + 1 = mean of the 8 children of t on grid s; e of grid s + 1 = 0
template <typename T>
__global__ void __launch_bounds__(256) k_lex_restrict(SmallDev<T> sm, int s) {
    pdl_trigger();
    pdl_wait();
    int q, cell;
    if (!lex_cell(sm, s + 1, blockIdx.x * (size_t)blockDim.x + threadIdx.x, q, cell)) return;
    const LexGrid<T> G{sm.dims[s][0], sm.dims[s][1], sm.dims[s][2]};
    const LexGrid<T> C{sm.dims[s + 1][0], sm.dims[s + 1][1], sm.dims[s + 1][2]};
    const int n = G.nx * G.ny * G.nz, nc_ = C.nx * C.ny * C.nz;
    const T *t = sm.t[s] + (size_t)q * 3 * n;
    const int x = cell % C.nx, y = (cell / C.nx) % C.ny, z = cell / (C.nx * C.ny);
    for (int c = 0; c < 3; c++) {
        T acc = 0;
        for (int dk = 0; dk < 2; dk++)
            for (int dj = 0; dj < 2; dj++)
                for (int di = 0; di < 2; di++) acc += t[G.id(c, 2 * x + di, 2 * y + dj, 2 * z + dk)];
        const size_t id = (size_t)q * 3 * nc_ + (size_t)c * nc_ + cell;
        sm.r[s + 1][id] = acc / T(8);
        sm.e[s + 1][id] = T(0);
    }
}

// e of grid s += trilinear interpolation of e of grid s + 1
template <typename T>
__global__ void __launch_bounds__(256) k_lex_prolong(SmallDev<T> sm, int s) {
    pdl_trigger();
    pdl_wait();
    int q, cell;
    if (!lex_cell(sm, s, blockIdx.x * (size_t)blockDim.x + threadIdx.x, q, cell)) return;
    const LexGrid<T> G{sm.dims[s][0], sm.dims[s][1], sm.dims[s][2]};
    const LexGrid<T> C{sm.dims[s + 1][0], sm.dims[s + 1][1], sm.dims[s + 1][2]};
    const int n = G.nx * G.ny * G.nz, nc_ = C.nx * C.ny * C.nz;
    const T *ec = sm.e[s + 1] + (size_t)q * 3 * nc_;
    T *e = sm.e[s] + (size_t)q * 3 * n;
    const int x = cell % G.nx, y = (cell / G.nx) % G.ny, z = cell / (G.nx * G.ny);
    const int px = x >> 1, py = y >> 1, pz = z >> 1;
    const int sx = (x & 1) ? 1 : -1, sy = (y & 1) ? 1 : -1, sz = (z & 1) ? 1 : -1;
    for (int c = 0; c < 3; c++) {
        T v = 0;
        for (int ak = 0; ak < 2; ak++)
            for (int aj = 0; aj < 2; aj++)
                for (int ai = 0; ai < 2; ai++) {
                    T wt = (ai ? T(0.25) : T(0.75)) * (aj ? T(0.25) : T(0.75)) * (ak ? T(0.25) : T(0.75));
                    v += wt * ec[C.id(c, px + ai * sx, py + aj * sy, pz + ak * sz)];
                }
        e[(size_t)c * n + cell] += v;
    }
}

template <typename T>
static unsigned lex_grid(const SmallDev<T> &sm, int s) {
    const size_t n = (size_t)sm.ninst * sm.dims[s][0] * sm.dims[s][1] * sm.dims[s][2];
    return (unsigned)((n + 255) / 256);
}

template <typename T>
cudaError_t launch_lex_sweeps(const SmallDev<T> &sm, int s, double lamdt, int nsweep, cudaStream_t st) {
    for (int i = 0; i < nsweep; i++) {
        launch_pdl(k_lex_pass<T>, lex_grid(sm, s), 256, 0, st, sm, s, lamdt, 0, 1);  // e -> t: red
        launch_pdl(k_lex_pass<T>, lex_grid(sm, s), 256, 0, st, sm, s, lamdt, 1, 0);  // t -> e: black
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_lex_resid_restrict(const SmallDev<T> &sm, int s, double lamdt, cudaStream_t st) {
    launch_pdl(k_lex_resid<T>, lex_grid(sm, s), 256, 0, st, sm, s, lamdt);
    launch_pdl(k_lex_restrict<T>, lex_grid(sm, s + 1), 256, 0, st, sm, s);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_lex_prolong(const SmallDev<T> &sm, int s, cudaStream_t st) {
    launch_pdl(k_lex_prolong<T>, lex_grid(sm, s), 256, 0, st, sm, s);
    return cudaGetLastError();
}
template cudaError_t launch_lex_sweeps<double>(const SmallDev<double> &, int, double, int, cudaStream_t);
template cudaError_t launch_lex_sweeps<float>(const SmallDev<float> &, int, double, int, cudaStream_t);
template cudaError_t launch_lex_resid_restrict<double>(const SmallDev<double> &, int, double, cudaStream_t);
template cudaError_t launch_lex_resid_restrict<float>(const SmallDev<float> &, int, double, cudaStream_t);
template cudaError_t launch_lex_prolong<double>(const SmallDev<double> &, int, cudaStream_t);
template cudaError_t launch_lex_prolong<float>(const SmallDev<float> &, int, cudaStream_t);

// Setup of the lexicographic grids: eta of each from the grid above it (mean of the 8 children),
// one launch per grid, and the inverse diagonals of all of them in one launch, a thread per
// instance and cell.  Bound by launch latency (the grids hold at most a few 10^5 cells); one
// thread block per instance, which did the whole chain before, was bound by one SM's float64
// units instead (the diagonal is formed in float64): 2421 us per call for the 60 x 52 x 44
// grid below 120 x 104 x 88, about 15 us now (two steps with a new eta each: 15.7 -> 6.05 ms).
template <typename T>
__global__ void __launch_bounds__(128) k_small_eta(SmallDev<T> sm, int s) {
    const size_t tid = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    const LexGrid<T> F{sm.dims[s - 1][0], sm.dims[s - 1][1], sm.dims[s - 1][2]};
    const LexGrid<T> C{sm.dims[s][0], sm.dims[s][1], sm.dims[s][2]};
    const int n = C.nx * C.ny * C.nz;
    if (tid >= (size_t)sm.ninst * n) return;
    const int q = (int)(tid / n), cell = (int)(tid - (size_t)q * n);
    const T *fine = sm.eta[s - 1] + (size_t)q * F.nx * F.ny * F.nz;
    const int x = cell % C.nx, y = (cell / C.nx) % C.ny, z = cell / (C.nx * C.ny);
    T acc = 0;
    for (int dk = 0; dk < 2; dk++)
        for (int dj = 0; dj < 2; dj++)
            for (int di = 0; di < 2; di++) acc += fine[F.id(0, 2 * x + di, 2 * y + dj, 2 * z + dk)];
    sm.eta[s][(size_t)q * n + cell] = acc / T(8);
}

template <typename T>
__global__ void __launch_bounds__(128) k_small_inv(SmallDev<T> sm, double lamdt) {
    size_t tid = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    int s = 0;
    for (; s < sm.n; s++) {  // the grid of this thread
        const size_t all = (size_t)sm.ninst * sm.dims[s][0] * sm.dims[s][1] * sm.dims[s][2];
        if (tid < all) break;
        tid -= all;
    }
    if (s == sm.n) return;
    const LexGrid<T> G{sm.dims[s][0], sm.dims[s][1], sm.dims[s][2]};
    const int n = G.nx * G.ny * G.nz;
    const int q = (int)(tid / n), cell = (int)(tid - (size_t)q * n);
    const int x = cell % G.nx, y = (cell / G.nx) % G.ny, z = cell / (G.nx * G.ny);
    const T *E = sm.eta[s] + (size_t)q * n;
    T *inv = sm.inv[s] + (size_t)q * 3 * n;
    const double lh2 = lamdt / (sm.h[s] * sm.h[s]);
    const double e0 = (double)E[cell];
    const double sa[3] = {0.5 * (e0 + (double)E[G.id(0, x + 1, y, z)]) + 0.5 * (e0 + (double)E[G.id(0, x - 1, y, z)]),
                          0.5 * (e0 + (double)E[G.id(0, x, y + 1, z)]) + 0.5 * (e0 + (double)E[G.id(0, x, y - 1, z)]),
                          0.5 * (e0 + (double)E[G.id(0, x, y, z + 1)]) + 0.5 * (e0 + (double)E[G.id(0, x, y, z - 1)])};
    for (int c = 0; c < 3; c++) {
        double al = 0.0;
        for (int ax = 0; ax < 3; ax++)
            if (ax != c) al += lh2 * sa[ax];
        inv[(size_t)c * n + cell] = (T)(sm.omega / (1.0 + al));
    }
}

template <typename T>
cudaError_t launch_small_eta(const SmallDev<T> &sm, cudaStream_t st) {
    for (int s = 1; s < sm.n; s++) {
        const size_t n = (size_t)sm.ninst * sm.dims[s][0] * sm.dims[s][1] * sm.dims[s][2];
        k_small_eta<T><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(sm, s);
    }
    return cudaGetLastError();
}
template cudaError_t launch_small_eta<double>(const SmallDev<double> &, cudaStream_t);
template cudaError_t launch_small_eta<float>(const SmallDev<float> &, cudaStream_t);

template <typename T>
cudaError_t launch_small_inv(const SmallDev<T> &sm, double lamdt, cudaStream_t st) {
    size_t n = 0;
    for (int s = 0; s < sm.n; s++) n += (size_t)sm.ninst * sm.dims[s][0] * sm.dims[s][1] * sm.dims[s][2];
    if (n == 0) return cudaSuccess;
    k_small_inv<T><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(sm, lamdt);
    return cudaGetLastError();
}
template cudaError_t launch_small_inv<double>(const SmallDev<double> &, double, cudaStream_t);
template cudaError_t launch_small_inv<float>(const SmallDev<float> &, double, cudaStream_t);

}  // namespace ohm
