// sphst_kernels.cuh -- CUDA kernels of the pair-sweep library (sm_103a).
//
// Rebuild (once per advection step, Section 3.3): cell assignment with Morton
// keys, a counting sort over the dense cell table (histogram by atomics,
// exclusive scan, scatter), a per-cell sort by insertion index that makes the
// order canonical, a gather of the particle arrays, the neighbour list of the
// frozen configuration and the interface band.
//
// Pair sweeps (gather-only: every particle's sum is owned by one thread, or by
// a group of 2-8 lanes that split its list, or its cells, and add their parts
// in a fixed order, so there are no atomics on particle data):
//   M  correction matrix B_i (Eq. 15; also over the own fluid for the
//      surface_corr reading)                             once per advection step
//   V  viscous acceleration (Eq. 13) + transport shift (Eq. 14)  once per advection step
//   A  colour gradient (Eq. 22); with the list over the interface band only
//                                                         every acoustic substep
//   S  surface stress + penalty (Eqs. 24, 26, 30, 33) of the interface band
//                                                         every substep (list cases)
//   B  pressure (Eqs. 7-12) (+ the surface terms with the cell walk) + kick
//                                                         every substep
//   C  continuity (Eq. 6) + drift                         every substep
// The list build, the band and M, V, B, C (and A with the cell walk) run
// over the fluid particles only (their ranks after each reorder); A and S of
// the list classes stride over the band list.  Time-step control (Eqs.
// 16-18) runs in FP64 in one-thread-per-case kernels.  A one-case engine
// launches B and C of the list classes with the case's constants in the launch
// parameters (MODE_ONE); their sums are explicitly rounded, so the results do
// not depend on that choice.
#pragma once

#include <cfloat>
#include <type_traits>
#include <utility>

#include <cuda_runtime.h>
#include <math_constants.h>
#include "sphst_internal.cuh"

// Tuning switches of the pair sweeps (compile-time):
//   SPHST_LIST_LDCS    1: read neighbour-list words with evict-first loads so the
//                      streamed list does not push particle data out of L2
//   SPHST_SWEEP_MINB   >0: minimum resident 256-thread blocks per SM for the
//                      sweeps (caps registers per thread)
//   SPHST_SWEEPB_MINB  the same for sweep B alone (default 4: 64 registers)
//   SPHST_SWEEPB_MINB_ONE  the same for the FP32 sweep B of a one-case engine
//                      (default 6: 42 registers, as its per-case constants are
//                      not in registers; 1M particles: 6 250 us, 5 271, 7 279)
//   SPHST_SWEEPAS_MINB the same for sweep A of the cell-walk classes
//   SPHST_LIST_NOALLOC 1: the list words are read without allocating L1 lines
//                      (measured +1% on the 3D drop)
#ifndef SPHST_LIST_LDCS
#define SPHST_LIST_LDCS 1
#endif
#ifndef SPHST_SWEEP_MINB
#define SPHST_SWEEP_MINB 0
#endif
#ifndef SPHST_SWEEPAS_MINB
#define SPHST_SWEEPAS_MINB 4
#endif
#ifndef SPHST_SWEEPB_MINB
#define SPHST_SWEEPB_MINB 4
#endif
#ifndef SPHST_LIST_NOALLOC
#define SPHST_LIST_NOALLOC 1
#endif
#ifndef SPHST_SWEEPB_MINB_ONE
#define SPHST_SWEEPB_MINB_ONE 6
#endif
#if SPHST_SWEEP_MINB > 0
#define SPH_SWEEP_BOUNDS __launch_bounds__(256, SPHST_SWEEP_MINB)
#else
#define SPH_SWEEP_BOUNDS __launch_bounds__(256)
#endif
// sweep B is latency-bound on neighbour gathers: capping it at 64 registers
// (4 blocks of 256 per SM) doubles its resident warps (measured 1.38 -> 0.96
// ms on 1.19M particles); the lighter sweeps A and C are faster uncapped
#if SPHST_SWEEPAS_MINB > 0
#define SPH_SWEEPAS_BOUNDS __launch_bounds__(256, SPHST_SWEEPAS_MINB)
#else
#define SPH_SWEEPAS_BOUNDS __launch_bounds__(256)
#endif
// sweep B of a one-case engine reads its per-case constants from the
// parameter block, which leaves it room for more resident blocks
#define SPH_SWEEPB_BOUNDS_M(T, LIST, L, MODE)                                                          \
    __launch_bounds__(256, (MODE) == 3 || (!(LIST) && (L) > 1) ? 1 : !(LIST) ? 4 : sizeof(T) == 8 ? 2 : (MODE) == 2 ? SPHST_SWEEPB_MINB_ONE                  \
                                                         : (SPHST_SWEEPB_MINB > 0 ? SPHST_SWEEPB_MINB : 1))
// sweep C of a batch with lists (FP32): with the constants in registers the
// compiler left its gathers no room (52 to 55 registers); at 64 (4 blocks per
// SM) a batch of 6M particles takes 582 us per launch in 3D against 719, with
// work lists 585 against 604 (2D 154 against 178; the tiled 2D form is better
// without, 147 against 167).  The two-lane cell walk in 3D (FP32) likewise
// takes what it asks for (76 instead of 58): 30k particles 60.4 us against
// 66.2, 125k 170 against 166.
#define SPH_SWEEPC_BOUNDS_M(T, D, LIST, L, MODE)                                                       \
    __launch_bounds__(256, (LIST) && sizeof(T) == 4 && ((MODE) == 1 || ((MODE) == 0 && (D) == 3)) ? 4                \
                         : !(LIST) && (L) > 1 && sizeof(T) == 4 && (D) == 3 ? 1 : SPHST_SWEEP_MINB)

namespace sphst {

// ------------------------------------------------------------------ helpers
// rho_i + rho_j and its product with rho_j are normal numbers, so the
// flush-to-zero reciprocal gives the same value without the scaling of
// denormal arguments.  So does the root for a normal r^2; for the others (r
// below 1.1e-19, where r_ij is cut off by FP32's range itself) there is rsq_full.
__device__ __forceinline__ float rsq(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsq_full(float x) { return rsqrtf(x); }
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ double rsq(double x) { return rsqrt(x); }
__device__ __forceinline__ double rsq_full(double x) { return rsqrt(x); }

template <typename T> __device__ __forceinline__ V4<T> ld4(const V4<T> *p) { return *p; }
template <> __device__ __forceinline__ V4<float> ld4<float>(const V4<float> *p) {
    float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return V4<float>{v.x, v.y, v.z, v.w};
}

// the same, issued where it stands: a gather that is to be in flight while
// other neighbours are evaluated (a plain load, used behind a branch or in the
// next iteration only, is moved down to its use by the compiler)
__device__ __forceinline__ V4<float> ld4_now(const V4<float> *p) {
    V4<float> v;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ V4<double> ld4_now(const V4<double> *p) {
    V4<double> v;
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2+16];" : "=d"(v.z), "=d"(v.w) : "l"(p));
    return v;
}

// a / b of the pair sums: in FP32 a times the SFU reciprocal (<= 2 ulp, for
// divisors below 2^126, which products of densities are) instead of the IEEE
// sequence; FP64 keeps IEEE division
__device__ __forceinline__ float vdiv(float a, float b) { return __fmul_rn(a, rcp_approx(b)); }
__device__ __forceinline__ double vdiv(double a, double b) { return a / b; }

// b - 1 as a floating-point value for a 2-bit field b (0..2), without an
// integer conversion: the bit pattern 2^23 + b (2^52 + b) is exact and the
// subtraction of 2^23 + 1 (2^52 + 1) is exact too
__device__ __forceinline__ float code_off(uint32_t b, float) {
    return __fsub_rn(__uint_as_float(0x4B000000u | b), 8388609.0f);
}
__device__ __forceinline__ double code_off(uint32_t b, double) {
    return __dsub_rn(__longlong_as_double(0x4330000000000000ll | (long long)b), 4503599627370497.0);
}

// Every operation of the pair sums is explicitly rounded, so a particle's
// sums have the same bits whichever kernel computes them and whatever its
// register allocation.
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }

// a ? x1 : x0 for the two fluid phases' constants (no indexed loads)
template <typename T> __device__ __forceinline__ T sel(uint32_t k, T x0, T x1) { return k ? x1 : x0; }

// A list word of the per-substep walks.  The list is streamed once per sweep
// while the neighbour records it points to are gathered ~80 times; its words
// are read without allocating L1 lines (SPHST_LIST_NOALLOC), so they take none
// from the gathered data (else as evict-first loads).
__device__ __forceinline__ uint32_t ld_list_walk(const uint32_t *p) {
#if SPHST_LIST_NOALLOC
    uint32_t v;
    asm("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
#else
    return __ldcs(p);
#endif
}

__device__ __forceinline__ uint32_t ld_list(const uint32_t *p) {
#if SPHST_LIST_LDCS
    return __ldcs(p);
#else
    return __ldg(p);
#endif
}

__device__ __forceinline__ double bits_to_d(unsigned long long b) { return __longlong_as_double((long long)b); }

// explicitly rounded operations for the pair geometry, so that every test of
// a pair, by the cell walk and by the list build, finds the same r^2
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
template <typename T, int D> __device__ __forceinline__ T norm2(T x, T y, T z) {
    return D == 3 ? fma_rn(x, x, fma_rn(y, y, mul_rn(z, z))) : fma_rn(x, x, mul_rn(y, y));
}

// |v|^2 in FP64 with a fixed operation order and no contraction
template <typename T> __device__ __forceinline__ double speed2(const V4<T> &v, int dim) {
    double x = (double)v.x, y = (double)v.y, z = (double)v.z;
    double s = __dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y));
    if (dim == 3) s = __dadd_rn(s, __dmul_rn(z, z));
    return s;
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    return v;
}

// Eq. 11 dissipation limiter, branch-free: min(max(k dU w, lo), hi) with the
// case's (k, lo, hi) = (3 / c0, 0, 1) for the density reading and the printed
// form, (0, 1, 1) for beta = 1 and (0, 0, 0) for beta = 0; w = 1, or for the
// printed form (P_L + P_R)/(rho_L + rho_R) of the pair
__device__ __forceinline__ float clamp_lh(float x, float lo, float hi) { return fminf(fmaxf(x, lo), hi); }
__device__ __forceinline__ double clamp_lh(double x, double lo, double hi) { return fmin(fmax(x, lo), hi); }
// the no-suction wall reading's floor
__device__ __forceinline__ float vpush(float x) { return x > 0.0f ? x : 0.0f; }
__device__ __forceinline__ double vpush(double x) { return x > 0.0 ? x : 0.0; }

// Neighbour cell index along axis a: wrapped on a periodic axis (the cells
// tile the period exactly, so the cell at -1 is the last one and lies one
// cell width before cell 0); false when it falls off a non-periodic axis.
__device__ __forceinline__ bool wrap_cell(const CaseDesc &d, int a, int &c) {
    if (c >= 0 && c < d.ncell[a]) return true;
    if (!((d.periodic >> a) & 1)) return false;
    c += c < 0 ? d.ncell[a] : -d.ncell[a];
    return true;
}

// First statement of every kernel of a step, which is launched while the one
// before it still runs out (programmatic dependent launch): waits until that
// one has finished and its writes are visible.  Nothing is read or written
// before the wait, so a kernel that has finished had all before it finished.
__device__ __forceinline__ void follow() { cudaGridDependencySynchronize(); }
// In the kernels of one or a few blocks: the next kernel's blocks may take
// their places at once.  Not in the others: blocks placed around a running
// kernel's leave the SMs unevenly filled (in every kernel, FP64 2D 6k
// particles 643 -> 817, 64k 1912 -> 2243 us a pass; in these alone 672 -> 542,
// 1775 -> 1735).
__device__ __forceinline__ void lead() { cudaTriggerProgrammaticLaunchCompletion(); }

// Launches a kernel that starts with follow() behind the kernel before it in
// the stream.  Plain launches against these: 2D 576 particles 319 -> 313 us a pass, FP64 2D 6k 643
// -> 635, shear flow of 37k 499 -> 474, 1M 12.74 -> 12.66 ms.
template <typename... P, typename... A>
void launch_next(void (*kernel)(P...), unsigned grid, dim3 block, size_t shared, cudaStream_t stream, A &&...args) {
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = shared;
    cfg.stream = stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);   // a failure stays for the caller's cudaGetLastError
}

// --------------------------------------------------------------- cell walk
// Calls f(j, snap_j, r_ij vector, r^2) for every j != i with 0 < r_ij < 2h in
// the 3^D cells around i's cell, x fastest, and next() after each cell (once
// for an odd number of cells that are off the grid).  r_ij = s_i - s_j - o cs,
// where o is the neighbour cell's offset, because both offsets are taken from
// their own cell origins.  OTHER: only particles of the other fluid, which is
// asked first (most of the fluid has none around).  Returns true when a
// coincident particle was met.
template <bool OTHER, typename T, int D, typename F, typename N>
__device__ __forceinline__ bool walk(const CaseDesc &d, const CasePhys<T> &cp,
                                     const uint32_t *__restrict__ starts,
                                     const V4<T> *__restrict__ snap, int64_t i,
                                     const V4<T> &si, uint32_t pki, F &&f, N &&next) {
    const int cx = cell_x<D>(pki), cy = cell_y<D>(pki), cz = cell_z<D>(pki);
    const uint32_t toff = (uint32_t)d.table_off, other = phase_of(pki) ^ 1u;
    const T cs = cp.cs, R2 = cp.four_h2;
    bool coincident = false;
    for (int oz = (D == 3 ? -1 : 0); oz <= (D == 3 ? 1 : 0); ++oz) {
        int nz = cz + oz;
        if (D == 3 && !wrap_cell(d, 2, nz)) { next(); continue; }
        const T sz = D == 3 ? sub_rn(si.z, mul_rn(T(oz), cs)) : T(0);
        for (int oy = -1; oy <= 1; ++oy) {
            int ny = cy + oy;
            if (!wrap_cell(d, 1, ny)) { next(); continue; }
            const T sy = sub_rn(si.y, mul_rn(T(oy), cs));
            for (int ox = -1; ox <= 1; ++ox) {
                int nx = cx + ox;
                if (wrap_cell(d, 0, nx)) {
                    const T sx = sub_rn(si.x, mul_rn(T(ox), cs));
                    const uint32_t m = toff + morton<D>(nx, ny, nz);
                    const uint32_t b = __ldg(starts + m), e = __ldg(starts + m + 1);
                    for (uint32_t j = b; j < e; ++j) {
                        const V4<T> sj = ld4(snap + j);
                        const T rx = sub_rn(sx, sj.x), ry = sub_rn(sy, sj.y);
                        const T rz = D == 3 ? sub_rn(sz, sj.z) : T(0);
                        const T r2 = norm2<T, D>(rx, ry, rz);
                        if ((!OTHER || phase_of(w_bits(sj.w)) == other) && r2 < R2 && j != (uint32_t)i) {
                            if (r2 > T(0)) f(j, sj, rx, ry, rz, r2);
                            else coincident = true;
                        }
                    }
                }
                next();
            }
        }
    }
    return coincident;
}
struct Nothing { __device__ __forceinline__ void operator()() const {} };

// Neighbour list of the frozen configuration.  A slot is one fluid particle,
// by its rank among them.  The slot of local number r holds entry k at word
// ((r / 32) K + k) 32 + r % 32 of its case's lists, K the list capacity: a
// warp's 32 slots own one contiguous block of K rows, a row of 32 words is one
// 128-byte line, and consecutive entries are one row apart whatever the case's
// size.  An entry is j << 6 | cell code, the code holding (o + 1) per axis in
// 2 bits, o the neighbour cell's offset.  Each list holds the neighbours of
// the other fluid phase first, then the rest, each part in increasing j;
// cnt[slot] = count | (other-phase count << 16),
// so the colour-gradient sweep reads only the first part.
constexpr uint32_t NBR_SHIFT = 6;
constexpr uint32_t CNT_MASK = 0xffffu;
constexpr int LROW = 32;                        // words between consecutive entries of a list
// first word of the list of global slot q
__device__ __forceinline__ int64_t list_word(const CaseDesc &d, int64_t q) {
    const int64_t r = q - d.f_begin;
    return d.nbr_base + (r >> 5) * ((int64_t)d.nbr_k * LROW) + (r & 31);
}
enum NbrPart { PART_ALL = 0, PART_OTHER = 1 };
template <int D>
__device__ __forceinline__ uint32_t cell_code(int ox, int oy, int oz) {
    return (uint32_t)(ox + 1) | ((uint32_t)(oy + 1) << 2) | (D == 3 ? ((uint32_t)(oz + 1) << 4) : 0u);
}

// r_ij = (s_i - o cs) - s_j of an entry or cell code e (o cs is exact): the
// operations of the cell walk.  Every test of a pair takes them, and the sums
// of the cell walk, so list and walk hold the same pairs.
template <typename T, int D>
__device__ __forceinline__ void pair_offset(uint32_t e, const V4<T> &si, const V4<T> &sj, T cs, T &rx, T &ry, T &rz) {
    rx = sub_rn(fma_rn(-code_off(e & 3u, T()), cs, si.x), sj.x);
    ry = sub_rn(fma_rn(-code_off((e >> 2) & 3u, T()), cs, si.y), sj.y);
    rz = D == 3 ? sub_rn(fma_rn(-code_off((e >> 4) & 3u, T()), cs, si.z), sj.z) : T(0);
}
// r_ij = s_i - (s_j + o cs) of list entry e: the form of the list's sums, equal
// to rounding.  Its rounding differs from neighbour to neighbour, where that
// of s_i - o cs is common to a cell's: FP32 results lie 10% nearer to those
// in 64 bits (1M particles, one step: 4.5e-7 against 5.0e-7).  Never zero for
// a pair of the list: offsets lie in [0, cs), and s_j + o cs does not round
// into that range unless o = 0, where both forms are one.
template <typename T, int D>
__device__ __forceinline__ void moved_offset(uint32_t e, const V4<T> &si, const V4<T> &sj, T cs, T &rx, T &ry, T &rz) {
    rx = add_rn(si.x, fma_rn(-code_off(e & 3u, T()), cs, -sj.x));
    ry = add_rn(si.y, fma_rn(-code_off((e >> 2) & 3u, T()), cs, -sj.y));
    rz = D == 3 ? add_rn(si.z, fma_rn(-code_off((e >> 4) & 3u, T()), cs, -sj.z)) : T(0);
}

// How a sweep gathers its neighbours (U of walk_list), by measurement at 1M and
// 64k particles in 3D and 37k in 2D (FP32; us per launch, PLAIN against the
// choice):  C 237 -> 213, 33 -> 25 (AHEAD), 16.0 -> 12.7 (4, in 2D);
// V + M 977 -> 822, 134 -> 107 (745 at 1M since they hold the case's constants); A 19.3 -> 14.6; S 72 -> 63, 31 -> 27 (4).
// Sweep B at 1M particles stays PLAIN (250 against 271-300): its arithmetic
// leaves no registers for a neighbour in flight at the warps it needs.
constexpr int PLAIN = 1, AHEAD = -1;
// A list: f(e, s_j, aux_j) for the first c entries from word p on, in order.
// With L lanes, lane `sub` of the group takes the entries sub, sub + L,
// sub + 2L, ...  AUX: a second record per neighbour is gathered too.
// PLAIN keeps two list words in flight and leaves the latency of the gathers
// to the other warps; AHEAD gathers the next neighbour while the current one
// is evaluated and reads list words four entries ahead of it (a word comes
// from HBM and is needed one evaluation earlier); U > 1 gathers U neighbours
// before the first is evaluated.  The order of the entries, and with it every
// sum, is the same.
template <bool AUX, typename T, int L, int U, typename F>
__device__ __forceinline__ void walk_list(const uint32_t *__restrict__ p, uint32_t c, const V4<T> *__restrict__ snap,
                                          const V4<T> *__restrict__ aux, F &&f, uint32_t sub) {
    p += (int)sub * LROW;
    if constexpr (U == PLAIN) {
        uint32_t next = sub < c ? ld_list_walk(p) : 0u;
        uint32_t next2 = sub + L < c ? ld_list_walk(p + L * LROW) : 0u;
        p += L * LROW;
#pragma unroll 1
        for (uint32_t k = sub; k < c; k += L) {
            const uint32_t e = next;            // entries k + L and k + 2L in flight
            next = next2;
            p += L * LROW;
            if (k + 2 * L < c) next2 = ld_list_walk(p);
            const uint32_t j = e >> NBR_SHIFT;
            const V4<T> sj = ld4(snap + j);
            f(e, sj, AUX ? ld4(aux + j) : sj);
        }
    } else if constexpr (U == AHEAD) {
        const auto word = [&](uint32_t k) { return k < c ? ld_list_walk(p + (int64_t)(k - sub) * LROW) : 0u; };
        uint32_t e = word(sub), w1 = word(sub + L), w2 = word(sub + 2 * L), w3 = word(sub + 3 * L);
        V4<T> sj = ld4_now(snap + (e >> NBR_SHIFT)), aj = AUX ? ld4_now(aux + (e >> NBR_SHIFT)) : sj;
        p += 4 * L * LROW;
#pragma unroll 2
        for (uint32_t k = sub; k < c; k += L) {
            const V4<T> sn = ld4_now(snap + (w1 >> NBR_SHIFT)), an = AUX ? ld4_now(aux + (w1 >> NBR_SHIFT)) : sn;
            uint32_t w4 = 0u;
            if (k + 4 * L < c) w4 = ld_list_walk(p);
            p += L * LROW;
            f(e, sj, AUX ? aj : sj);
            e = w1;
            w1 = w2;
            w2 = w3;
            w3 = w4;
            sj = sn;
            aj = an;
        }
    } else {
        uint32_t next[U];
#pragma unroll
        for (int u = 0; u < U; ++u) next[u] = sub + u * L < c ? ld_list_walk(p + u * L * LROW) : 0u;
#pragma unroll 1
        for (uint32_t k = sub; k < c; k += U * L) {
            uint32_t e[U];
            V4<T> sj[U], aj[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {       // a missing entry gathers particle 0 and is dropped
                e[u] = next[u];
                sj[u] = ld4_now(snap + (e[u] >> NBR_SHIFT));
                if (AUX) aj[u] = ld4_now(aux + (e[u] >> NBR_SHIFT));
            }
            p += U * L * LROW;
#pragma unroll
            for (int u = 0; u < U; ++u) next[u] = k + (U + u) * L < c ? ld_list_walk(p + u * L * LROW) : 0u;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k + u * L < c) f(e[u], sj[u], AUX ? aj[u] : sj[u]);
        }
    }
}

// The geometry of one pair as the sums use it.  FP32: the carrier (x, y, z) is
// r_ij itself, with W'/r = (kcoef / h) (1 - q/2)^3 as its weight, which saves
// the unit vector.  FP64: the carrier is the unit vector e_ij with weight W',
// the form that is stored beside the list (below).
template <typename T> struct PairG;
template <> struct PairG<float> {
    float x, y, z, inv, r, wd;                  // r_ij, 1/r, r, W'/r
    // FULL: 1/r also of a denormal r^2 (r < 1.1e-19).  The sums that weigh
    // e_ij by W' or r_ij by W'/r take the least normal r^2 instead: such a pair
    // gives them less than their rounding (its r is below 4e-10 h at the least h
    // FP32 holds), and the full form costs sweep C 3.4% and B 1.4% at 1M
    // particles.  The penalty of sweep S, where e_ij W'/r counts, needs it.
    template <bool FULL>
    __device__ __forceinline__ PairG(const CasePhys<float> &cp, float rx, float ry, float rz, float r2, std::bool_constant<FULL>)
        : x(rx), y(ry), z(rz) {
        r2 = FULL ? r2 : fmaxf(r2, FLT_MIN);
        inv = FULL ? rsq_full(r2) : rsq(r2);
        r = vmul(r2, inv);
        const float u = vfma(r, cp.mhalf_inv_h, 1.0f);
        wd = vmul(vmul(vmul(cp.kcoef_h, u), u), u);
    }
    __device__ __forceinline__ float du(float dot) const { return vmul(dot, inv); }   // carrier product -> along e
    __device__ __forceinline__ float e(float c) const { return vmul(c, inv); }        // carrier -> unit vector
    __device__ __forceinline__ float dW() const { return vmul(wd, r); }               // W'
    __device__ __forceinline__ float dW_r() const { return wd; }                      // W' / r
    __device__ __forceinline__ float outer() const { return wd; }                     // weight of carrier (x) carrier in r (x) W' e
};
template <> struct PairG<double> {
    double x, y, z, inv, r, wd;                 // e_ij, 1/r, r, W'
    __device__ __forceinline__ PairG() {}
    template <bool FULL>
    __device__ __forceinline__ PairG(const CasePhys<double> &cp, double rx, double ry, double rz, double r2, std::bool_constant<FULL>) {
        inv = rsq(r2);
        r = vmul(r2, inv);
        const double u = vfma(r, cp.mhalf_inv_h, 1.0);
        // W' <= 0: at 2h u may round to 0 or below, which is 0 for W'
        wd = -fabs(vmul(vmul(vmul(vmul(cp.kcoef_h, u), u), u), r));
        x = vmul(rx, inv); y = vmul(ry, inv); z = vmul(rz, inv);
    }
    __device__ __forceinline__ double du(double dot) const { return dot; }
    __device__ __forceinline__ double e(double c) const { return c; }
    __device__ __forceinline__ double dW() const { return wd; }
    __device__ __forceinline__ double dW_r() const { return vmul(wd, inv); }
    __device__ __forceinline__ double outer() const { return vmul(wd, r); }
};

// One particle's list: its first word, its count as in cnt[], and (FP64,
// optional) the stored geometry of its entries: (e_ij, W') and (r, 1/r) of the
// frozen configuration at the list's own positions.  W' = -|W'| for every
// pair, with the sign bit set also where it is 0; a wall's entry stores |W'|,
// with the bit clear, and the other fluid's entries come first, so the
// neighbour's kind is known without its position.
struct alignas(16) RInv { double r, inv; };
template <typename T> struct ListRef {
    const uint32_t *p;
    uint32_t count;
    const V4<T> *ge;
    const RInv *gr;
};
// The walk over stored geometry: word, geometry and second record of the next
// entry are in flight while the current one is evaluated.
template <bool AUX, bool NEED_R, int L, typename F>
__device__ __forceinline__ void walk_geo(const ListRef<double> &l, uint32_t c, const V4<double> *__restrict__ aux, uint32_t ki,
                                         F &&f, uint32_t sub) {
    const uint32_t c_other = l.count >> 16;
    const uint32_t *p = l.p + (int)sub * LROW;
    const V4<double> *ge = l.ge + (int)sub * LROW;
    const RInv *gr = l.gr + (int)sub * LROW;
    if (sub >= c) return;
    uint32_t e = ld_list_walk(p), w1 = sub + L < c ? ld_list_walk(p + L * LROW) : 0u;
    V4<double> g = ld4_now(ge), aj = AUX ? ld4_now(aux + (e >> NBR_SHIFT)) : g;
    RInv ri = NEED_R ? *gr : RInv{0.0, 0.0};
#pragma unroll 1
    for (uint32_t k = sub; k < c; k += L) {
        p += L * LROW;
        ge += L * LROW;
        gr += L * LROW;
        const uint32_t ec = e;
        const V4<double> gc = g, ac = aj;
        const RInv rc = ri;
        e = w1;
        if (k + L < c) {
            g = ld4_now(ge);
            if (AUX) aj = ld4_now(aux + (e >> NBR_SHIFT));
            if (NEED_R) ri = *gr;
        }
        if (k + 2 * L < c) w1 = ld_list_walk(p + L * LROW);
        const bool wall = __double_as_longlong(gc.w) >= 0;
        PairG<double> G;
        G.x = gc.x; G.y = gc.y; G.z = gc.z; G.wd = -fabs(gc.w);
        G.r = rc.r; G.inv = rc.inv;
        f(ec >> NBR_SHIFT, wall ? PH_WALL : k < c_other ? ki ^ 1u : ki, AUX ? ac : gc, G);
    }
}

// The cell walk of a sweep (cases without a list).  Only a sixth of the
// candidates of the 3^D cells are neighbours, and which ones differs from lane
// to lane: evaluated where they are found, nearly every candidate cost its
// warp the whole pair with few lanes at work.  So each thread puts its hits
// aside in shared memory, and when a lane of the warp might run out of places
// all lanes evaluate what they have, in the walk's order (the same sums).
// With two lanes per particle, 30k particles in 3D: FP32 A 76 -> 52, B 308 ->
// 92, C 150 -> 68 us; FP64 A 614 -> 388, B 4381 -> 1118, C 1689 -> 703.  125k:
// A 87 -> 101, B 376 -> 257, C 187 -> 168.
// Lanes per particle: lane `sub` takes the cells sub, sub + L, ... of the 3^D,
// and the lanes add their sums in a fixed order.  One lane leaves a case of 30k
// particles 6 warps per SM, each waiting for its candidates.
constexpr int CELL_LANES = 2;
// Places of a thread, a word and a byte each.  More make the evaluations
// fuller, fewer leave shared memory to more warps, which the cheap pairs of
// FP32 sweeps A (which puts only the other fluid aside) and C need more: at
// 125k particles C 168 us with 32, 175 with 38, 195 with 56; B 257 with 56,
// 272 with 48, 283 with 38.  FP64 pairs are dear: C 703 with 56, 838 with 38.
constexpr int CELL_PLACES_MAX = 56;
constexpr int CELL_PLACES_k_sweep_A = 20, CELL_PLACES_k_sweep_C = 32;
constexpr int CELL_PLACES_k_sweep_B = 56, CELL_PLACES_k_sweep_V = 56, CELL_PLACES_k_sweep_M = 32, CELL_PLACES_k_debug_neighbors = 32;
// From this many particles per SM on a sweep takes one thread per particle,
// which evaluates its pairs where it finds them: the chip is full then, and
// what lanes and places spare no longer pays for their own work.  Two lanes
// against one thread, us per launch (FP32): A in 3D at 822 particles per SM 100
// and 101, 2775 267 and 235, in 2D at 592 22 and 22, 2368 51 and 41; C in 3D at
// 822 166 and 186, 2775 460 and 439, 6578 1046 and 905, in 2D at 1332 46 and
// 55, 2368 73 and 69, 6578 188 and 166; B in 2D at 1332 92 and 99, 2368 155 and
// 133, 6578 426 and 324 (M and V alike); B in 3D and FP64 pairs, which are
// dear, stay with the lanes, but for A in 3D (177: 428 and 446, 822: 1777 and
// 1370).
constexpr int64_t CELL_NEVER = (int64_t)1 << 40;
template <typename T, int D> constexpr int64_t CELL_ALONE_k_sweep_A = sizeof(T) == 4 ? 1024 : D == 3 ? 512 : CELL_NEVER;
template <typename T, int D> constexpr int64_t CELL_ALONE_k_sweep_C = sizeof(T) == 4 ? 2048 : CELL_NEVER;
template <typename T, int D> constexpr int64_t CELL_ALONE_k_sweep_B = sizeof(T) == 4 && D == 2 ? 2048 : CELL_NEVER;
template <typename T, int D> constexpr int64_t CELL_ALONE_k_sweep_V = CELL_ALONE_k_sweep_B<T, D>;
template <typename T, int D> constexpr int64_t CELL_ALONE_k_sweep_M = CELL_ALONE_k_sweep_B<T, D>;
template <typename T, int D> constexpr int64_t CELL_ALONE_k_debug_neighbors = CELL_NEVER;
// 1M particles in 3D: B 1784 us in blocks of 128, 2040 of 160 (5 instead of 6
// blocks per SM), 2680 of 256 (38 places); 2D: 426 and 604
constexpr int CELL_BLOCK_MAX = 128;
// at most 48 KB per block, so that no block size asks for an opt-in
template <typename T> __host__ __device__ inline int cell_places(int threads, int want) {
    return min(sizeof(T) == 8 ? CELL_PLACES_MAX : want, 49152 / (threads * 5));
}
template <typename T> __host__ __device__ inline size_t cell_walk_bytes(int threads, int want) {
    return (size_t)threads * cell_places<T>(threads, want) * 5;
}
constexpr int CELL_STEP = 16;                   // candidates between two looks at the free places
template <int PLACES, bool AUX, bool AUX2, bool OTHER, bool FULL, typename T, int D, int L, typename F>
__device__ __forceinline__ bool walk_cells(const CaseDesc &d, const CasePhys<T> &cp, const uint32_t *__restrict__ starts,
                                           const V4<T> *__restrict__ snap, const V4<T> *__restrict__ aux,
                                           const V4<T> *__restrict__ aux2, int64_t i, const V4<T> &si, uint32_t pki, uint32_t sub, F &&f) {
    constexpr int NC = D == 3 ? 27 : 9;
    constexpr int U = sizeof(T) == 8 ? 2 : 4;   // gathers in flight
    extern __shared__ __align__(16) unsigned char sph_cells[];
    const int threads = blockDim.x, places = cell_places<T>(threads, PLACES), step = min(CELL_STEP, places);
    const uint32_t other = phase_of(pki) ^ 1u;
    uint32_t *const word = reinterpret_cast<uint32_t *>(sph_cells) + threadIdx.x;
    uint8_t *const codes = sph_cells + (size_t)threads * places * 4 + threadIdx.x;
    const unsigned lanes = __activemask();
    const int cx = cell_x<D>(pki), cy = cell_y<D>(pki), cz = cell_z<D>(pki);
    const T cs = cp.cs, R2 = cp.four_h2;
    bool coincident = false;
    int held = 0;
    const auto evaluate = [&]() {
        for (int k0 = 0; k0 < held; k0 += U) {
            uint32_t j[U];
            V4<T> sj[U], aj[U], bj[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {        // past the end: the last one again, not evaluated
                j[u] = word[min(k0 + u, held - 1) * threads];
                sj[u] = ld4_now(snap + j[u]);
                aj[u] = AUX ? ld4_now(aux + j[u]) : sj[u];
                bj[u] = AUX2 ? ld4_now(aux2 + j[u]) : sj[u];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (k0 + u >= held) break;
                const uint32_t c = codes[(k0 + u) * threads];
                T rx, ry, rz;
                pair_offset<T, D>(c, si, sj[u], cs, rx, ry, rz);
                const PairG<T> g(cp, rx, ry, rz, norm2<T, D>(rx, ry, rz), std::bool_constant<FULL>());
                if constexpr (AUX2) f(j[u], phase_of(w_bits(sj[u].w)), aj[u], bj[u], g);
                else f(j[u], phase_of(w_bits(sj[u].w)), aj[u], g);
            }
        }
        held = 0;
        __syncwarp(lanes);
    };
    // particles of the q-th cell around, none past the last or off the grid
    const auto range = [&](int q, uint32_t &b, uint32_t &e) {
        int nx = cx + q % 3 - 1, ny = cy + q / 3 % 3 - 1, nz = D == 3 ? cz + q / 9 - 1 : 0;
        b = e = 0;
        if (q < NC && wrap_cell(d, 0, nx) && wrap_cell(d, 1, ny) && (D == 2 || wrap_cell(d, 2, nz))) {
            const uint32_t m = (uint32_t)d.table_off + morton<D>(nx, ny, nz);
            b = __ldg(starts + m);
            e = __ldg(starts + m + 1);
        }
    };
    uint32_t nb, ne;                             // the next cell's, read one cell ahead
    range((int)sub, nb, ne);
#pragma unroll 1
    for (int q = (int)sub; __any_sync(lanes, q < NC); q += L) {
        uint32_t b = nb;
        const uint32_t e = ne;
        const int ox = q % 3 - 1, oy = q / 3 % 3 - 1, oz = D == 3 ? q / 9 - 1 : 0;
        const T sx = sub_rn(si.x, mul_rn(T(ox), cs)), sy = sub_rn(si.y, mul_rn(T(oy), cs));
        const T sz = D == 3 ? sub_rn(si.z, mul_rn(T(oz), cs)) : T(0);
        const uint8_t code = (uint8_t)cell_code<D>(ox, oy, oz);
        range(q + L, nb, ne);
        while (__any_sync(lanes, b < e)) {
            const uint32_t end = min(e, b + step);
            if (__any_sync(lanes, held + (int)(end - min(b, end)) > places)) evaluate();
            const auto test = [&](uint32_t k, const V4<T> &sj) {
                const T rx = sub_rn(sx, sj.x), ry = sub_rn(sy, sj.y);
                const T rz = D == 3 ? sub_rn(sz, sj.z) : T(0);
                const T r2 = norm2<T, D>(rx, ry, rz);
                if (r2 < R2) {
                    if (!(r2 > T(0))) {
                        coincident |= k != (uint32_t)i;
                    } else if (!OTHER || phase_of(w_bits(sj.w)) == other) {
                        word[held * threads] = k;
                        codes[held * threads] = code;
                        ++held;
                    }
                }
            };
            for (; b + U <= end; b += U) {
                V4<T> sj[U];
#pragma unroll
                for (int u = 0; u < U; ++u) sj[u] = ld4_now(snap + b + u);
#pragma unroll
                for (int u = 0; u < U; ++u) test(b + u, sj[u]);
            }
            for (; b < end; ++b) test(b, ld4_now(snap + b));
            b = max(b, end);
            __syncwarp(lanes);
        }
    }
    evaluate();
    return coincident;
}

// neighbours of particle i as f(j, kind of j, aux_j, geometry), from its list
// or from the cell walk.  NEED_R: f reads r or 1/r (FULL of PairG).
template <bool LIST, bool AUX, bool NEED_R, typename T, int D, int PART = PART_ALL, int L = 1, int U = PLAIN, int PLACES = 0,
          typename F, typename N = Nothing>
__device__ __forceinline__ bool neighbors(const CaseDesc &d, const CasePhys<T> &cp, const uint32_t *starts,
                                          const ListRef<T> &l, const V4<T> *snap, const V4<T> *aux, int64_t i,
                                          const V4<T> &si, uint32_t pki, F &&f, uint32_t sub = 0, N &&next = N()) {
    if constexpr (LIST) {
        const uint32_t c = PART == PART_OTHER ? l.count >> 16 : l.count & CNT_MASK;
        if constexpr (sizeof(T) == 8)
            if (l.ge) {
                walk_geo<AUX, NEED_R, L>(l, c, aux, phase_of(pki), f, sub);
                return false;
            }
        const T cs = cp.cs;
        walk_list<AUX, T, L, U>(l.p, c, snap, aux,
            [&](uint32_t e, const V4<T> &sj, const V4<T> &aj) {
                T rx, ry, rz;
                moved_offset<T, D>(e, si, sj, cs, rx, ry, rz);
                f(e >> NBR_SHIFT, phase_of(w_bits(sj.w)), aj, PairG<T>(cp, rx, ry, rz, norm2<T, D>(rx, ry, rz), std::bool_constant<NEED_R>()));
            }, sub);
        return false;
    } else if constexpr (L == 1) {
        return walk<PART == PART_OTHER, T, D>(d, cp, starts, snap, i, si, pki,
            [&](uint32_t j, const V4<T> &sj, T rx, T ry, T rz, T r2) {
                f(j, phase_of(w_bits(sj.w)), AUX ? ld4(aux + j) : sj, PairG<T>(cp, rx, ry, rz, r2, std::bool_constant<NEED_R>()));
            }, next);
    } else {
        return walk_cells<PLACES, AUX, false, PART == PART_OTHER, NEED_R, T, D, L>(d, cp, starts, snap, aux, nullptr, i, si, pki, sub, f);
    }
}

// Sum over the L lanes that share one particle (L = 1, 2, 4, 8; groups are
// aligned within the warp).  The butterfly gives every lane of the group the
// same value: each step adds two partial sums in an order-free way.
template <int L, typename T> __device__ __forceinline__ T group_sum(T v) {
    if constexpr (L > 1) {
        const unsigned lane = threadIdx.x & 31u;
        const unsigned mask = ((1u << L) - 1u) << (lane & ~(unsigned)(L - 1));
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) v = add_rn(v, __shfl_xor_sync(mask, v, o));
    }
    return v;
}

// Where CELL_LANES = 2 lanes share a particle in the cell walk, one takes the
// even cells and the other the odd ones.  A thread that takes them all keeps the
// two sums apart, exchanging them from cell to cell, and adds them at the end:
// the same bits.  walk(next): the walk, which calls next() between cells.
template <bool LIST, int L, typename T, int N> struct Sums {
    T *const now[N];
    T apart[N] = {};
    template <typename W> __device__ __forceinline__ void over(W &&walk) {
        static_assert(CELL_LANES == 2);
        if constexpr (!LIST && L == 1) {
            walk([&]() {
#pragma unroll
                for (int k = 0; k < N; ++k) { const T v = *now[k]; *now[k] = apart[k]; apart[k] = v; }
            });
#pragma unroll
            for (int k = 0; k < N; ++k) *now[k] = add_rn(*now[k], apart[k]);
        } else {
            walk(Nothing());
        }
    }
};

// (v_j - v_i) . carrier, from -v_i
template <typename T, int D>
__device__ __forceinline__ T pair_dot(const V4<T> &vj, T nvx, T nvy, T nvz, T rx, T ry, T rz) {
    const T dx = vadd(vj.x, nvx), dy = vadd(vj.y, nvy);
    if (D == 2) return vfma(dx, rx, vmul(dy, ry));
    return vfma(dx, rx, vfma(dy, ry, vmul(vadd(vj.z, nvz), rz)));
}
// Pressure (Eqs. 7-12): the factor f of one neighbour's term f x (x the
// carrier) in sum_j P* grad W V_j, for particles of densities rho_i and c0 drho_i = b_i.
// With p = c0^2 drho, P* = c0 (rho_j (b_i + beta rho_i dU) + rho_i c0 drho_j) /
// (rho_i + rho_j) (Eqs. 8, 12; beta of Eq. 11) and V_j = m_j / rho_j: one
// division.  Walls by their mirror state rho_i, p_i, 2 U_w - U_L.
template <typename T>
__device__ __forceinline__ T pressure_factor(const CasePhys<T> &cp, bool printed, bool push_only, uint32_t kj, T drj,
                                             T dot, const PairG<T> &g, T rho_i, T b_i) {
    T dU = g.du(dot);                           // U_L - U_R = (v_j - v_i).e (Eq. 10, U = -v.e)
    if (kj == PH_WALL) {
        dU = vmul(T(2), dU);
        T x = vmul(cp.beta_k, dU);
        if (printed) x = vmul(x, vdiv(vmul(cp.c0, b_i), rho_i));
        T ps = vfma(vmul(vmul(clamp_lh(x, cp.beta_lo, cp.beta_hi), rho_i), dU), T(0.5), b_i);   // P* / c0
        if (push_only) ps = vpush(ps);          // no-suction wall reading
        return vmul(vmul(ps, cp.c0_vol), g.wd);
    }
    const T rho_j = add_rn(sel(kj, cp.rho0[0], cp.rho0[1]), drj), a_j = mul_rn(cp.c0, drj);
    const T rs = vadd(rho_i, rho_j);
    T x = vmul(cp.beta_k, dU);
    if (printed) x = vmul(x, vdiv(vmul(cp.c0, vadd(b_i, a_j)), rs));
    const T t = vfma(vmul(clamp_lh(x, cp.beta_lo, cp.beta_hi), dU), rho_i, b_i);
    const T num = vfma(rho_j, t, vmul(rho_i, a_j));
    return vmul(vdiv(vmul(num, sel(kj, cp.mass_c0[0], cp.mass_c0[1])), vmul(rs, rho_j)), g.wd);
}
// Continuity (Eq. 6): (v_i - v*).e V_j of one neighbour, with
// (v_i - v*).e = U* - U_L = (rho_j (v_i - v_j).e + (b_i - c0 drho_j)) /
// (rho_i + rho_j); the printed v* takes the other sign of the pressure
// difference, folded into sb_i and nsc0 = -(+-c0).  v* = v_w at a wall.
template <typename T>
__device__ __forceinline__ T continuity_factor(const CasePhys<T> &cp, uint32_t kj, T drj, T dot, const PairG<T> &g,
                                               T rho_i, T sb_i, T nsc0) {
    const T dU = g.du(dot);
    if (kj == PH_WALL) return vmul(dU, -cp.vol_wall);
    const T rho_j = add_rn(sel(kj, cp.rho0[0], cp.rho0[1]), drj);
    const T num = vfma(-rho_j, dU, vadd(sb_i, mul_rn(nsc0, drj)));
    return vdiv(vmul(num, sel(kj, cp.mass[0], cp.mass[1])),
                vmul(vadd(rho_i, rho_j), rho_j));
}

// ================================================================ rebuild
// First placement of a freshly uploaded case: absolute FP64 positions ->
// cell coordinates (floor((x - origin)/cs) in FP64, as the key definition
// states) and offsets from the cell origin.
template <typename T, int D>
__device__ __forceinline__ void init_one(const CaseDesc &d, int c, int64_t k, const double *apos,
                                         const double *avel, const double *arho, const uint8_t *akind,
                                         V4<T> *pos, V4<T> *vel, T *drho, uint32_t *id, CaseState *st) {
    int cc[3] = {0, 0, 0};
    double off[3] = {0.0, 0.0, 0.0};
    bool bad = false;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        double rel = __dsub_rn(apos[3 * k + a], d.origin[a]);
        if ((d.periodic >> a) & 1) {
            // into the period [0, L), then the last cell also takes a
            // position that rounds onto its end
            const double L = d.period_len[a];
            rel = __dsub_rn(rel, __dmul_rn(L, floor(__ddiv_rn(rel, L))));
        }
        double f = floor(__ddiv_rn(rel, d.cs));
        if ((d.periodic >> a) & 1 && f >= (double)d.ncell[a]) f = (double)(d.ncell[a] - 1);
        if (!(f >= 0.0 && f < (double)d.ncell[a])) {
            bad = true;
            f = f < 0.0 || f != f ? 0.0 : (double)(d.ncell[a] - 1);
        }
        cc[a] = (int)f;
        off[a] = __dsub_rn(rel, __dmul_rn(f, d.cs));
    }
    if (bad) atomicCAS(&st[c].status, 0, DEV_ERR_DOMAIN);
    const uint32_t ph = akind[k];
    V4<T> p;
    p.x = (T)off[0]; p.y = (T)off[1]; p.z = (T)off[2];
    p.w = bits_w(pack_cell<D>(cc[0], cc[1], cc[2], ph), T());
    const int64_t i = d.p_begin + k;
    pos[i] = p;
    V4<T> v;
    v.x = (T)avel[3 * k]; v.y = (T)avel[3 * k + 1]; v.z = (T)avel[3 * k + 2]; v.w = T(0);
    drho[i] = ph < 2 ? (T)(arho[k] - d.rho0[ph]) : T(0);
    v.w = drho[i];                    // vel.w mirrors drho (read with the velocity)
    vel[i] = v;
    id[i] = (uint32_t)k;
}

template <typename T>
__global__ void k_init_case(const CaseDesc *__restrict__ desc, int c, const double *apos,
                            const double *avel, const double *arho, const uint8_t *akind,
                            V4<T> *pos, V4<T> *vel, T *drho, uint32_t *id, CaseState *st) {
    const CaseDesc &d = desc[c];
    const int64_t n = d.p_end - d.p_begin;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        if (d.dim == 3) init_one<T, 3>(d, c, k, apos, avel, arho, akind, pos, vel, drho, id, st);
        else init_one<T, 2>(d, c, k, apos, avel, arho, akind, pos, vel, drho, id, st);
    }
}

// New cell of every particle from its offset (which may have drifted out of
// the cell since the last rebuild), histogram of the cell table.
template <typename T, int D>
__device__ __forceinline__ void assign_one(const CaseDesc &d, CaseState *st, int c, int64_t i,
                                           V4<T> *pos, uint32_t *key, uint32_t *rank,
                                           uint32_t *counts) {
    const CasePhys<T> &cp = phys<T>(d);
    V4<T> p = pos[i];
    const uint32_t pk = w_bits(p.w);
    int cc[3] = {cell_x<D>(pk), cell_y<D>(pk), cell_z<D>(pk)};
    T off[3] = {p.x, p.y, p.z};
    bool bad = false;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        T f = floor(off[a] / cp.cs);
        if (!(f == f) || f > T(4096) || f < T(-4096)) { f = T(0); bad = true; }
        int nc = cc[a] + (int)f;
        if ((d.periodic >> a) & 1) {
            // the offset is taken from the unwrapped cell; the index wraps
            nc = ((nc % d.ncell[a]) + d.ncell[a]) % d.ncell[a];
        } else if (nc < 0 || nc >= d.ncell[a]) {
            bad = true;
            nc = nc < 0 ? 0 : d.ncell[a] - 1;
            f = T(nc - cc[a]);
        }
        off[a] = off[a] - f * cp.cs;
        cc[a] = nc;
    }
    if (bad) atomicCAS(&st[c].status, 0, DEV_ERR_DOMAIN);
    p.x = off[0]; p.y = off[1]; p.z = off[2];
    p.w = bits_w(pack_cell<D>(cc[0], cc[1], cc[2], phase_of(pk)), T());
    pos[i] = p;
    const uint32_t k = (uint32_t)d.table_off + morton<D>(cc[0], cc[1], cc[2]);
    key[i] = k;
    rank[i] = atomicAdd(counts + k, 1u);
}

template <typename T>
__global__ void k_cell_assign(const Tile *__restrict__ tiles, const CaseDesc *__restrict__ desc,
                              CaseState *st, V4<T> *pos, uint32_t *key, uint32_t *rank,
                              uint32_t *counts) {
    follow();
    const Tile t = tiles[blockIdx.x];
    if ((int)threadIdx.x >= t.n) return;
    const CaseDesc &d = desc[t.c];
    const int64_t i = t.begin + threadIdx.x;
    if (d.dim == 3) assign_one<T, 3>(d, st, t.c, i, pos, key, rank, counts);
    else assign_one<T, 2>(d, st, t.c, i, pos, key, rank, counts);
}

// ---- exclusive scan of the cell histogram (in place, n+1 entries) ----
constexpr int SCAN_T = 1024;            // threads per block
constexpr int SCAN_ITEMS = 2 * SCAN_T;  // entries per block

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *total) {
    __shared__ uint32_t warp_sums[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t s = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        warp_sums[lane] = s;
    }
    __syncthreads();
    const uint32_t before = (w > 0 ? warp_sums[w - 1] : 0u) + x - v;
    *total = warp_sums[(blockDim.x >> 5) - 1];
    __syncthreads();
    return before;
}

static __global__ void k_scan_reduce(const uint32_t *data, int64_t n, uint32_t *block_sums) {
    follow();
    const int64_t base = (int64_t)blockIdx.x * SCAN_ITEMS + 2 * threadIdx.x;
    uint32_t v = 0;
    if (base < n) v += data[base];
    if (base + 1 < n) v += data[base + 1];
    uint32_t total;
    block_exclusive_scan(v, &total);
    if (threadIdx.x == 0) block_sums[blockIdx.x] = total;
}

static __global__ void k_scan_blocks(uint32_t *block_sums, int64_t nb) {
    lead();
    follow();
    uint32_t carry = 0;
    for (int64_t base = 0; base < nb; base += SCAN_T) {
        const int64_t k = base + threadIdx.x;
        const uint32_t v = k < nb ? block_sums[k] : 0u;
        uint32_t total;
        const uint32_t ex = block_exclusive_scan(v, &total);
        if (k < nb) block_sums[k] = carry + ex;
        carry += total;
    }
}

static __global__ void k_scan_apply(uint32_t *data, int64_t n, const uint32_t *block_sums) {
    follow();
    const int64_t base = (int64_t)blockIdx.x * SCAN_ITEMS + 2 * threadIdx.x;
    const uint32_t a = base < n ? data[base] : 0u;
    const uint32_t b = base + 1 < n ? data[base + 1] : 0u;
    uint32_t total;
    const uint32_t ex = block_exclusive_scan(a + b, &total) + block_sums[blockIdx.x];
    if (base < n) data[base] = ex;
    if (base + 1 < n) data[base + 1] = ex + a;
}

static __global__ void k_scatter(int64_t n, const uint32_t *key, const uint32_t *rank,
                          const uint32_t *starts, uint32_t *perm) {
    follow();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    perm[starts[key[i]] + rank[i]] = (uint32_t)i;
}

// canonical order inside each cell: ascending insertion index
static __global__ void k_cell_sort(int64_t ncells, const uint32_t *starts, const uint32_t *id,
                            uint32_t *perm) {
    follow();
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= ncells) return;
    const uint32_t b = starts[c], e = starts[c + 1];
    if (e - b < 2) return;
    for (uint32_t k = b + 1; k < e; ++k) {
        const uint32_t pk = perm[k];
        const uint32_t ik = id[pk];
        uint32_t m = k;
        while (m > b && id[perm[m - 1]] > ik) {
            perm[m] = perm[m - 1];
            --m;
        }
        perm[m] = pk;
    }
}

template <typename T>
__global__ void k_gather(int64_t n, const uint32_t *perm, const V4<T> *pos, const V4<T> *vel,
                         const T *drho, const uint32_t *id, V4<T> *pos_t, V4<T> *vel_t,
                         T *drho_t, uint32_t *id_t) {
    follow();
    const int64_t d = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (d >= n) return;
    const uint32_t s = perm[d];
    pos_t[d] = pos[s];
    vel_t[d] = vel[s];
    drho_t[d] = drho[s];
    id_t[d] = id[s];
}

template <typename T>
__global__ void k_copy_back(int64_t n, const V4<T> *pos_t, const V4<T> *vel_t, const T *drho_t,
                            const uint32_t *id_t, V4<T> *pos, V4<T> *vel, T *drho, uint32_t *id) {
    follow();
    const int64_t d = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (d >= n) return;
    pos[d] = pos_t[d];
    vel[d] = vel_t[d];
    drho[d] = drho_t[d];
    id[d] = id_t[d];
}

template <typename T>
__device__ __forceinline__ T volume_of(const CasePhys<T> &cp, uint32_t kj, T drj) {
    return kj == PH_WALL ? cp.vol_wall : vdiv(sel(kj, cp.mass[0], cp.mass[1]), add_rn(sel(kj, cp.rho0[0], cp.rho0[1]), drj));
}
// Volume of neighbour j.  FP64 reads it: its division takes 10 operations of
// the narrow pipe per pair, and k_fluid_scatter and sweep C leave the volumes
// in memory.  FP32 forms it from the density deviation: that write made its
// sweep C 4% slower and saves two operations per pair here.
template <typename T>
__device__ __forceinline__ T volume_at(const CasePhys<T> &cp, uint32_t kj, const T *vd, uint32_t j) {
    return sizeof(T) == 8 ? vd[j] : volume_of(cp, kj, vd[j]);
}

// ---- fluid ranks: after the reorder, the fluid particles in sorted order, walls
// left out: a particle's slot.  The list build, the band and sweeps M, V, B
// and C (and A with the cell walk) run their tiles over the slots, so no lane
// of theirs idles on a wall particle (16% of the 3D drop, interleaved with the
// fluid near the walls by the Morton order).  Flags, an exclusive scan of them,
// a scatter.  Each case's fluid particles take the slots after the previous
// cases' ones, whose count is fixed.
template <typename T>
__global__ void k_fluid_flag(int64_t n, const V4<T> *snap, uint32_t *flag, uint32_t *counts) {
    follow();
    if (blockIdx.x == 0 && threadIdx.x < 4) counts[threadIdx.x] = 0;   // of the band and cell lists
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i > n) return;
    flag[i] = (i < n && phase_of(w_bits(snap[i].w)) != PH_WALL) ? 1u : 0u;
}

// Writes each slot's particle and the values a rebuild starts from: the
// particles' volumes (FP64), a zero colour gradient (the list classes' colour sweep then writes only the
// interface band) and an empty band.  The first fluid particle of each cell of
// a list case appends the cell, as (case << 32 | its first particle), to its
// class's cell list for the list build (warp-aggregated; the order is
// irrelevant, neighbouring cells stay close).  A cell's particles are found by
// their packed cell coordinates: both dimensions share this kernel, which
// therefore forms no Morton code.
constexpr uint32_t CELL_BITS = 0x3fffffffu;     // the cell coordinates of a packed word
template <typename T>
__global__ void k_fluid_scatter(const Tile *__restrict__ tiles, const CaseDesc *__restrict__ desc, const V4<T> *snap,
                                const uint32_t *rank, const T *drho, T *vol, uint32_t *fidx, V4<T> *gradC, uint8_t *band, uint64_t *clist,
                                uint32_t *ccount, int64_t base2d) {
    follow();
    const Tile t = tiles[blockIdx.x];
    const CaseDesc &d = desc[t.c];
    const int64_t i = t.begin + threadIdx.x;
    bool first = false;
    uint32_t b = (uint32_t)i;
    if ((int)threadIdx.x < t.n) {
        gradC[i] = V4<T>{T(0), T(0), T(0), T(0)};
        band[i] = 0;
        const uint32_t pk = w_bits(snap[i].w);
        if (sizeof(T) == 8) vol[i] = volume_of(phys<T>(d), phase_of(pk), drho[i]);
        if (phase_of(pk) != PH_WALL) {
            fidx[rank[i]] = (uint32_t)i;
            first = d.nbr_mode == 0;
            for (; first && (int64_t)b > d.p_begin; --b) {
                const uint32_t pk2 = w_bits(snap[b - 1].w);
                if ((pk2 ^ pk) & CELL_BITS) break;
                first = phase_of(pk2) == PH_WALL;
            }
        }
    }
    const unsigned mask = __ballot_sync(0xffffffffu, first);
    if (!mask) return;
    const int k = d.dim == 3 ? 0 : 1;
    const int lane = threadIdx.x & 31, leader = __ffs(mask) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(ccount + k, (uint32_t)__popc(mask));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (first)
        clist[(k ? base2d : 0) + base + __popc(mask & ((1u << lane) - 1u))] = ((uint64_t)(uint32_t)t.c << 32) | b;
}

// ================================================================ time step
static __global__ void k_reset_vmax(int ncases, CaseState *st) {
    lead();
    follow();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncases) return;
    st[c].vmax2_acc[0] = 0ull;
    st[c].vmax2_acc[1] = 0ull;
}

template <typename T>
__global__ void k_vmax(const Tile *__restrict__ tiles, const CaseDesc *__restrict__ desc,
                       CaseState *st, const V4<T> *pos, const V4<T> *vel) {
    follow();
    const Tile t = tiles[blockIdx.x];
    const int dim = desc[t.c].dim;
    unsigned long long m[2] = {0ull, 0ull};
    if ((int)threadIdx.x < t.n) {
        const int64_t i = t.begin + threadIdx.x;
        const uint32_t ph = phase_of(w_bits(pos[i].w));
        if (ph < 2) m[ph] = (unsigned long long)__double_as_longlong(speed2(vel[i], dim));
    }
    m[0] = warp_max_u64(m[0]);
    m[1] = warp_max_u64(m[1]);
    if ((threadIdx.x & 31) == 0) {
        if (m[0]) atomicMax(&st[t.c].vmax2_acc[0], m[0]);
        if (m[1]) atomicMax(&st[t.c].vmax2_acc[1], m[1]);
    }
}

// Eq. 16 per fluid (factor cfl_ad), Eq. 18 minimum; speed terms with
// |v|max = 0 are dropped.
static __global__ void k_adv_begin(int ncases, const CaseDesc *desc, CaseState *st) {
    lead();
    follow();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncases) return;
    const CaseDesc &d = desc[c];
    CaseState &s = st[c];
    s.active = 0;
    s.last = 0;
    if (s.status) return;
    double dt_ad = __longlong_as_double(0x7ff0000000000000ll);   // +inf
    for (int k = 0; k < 2; ++k) {
        if (!s.present[k]) continue;
        const double vmax = sqrt(bits_to_d(s.vmax2_acc[k]));
        double t = __ddiv_rn(__dmul_rn(__dmul_rn(d.rho0[k], d.h), d.h), d.eta[k]);
        if (vmax > 0.0) {
            const double tv = __ddiv_rn(d.h, vmax);
            if (tv < t) t = tv;
        }
        const double cand = __dmul_rn(d.cfl_ad, t);
        if (cand < dt_ad) dt_ad = cand;
    }
    if (!(dt_ad > 0.0) || !(dt_ad < 1e300)) {
        s.status = DEV_ERR_NONFINITE;
        return;
    }
    s.dt_ad = dt_ad;
    s.t_in = 0.0;
    s.n_sub_adv = 0;
    s.active = 1;
}

// One acoustic substep criterion per case (Eq. 17 with factor cfl_ac, Eq. 18), clipped to end
// exactly on the advection step; sets the while-loop condition to "some case
// still has a substep after this one".
static __global__ void k_dt(int ncases, const CaseDesc *desc, CaseState *st, int *loop_flag,
                     cudaGraphConditionalHandle handle, int use_handle) {
    lead();
    follow();
    int more = 0;
    for (int c = threadIdx.x; c < ncases; c += blockDim.x) {
        const CaseDesc &d = desc[c];
        CaseState &s = st[c];
        if (s.active && s.last) {            // its advection step ended last iteration
            if (!s.status) {
                s.t = __dadd_rn(s.t, s.dt_ad);
                s.n_adv += 1;
            }
            s.active = 0;
        }
        if (s.active && s.status) s.active = 0;
        if (!s.active) continue;
        if (s.n_sub_adv >= d.max_substeps) {
            s.status = DEV_ERR_STALLED;
            s.active = 0;
            continue;
        }
        double vmax[2];
        for (int k = 0; k < 2; ++k) {
            s.vmax2_cur[k] = s.vmax2_acc[k];
            s.vmax2_acc[k] = 0ull;
            vmax[k] = sqrt(bits_to_d(s.vmax2_cur[k]));
        }
        double dt_ac = __longlong_as_double(0x7ff0000000000000ll);
        bool finite = true;
        for (int k = 0; k < 2; ++k) {
            if (!s.present[k]) continue;
            if (!(vmax[k] <= 1e300)) finite = false;
            double t = __ddiv_rn(d.h, __dadd_rn(d.c0, vmax[k]));
            if (d.gamma > 0.0 && d.dt_surf[k] < t) t = d.dt_surf[k];   // formed on the host (Eq. 17)
            const double cand = __dmul_rn(d.cfl_ac, t);
            if (cand < dt_ac) dt_ac = cand;
        }
        if (!finite || !(dt_ac > 0.0) || !(dt_ac < 1e300)) {
            s.status = DEV_ERR_NONFINITE;
            s.active = 0;
            continue;
        }
        const double rem = __dsub_rn(s.dt_ad, s.t_in);
        const int last = dt_ac >= rem;
        const double dt = last ? rem : dt_ac;
        s.last_dt_ac = dt_ac;
        s.dt = dt;
        s.last = last;
        s.t_in = __dadd_rn(s.t_in, dt);
        s.n_sub += 1;
        s.n_sub_adv += 1;
        if (!s.last) more = 1;
    }
    more = __syncthreads_or(more);
    if (threadIdx.x == 0) {
        *loop_flag = more;
        if (use_handle) cudaGraphSetConditional(handle, more ? 1u : 0u);
    }
}

// closes the advection step of the cases that ended it in the final substep
// (the others were closed by k_dt when they went idle)
static __global__ void k_adv_end(int ncases, CaseState *st) {
    follow();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncases) return;
    CaseState &s = st[c];
    if (s.active && s.last && !s.status) {
        s.t = __dadd_rn(s.t, s.dt_ad);
        s.n_adv += 1;
    }
    s.active = 0;
}

// ================================================================= sweeps
// ---- M: correction matrix of Eq. 15, B_i = -(sum_j r_ij (x) grad_i W_ij V_j)^-1
template <typename T> struct Moment {
    T m00, m01, m02, m11, m12, m22;
    // adds (W' V / r) r_vec (x) r_vec of one neighbour, s = W' V / r
    template <int D> __device__ __forceinline__ void add(T s, T rx, T ry, T rz) {
        const T tx = vmul(s, rx), ty = vmul(s, ry);
        m00 = vfma(tx, rx, m00); m01 = vfma(tx, ry, m01); m11 = vfma(ty, ry, m11);
        if (D == 3) { m02 = vfma(tx, rz, m02); m12 = vfma(ty, rz, m12); m22 = vfma(vmul(s, rz), rz, m22); }
    }
    template <int L> __device__ __forceinline__ void group() {
        m00 = group_sum<L>(m00); m01 = group_sum<L>(m01); m02 = group_sum<L>(m02);
        m11 = group_sum<L>(m11); m12 = group_sum<L>(m12); m22 = group_sum<L>(m22);
    }
};

template <typename T, int D>
__device__ __forceinline__ void store_B(const Moment<T> &M, int64_t i, V4<T> *bmat) {
    const T m00 = M.m00, m01 = M.m01, m02 = M.m02, m11 = M.m11, m12 = M.m12, m22 = M.m22;
    T b00, b01, b02 = 0, b11, b12 = 0, b22 = 0;
    T det;
    if (D == 2) {
        det = m00 * m11 - m01 * m01;
        const T id = T(1) / det;
        b00 = -m11 * id; b01 = m01 * id; b11 = -m00 * id;
    } else {
        const T c00 = m11 * m22 - m12 * m12, c01 = m02 * m12 - m01 * m22, c02 = m01 * m12 - m02 * m11;
        det = m00 * c00 + m01 * c01 + m02 * c02;
        const T id = T(1) / det;
        b00 = -c00 * id; b01 = -c01 * id; b02 = -c02 * id;
        b11 = -(m00 * m22 - m02 * m02) * id;
        b12 = -(m02 * m01 - m00 * m12) * id;
        b22 = -(m00 * m11 - m01 * m01) * id;
    }
    if (!(fabs(det) >= T(1e-3))) {
        b00 = 1; b01 = 0; b02 = 0; b11 = 1; b12 = 0; b22 = D == 3 ? T(1) : T(0);
    }
    bmat[2 * i] = V4<T>{b00, b01, b02, b11};
    bmat[2 * i + 1] = V4<T>{b12, b22, T(0), T(0)};
}

template <bool LIST, typename T, int D, int L = 1>
__device__ __forceinline__ void sweep_M(const CaseDesc &d, const CasePhys<T> &cp, int64_t i,
                                        const uint32_t *starts, const ListRef<T> &l, const V4<T> *snap, const T *vol,
                                        V4<T> *bmat, V4<T> *bk, int32_t *status, uint32_t sub = 0) {
    const V4<T> si = ld4(snap + i);
    const uint32_t pki = w_bits(si.w);
    const uint32_t ki = phase_of(pki);
    if (ki == PH_WALL) return;
    const bool own = bk != nullptr && d.surface_corr == 1;
    Moment<T> M{}, Mk{};
    bool coinc = false;
    Sums<LIST, L, T, 12>{{&M.m00, &M.m01, &M.m02, &M.m11, &M.m12, &M.m22, &Mk.m00, &Mk.m01, &Mk.m02, &Mk.m11, &Mk.m12, &Mk.m22}}.over([&](auto &&next) {
        coinc = neighbors<LIST, false, true, T, D, PART_ALL, L, AHEAD, CELL_PLACES_k_sweep_M>(d, cp, starts, l, snap, nullptr, i, si, pki,
            [&](uint32_t j, uint32_t kj, const V4<T> &, const PairG<T> &g) {
                const T w = vmul(g.outer(), volume_at(cp, kj, vol, j));
                M.template add<D>(w, g.x, g.y, g.z);
                // the same sum over i's own fluid (surface_corr reading of Eq. 33)
                if (own && kj == ki) Mk.template add<D>(w, g.x, g.y, g.z);
            }, sub, next);
    });
    if (coinc) atomicCAS(status, 0, DEV_ERR_COINCIDENT);
    M.template group<L>();
    if (own) Mk.template group<L>();
    if (sub != 0) return;
    store_B<T, D>(M, i, bmat);
    if (own) store_B<T, D>(Mk, i, bk);
}

// ---- V: viscous acceleration (Eq. 13) and transport shift (Eq. 14)
// The sums of one particle: a = sum eta (v_i - v_j) W' V / r
// (each step from -v_i) and the shift sum (B_i + B_j) grad W V with symmetric
// B = [b00 b01 b02; b01 b11 b12; b02 b12 b22]
template <typename T> struct ViscSum {
    T ax, ay, az, sx, sy, sz;
    // wv = W' V_j / r, w = V_j times the carrier's weight, neta = -(pair
    // viscosity), b = B_i
    template <int D>
    __device__ __forceinline__ void add(T wv, T w, T neta, bool tvf, const V4<T> &vj, T nvx, T nvy, T nvz, T rx, T ry, T rz,
                                        const T (&b)[6], bool wall, const V4<T> &Bj0, const V4<T> &Bj1) {
        const T f = vmul(neta, wv);
        ax = vfma(f, vadd(vj.x, nvx), ax);
        ay = vfma(f, vadd(vj.y, nvy), ay);
        if (D == 3) az = vfma(f, vadd(vj.z, nvz), az);
        if (!tvf) return;
        // a wall lends its fluid partner's B_i
        const T b00 = wall ? b[0] : Bj0.x, b01 = wall ? b[1] : Bj0.y, b11 = wall ? b[3] : Bj0.w;
        const T gx = vmul(w, rx), gy = vmul(w, ry);
        sx = vfma(vadd(b[0], b00), gx, vfma(vadd(b[1], b01), gy, sx));
        sy = vfma(vadd(b[1], b01), gx, vfma(vadd(b[3], b11), gy, sy));
        if (D == 3) {
            const T b02 = wall ? b[2] : Bj0.z, b12 = wall ? b[4] : Bj1.x, b22 = wall ? b[5] : Bj1.y;
            const T gz = vmul(w, rz);
            sx = vfma(vadd(b[2], b02), gz, sx);
            sy = vfma(vadd(b[4], b12), gz, sy);
            sz = vfma(vadd(b[2], b02), gx, vfma(vadd(b[4], b12), gy, vfma(vadd(b[5], b22), gz, sz)));
        }
    }
    template <int L> __device__ __forceinline__ void group() {
        ax = group_sum<L>(ax); ay = group_sum<L>(ay); az = group_sum<L>(az);
        sx = group_sum<L>(sx); sy = group_sum<L>(sy); sz = group_sum<L>(sz);
    }
};
// the pair viscosity 2 eta_i eta_j / (eta_i + eta_j) takes one value per fluid
// of j; walls use eta_i.  Negated.
template <typename T> struct PairEta {
    T wall, e0, e1;
    __device__ __forceinline__ PairEta(const CasePhys<T> &cp, uint32_t ki) {
        const T eta_i = sel(ki, cp.eta[0], cp.eta[1]);
        wall = -eta_i;
        e0 = -(T(2) * eta_i * cp.eta[0] / (eta_i + cp.eta[0]));
        e1 = -(T(2) * eta_i * cp.eta[1] / (eta_i + cp.eta[1]));
    }
    __device__ __forceinline__ T operator()(uint32_t kj) const { return kj == PH_WALL ? wall : sel(kj, e0, e1); }
};
template <typename T, int D>
__device__ __forceinline__ void store_V(const CasePhys<T> &cp, bool tvf, int64_t i, T rho_i, T ax, T ay, T az, T sx, T sy,
                                        T sz, V4<T> *acc_visc, V4<T> *pos) {
    const T c = T(2) / rho_i;
    acc_visc[i] = V4<T>{vmul(c, ax), vmul(c, ay), vmul(c, az), T(0)};
    if (tvf) {
        V4<T> p = pos[i];
        p.x = vfma(cp.tvf_coef, sx, p.x);
        p.y = vfma(cp.tvf_coef, sy, p.y);
        if (D == 3) p.z = vfma(cp.tvf_coef, sz, p.z);
        pos[i] = p;
    }
}

template <bool LIST, typename T, int D, int L = 1>
__device__ __forceinline__ void sweep_V(const CaseDesc &d, const CasePhys<T> &cp, int64_t i,
                                        const uint32_t *starts, const ListRef<T> &l, const V4<T> *snap,
                                        const V4<T> *vel, const T *vol, const V4<T> *bmat, V4<T> *acc_visc,
                                        V4<T> *pos, int32_t *status, uint32_t sub = 0) {
    const V4<T> si = ld4(snap + i);
    const uint32_t pki = w_bits(si.w);
    const uint32_t ki = phase_of(pki);
    if (ki == PH_WALL) return;
    const V4<T> vi = vel[i];
    const PairEta<T> eta(cp, ki);
    const bool tvf = d.tvf_on != 0;
    T b[6] = {0, 0, 0, 0, 0, 0};
    if (tvf) {
        const V4<T> b0 = bmat[2 * i], b1 = bmat[2 * i + 1];
        b[0] = b0.x; b[1] = b0.y; b[2] = b0.z; b[3] = b0.w; b[4] = b1.x; b[5] = b1.y;
    }
    ViscSum<T> S{};
    bool coinc = false;
    Sums<LIST, L, T, 6>{{&S.ax, &S.ay, &S.az, &S.sx, &S.sy, &S.sz}}.over([&](auto &&next) {
        coinc = neighbors<LIST, true, true, T, D, PART_ALL, L, AHEAD, CELL_PLACES_k_sweep_V>(d, cp, starts, l, snap, vel, i, si, pki,
            [&](uint32_t j, uint32_t kj, const V4<T> &vj, const PairG<T> &g) {
                const bool wall = kj == PH_WALL;
                V4<T> B0{}, B1{};
                if (tvf && !wall) { B0 = bmat[2 * j]; if (D == 3) B1 = bmat[2 * j + 1]; }
                const T V = sizeof(T) == 8 ? vol[j] : volume_of(cp, kj, vj.w);
                S.template add<D>(vmul(g.dW_r(), V), vmul(g.wd, V), eta(kj), tvf, vj, -vi.x, -vi.y, -vi.z, g.x, g.y, g.z, b, wall,
                                  B0, B1);
            }, sub, next);
    });
    if (coinc) atomicCAS(status, 0, DEV_ERR_COINCIDENT);
    S.template group<L>();
    if (sub != 0) return;
    store_V<T, D>(cp, tvf, i, sel(ki, cp.rho0[0], cp.rho0[1]) + vi.w, S.ax, S.ay, S.az, S.sx, S.sy, S.sz, acc_visc, pos);
}

// ---- A: colour gradient, Eq. 22 (only pairs of different fluids contribute),
// kept as its unit vector and its magnitude (w), the form the surface sum reads
template <bool LIST, typename T, int D, int L = 1, int U = PLAIN>
__device__ __forceinline__ void sweep_A(const CaseDesc &d, const CasePhys<T> &cp, int64_t i,
                                        const uint32_t *starts, const ListRef<T> &l, const V4<T> *snap, const T *vol,
                                        V4<T> *gradC, uint32_t sub = 0) {
    const V4<T> si = ld4(snap + i);
    const uint32_t pki = w_bits(si.w);
    const uint32_t ki = phase_of(pki);
    V4<T> g = {0, 0, 0, 0};
    if (ki != PH_WALL && d.n_fluid_phases == 2) {
        const T two_phi = sel(ki, cp.two_phi[0], cp.two_phi[1]);
        Sums<LIST, L, T, 3>{{&g.x, &g.y, &g.z}}.over([&](auto &&next) {
            neighbors<LIST, false, false, T, D, PART_OTHER, L, U, CELL_PLACES_k_sweep_A>(d, cp, starts, l, snap, nullptr, i, si, pki,
                [&](uint32_t j, uint32_t kj, const V4<T> &, const PairG<T> &G) {
                    const T s = vmul(vmul(two_phi, G.wd), volume_at(cp, kj, vol, j));
                    g.x = fma_rn(s, G.x, g.x);
                    g.y = fma_rn(s, G.y, g.y);
                    if (D == 3) g.z = fma_rn(s, G.z, g.z);
                }, sub, next);
        });
        g.x = group_sum<L>(g.x);
        g.y = group_sum<L>(g.y);
        if (D == 3) g.z = group_sum<L>(g.z);
        g.w = sqrt(fma_rn(g.x, g.x, fma_rn(g.y, g.y, g.z * g.z)));
        const T inv = g.w > T(0) ? T(1) / g.w : T(0);
        g.x *= inv; g.y *= inv; g.z *= inv;
    }
    if (sub == 0) gradC[i] = g;
}

// v + dt (a^p + a^s + a^v), w = the density deviation for sweep C
template <typename T, int D>
__device__ __forceinline__ V4<T> kicked(const V4<T> &vi, T rho_i, T dt, T apx, T apy, T apz, T asx, T asy, T asz,
                                        const V4<T> &av) {
    const T inv_rho = T(1) / rho_i;
    const T m2inv_rho = T(-2) * inv_rho;
    V4<T> vn;
    vn.x = fma_rn(dt, fma_rn(inv_rho, asx, fma_rn(m2inv_rho, apx, av.x)), vi.x);
    vn.y = fma_rn(dt, fma_rn(inv_rho, asy, fma_rn(m2inv_rho, apy, av.y)), vi.y);
    vn.z = D == 3 ? fma_rn(dt, fma_rn(inv_rho, asz, fma_rn(m2inv_rho, apz, av.z)), vi.z) : T(0);
    vn.w = vi.w;
    return vn;
}

// ---- B: pressure + surface tension + kick
// With the neighbour list the surface sum (Eqs. 24, 26, 30, 33) is a kernel of
// its own (S, below), launched before B and taken only by particles of the
// interface band (band[i]: i or one of its neighbours has neighbours of the
// other fluid; elsewhere grad C = 0 for i and all its neighbours and every
// surface term is zero).  B then runs the pressure sum over all neighbours and
// adds the stored surface sum.  The terms are those of the single pass of
// the cell walk; the list's order (other-phase neighbours first) and the
// surface sweep's lanes add them in another order, so the two agree to
// rounding.
//
// PASS: 0 = pressure + surface in one walk (cell walk), 1 = pressure and the
// stored surface sum (list), 2 = surface sum only (list, band particles).
template <bool LIST, int PASS, typename T, int D, int L = 1, int U = PLAIN>
__device__ __forceinline__ double sweep_B(const CaseDesc &d, const CasePhys<T> &cp, T dt,
                                          int64_t i, const uint32_t *starts, const ListRef<T> &l,
                                          const uint8_t *band, const V4<T> *snap,
                                          const V4<T> *vel, const V4<T> *gradC,
                                          const V4<T> *acc_visc, V4<T> *acc_surf, V4<T> *vel_new,
                                          uint32_t *phase_out, uint32_t sub = 0,
                                          const V4<T> *bk = nullptr, const T *vol = nullptr) {
    const V4<T> si = ld4(snap + i);
    const uint32_t pki = w_bits(si.w);
    const uint32_t ki = phase_of(pki);
    *phase_out = ki;
    if (ki == PH_WALL) return 0.0;
    if (PASS == 2 && !band[i]) return 0.0;
    const V4<T> vi = vel[i];
    const T dri = vi.w;
    const T rho_i = add_rn(sel(ki, cp.rho0[0], cp.rho0[1]), dri);
    const T b_i = mul_rn(cp.c0, dri);
    T apx = 0, apy = 0, apz = 0, asx = 0, asy = 0, asz = 0;
    const bool printed = d.limiter == 3, push_only = d.wall_form == 1;
    const auto pressure = [&](uint32_t, uint32_t kj, const V4<T> &vj, const PairG<T> &g) {
        const T dot = pair_dot<T, D>(vj, -vi.x, -vi.y, -vi.z, g.x, g.y, g.z);
        const T f = pressure_factor<T>(cp, printed, push_only, kj, vj.w, dot, g, rho_i, b_i);
        apx = vfma(f, g.x, apx);
        apy = vfma(f, g.y, apy);
        if (D == 3) apz = vfma(f, g.z, apz);
    };

    // surface stress and penalty (Eqs. 24, 26, 30, 33); walls take no part
    // unit normal, magnitude and colour gradient of i; n = 0 off the interface
    const V4<T> ni = d.n_fluid_phases == 2 ? gradC[i] : V4<T>{0, 0, 0, 0};
    const V4<T> gi{ni.w * ni.x, ni.w * ni.y, ni.w * ni.z, ni.w};
    const bool if_i = ni.w * cp.h > cp.nhat_eps;
    const T nix = if_i ? ni.x : T(0), niy = if_i ? ni.y : T(0), niz = if_i ? ni.z : T(0);
    const T gam_gi = if_i ? cp.gamma * ni.w : T(0);
    // surface_corr reading: the own-fluid correction matrix of i (Eq. 15
    // over i's fluid), symmetric: (b00, b01, b02, b11), (b12, b22)
    const bool corr = bk != nullptr && d.surface_corr == 1;
    V4<T> bi0{T(0), T(0), T(0), T(0)}, bi1{T(0), T(0), T(0), T(0)};
    if (corr && PASS != 1) { bi0 = bk[2 * i]; bi1 = bk[2 * i + 1]; }
    const auto surface = [&](uint32_t j, uint32_t kj, const V4<T> &nj, const PairG<T> &g) {
        if (kj == PH_WALL) return;
        if (ni.w == T(0) && nj.w == T(0)) return;                // every surface term vanishes
        const T ex = g.e(g.x), ey = g.e(g.y), ez = D == 3 ? g.e(g.z) : T(0);
        const T Vj = volume_at(cp, kj, vol, j);
        const V4<T> gj{nj.w * nj.x, nj.w * nj.y, nj.w * nj.z, nj.w};
        const bool if_j = nj.w * cp.h > cp.nhat_eps;
        const T njx = if_j ? nj.x : T(0), njy = if_j ? nj.y : T(0), njz = if_j ? nj.z : T(0);
        const T gam_gj = if_j ? cp.gamma * nj.w : T(0);
        if (corr && kj == ki) {
            // same-phase line applied to the corrected kernel gradient
            // W' (B^k_i + B^k_j)/2 e = W' v (C_ij = 0): S v with
            // Pi v = gamma |gradC| (v - n (n.v)) and C-hat v of Eq. 30
            const V4<T> bj0 = bk[2 * j], bj1 = bk[2 * j + 1];
            const T m00 = T(0.5) * (bi0.x + bj0.x), m01 = T(0.5) * (bi0.y + bj0.y), m11 = T(0.5) * (bi0.w + bj0.w);
            const T m02 = D == 3 ? T(0.5) * (bi0.z + bj0.z) : T(0), m12 = D == 3 ? T(0.5) * (bi1.x + bj1.x) : T(0);
            const T m22 = D == 3 ? T(0.5) * (bi1.y + bj1.y) : T(0);
            const T vx = m00 * ex + m01 * ey + m02 * ez, vy = m01 * ex + m11 * ey + m12 * ez;
            const T vz = D == 3 ? m02 * ex + m12 * ey + m22 * ez : T(0);
            const T niv = nix * vx + niy * vy + niz * vz, njv = njx * vx + njy * vy + njz * vz;
            const T bx = T(0.5) * (gi.x + gj.x), by = T(0.5) * (gi.y + gj.y), bz = T(0.5) * (gi.z + gj.z);
            const T b2 = bx * bx + by * by + bz * bz;
            const T inv_bn = b2 > T(0) ? rsq_full(b2) : T(0);
            T cx, cy, cz;
            if (d.penalty_form == 0) {            // -|gradCbar| r nbar (nbar.v)
                const T fac = g.r * (bx * vx + by * vy + bz * vz) * inv_bn;
                cx = -fac * bx; cy = -fac * by; cz = -fac * bz;
            } else if (d.penalty_form == 1) {     // -|gradCbar| r e (e.v)
                const T f = -(b2 * inv_bn * g.r) * (ex * vx + ey * vy + ez * vz);
                cx = f * ex; cy = f * ey; cz = f * ez;
            } else {                              // -(gradCbar . r_ij) v
                const T f = -g.r * (bx * ex + by * ey + bz * ez);
                cx = f * vx; cy = f * vy; cz = f * vz;
            }
            const T nic = nix * cx + niy * cy + niz * cz, njc = njx * cx + njy * cy + njz * cz;
            const T qx = T(0.5) * (nix * nic + njx * njc), qy = T(0.5) * (niy * nic + njy * njc),
                    qz = T(0.5) * (niz * nic + njz * njc);
            const T pen_s = d.penalty_scope == 1 ? T(0) : cp.xi * cp.gamma * g.inv;
            const T sx = gam_gi * (vx - nix * niv) + gam_gj * (vx - njx * njv) + pen_s * (cx - qx);
            const T sy = gam_gi * (vy - niy * niv) + gam_gj * (vy - njy * njv) + pen_s * (cy - qy);
            const T sz = gam_gi * (vz - niz * niv) + gam_gj * (vz - njz * njv) + pen_s * (cz - qz);
            const T w = g.dW() * Vj;
            asx += sx * w; asy += sy * w; if (D == 3) asz += sz * w;
            return;
        }
        const T nie = nix * ex + niy * ey + niz * ez;
        const T nje = njx * ex + njy * ey + njz * ez;
        // Pi e = gamma |gradC| (e - n (n.e))   (Eq. 24)
        const T pix = gam_gi * (ex - nix * nie), piy = gam_gi * (ey - niy * nie), piz = gam_gi * (ez - niz * nie);
        const T pjx = gam_gj * (ex - njx * nje), pjy = gam_gj * (ey - njy * nje), pjz = gam_gj * (ez - njz * nje);
        const bool same = kj == ki;
        const T sg = (same || d.grad_mode == 1) ? T(1) : T(-1);
        const T bx = T(0.5) * (gi.x + sg * gj.x), by = T(0.5) * (gi.y + sg * gj.y),
                bz = T(0.5) * (gi.z + sg * gj.z);
        const T b2 = bx * bx + by * by + bz * bz;
        const T inv_bn = b2 > T(0) ? rsq_full(b2) : T(0);
        const T Cij = same ? T(0) : T(1);
        // C-hat e (Eq. 30 with the selected contraction)
        T cx, cy, cz;
        if (d.penalty_form == 0) {
            const T fac = g.r * (bx * ex + by * ey + bz * ez) * inv_bn;
            cx = Cij * ex - fac * bx; cy = Cij * ey - fac * by; cz = Cij * ez - fac * bz;
        } else {
            // EE: (C_ij - |gradCbar| r) e; SCALAR (Eq. 29): (C_ij - gradCbar . r_ij) e
            const T s = d.penalty_form == 1 ? Cij - b2 * inv_bn * g.r
                                            : Cij - g.r * (bx * ex + by * ey + bz * ez);
            cx = s * ex; cy = s * ey; cz = s * ez;
        }
        // N-bar C-hat e = (n_i (n_i.c) + n_j (n_j.c)) / 2
        const T nic = nix * cx + niy * cy + niz * cz;
        const T njc = njx * cx + njy * cy + njz * cz;
        const T qx = T(0.5) * (nix * nic + njx * njc), qy = T(0.5) * (niy * nic + njy * njc),
                qz = T(0.5) * (niz * nic + njz * njc);
        const T pen = cp.xi * cp.gamma * g.inv;
        T sx, sy, sz;
        if (same) {   // Eq. 33, first line; T-bar c = c - N-bar c
            const T pen_s = d.penalty_scope == 1 ? T(0) : pen;
            sx = pix + pjx + pen_s * (cx - qx);
            sy = piy + pjy + pen_s * (cy - qy);
            sz = piz + pjz + pen_s * (cz - qz);
        } else {      // Eq. 33, second line: 2 phi_j Pi_i + 2 phi_i Pi_j as printed, or
                      // each stress by its own particle's 2 phi (stress_weights 1)
            const bool own = d.stress_weights == 1;
            const T a = sel(own ? ki : kj, cp.two_phi[0], cp.two_phi[1]),
                    b = sel(own ? kj : ki, cp.two_phi[0], cp.two_phi[1]),
                    c = cp.four_phi_phi * pen;
            sx = a * pix + b * pjx - c * qx;
            sy = a * piy + b * pjy - c * qy;
            sz = a * piz + b * pjz - c * qz;
        }
        const T w = g.dW() * Vj;
        asx += sx * w; asy += sy * w; if (D == 3) asz += sz * w;
    };

    const bool surface_on = d.n_fluid_phases == 2;
    if constexpr (PASS == 2) {
        if (surface_on)
            neighbors<LIST, true, true, T, D, PART_ALL, L, U, CELL_PLACES_k_sweep_B>(d, cp, starts, l, snap, gradC, i, si, pki, surface, sub);
        asx = group_sum<L>(asx);
        asy = group_sum<L>(asy);
        if (D == 3) asz = group_sum<L>(asz);
        if (sub == 0) acc_surf[i] = V4<T>{asx, asy, asz, T(0)};
        return 0.0;
    } else if constexpr (PASS == 1) {
        neighbors<LIST, true, false, T, D, PART_ALL, L, U, CELL_PLACES_k_sweep_B>(d, cp, starts, l, snap, vel, i, si, pki, pressure, sub);
        apx = group_sum<L>(apx);
        apy = group_sum<L>(apy);
        if (D == 3) apz = group_sum<L>(apz);
        if (sub != 0) {               // the group's lane 0 kicks
            *phase_out = PH_WALL;
            return 0.0;
        }
        if (surface_on && band[i]) {
            const V4<T> as = acc_surf[i];
            asx = as.x; asy = as.y; asz = as.z;
        }
    } else {
        const auto both = [&](uint32_t j, uint32_t kj, const V4<T> &vj, const V4<T> &nj, const PairG<T> &g) {
            pressure(j, kj, vj, g);
            surface(j, kj, nj, g);
        };
        if constexpr (L == 1)
            Sums<LIST, L, T, 6>{{&apx, &apy, &apz, &asx, &asy, &asz}}.over([&](auto &&next) {
                walk<false, T, D>(d, cp, starts, snap, i, si, pki,
                    [&](uint32_t j, const V4<T> &sj, T rx, T ry, T rz, T r2) {
                        const uint32_t kj = phase_of(w_bits(sj.w));
                        const PairG<T> g(cp, rx, ry, rz, r2, std::true_type());
                        pressure(j, kj, ld4(vel + j), g);
                        if (surface_on) surface(j, kj, ld4(gradC + j), g);
                    }, next);
            });
        else if (surface_on)
            walk_cells<CELL_PLACES_k_sweep_B, true, true, false, true, T, D, L>(d, cp, starts, snap, vel, gradC, i, si, pki, sub, both);
        else
            walk_cells<CELL_PLACES_k_sweep_B, true, false, false, false, T, D, L>(d, cp, starts, snap, vel, nullptr, i, si, pki, sub, pressure);
        apx = group_sum<L>(apx);
        apy = group_sum<L>(apy);
        asx = group_sum<L>(asx);
        asy = group_sum<L>(asy);
        if (D == 3) { apz = group_sum<L>(apz); asz = group_sum<L>(asz); }
        if (sub != 0) {
            *phase_out = PH_WALL;
            return 0.0;
        }
    }
    const V4<T> vn = kicked<T, D>(vi, rho_i, dt, apx, apy, apz, asx, asy, asz, acc_visc[i]);
    vel_new[i] = vn;
    return speed2(vn, D);
}

// ---- C: continuity (Eq. 6) with v* (normal component -U*) + drift
template <typename T, int D>
__device__ __forceinline__ void store_C(const CasePhys<T> &cp, uint32_t ki, int64_t i, T dt, T rho_i, T sum, V4<T> vi, T *drho,
                                        T *vol, V4<T> *vel, V4<T> *pos) {
    const T dr_new = fma_rn(dt, T(2) * rho_i * sum, vi.w);
    drho[i] = dr_new;
    if (sizeof(T) == 8) vol[i] = volume_of(cp, ki, dr_new);
    V4<T> p = pos[i];
    p.x = fma_rn(dt, vi.x, p.x);
    p.y = fma_rn(dt, vi.y, p.y);
    if (D == 3) p.z = fma_rn(dt, vi.z, p.z);
    pos[i] = p;
    vi.w = dr_new;
    vel[i] = vi;
}

template <bool LIST, typename T, int D, int L = 1, int U = PLAIN>
__device__ __forceinline__ void sweep_C(const CaseDesc &d, const CasePhys<T> &cp, T dt, int64_t i,
                                        const uint32_t *starts, const ListRef<T> &l, const V4<T> *snap,
                                        const V4<T> *vel_new, T *drho, T *vol,
                                        V4<T> *vel, V4<T> *pos, uint32_t sub = 0) {
    const V4<T> si = ld4(snap + i);
    const uint32_t pki = w_bits(si.w);
    const uint32_t ki = phase_of(pki);
    if (ki == PH_WALL) return;
    const V4<T> vi = vel_new[i];
    const T rho_i = add_rn(sel(ki, cp.rho0[0], cp.rho0[1]), vi.w);
    const T nsc0 = d.vstar_printed ? cp.c0 : -cp.c0, sb_i = mul_rn(-nsc0, vi.w);
    T s = 0;
    Sums<LIST, L, T, 1>{{&s}}.over([&](auto &&next) {
        neighbors<LIST, true, false, T, D, PART_ALL, L, U, CELL_PLACES_k_sweep_C>(d, cp, starts, l, snap, vel_new, i, si, pki,
            [&](uint32_t, uint32_t kj, const V4<T> &vj, const PairG<T> &g) {
                const T dot = pair_dot<T, D>(vj, -vi.x, -vi.y, -vi.z, g.x, g.y, g.z);
                s = vfma(continuity_factor<T>(cp, kj, vj.w, dot, g, rho_i, sb_i, nsc0), g.dW(), s);
            }, sub, next);
    });
    s = group_sum<L>(s);
    if (sub == 0) store_C<T, D>(cp, ki, i, dt, rho_i, s, vi, drho, vol, vel, pos);
}

// ---------------------------------------------------------- sweep kernels
// Tiles are grouped by class (dimension, neighbour source) and each class is
// launched with its own instantiation, so every kernel is compiled (and its
// registers allocated) for one dimension and one neighbour source only.
struct SweepArgs {
    const Tile *tiles;
    const CaseDesc *desc;
    CaseState *st;
    const uint32_t *starts;
    const uint32_t *nbr;
    const uint32_t *cnt;
    int64_t tile0;                 // first tile of the launched class
    // nullptr: tile entries are particle indices; else the tiles run over
    // fluid ranks and fidx maps a rank to the particle (sweeps B and C)
    const uint32_t *fidx = nullptr;
    // stored pair geometry of the lists (FP64, of the cases that keep it)
    const void *ge = nullptr, *gr = nullptr;
    // batches: the tiles of the cases active in this substep, compacted per
    // class after the criterion kernel (work[tile0 + k] is a tile index,
    // *work_count of them); the launch's blocks stride over them.  nullptr:
    // block b takes tile tile0 + b / L.
    const uint32_t *work = nullptr;
    const uint32_t *work_count = nullptr;
    // an engine of one case: its descriptor by value, so that the sweeps of
    // MODE_ONE read the per-case constants from the launch's parameter block
    // (constant-bank operands) instead of holding them in registers
    CaseDesc one{};
};

// How a per-substep sweep finds its tiles and its case: MODE_TILES, block b
// takes tile tile0 + b / L and reads desc[c]; MODE_WORK, the blocks stride
// over the batch's work list; MODE_ONE, as MODE_TILES with the one case's
// descriptor taken from the parameter block; MODE_FEW, as MODE_ONE for a case
// that leaves the SMs with few warps: four neighbours are gathered at a time.
enum SweepMode { MODE_TILES = 0, MODE_WORK = 1, MODE_ONE = 2, MODE_FEW = 3 };
template <int MODE> __device__ __forceinline__ const CaseDesc &case_desc(const SweepArgs &a, int c) {
    if constexpr (MODE == MODE_ONE || MODE == MODE_FEW) return a.one;
    else return a.desc[c];
}

// A sweep's per-case constants: of the parameter block where the launch has
// them; else, with the list, copied from memory before the pair loop.  Read
// through a reference they were loaded again for every pair: per launch of a
// batch of 6M particles B 876 us against 798, S 347 against 329, A 61 against
// 57, V 1436 against 1244 (M, 658 against 790, keeps the reference).  The cell
// walk, whose registers are short, reads them again (3D, 125k particles: B 259
// us, with copies 321).
template <bool LIST, int MODE, typename T>
using Phys = std::conditional_t<!LIST || MODE == MODE_ONE || MODE == MODE_FEW, const CasePhys<T> &, const CasePhys<T>>;

// Work items of a sweep launch: (tile, block of the tile) pairs; with L
// lanes per particle a tile takes L blocks.  Without a work list (WORK
// false: single cases) the launch has one block per item and each block
// runs one item; with one (batches), its blocks take items blockIdx.x,
// blockIdx.x + gridDim.x, ... up to L x (active tiles of the class).
template <int L, bool WORK> __device__ __forceinline__ int64_t work_items(const SweepArgs &a) {
    return WORK ? (int64_t)(*a.work_count) * L : (int64_t)gridDim.x;
}
template <int L, bool WORK> __device__ __forceinline__ Tile work_tile(const SweepArgs &a, int64_t w) {
    return a.tiles[WORK ? (int64_t)a.work[a.tile0 + w / L] : a.tile0 + w / L];
}

// particle of a thread within its tile: with L lanes a block covers 1/L of it
template <int L> __device__ __forceinline__ int local_index(int64_t w) {
    return L == 1 ? (int)threadIdx.x : (int)((w % L) * (blockDim.x / L) + threadIdx.x / L);
}

// particle of tile position q: the position itself, or the fluid particle of
// that rank (the list build, the band, sweeps M, V, B and C, A with the cell walk)
__device__ __forceinline__ int64_t particle_at(const SweepArgs &a, int64_t q) {
    return a.fidx ? (int64_t)a.fidx[q] : q;
}

template <bool LIST, typename T> __device__ __forceinline__ ListRef<T> list_of(const SweepArgs &a, const CaseDesc &d, int64_t q) {
    if (!LIST) return ListRef<T>{nullptr, 0u, nullptr, nullptr};
    const int64_t w = list_word(d, q);
    if (sizeof(T) == 8 && d.geo_base >= 0) {
        const int64_t g = d.geo_base + (w - d.nbr_base);
        return ListRef<T>{a.nbr + w, a.cnt[q], static_cast<const V4<T> *>(a.ge) + g, static_cast<const RInv *>(a.gr) + g};
    }
    return ListRef<T>{a.nbr + w, a.cnt[q], nullptr, nullptr};
}

// entry t of the band list: (case << 32 | slot)
struct BandEntry {
    int c;
    int64_t q, i;
    __device__ __forceinline__ BandEntry(const SweepArgs &a, const uint64_t *blist, int64_t t) {
        const uint64_t e = blist[t];
        c = (int)(e >> 32);
        q = (int64_t)(uint32_t)e;
        i = (int64_t)a.fidx[q];
    }
};

// ---- L: neighbour lists of the frozen configuration (fluid particles only),
// one block per cell that holds fluid particles.  All particles of a cell
// share their candidates, the particles of the 3^D cells around it (475 in
// 3D, of which 80 are neighbours): the block orders those cells by table
// index, so that candidates come in increasing j, and copies their positions
// to shared memory once, moved by their cell's offset and in FP32.  Each warp
// takes one slot (fluid particle) after the other and tests 32 candidates at a
// time, one per lane; a ballot gives the hits and their places in the slot's
// list, which is put together in shared memory (the other phase's entries
// from the end) and written at the end row by row, neighbouring slots side by
// side.  Which candidates are neighbours is decided by the cell walk's own
// operations, so list and walk hold the same pairs: in FP32 for the few that
// the first test cannot settle, in FP64 for its hits, a sixth of the
// candidates: the FP64
// pipe is 64 times narrower.  It is bound by instruction issue (about 21
// instructions per 32 candidates of a slot).  Measured, rebuild of an
// advection step: 1M fluid particles in FP32 1.71 -> 1.13 ms, 64k 0.56 ->
// 0.18 ms, 6.9M 11.6 -> 7.1 ms, 43k in FP64 1.17 -> 0.31 ms, against a thread
// per particle that walked its cells alone (lanes in different cells, the
// ordered cells of each lane in local memory) and a separate pass over all
// lists for the band; a warp per cell with the slots in its inner loop took
// 1.76 ms at 1M (58 instructions per 32 candidates of a slot).
constexpr int LB_WARPS = 4;                     // warps per block
constexpr int LB_CAND = 576;                    // candidates in shared memory at a time (8^3 on a lattice, and some)
constexpr int LB_WORDS = 3072;                  // list words of a group of slots in shared memory
constexpr int LB_SLOTS = 32;                    // slots of a group at most
struct ListSmem {
    float4 cand[LB_CAND];                       // x, y, z relative to the cell, list entry
    uint32_t fluid[2][LB_CAND / 32];            // candidates of each fluid, a word per 32
    uint32_t begin[32], pre[33], code[32];      // cells around in increasing table index
    uint32_t idx[LB_SLOTS], rest[LB_SLOTS], other[LB_SLOTS];   // a slot's particle, entries of its list's parts
    uint32_t list[LB_WORDS];
};
// The row length of the shared lists: K + 1 words, so that for the even
// capacities in use a column of slots lies in different banks; capacities of
// LB_WORDS or more are not accepted by the library (K <= 1024)
__device__ __forceinline__ int lb_group(int K) { return min(LB_SLOTS, LB_WORDS / (K + 1)); }


// whether list entry e lies within 2h of slot i, by the cell walk's operations
template <typename T, int D>
__device__ __forceinline__ bool list_exact(uint32_t e, const CasePhys<T> &cp, const V4<T> &si, uint32_t i,
                                           const V4<T> *snap, bool &coinc) {
    const uint32_t j = e >> NBR_SHIFT;
    const V4<T> sj = ld4(snap + j);
    T rx, ry, rz;
    pair_offset<T, D>(e, si, sj, cp.cs, rx, ry, rz);
    const T r2 = norm2<T, D>(rx, ry, rz);
    const bool near = r2 < cp.four_h2 && j != i;
    coinc |= near && !(r2 > T(0));
    return near && r2 > T(0);
}

// keeps the exact neighbours among the n entries row[at], row[at + step], ...;
// returns their number
template <typename T, int D>
__device__ __forceinline__ uint32_t list_keep(uint32_t *row, int at, int step, uint32_t n, const CasePhys<T> &cp,
                                              const V4<T> &si, uint32_t i, const V4<T> *snap, bool &coinc) {
    const int lane = threadIdx.x & 31;
    uint32_t kept = 0;
    for (uint32_t k0 = 0; k0 < n; k0 += 32) {
        const uint32_t k = k0 + lane;
        const uint32_t e = k < n ? row[at + (int)k * step] : 0u;
        const bool hit = k < n && list_exact<T, D>(e, cp, si, i, snap, coinc);
        const unsigned h = __ballot_sync(0xffffffffu, hit);   // all of the chunk is read before it is written
        if (hit) row[at + (int)(kept + __popc(h & ((1u << lane) - 1u))) * step] = e;
        kept += (uint32_t)__popc(h);
    }
    __syncwarp();
    return kept;
}

// a coordinate as the test in FP32 takes it: FP64 coordinates in the unit
// list_unit, so that they and their squares lie within FP32 whatever the
// case's unit of length is
__device__ __forceinline__ float list_coord(float x, float) { return x; }
__device__ __forceinline__ float list_coord(double x, double unit) { return (float)(x * unit); }

// Margin of the first test's r^2 against the cell walk's, of (2h)^2: it takes
// s_i - (s_j + o cs), with coordinates up to 2 cs <= 8/3 (2h) in FP32, which
// moves r^2 by less than 1.7e-6
constexpr float LIST_MARGIN = 4e-6f;

// tests nc staged candidates (a multiple of 32) against slot i and appends the
// hits to its shared list.  The first test settles all but the candidates
// within its margin of 2h or of 0; in FP32 those (about one in 10^5, and the
// slot's own particle) are tested by the cell walk's operations at once, in
// FP64 the caller tests all hits.  EXACT: every hit is tested so.
template <typename T, int D, bool MIXED, bool EXACT>
__device__ __forceinline__ void list_scan(const ListSmem &S, uint32_t *row, int K, int nc, const CasePhys<T> &cp,
                                          const V4<T> &si, T unit, uint32_t i, uint32_t ki, float R2, const V4<T> *snap,
                                          uint32_t &c_rest, uint32_t &c_other, bool &coinc) {
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const float sx = list_coord(si.x, unit), sy = list_coord(si.y, unit), sz = list_coord(si.z, unit);
    const float R2w = R2 * (1.0f + LIST_MARGIN), mid = R2 * 0.5f, half = mid * (1.0f - 2.0f * LIST_MARGIN);
    uint32_t cr = c_rest, co = c_other;
#pragma unroll 3
    for (int q = 0; q < nc; q += 32) {
        const float4 s = S.cand[q + lane];
        const float r2 = norm2<float, D>(sub_rn(sx, s.x), sub_rn(sy, s.y), D == 3 ? sub_rn(sz, s.z) : 0.0f);
        const uint32_t e = __float_as_uint(s.w);
        bool hit = r2 < R2w;
        if (EXACT) {
            hit = hit && list_exact<T, D>(e, cp, si, i, snap, coinc);
        } else if (sizeof(T) == 4) {
            const bool open = hit && !(fabsf(r2 - mid) < half);
            if (__any_sync(0xffffffffu, open)) {
                if (open) hit = (e >> NBR_SHIFT) != i && list_exact<T, D>(e, cp, si, i, snap, coinc);
                __syncwarp();
            }
        }
        const unsigned h = __ballot_sync(0xffffffffu, hit);
        if (MIXED) {
            const unsigned ho = h & S.fluid[ki ^ 1u][q >> 5], hr = h & ~ho;
            const uint32_t nr = (uint32_t)__popc(hr), no = (uint32_t)__popc(ho);
            const uint32_t at = (ho >> lane) & 1u ? K - 1 - (co + __popc(ho & below)) : cr + __popc(hr & below);
            if (hit && cr + nr + co + no <= (uint32_t)K) row[at] = e;
            cr += nr;
            co += no;
        } else {
            const uint32_t at = cr + __popc(h & below);
            if (hit && at + co < (uint32_t)K) row[at] = e;
            cr += (uint32_t)__popc(h);
        }
    }
    __syncwarp();
    c_rest = cr;
    c_other = co;
}

template <typename T, int D>
__device__ __forceinline__ void build_cell(const CaseDesc &d, const CasePhys<T> &cp, uint32_t b, ListSmem &S,
                                           const uint32_t *starts, const uint32_t *rank, const uint32_t *fidx,
                                           const V4<T> *snap, uint32_t *nbr, uint32_t *cnt, uint8_t *band,
                                           int32_t *status) {
    constexpr int NC = D == 3 ? 27 : 9;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int K = d.nbr_k, LS = K + 1, G = lb_group(K);
    const uint32_t pk = w_bits(snap[b].w), m = (uint32_t)d.table_off + morton_of_packed<D>(pk);
    const uint32_t f0 = rank[b], f1 = rank[starts[m + 1]];
    __syncthreads();                            // the previous cell's shared data is done with
    if (warp == 0) {
        // the 3^D cells around, one per lane, in increasing table index
        uint32_t mq = 0xffffffffu, bq = 0, nq = 0, code = 0;
        if (lane < NC) {
            const int ox = lane % 3 - 1, oy = lane / 3 % 3 - 1, oz = D == 3 ? lane / 9 - 1 : 0;
            int nx = cell_x<D>(pk) + ox, ny = cell_y<D>(pk) + oy, nz = cell_z<D>(pk) + oz;
            if (wrap_cell(d, 0, nx) && wrap_cell(d, 1, ny) && (D == 2 || wrap_cell(d, 2, nz))) {
                mq = (uint32_t)d.table_off + morton<D>(nx, ny, nz);
                bq = starts[mq];
                nq = starts[mq + 1] - bq;
                code = cell_code<D>(ox, oy, oz);
            }
        }
        int place = 0;
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            const uint32_t o = __shfl_sync(0xffffffffu, mq, q);
            place += o < mq || (o == mq && q < lane);
        }
        if (lane < NC) { S.begin[place] = bq; S.pre[place] = nq; S.code[place] = code; }
        __syncwarp();
        const uint32_t own = lane < NC ? S.pre[lane] : 0u;
        uint32_t x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        __syncwarp();
        S.pre[lane] = x - own;                  // candidates before cell `lane`
        if (lane == 31) S.pre[32] = x;          // all of them
    }
    __syncthreads();
    const uint32_t total = S.pre[32];
    const T unit = sizeof(T) == 8 ? (T)d.list_unit : T(1);
    const float R2 = (float)(cp.four_h2 * unit * unit);
    bool coinc = false, overflow = false, has0 = false, has1 = false;
    for (uint32_t g0 = f0; g0 < f1; g0 += G) {
        const int ns = (int)min((uint32_t)G, f1 - g0);
        // a group with a list that does not fit is built again with every hit
        // tested by the cell walk's operations: only what they count overflows
        bool exact = false;
    again:
        bool full = false;
        for (uint32_t c0 = 0; c0 < total; c0 += LB_CAND) {
            const int nc = ((int)min((uint32_t)LB_CAND, total - c0) + 31) / 32 * 32;
            if ((g0 == f0 && !exact) || total > LB_CAND) {
                __syncthreads();
                bool p0 = false, p1 = false;
                for (int q = threadIdx.x; q < nc; q += LB_WARPS * 32) {
                    const uint32_t t = c0 + q;
                    float4 s = make_float4(CUDART_NAN_F, CUDART_NAN_F, CUDART_NAN_F, 0.0f);   // near no slot
                    uint32_t pj = PH_WALL;
                    if (t < total) {
                        int cell = 0;
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1)
                            if (cell + o < NC && S.pre[cell + o] <= t) cell += o;
                        const uint32_t j = S.begin[cell] + (t - S.pre[cell]), cj = S.code[cell];
                        const V4<T> sj = ld4(snap + j);
                        pj = phase_of(w_bits(sj.w));
                        s.x = list_coord(fma_rn(code_off(cj & 3u, T()), cp.cs, sj.x), unit);
                        s.y = list_coord(fma_rn(code_off((cj >> 2) & 3u, T()), cp.cs, sj.y), unit);
                        if (D == 3) s.z = list_coord(fma_rn(code_off((cj >> 4) & 3u, T()), cp.cs, sj.z), unit);
                        s.w = __uint_as_float((j << NBR_SHIFT) | cj);
                    }
                    S.cand[q] = s;
                    const unsigned m0 = __ballot_sync(0xffffffffu, pj == 0), m1 = __ballot_sync(0xffffffffu, pj == 1);
                    if (lane == 0) { S.fluid[0][q >> 5] = m0; S.fluid[1][q >> 5] = m1; }
                    p0 |= m0 != 0;
                    p1 |= m1 != 0;
                }
                has0 = __syncthreads_or(p0);
                has1 = __syncthreads_or(p1);
            }
            for (int s = warp; s < ns; s += LB_WARPS) {
                const uint32_t i = fidx[g0 + s];
                const V4<T> si = ld4(snap + i);
                const uint32_t ki = phase_of(w_bits(si.w));
                const bool mixed = ki == 0 ? has1 : has0;
                const uint32_t r0 = c0 ? S.rest[s] : 0u, o0 = c0 ? S.other[s] : 0u;
                uint32_t cr = r0, co = o0;
                uint32_t *row = S.list + s * LS;
                if (exact) {
                    list_scan<T, D, true, true>(S, row, K, nc, cp, si, unit, i, ki, R2, snap, cr, co, coinc);
                } else {
                    if (mixed) list_scan<T, D, true, false>(S, row, K, nc, cp, si, unit, i, ki, R2, snap, cr, co, coinc);
                    else list_scan<T, D, false, false>(S, row, K, nc, cp, si, unit, i, ki, R2, snap, cr, co, coinc);
                    if (sizeof(T) == 8 && cr + co <= (uint32_t)K) {
                        cr = r0 + list_keep<T, D>(row, (int)r0, 1, cr - r0, cp, si, i, snap, coinc);
                        if (co > o0) co = o0 + list_keep<T, D>(row, K - 1 - (int)o0, -1, co - o0, cp, si, i, snap, coinc);
                    }
                }
                full |= cr + co > (uint32_t)K;
                if (lane == 0) { S.idx[s] = i; S.rest[s] = cr; S.other[s] = co; }
            }
        }
        if (__syncthreads_or(full) && !exact) {
            exact = true;
            goto again;
        }
        // rows of 32 slots; a slot with more neighbours than its list holds
        // keeps none (its case stops).  A particle with neighbours of the
        // other fluid and all its neighbours form the interface band
        const int s = lane;
        if (s < ns) {
            uint32_t co = S.other[s], c = S.rest[s] + co;
            if (c > (uint32_t)K) {
                overflow = true;
                c = co = 0;
            }
            const uint32_t *src = S.list + s * LS;
            if (warp == 0) {
                cnt[g0 + s] = c | (co << 16);
                if (co) band[S.idx[s]] = 1;
            }
            uint32_t *dst = nbr + list_word(d, (int64_t)g0 + s);
            for (uint32_t k = warp; k < c; k += LB_WARPS) {
                const uint32_t e = src[k < co ? K - 1 - k : k - co];
                dst[k * LROW] = e;
                if (co) band[e >> NBR_SHIFT] = 1;
            }
        }
        __syncthreads();
    }
    if (coinc) atomicCAS(status, 0, DEV_ERR_COINCIDENT);
    if (overflow) atomicCAS(status, 0, DEV_ERR_NBR_OVERFLOW);
}

template <typename T, int D>
__global__ void __launch_bounds__(LB_WARPS * 32) k_build_list(SweepArgs a, const uint64_t *clist, const uint32_t *ccount,
                                                              const uint32_t *rank, const V4<T> *snap,
                                                              uint32_t *nbr, uint32_t *cnt, uint8_t *band) {
    follow();
    __shared__ ListSmem S;
    const uint32_t cells = *ccount;
    for (uint32_t e = blockIdx.x; e < cells; e += gridDim.x) {
        const uint64_t cm = clist[e];
        const int c = (int)(cm >> 32);
        if (!a.st[c].active) continue;          // uniform per block
        const CaseDesc &d = a.desc[c];
        build_cell<T, D>(d, phys<T>(d), (uint32_t)cm, S, a.starts, rank, a.fidx, snap, nbr, cnt, band, &a.st[c].status);
    }
}

// ---- interface band of the frozen configuration: the list build has marked
// the particles that have neighbours of the other fluid phase and all their
// neighbours.  The marked fluid particles are appended, as
// (case << 32 | slot), to the class's list that the surface and colour sweeps
// walk (warp-aggregated atomics; the order is irrelevant because every
// particle's sum is its own).
static __global__ void __launch_bounds__(256) k_band(SweepArgs a, const uint8_t *band, uint64_t *blist, uint32_t *bcount) {
    follow();
    const Tile t = a.tiles[a.tile0 + blockIdx.x];
    const int64_t q = t.begin + threadIdx.x;
    const bool b = (int)threadIdx.x < t.n && a.st[t.c].active && band[particle_at(a, q)];
    const unsigned m = __ballot_sync(0xffffffffu, b);
    if (!m) return;
    const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(bcount, (uint32_t)__popc(m));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (b) blist[base + __popc(m & ((1u << lane) - 1u))] = ((uint64_t)(uint32_t)t.c << 32) | (uint64_t)(uint32_t)q;
}

// ---- G: the stored geometry of the lists (FP64), once per advection step.  A
// block takes a tile's slots 32 at a time, its warps the rows.  FP64 sweeps
// are bound by their arithmetic (2 FP64 lanes per clock and SM), of which the
// pair geometry is half: 26 of 59 operations in B, of 49 in C; reading 32 bytes
// per pair instead costs 1/10 of that time.
constexpr int LG_WARPS = 8;
template <int D>
__global__ void __launch_bounds__(32 * LG_WARPS) k_list_geo(SweepArgs a, const V4<double> *snap, V4<double> *ge, RInv *gr) {
    follow();
    const Tile t = a.tiles[a.tile0 + blockIdx.x];
    if (!a.st[t.c].active) return;
    const CaseDesc &d = a.desc[t.c];
    if (d.geo_base < 0) return;
    const CasePhys<double> &cp = d.pd;
    ge += d.geo_base - d.nbr_base;
    gr += d.geo_base - d.nbr_base;
    for (int s = threadIdx.x; s < t.n; s += 32) {
        const int64_t q = t.begin + s, i = particle_at(a, q), w = list_word(d, q);
        const V4<double> si = ld4(snap + i);
        const uint32_t c = a.cnt[q] & CNT_MASK;
        for (uint32_t k = threadIdx.y; k < c; k += LG_WARPS) {
            const int64_t at = w + (int64_t)k * LROW;
            const uint32_t e = ld_list(a.nbr + at);
            const V4<double> sj = ld4(snap + (e >> NBR_SHIFT));
            double rx, ry, rz;
            moved_offset<double, D>(e, si, sj, cp.cs, rx, ry, rz);
            const PairG<double> g(cp, rx, ry, rz, norm2<double, D>(rx, ry, rz), std::true_type());
            ge[at] = V4<double>{g.x, g.y, g.z, phase_of(w_bits(sj.w)) == PH_WALL ? fabs(g.wd) : g.wd};
            gr[at] = RInv{g.r, g.inv};
        }
    }
}

template <typename T, int D, bool LIST, int L = 1>
__global__ void SPH_SWEEP_BOUNDS k_sweep_M(SweepArgs a, const V4<T> *snap, const T *vol, V4<T> *bmat,
                                           V4<T> *bk) {
    follow();
    const Tile t = work_tile<L, false>(a, blockIdx.x);
    const int li = local_index<L>(blockIdx.x);
    if (li >= t.n || !a.st[t.c].active) return;
    const CaseDesc &d = a.desc[t.c];
    if (!d.tvf_on && d.surface_corr != 1) return;
    const CasePhys<T> &cp = phys<T>(d);
    const int64_t q = t.begin + li, i = particle_at(a, q);
    sweep_M<LIST, T, D, L>(d, cp, i, a.starts, list_of<LIST, T>(a, d, q), snap, vol, bmat, bk, &a.st[t.c].status, threadIdx.x % L);
}

template <typename T, int D, bool LIST, int L = 1>
__global__ void SPH_SWEEP_BOUNDS k_sweep_V(SweepArgs a, const V4<T> *snap, const V4<T> *vel, const T *vol,
                                           const V4<T> *bmat, V4<T> *acc_visc, V4<T> *pos) {
    follow();
    const Tile t = work_tile<L, false>(a, blockIdx.x);
    const int li = local_index<L>(blockIdx.x);
    if (li >= t.n || !a.st[t.c].active) return;
    const CaseDesc &d = a.desc[t.c];
    Phys<LIST, MODE_TILES, T> cp = phys<T>(d);
    const int64_t q = t.begin + li, i = particle_at(a, q);
    sweep_V<LIST, T, D, L>(d, cp, i, a.starts, list_of<LIST, T>(a, d, q), snap, vel, vol, bmat, acc_visc, pos,
                        &a.st[t.c].status, threadIdx.x % L);
}

// Sweeps B and C (and A with the cell walk) take L lanes per particle (L = 1,
// 2, 4, 8; list classes): L blocks share one tile, block b takes its part
// b % L of blockDim / L particles, and lane threadIdx % L of a particle's
// group walks every L-th list entry.  local_index gives the particle's index
// within its tile.  Sweeps S and A of the list classes do the same per entry
// of their band list.

template <typename T, int D, bool LIST, int L = 1, int MODE = MODE_TILES>
__global__ void SPH_SWEEPAS_BOUNDS k_sweep_A(SweepArgs a, const V4<T> *snap, const T *vol, V4<T> *gradC) {
    follow();
    const auto item = [&](int64_t w) {
        const Tile t = work_tile<L, MODE == MODE_WORK>(a, w);
        const int li = local_index<L>(w);
        if (li >= t.n || !a.st[t.c].active) return;
        const CaseDesc &d = case_desc<MODE>(a, t.c);
        Phys<LIST, MODE, T> cp = phys<T>(d);
        const int64_t q = t.begin + li, i = particle_at(a, q);
        sweep_A<LIST, T, D, L>(d, cp, i, a.starts, list_of<LIST, T>(a, d, q), snap, vol, gradC,
                               threadIdx.x % L);
    };
    if constexpr (MODE == MODE_WORK) {
        const int64_t items = work_items<L, true>(a);
        for (int64_t w = blockIdx.x; w < items; w += gridDim.x) item(w);
    } else {
        item(blockIdx.x);
    }
}

// colour gradient of the band particles (list classes): one thread (L lanes)
// per entry of the class's compacted band list, as in S; the launch's
// threads stride over the list (the grid is a few blocks per SM, since the
// list's length is known only on the device).  A particle outside
// the band has no neighbour of the other fluid, so its colour gradient is the
// zero written at the start of the advection step.
template <typename T, int D, int L = 1>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 1 : 4) k_sweep_A_band(SweepArgs a, const uint64_t *blist, const uint32_t *bcount,
                                                const V4<T> *snap, const T *vol, V4<T> *gradC) {
    follow();
    const int64_t items = (int64_t)*bcount * L;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < items; t += (int64_t)gridDim.x * blockDim.x) {
        const BandEntry e(a, blist, t / L);
        if (!a.st[e.c].active) continue;
        const CaseDesc &d = a.desc[e.c];
        const CasePhys<T> cp = phys<T>(d);
        sweep_A<true, T, D, L, AHEAD>(d, cp, e.i, a.starts, list_of<true, T>(a, d, e.q), snap, vol, gradC, threadIdx.x % L);
    }
}

// surface sum of the band particles (list classes only), before B: one
// thread (L lanes) per entry of the class's compacted band list, so warps
// are full of band particles; the threads stride over the list (a group of
// L lanes stays together: the stride is a multiple of L)
template <typename T, int D, int L = 1>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 1 : 2) k_sweep_S(SweepArgs a, const uint64_t *blist, const uint32_t *bcount,
                                           const uint8_t *band, const V4<T> *snap, const V4<T> *vel,
                                           const V4<T> *gradC, V4<T> *acc_surf, const V4<T> *bk, const T *vol) {
    follow();
    const int64_t items = (int64_t)*bcount * L;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < items; t += (int64_t)gridDim.x * blockDim.x) {
        const BandEntry e(a, blist, t / L);
        if (!a.st[e.c].active) continue;
        const CaseDesc &d = a.desc[e.c];
        const CasePhys<T> cp = phys<T>(d);
        uint32_t ph;
        sweep_B<true, 2, T, D, L, 4>(d, cp, T(0), e.i, a.starts, list_of<true, T>(a, d, e.q), band, snap, vel, gradC,
                                          nullptr, acc_surf, nullptr, &ph, threadIdx.x % L, bk, vol);
    }
}

// largest |v|^2 (its bits) per fluid of a block's case; all threads of a warp
// take part
__device__ __forceinline__ void reduce_vmax(const SweepArgs &a, int c, uint32_t ph, unsigned long long v2) {
    unsigned long long m0 = ph == 0 ? v2 : 0ull, m1 = ph == 1 ? v2 : 0ull;
    m0 = warp_max_u64(m0);
    m1 = warp_max_u64(m1);
    if ((threadIdx.x & 31) == 0) {
        if (m0) atomicMax(&a.st[c].vmax2_acc[0], m0);
        if (m1) atomicMax(&a.st[c].vmax2_acc[1], m1);
    }
}

template <typename T, int D, bool LIST, int L = 1, int MODE = MODE_TILES>
__global__ void SPH_SWEEPB_BOUNDS_M(T, LIST, L, MODE) k_sweep_B(SweepArgs a, const uint8_t *band, const V4<T> *snap, const V4<T> *vel,
                                            const V4<T> *gradC, const V4<T> *acc_visc, V4<T> *acc_surf,
                                            V4<T> *vel_new, const V4<T> *bk, const T *vol) {
    follow();
    const auto item = [&](int64_t w) {
        const Tile t = work_tile<L, MODE == MODE_WORK>(a, w);
        if (!a.st[t.c].active) return;             // uniform per block
        const CaseDesc &d = case_desc<MODE>(a, t.c);
        double v2 = 0.0;
        uint32_t ph = PH_WALL;
        const int li = local_index<L>(w);
        if (li < t.n) {
            Phys<LIST, MODE, T> cp = phys<T>(d);
            const int64_t q = t.begin + li, i = particle_at(a, q);
            const T dt = (T)a.st[t.c].dt;
            v2 = sweep_B<LIST, LIST ? 1 : 0, T, D, L, MODE == MODE_FEW ? 4 : PLAIN>(d, cp, dt, i, a.starts, list_of<LIST, T>(a, d, q), band, snap, vel,
                                                      gradC, acc_visc, acc_surf, vel_new, &ph, threadIdx.x % L,
                                                      LIST ? nullptr : bk, vol);
        }
        reduce_vmax(a, t.c, ph, (unsigned long long)__double_as_longlong(v2));
    };
    if constexpr (MODE == MODE_WORK) {
        const int64_t items = work_items<L, true>(a);
        for (int64_t w = blockIdx.x; w < items; w += gridDim.x) item(w);
    } else {
        item(blockIdx.x);
    }
}

template <typename T, int D, bool LIST, int L = 1, int MODE = MODE_TILES>
__global__ void SPH_SWEEPC_BOUNDS_M(T, D, LIST, L, MODE) k_sweep_C(SweepArgs a, const V4<T> *snap, const V4<T> *vel_new, T *drho, T *vol,
                                           V4<T> *vel, V4<T> *pos) {
    follow();
    const auto item = [&](int64_t w) {
        const Tile t = work_tile<L, MODE == MODE_WORK>(a, w);
        const int li = local_index<L>(w);
        if (li >= t.n || !a.st[t.c].active) return;
        const CaseDesc &d = case_desc<MODE>(a, t.c);
        Phys<LIST, MODE, T> cp = phys<T>(d);
        const int64_t q = t.begin + li, i = particle_at(a, q);
        const T dt = (T)a.st[t.c].dt;
        sweep_C<LIST, T, D, L, MODE == MODE_FEW && D == 2 ? 4 : AHEAD>(d, cp, dt, i, a.starts, list_of<LIST, T>(a, d, q),
                               snap, vel_new, drho, vol, vel, pos,
                               threadIdx.x % L);
    };
    if constexpr (MODE == MODE_WORK) {
        const int64_t items = work_items<L, true>(a);
        for (int64_t w = blockIdx.x; w < items; w += gridDim.x) item(w);
    } else {
        item(blockIdx.x);
    }
}

// ---- work lists of the per-substep sweeps in a batch: after the criterion
// kernel has set each case's active flag, the fluid tiles of the active
// cases are listed per class.  Scan (one block): case c's tiles go to
// positions off[c] .. off[c] + ftn[c] - 1 of its class's list, and
// count[k] receives the length of class k's list.  Fill: every fluid tile of
// an active case writes its index there.  Tiles of class k start at cls0[k]
// in the tile array and in the list alike.
static __global__ void k_work_scan(int ncases, const int32_t *cls_of, const uint32_t *ftn, const CaseState *st,
                                   uint32_t *off, uint32_t *count) {
    lead();
    follow();
    uint32_t base[4] = {0u, 0u, 0u, 0u};
    for (int c0 = 0; c0 < ncases; c0 += (int)blockDim.x) {
        const int c = c0 + (int)threadIdx.x;
        const int k = c < ncases ? cls_of[c] : -1;
        const uint32_t n = c < ncases && st[c].active ? ftn[c] : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t total;
            const uint32_t before = block_exclusive_scan(k == q ? n : 0u, &total);
            if (k == q) off[c] = base[q] + before;
            base[q] += total;
        }
    }
    if (threadIdx.x < 4) count[threadIdx.x] = base[threadIdx.x];
}
static __global__ void k_work_fill(int64_t n_ftiles, const Tile *ftiles, const int64_t *ft_first,
                                   const int64_t *cls0, const int32_t *cls_of, const uint32_t *off,
                                   const CaseState *st, uint32_t *work) {
    follow();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n_ftiles) return;
    const int c = ftiles[t].c;
    if (!st[c].active) return;
    work[cls0[cls_of[c]] + off[c] + (t - ft_first[c])] = (uint32_t)t;
}

// ---------------------------------------------------------- diagnostics
// FP64 sums over one case's fluid particles: per-block partials (warp
// shuffles, then the block's warps in order), then one block adds the
// partials in block order, so the result does not depend on scheduling.
// Quantities: 0-2 momentum, 3 kinetic, 4-5 count per phase, 6-8 first
// moments, 9-14 second moments, 15 p_in, 16 p_out, 17 n_in, 18 n_out,
// 19 non-finite count.

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

template <typename T>
__global__ void __launch_bounds__(256) k_diag_partial(const CaseDesc *desc, int c, const V4<T> *pos,
                                                      const V4<T> *vel, const T *drho, double cx, double cy,
                                                      double cz, double r_in2, double r_out2, double *partial) {
    const CaseDesc &d = desc[c];
    const int64_t n = d.p_end - d.p_begin;
    const int dim = d.dim;
    double q[DIAG_Q];
#pragma unroll
    for (int k = 0; k < DIAG_Q; ++k) q[k] = 0.0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = d.p_begin + k;
        const V4<T> p = pos[i];
        const uint32_t pk = w_bits(p.w);
        const uint32_t ph = phase_of(pk);
        if (ph > 1) continue;
        const int cc[3] = {dim == 3 ? cell_x<3>(pk) : cell_x<2>(pk), dim == 3 ? cell_y<3>(pk) : cell_y<2>(pk),
                           dim == 3 ? cell_z<3>(pk) : 0};
        const double off[3] = {(double)p.x, (double)p.y, (double)p.z};
        double x[3] = {0.0, 0.0, 0.0};
        for (int a = 0; a < dim; ++a) x[a] = d.origin[a] + (double)cc[a] * d.cs + off[a];
        const V4<T> v4 = vel[i];
        const double v[3] = {(double)v4.x, (double)v4.y, dim == 3 ? (double)v4.z : 0.0};
        const double dr = (double)drho[i];
        const double m = d.mass[ph];
        const bool finite = isfinite(x[0]) && isfinite(x[1]) && isfinite(x[2]) && isfinite(v[0]) &&
                            isfinite(v[1]) && isfinite(v[2]) && isfinite(dr);
        if (!finite) { q[19] += 1.0; continue; }
        q[0] += m * v[0]; q[1] += m * v[1]; q[2] += m * v[2];
        q[3] += 0.5 * m * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
        q[4 + ph] += 1.0;
        const double rx = x[0] - cx, ry = x[1] - cy, rz = dim == 3 ? x[2] - cz : 0.0;
        const double r2 = rx * rx + ry * ry + rz * rz;
        const double pr = d.c0 * d.c0 * dr;
        if (ph == 0) {
            q[6] += x[0]; q[7] += x[1]; q[8] += x[2];
            q[9] += x[0] * x[0]; q[10] += x[1] * x[1]; q[11] += x[2] * x[2];
            q[12] += x[0] * x[1]; q[13] += x[0] * x[2]; q[14] += x[1] * x[2];
            if (r2 < r_in2) { q[15] += pr; q[17] += 1.0; }
        } else if (r2 > r_out2) {
            q[16] += pr; q[18] += 1.0;
        }
    }
    __shared__ double sh[8][DIAG_Q];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < DIAG_Q; ++k) {
        const double t = warp_sum_d(q[k]);
        if (lane == 0) sh[w][k] = t;
    }
    __syncthreads();
    if (threadIdx.x < DIAG_Q) {
        double t = 0.0;
        for (int ww = 0; ww < (int)(blockDim.x >> 5); ++ww) t += sh[ww][threadIdx.x];
        partial[(int64_t)blockIdx.x * DIAG_Q + threadIdx.x] = t;
    }
}

static __global__ void k_diag_final(const double *partial, int nblocks, double *out) {
    if (threadIdx.x < DIAG_Q) {
        double t = 0.0;
        for (int b = 0; b < nblocks; ++b) t += partial[(int64_t)b * DIAG_Q + threadIdx.x];
        out[threadIdx.x] = t;
    }
}

// ------------------------------------------------------------ read-back
// field values of one case into a device buffer in insertion order (FP64)
template <typename T>
__global__ void k_read_field(const CaseDesc *desc, int c, int field, const V4<T> *pos,
                             const V4<T> *vel, const T *drho, const V4<T> *gradC,
                             const V4<T> *acc_visc, const uint32_t *id, double *out) {
    const CaseDesc &d = desc[c];
    const int64_t n = d.p_end - d.p_begin;
    const int dim = d.dim;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = d.p_begin + k;
        const int64_t o = id[i];
        const V4<T> p = pos[i];
        const uint32_t pk = w_bits(p.w);
        const uint32_t ph = phase_of(pk);
        switch (field) {
        case 0: {
            const int cc[3] = {dim == 3 ? cell_x<3>(pk) : cell_x<2>(pk),
                               dim == 3 ? cell_y<3>(pk) : cell_y<2>(pk),
                               dim == 3 ? cell_z<3>(pk) : 0};
            const double off[3] = {(double)p.x, (double)p.y, (double)p.z};
            for (int a = 0; a < dim; ++a)
                out[o * dim + a] = d.origin[a] + (double)cc[a] * d.cs + off[a];
            break;
        }
        case 1: {
            const V4<T> v = vel[i];
            const double vv[3] = {(double)v.x, (double)v.y, (double)v.z};
            for (int a = 0; a < dim; ++a) out[o * dim + a] = vv[a];
            break;
        }
        case 2: out[o] = ph < 2 ? d.rho0[ph] + (double)drho[i] : d.rho0[0]; break;
        case 3: out[o] = ph < 2 ? d.c0 * d.c0 * (double)drho[i] : 0.0; break;
        case 5: {
            const V4<T> g = gradC[i];
            const double gg[3] = {(double)g.x, (double)g.y, (double)g.z};   // unit vector; w the magnitude
            for (int a = 0; a < dim; ++a) out[o * dim + a] = (double)g.w * gg[a];
            break;
        }
        case 6: {
            const V4<T> g = acc_visc[i];
            const double gg[3] = {(double)g.x, (double)g.y, (double)g.z};
            for (int a = 0; a < dim; ++a) out[o * dim + a] = gg[a];
            break;
        }
        default: break;
        }
    }
}

// Morton key (from the packed cell of the last rebuild) and insertion id of
// every particle of case c in device order
template <typename T>
__global__ void k_debug_keys(const CaseDesc *desc, int c, const V4<T> *snap, const uint32_t *id,
                             unsigned long long *keys, long long *ids) {
    const CaseDesc &d = desc[c];
    const int64_t n = d.p_end - d.p_begin;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = d.p_begin + k;
        const uint32_t pk = w_bits(snap[i].w);
        keys[k] = d.dim == 3 ? morton_of_packed<3>(pk) : morton_of_packed<2>(pk);
        ids[k] = id[i];
    }
}

template <typename T, int D>
__device__ void count_nbrs(const CaseDesc &d, int64_t i, const uint32_t *starts, const V4<T> *snap,
                           const uint32_t *id, int *out) {
    const V4<T> si = ld4(snap + i);
    int cnt = 0;
    walk<false, T, D>(d, phys<T>(d), starts, snap, i, si, w_bits(si.w),
               [&](uint32_t, const V4<T> &, T, T, T, T) { ++cnt; }, Nothing());
    out[id[i]] = cnt;
}

template <typename T>
__global__ void k_debug_counts(const CaseDesc *desc, int c, const uint32_t *starts,
                               const V4<T> *snap, const uint32_t *id, int *out) {
    const CaseDesc &d = desc[c];
    const int64_t n = d.p_end - d.p_begin;
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n) return;
    if (d.dim == 3) count_nbrs<T, 3>(d, d.p_begin + k, starts, snap, id, out);
    else count_nbrs<T, 2>(d, d.p_begin + k, starts, snap, id, out);
}

// neighbours of case c's fluid particles as the sweeps find them (its lists,
// or the cell walk), by insertion index: counts and the first `width` of each
template <typename T, int D, bool LIST, int L = 1>
__global__ void __launch_bounds__(256) k_debug_neighbors(SweepArgs a, int c, const V4<T> *snap, const uint32_t *id, int64_t width,
                                                         int *counts, long long *ids) {
    follow();
    const Tile t = work_tile<L, false>(a, blockIdx.x);
    const int li = local_index<L>(blockIdx.x);
    if (li >= t.n || t.c != c) return;
    const CaseDesc &d = a.desc[c];
    const int64_t q = t.begin + li, i = particle_at(a, q), o = id[i];
    const V4<T> si = ld4(snap + i);
    neighbors<LIST, false, false, T, D, PART_ALL, L, PLAIN, CELL_PLACES_k_debug_neighbors>(
        d, phys<T>(d), a.starts, list_of<LIST, T>(a, d, q), snap, nullptr, i, si, w_bits(si.w),
        [&](uint32_t j, uint32_t, const V4<T> &, const PairG<T> &) {
            const int k = atomicAdd(counts + o, 1);
            if (k < width) ids[o * width + k] = id[j];
        }, threadIdx.x % L);
}

}  // namespace sphst
