// kernels.cuh -- CUDA kernels of one MTPT time step (Sec. 3) for sm_103a.
//
// GB300 issues every binary64 instruction (arithmetic, compares, f32<->f64
// conversions) at about 1/70 of the binary32 rate, so the kernels keep
// binary64 to the operations whose results must match the binary64 method
// bit for bit (the walk's x + sigma xi, and the pair test inside a narrow
// band around the cutoff) or carry the binary64 form's accuracy (its pair
// terms and sums), and do everything else in binary32 and integer
// arithmetic.
//
// Data layout (structure of arrays, `stride` = capacity >= n):
//   pos[a * stride + s]  binary64 coordinates, particles in cell order
//   mass[s], id[s]       binary64 mass, uint32 input index (keys the walk)
//   cell[s]              linear cell index of particle s (written and read in 3-d
//                        only: below 3-d the record carries the cell coordinates)
//   rec (load_rec)       float4: binary32 offsets of the particle from its
//                        cell's lower corner (x, y, z), and in .w the cell's
//                        x index (a small integer, exact in binary32); in
//                        2-d, .z (no offset there) holds the cell's y index.
//                        Stored two particles a 32-byte block, component by
//                        component: {x0 x1 w0 w1 y0 y1 z0 z1}
//   start[c]             first particle of cell c (exclusive prefix sum)
// Cells are row-major (x fastest), so the three cells (cx-1..cx+1) of one
// neighbour row are one contiguous particle range; inside a cell particles
// are ordered by x (then id), so that range is sorted by x up to rounding.
#pragma once
#include <cstdint>
#include <type_traits>

#include "expneg.cuh"
#include "rng.cuh"

namespace mtpt {

enum : uint32_t { kStatusNonFinite = 1u, kStatusOutOfDomain = 2u };

// Generator ids are below 2^31; a tile marks its ghost copies of other tiles'
// particles with this bit (see tiles.cuh).
constexpr uint32_t kGhostBit = 0x80000000u;

// Bounds-checked build (compiled with -DMTPT_CHECKED; the tests load it as a
// second library): index invariants that hold by construction are verified at
// run time; a violation sets its bit in a device word and the access is
// skipped.  The normal build compiles every check to `true`.
enum : uint32_t {
    kChkCell = 1u,       // walk: cell index inside the realisation's cells
    kChkSlot = 2u,       // scatter: counting-sort slot inside [0, n)
    kChkGather = 4u,     // gather: source and in-cell rank inside the cell's range
    kChkRow = 8u,        // pair search: neighbour row inside the realisation's cells
    kChkSegment = 16u,   // dense pair passes: a particle's words hold all its neighbours
    kChkOutput = 32u,    // outputs: particle id inside [0, n)
};
#ifdef MTPT_CHECKED
__device__ uint32_t g_check_word;
__device__ __forceinline__ bool check(bool ok, uint32_t bit) {
    if (!ok) atomicOr(&g_check_word, bit);
    return ok;
}
#else
__device__ __forceinline__ constexpr bool check(bool, uint32_t) { return true; }
#endif

constexpr int kBlock = 256;
constexpr int kScanThreads = 1024;
constexpr int kScanPerThread = 16;                        // cells per scan thread
constexpr int kScanTile = kScanPerThread * kScanThreads;  // cells per scan block

// The kernels of a time step are launched with programmatic stream
// serialisation (`launch` in mtpt.cu): a kernel may be set up, and its blocks
// may start, once the blocks of the kernel before it on the stream have ended,
// before that kernel is complete.  So each of them first waits until the one
// before is complete and its writes are visible, and only then touches memory.
// That takes the set-up of each launch out of the chain: one step of 1e4 particles
// and its two reads 55.7 -> 38 us (eight kernels), the adjoint's 200 steps of 250,000
// 44.5 -> 38.8 ms.
// (No griddepcontrol.launch_dependents: with the next kernel's blocks resident
// from the start of this one, a grid of two to six blocks an SM spread unevenly over
// the SMs: 36.7 instead of 30.7 us a step at 1e5 particles in 2-d, 49.4 instead of 39.9 in
// 3-d, precision form; the same within 1 % below 2e4 and above 4e5.)
// (after_previous itself is for kernels that only update a word in place: what is
// read through a pointer to const takes its index from ordered_index.)
__device__ __forceinline__ void after_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
// The thread's global index, after after_previous(): passing through the asm, it
// keeps every access that depends on it (loads without a memory clobber of their
// own too) behind the wait.
__device__ __forceinline__ uint32_t ordered_index() {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    asm volatile("griddepcontrol.wait;\n\tmov.b32 %0, %0;" : "+r"(i)::"memory");
    return i;
}

// Loads of what the kernels of a step write.  Such a kernel's lifetime overlaps
// the writer's, so the read-only path (ld.global.nc, __ldg, pointers to const
// declared __restrict__), which wants memory that stays the same for as long as
// the kernel lives, is for the constants of a run alone: the corner tables and the
// exponential's table.  These are ordinary loads, after the wait by their address.
__device__ __forceinline__ float ld_global(const float* p) {
    float v;
    asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 ld_global(const float2* p) {
    float2 v;
    asm("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ld_global(const float4* p) {
    float4 v;
    asm("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(p));
    return v;
}
__device__ __forceinline__ double ld_global(const double* p) {
    double v;
    asm("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 ld_global(const double2* p) {
    double2 v;
    asm("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_global(const uint32_t* p) {
    uint32_t v;
    asm("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ld_global(const uint2* p) {
    uint2 v;
    asm("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint64_t ld_global(const uint64_t* p) {
    uint64_t v;
    asm("ld.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

struct Box {
    double lo[3], hi[3];
    long long lo_key[3], hi_key[3];   // order-preserving integer images of lo, hi
};

struct Grid {
    int n[3];          // cells per axis of this grid (1 on unused axes)
    int nglob[3];      // cells per axis of the whole box's grid (equal to n unless
                       // the grid is one tile's part of it)
    int off[3];        // global index of this grid's first cell per axis (0 unless tiled)
    double lo[3];      // lower corner of the box
    double w[3];       // cell width per axis, >= psi
    double inv_w[3];   // 1 / w
    float wf[3];       // w rounded to binary32
    float lo_f[3];     // lo rounded to binary32 (binary32 cell index)
    float inv_w_f[3];  // 1 / w in binary32
    int cell_f32;      // 1: cell index from binary32 arithmetic (margin in w), 0: binary64
    int reach;         // cells a neighbour can be away per axis: 1 (w >= psi) or 2 (w >= psi / 2)
    int corner_off[3]; // offset of axis a's corner table in `corners`
};

struct PairParams {
    double psi2;       // cutoff squared: the exact binary64 test d2 <= psi2
    float band_lo;     // binary32 d2 below this: certainly a neighbour; >= +0 (pair_band)
    float band_hi;     // binary32 d2 above this: certainly not a neighbour
    float reach2;      // band_hi (1 + 2^-16): bounds dx^2 + dy^2 (+ dz^2) of a neighbour
    float trim_eps;    // slack of the per-row candidate windows (see for_each_row)
    double a;          // 1 / (2 h^2)
    float a_log2e;     // a * log2(e) in binary32 (precision form)
    double beta;
    KernelConsts kc;   // of the binary64 form's fixed-point kernel
};

// Everything one realisation's kernels need.  A single run passes one by
// value (SingleView); a batch of independent realisations keeps a table in
// device memory and a realisation index per particle (BatchView).
struct RealParams {
    Box box;
    Grid g;
    PairParams pp;
    double sigma;        // walk scale sqrt(2 D_RW dt)
    double kernel_norm;  // (2 pi h^2)^(-d/2)
    uint64_t seed;       // generator key of the walk
    uint32_t id_offset;  // first global particle index of the realisation
    uint32_t cell_base;  // first global cell of the realisation
    int32_t transfer;    // 1 when D_MT > 0 (pair passes run)
    int32_t walk;        // 1 when sigma > 0 or a velocity component is nonzero
    double vdt[3];       // v dt per axis (advection)
    uint32_t advect;     // bit a set when v[a] != 0
    double dsigma_dD;    // d sigma / dD = sigma / (2 D) (adjoint)
    double h2;           // 2 D_MT dt / beta (adjoint)
    double inv_2D;       // 1 / (2 D) (adjoint)
    double inv_h2;       // 1 / h^2 (adjoint)
};

struct SingleView {
    static constexpr bool kBatch = false;
    RealParams p;
    __device__ __forceinline__ const RealParams& of_input(uint32_t) const { return p; }
    __device__ __forceinline__ const RealParams& of_sorted(uint32_t) const { return p; }
};

struct BatchView {
    static constexpr bool kBatch = true;
    const RealParams* tbl;
    const uint32_t* rid_input;    // realisation of each particle before the sort
    const uint32_t* rid_sorted;   // realisation of each particle in cell order
    __device__ __forceinline__ const RealParams& of_input(uint32_t i) const {
        return tbl[ld_global(rid_input + i)];
    }
    __device__ __forceinline__ const RealParams& of_sorted(uint32_t s) const {
        return tbl[ld_global(rid_sorted + s)];
    }
};

// ---------------------------------------------------------------------------
// Integer helpers for binary64 values.
// ---------------------------------------------------------------------------

// Order-preserving image of a binary64 value in int64: for non-NaN x, y,
// key(x) < key(y) implies x <= y (-0 sorts below +0).
__device__ __forceinline__ long long order_key(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}

// A particle's record rec (see the layout above).
__device__ __forceinline__ size_t rec_at(uint32_t j) { return size_t(j & ~1u) * 4u + (j & 1u); }
__device__ __forceinline__ float4 load_rec(const float* rec, uint32_t j) {
    const float* q = rec + rec_at(j);
    return make_float4(ld_global(q), ld_global(q + 4), ld_global(q + 6), ld_global(q + 2));
}
__device__ __forceinline__ void store_rec(float* __restrict__ rec, uint32_t j, const float4& v) {
    float* q = rec + rec_at(j);
    q[0] = v.x;
    q[2] = v.w;
    q[4] = v.y;
    q[6] = v.z;
}

// Two binary32 values in one register pair, one operation on both: each rounds as the scalar one.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
    return v;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// The records of particles j and j + 1, j even, as one 32-byte load.
struct RecPair {
    uint64_t x, w, y, z;
};
__device__ __forceinline__ RecPair load_rec_pair(const float* rec, uint32_t j) {
    RecPair r;
    asm("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
        : "=l"(r.x), "=l"(r.w), "=l"(r.y), "=l"(r.z)
        : "l"(rec + size_t(j) * 4u));
    return r;
}

// x split as hi + lo with hi = x truncated to binary32 (integer operations
// only: no binary64 instruction) and lo the binary32 nearest to the exact
// remainder x - hi (|lo| < 2^-23 |x|).  Values below 2^-126 in magnitude give
// hi = lo = 0; |x| must be below 2^127.
__device__ __forceinline__ void split_double(double x, float* hi, float* lo) {
    const uint32_t whi = uint32_t(__double2hiint(x));
    const uint32_t wlo = uint32_t(__double2loint(x));
    const int e = int((whi >> 20) & 0x7ffu);
    const uint32_t sign = whi & 0x80000000u;
    if (e < 949) {   // |x| < 2^-74: residual below binary32's normal range
        *hi = e < 897 ? __uint_as_float(sign)
                      : __uint_as_float(sign | (uint32_t(e - 896) << 23) | ((whi & 0xfffffu) << 3) | (wlo >> 29));
        *lo = __uint_as_float(sign);
        return;
    }
    *hi = __uint_as_float(sign | (uint32_t(e - 896) << 23) | ((whi & 0xfffffu) << 3) | (wlo >> 29));
    const float m = __uint2float_rn(wlo & 0x1fffffffu);           // remainder mantissa
    const float scale = __uint_as_float(uint32_t(e - 948) << 23);  // 2^(e - 1075)
    *lo = __uint_as_float(__float_as_uint(__fmul_rn(m, scale)) | sign);
}

// Exact binary32 -> binary64 conversion by integer operations (no binary64
// pipe instruction) for zero and normal values; subnormal inputs take the
// hardware conversion.
__device__ __forceinline__ double f32_to_f64(float f) {
    const uint32_t b = __float_as_uint(f);
    const uint32_t sign = b & 0x80000000u;
    const uint32_t mag = b & 0x7fffffffu;
    if (mag == 0u) return __hiloint2double(int(sign), 0);
    const uint32_t e = mag >> 23;
    if (e == 0u || e == 255u) return double(f);
    const uint32_t m = mag & 0x7fffffu;
    return __hiloint2double(int(sign | ((e + 896u) << 20) | (m >> 3)), int(m << 29));
}

// True when x is an infinity or a NaN (integer test on the exponent field).
__device__ __forceinline__ bool not_finite(double x) {
    return (uint32_t(__double2hiint(x)) & 0x7ff00000u) == 0x7ff00000u;
}

// ---------------------------------------------------------------------------
// Step 1: random walk with reflecting walls, then the particle's cell.
// ---------------------------------------------------------------------------

// Elastic reflection in the walls lo and hi; more than 64 mirrors (a jump of
// over 64 box lengths) puts the coordinate on the nearest wall.
__device__ __forceinline__ double reflect(double x, double lo, double hi) {
    for (int it = 0; it < 64; ++it) {
        if (x < lo) x = __dsub_rn(__dmul_rn(2.0, lo), x);
        else if (x > hi) x = __dsub_rn(__dmul_rn(2.0, hi), x);
        else return x;
    }
    return x < lo ? lo : (x > hi ? hi : x);
}

// As reflect(), also reporting the derivative of the result with respect to
// the unreflected coordinate: -1 after an odd number of mirrors, +1 after an
// even number, 0 when the coordinate was put on a wall.
__device__ __forceinline__ double reflect_parity(double x, double lo, double hi, double* sign) {
    double sg = 1.0;
    for (int it = 0; it < 64; ++it) {
        if (x < lo) x = __dsub_rn(__dmul_rn(2.0, lo), x);
        else if (x > hi) x = __dsub_rn(__dmul_rn(2.0, hi), x);
        else { *sign = sg; return x; }
        sg = -sg;
    }
    *sign = 0.0;
    return x < lo ? lo : (x > hi ? hi : x);
}

__device__ __forceinline__ int clamp_cell(float u, int n) {
    // u is finite here; truncation equals floor for u >= 0
    return u <= 0.0f ? 0 : (u >= float(n - 1) ? n - 1 : int(u));
}

template <int DIM>
__device__ __forceinline__ uint32_t cell_of(const double* x, const Grid& g, bool* bad) {
    uint32_t lin = 0, mult = 1;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        int c = 0;
        if (g.cell_f32) {
            float hi, lo;
            split_double(x[a], &hi, &lo);
            const float u = __fmul_rn(__fsub_rn(hi, g.lo_f[a]), g.inv_w_f[a]);
            if (!not_finite(x[a])) c = clamp_cell(u, g.nglob[a]);
        } else {
            const double u = __dmul_rn(__dsub_rn(x[a], g.lo[a]), g.inv_w[a]);
            if (u == u) c = u <= 0.0 ? 0 : (u >= double(g.nglob[a] - 1) ? g.nglob[a] - 1 : __double2int_rz(u));
            else *bad = true;
        }
        // the whole box's cell index, then this grid's part of it
        c -= g.off[a];
        c = c < 0 ? 0 : (c >= g.n[a] ? g.n[a] - 1 : c);
        if (not_finite(x[a])) *bad = true;
        lin += uint32_t(c) * mult;
        mult *= uint32_t(g.n[a]);
    }
    return lin;
}

// One particle's move of the random walk (Sec. 3: x + sigma xi per axis,
// then the reflecting walls), in place on x[DIM].  With TANGENT, also
// carries the pathwise derivative of the positions with respect to D (tan,
// same layout as pos, particle i): the walk adds dsigma/dD xi and a mirror
// flips the sign, exactly as it maps the coordinate.  ADVECT compiles the
// velocity term in (launched when some realisation has v != 0), so the
// binary64 pipe of a walk without one carries only its two operations per
// axis.
template <int DIM, bool TANGENT, bool ADVECT>
__device__ __forceinline__ void walk_particle(const RealParams& P, uint32_t gen_id, uint64_t step,
                                              double* x, double* __restrict__ tan, int64_t stride,
                                              int i) {
    const float4 z4 = normals4(P.seed, gen_id, step);
    const float z[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const double za = f32_to_f64(z[a]);
        // move sigma xi, or v dt + sigma xi with a velocity on this axis
        double disp = __dmul_rn(P.sigma, za);
        if constexpr (ADVECT) {
            if (P.advect & (1u << a)) disp = __dadd_rn(P.vdt[a], disp);
        }
        double xv = __dadd_rn(x[a], disp);
        const long long k = order_key(xv);
        // strictly inside in the integer order => inside in binary64, no
        // mirror needed; anything else (walls, outside, NaN) takes the
        // binary64 reflection
        if constexpr (TANGENT) {
            double sign = 1.0;
            if (!(k > P.box.lo_key[a] && k < P.box.hi_key[a]))
                xv = reflect_parity(xv, P.box.lo[a], P.box.hi[a], &sign);
            const double t = __fma_rn(P.dsigma_dD, za, tan[a * stride + i]);
            tan[a * stride + i] = __dmul_rn(sign, t);
        } else {
            if (!(k > P.box.lo_key[a] && k < P.box.hi_key[a]))
                xv = reflect(xv, P.box.lo[a], P.box.hi[a]);
        }
        x[a] = xv;
    }
}

// The particle's cell (global index) into *key_out and its cell count; a
// coordinate that is not finite sets the status bit.
template <int DIM>
__device__ __forceinline__ void key_particle(const RealParams& P, const double* x,
                                             uint32_t* __restrict__ status,
                                             uint32_t* __restrict__ key_out,
                                             uint32_t* __restrict__ count) {
    bool bad = false;
    const uint32_t c = P.cell_base + cell_of<DIM>(x, P.g, &bad);
    if (bad) atomicOr(status, kStatusNonFinite);
    if (!check(c - P.cell_base < uint32_t(P.g.n[0]) * uint32_t(P.g.n[1]) * uint32_t(P.g.n[2]),
               kChkCell))
        return;
    *key_out = c;
    atomicAdd(&count[c], 1u);
}

// Step 1 over all particles, in place: the walk (with do_walk) and the
// cell keys and counts of the counting sort (with do_key).
template <int DIM, class View, bool TANGENT = false, bool ADVECT = false>
__global__ void __launch_bounds__(kBlock)
k_walk_key(int n, int64_t stride, double* __restrict__ pos, const uint32_t* id,
           const unsigned long long* step_dev, int do_walk, int do_key,
           const __grid_constant__ View v, uint32_t* __restrict__ key,
           uint32_t* __restrict__ count, uint32_t* __restrict__ status,
           double* __restrict__ tan = nullptr) {
    const int i = int(ordered_index());
    if (i >= n) return;
    const uint64_t step = ld_relaxed_u64(step_dev);   // (behind the wait)
    const RealParams& P = v.of_input(uint32_t(i));
    double x[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) x[a] = pos[a * stride + i];
    if (do_walk && P.walk) {
        walk_particle<DIM, TANGENT, ADVECT>(P, id[i] - P.id_offset, step, x, tan, stride, i);
#pragma unroll
        for (int a = 0; a < DIM; ++a) pos[a * stride + i] = x[a];
    }
    if (do_key) key_particle<DIM>(P, x, status, key + i, count);
}

// Check of host-loaded input in its device copy (positions dim x n with
// stride `stride`, masses n): a position outside its realisation's box
// [lo, hi] (NaN included) sets bit 1, a mass that is not finite or above
// mass_limit in magnitude sets bit 2.  box holds lo[3], hi[3] per
// realisation; first[k] is realisation k's first particle (first[nreal] = n).
// With id_out, also writes the particle ids 0..n-1 there.
template <int DIM>
__global__ void __launch_bounds__(kBlock)
k_check_input(int n, int64_t stride, int nreal, const double* __restrict__ pos,
              const double* __restrict__ mass, const double* __restrict__ box,
              const uint32_t* __restrict__ first, double mass_limit,
              uint32_t* __restrict__ flags, uint32_t* __restrict__ id_out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t bad = 0;
    if (i < n) {
        int k = 0;
        if (nreal > 1) {   // last k with first[k] <= i
            int lo = 0, hi = nreal - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (first[mid] <= uint32_t(i)) lo = mid; else hi = mid - 1;
            }
            k = lo;
        }
        const double* b = box + 6 * k;
        // integer tests only (the binary64 unit is slow): x inside [lo, hi]
        // through the order keys (a NaN fails the finiteness test), |m| <=
        // mass_limit through the magnitude bits (ordered like the values)
        // (-0 and +0 compare equal, so both map to key 0)
        auto key0 = [](double v) {
            return (__double_as_longlong(v) & 0x7fffffffffffffffLL) == 0 ? 0LL : order_key(v);
        };
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            const double x = pos[int64_t(a) * stride + i];
            const long long kx = key0(x);
            if (not_finite(x) || kx < key0(b[a]) || kx > key0(b[3 + a])) bad |= 1u;
        }
        const double m = mass[i];
        const long long mag = __double_as_longlong(m) & 0x7fffffffffffffffLL;
        if (not_finite(m) || mag > __double_as_longlong(mass_limit)) bad |= 2u;
        if (id_out) id_out[i] = uint32_t(i);
    }
    const uint32_t any = __reduce_or_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0 && any) atomicOr(flags, any);
}

// Domain check of positions loaded from device memory.
template <int DIM, class View>
__global__ void k_check_domain(int n, int64_t stride, const double* __restrict__ pos,
                               const __grid_constant__ View v, uint32_t* __restrict__ status) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const RealParams& P = v.of_input(uint32_t(i));
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const double x = pos[a * stride + i];
        if (!(x >= P.box.lo[a] && x <= P.box.hi[a])) atomicOr(status, kStatusOutOfDomain);
    }
}

// Cell-corner tables: entry P.g.corner_off[a] + c holds lo_a + c w_a of
// realisation P as a binary32 head (nearest) and tail (nearest to the
// remainder).  One thread per (realisation, axis, cell) entry; `first[k]` is
// the first entry of realisation k (first[nreal] = total).
__global__ void k_corners(int total, int nreal, int dim, const RealParams* __restrict__ tbl,
                          const int* __restrict__ first, float2* __restrict__ out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    int lo = 0, hi = nreal - 1;            // realisation: last k with first[k] <= t
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= t) lo = mid; else hi = mid - 1;
    }
    const Grid& g = tbl[lo].g;
    int a = 0;
    while (a + 1 < dim && t >= g.corner_off[a + 1]) ++a;
    const int c = t - g.corner_off[a];
    const double corner = __dadd_rn(g.lo[a], __dmul_rn(double(c + g.off[a]), g.w[a]));
    const float hi_f = __double2float_rn(corner);
    out[t] = make_float2(hi_f, __double2float_rn(__dsub_rn(corner, double(hi_f))));
}

__global__ void k_iota(int n, uint32_t* __restrict__ id) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) id[i] = uint32_t(i);
}

// ---------------------------------------------------------------------------
// Step 2a: exclusive prefix sum of the cell counts in one launch.  Each block
// scans a tile of 16 cells per thread, publishes the tile's total, and adds
// the totals of all tiles before it, which every block publishes before it
// waits on anyone (so no wait is chained behind another: the reduce-then-scan
// pair of launches fused by single-pass publication, in the manner of D.
// Merrill and M. Garland's decoupled look-back, NVIDIA technical report
// NVR-2016-002).  The count array is padded with zeros to whole tiles, so
// start[n_cells] = n.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
    __shared__ uint32_t warp_sums[32];
    __shared__ uint32_t block_total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        uint32_t ws = lane < nw ? warp_sums[lane] : 0u;
        uint32_t wi = ws;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        if (lane < nw) warp_sums[lane] = wi - ws;
        if (lane == 31) block_total = wi;     // lane 31's inclusive sum covers every warp
    }
    __syncthreads();
    const uint32_t excl = warp_sums[warp] + inc - v;
    *total = block_total;
    __syncthreads();
    return excl;
}

// A tile's published word: tag << 32 | total.  The tag is the launch's number
// (ticket / tiles) mod 2^32 - 1, plus one: every launch rewrites every tile's
// word, so a word still holding the previous launch's tag, or the zero the
// host writes when the grid changes, is told apart from this launch's.
constexpr unsigned long long kScanTagMod = 0xffffffffull;
// Polls before a block stops waiting for an earlier tile's total and sums
// that tile's counts itself (tens of milliseconds; the tiles it waits on took
// their tickets first, so they are running: a safety net, not a path the
// scan takes).
constexpr int kScanWaitLimit = 1 << 17;
__device__ unsigned long long g_scan_waits_given_up;

// state[0, ntiles) are the tiles' words, state[ntiles] the ticket (both zeroed
// by the host whenever the grid changes).  The block of the last tile
// advances the walk's step counter (device-resident, so a captured graph of
// steps replays with the right counters) when `advance` is set: every kernel
// of the step that reads it has completed.  A tile equal to `hold` never
// publishes (a test hook: the tiles after it then run out of polls).
__global__ void __launch_bounds__(kScanThreads)
k_scan(const uint4* count4, uint4* __restrict__ start4,
       unsigned long long* __restrict__ state, int ntiles,
       unsigned long long* __restrict__ step_dev, int advance, int hold) {
    constexpr int kVec = kScanPerThread / 4;
    __shared__ uint32_t s_tile;
    __shared__ unsigned long long s_tag;
    // (one block a tile: its threads' indexes, behind the wait)
    const uint32_t thread = ordered_index() % uint32_t(kScanThreads);
    // (a grid of one tile, the small runs', has no tile to wait for or to tell)
    const bool single = ntiles == 1;
    if (thread == 0 && !single) {
        // tiles in ticket order: a block only ever waits on blocks that started
        const unsigned long long t = atomicAdd(state + ntiles, 1ull);
        s_tile = uint32_t(t % unsigned(ntiles));
        s_tag = (t / unsigned(ntiles)) % kScanTagMod + 1ull;
    }
    if (!single) __syncthreads();
    const uint32_t tile = single ? 0u : s_tile;
    const unsigned long long tag = single ? 0ull : s_tag;
    // this thread's 16 consecutive cells
    const size_t base = (size_t(tile) * kScanThreads + thread) * kVec;
    uint4 c[kVec];
    uint32_t own = 0;
#pragma unroll
    for (int k = 0; k < kVec; ++k) {
        c[k] = count4[base + k];
        own += c[k].x + c[k].y + c[k].z + c[k].w;
    }
    uint32_t total;
    const uint32_t excl = block_exclusive_scan(own, &total);
    if (thread == 0 && !single && int(tile) != hold) st_relaxed_u64(state + tile, (tag << 32) | total);
    // the totals of every earlier tile, one word per thread at a time
    uint32_t part = 0;
    bool gave_up = false;
    for (uint32_t p = thread; p < tile; p += kScanThreads) {
        unsigned long long w = ld_relaxed_u64(state + p);
        for (int polls = 0; (w >> 32) != tag && polls < kScanWaitLimit; ++polls) {
            __nanosleep(64);
            w = ld_relaxed_u64(state + p);
        }
        if ((w >> 32) == tag) {
            part += uint32_t(w);
        } else {
            gave_up = true;
            const uint4* q = count4 + size_t(p) * (kScanTile / 4);
            for (int k = 0; k < kScanTile / 4; ++k) part += q[k].x + q[k].y + q[k].z + q[k].w;
        }
    }
    if (gave_up) atomicAdd(&g_scan_waits_given_up, 1ull);
    uint32_t prefix = 0;
    if (!single) block_exclusive_scan(part, &prefix);
    if (advance && thread == 0 && tile == uint32_t(ntiles - 1)) *step_dev += 1ull;
    uint32_t e = prefix + excl;
#pragma unroll
    for (int k = 0; k < kVec; ++k) {
        start4[base + k] = make_uint4(e, e + c[k].x, e + c[k].x + c[k].y, e + c[k].x + c[k].y + c[k].z);
        e += c[k].x + c[k].y + c[k].z + c[k].w;
    }
}

// Step counter updates for steps without a scan (walk only) and for resets.
__global__ void k_advance_step(unsigned long long* step_dev) {
    after_previous();
    *step_dev += 1ull;
}
__global__ void k_set_step(unsigned long long* step_dev, unsigned long long value) {
    after_previous();
    *step_dev = value;
}

// Realisation index of every particle of a batch: the last k with
// first[k] <= i (first[nreal] = n).
__global__ void k_fill_rid(int n, int nreal, const uint32_t* __restrict__ first,
                           uint32_t* __restrict__ rid) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo = 0, hi = nreal - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= uint32_t(i)) lo = mid; else hi = mid - 1;
    }
    rid[i] = uint32_t(lo);
}

// ---------------------------------------------------------------------------
// Step 2b: counting-sort scatter.  Each particle takes a slot of its cell
// (decrementing the count returns every count to zero for the next step) and
// stores there its index and a 16-byte sort key: x, and id | cell << 32, all
// that the in-cell ranking of the gather reads.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlock)
k_scatter(int n, const uint32_t* key, const uint32_t* start,
          uint32_t* __restrict__ count, const double* x,
          const uint32_t* id, uint32_t* __restrict__ perm,
          double2* __restrict__ sortkey) {
    const int i = int(ordered_index());
    if (i >= n) return;
    const uint32_t c = key[i];
    const double xi = x[i];
    const uint32_t idi = id[i];
    const uint32_t left = atomicSub(&count[c], 1u);
    const uint32_t slot = start[c] + left - 1u;
    if (!check(left >= 1u && slot < uint32_t(n), kChkSlot)) return;
    perm[slot] = uint32_t(i);
    sortkey[slot] = make_double2(xi, __longlong_as_double((long long)(uint64_t(idi) |
                                                                      (uint64_t(c) << 32))));
}

// Cell coordinates of a realisation-local cell index (the last axis needs
// no modulo).
template <int DIM>
__device__ __forceinline__ void cell_coords_of(uint32_t local, const Grid& g, int* c) {
    c[0] = c[1] = c[2] = 0;
    if constexpr (DIM == 1) {
        c[0] = int(local);
    } else if constexpr (DIM == 2) {
        const uint32_t q = local / uint32_t(g.n[0]);
        c[0] = int(local - q * uint32_t(g.n[0]));
        c[1] = int(q);
    } else {
        const uint32_t q = local / uint32_t(g.n[0]);
        c[0] = int(local - q * uint32_t(g.n[0]));
        const uint32_t r = q / uint32_t(g.n[1]);
        c[1] = int(q - r * uint32_t(g.n[1]));
        c[2] = int(r);
    }
}

// The same from a particle's record: its x (and, in 2-d, y) cell index is
// there, so only 3-d reads the cell array (`cell` is cell[s], unused below 3-d).
template <int DIM>
__device__ __forceinline__ void cell_coords_rec(uint32_t cell, const float4& me, const RealParams& P,
                                                int* c) {
    if constexpr (DIM == 3) {
        cell_coords_of<3>(cell - P.cell_base, P.g, c);
    } else {
        c[0] = int(me.w);
        c[1] = DIM == 2 ? int(me.z) : 0;
        c[2] = 0;
    }
}

// cell[s] where the pair searches need it (3-d), else nothing is read.
template <int DIM>
__device__ __forceinline__ uint32_t cell_arg(const uint32_t* cell, uint32_t s) {
    return DIM == 3 ? cell[s] : 0u;
}

// Step 2c: gather into cell order.  The slot order the atomics gave inside a
// cell is replaced by the rank of (x, id) -- binary64 x in its integer order,
// the id breaking ties -- so the layout (and every sum over it) is identical
// run to run, and each neighbour row (cells cx-1..cx+1 of one y (, z)) is
// sorted by x up to the cells' rounding slack, which the pair search uses.
// The rank reads the sort keys of the cell's slots, next to the particle's
// own; the rest of the payload comes from the source index.  Also writes the
// particle's cell, its binary32 offset from the cell corner (from the
// binary32 head/tail split of the coordinate and of the corner: error below
// 2^-23 w, no binary64 instruction).
template <int DIM, class View, bool TANGENT = false>
__global__ void __launch_bounds__(kBlock)
k_gather(int n, int64_t stride, const uint32_t* perm,
         const double2* sortkey, const uint32_t* start,
         const double* pos_in, const double* mass_in,
         uint32_t* __restrict__ id_out, double* __restrict__ pos_out,
         double* __restrict__ mass_out, uint32_t* __restrict__ cell_out,
         float* __restrict__ rec_out,
         const float2* __restrict__ corners, uint32_t* __restrict__ rid_out,
         const __grid_constant__ View v, const double* tan_in = nullptr,
         double* __restrict__ tan_out = nullptr, const double* mass_b_in = nullptr,
         double* __restrict__ mass_b_out = nullptr, uint64_t* __restrict__ image_out = nullptr) {
    const int s = int(ordered_index());
    if (s >= n) return;
    const uint32_t src = perm[s];
    const double2 me = sortkey[s];
    if (!check(src < uint32_t(n), kChkGather)) return;
    // payload loads first: independent of the ranking below
    double xa[3] = {me.x, 0.0, 0.0};
#pragma unroll
    for (int a = 1; a < DIM; ++a) xa[a] = pos_in[a * stride + src];
    const double m = mass_in[src];
    const unsigned long long idc = (unsigned long long)__double_as_longlong(me.y);
    const uint32_t my_id = uint32_t(idc), c = uint32_t(idc >> 32);
    const uint32_t b = start[c], e = start[c + 1];
    if (!check(b <= uint32_t(s) && uint32_t(s) < e && e <= uint32_t(n), kChkGather)) return;
    const long long my_x = order_key(me.x);
    const uint32_t my_rank_id = my_id & ~kGhostBit;   // ghosts rank by their own id
    uint32_t rank = 0;
    for (uint32_t k = b; k < e; ++k) {
        const double2 q = sortkey[k];
        const long long xo = order_key(q.x);
        const uint32_t ido = uint32_t(__double_as_longlong(q.y)) & ~kGhostBit;
        rank += (xo < my_x || (xo == my_x && ido < my_rank_id)) ? 1u : 0u;
    }
    const uint32_t dst = b + rank;
    if (!check(dst < e, kChkGather)) return;
    id_out[dst] = my_id;
    if constexpr (DIM == 3) cell_out[dst] = c;   // only the 3-d searches read it
    if constexpr (View::kBatch) rid_out[dst] = ld_global(v.rid_input + src);
    if (mass_b_out) mass_b_out[dst] = mass_b_in[src];   // second species (reactions)
    const RealParams& P = v.of_input(src);
    mass_out[dst] = m;
    float off[3] = {0.0f, 0.0f, 0.0f};
    int cc[3];
    cell_coords_of<DIM>(c - P.cell_base, P.g, cc);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const uint32_t ca = uint32_t(cc[a]);
        const double x = xa[a];
        pos_out[a * stride + dst] = x;
        if constexpr (TANGENT) tan_out[a * stride + dst] = tan_in[a * stride + src];
        if (image_out) image_out[a * stride + dst] = x_image(x, P.pp.kc.x_shift);
        if (P.transfer) {
            float xh, xlo;
            split_double(x, &xh, &xlo);
            const float2 cr = __ldg(corners + P.g.corner_off[a] + ca);
            off[a] = __fadd_rn(__fsub_rn(xh, cr.x), __fsub_rn(xlo, cr.y));
        }
    }
    store_rec(rec_out, dst,
              make_float4(off[0], off[1], DIM == 2 ? float(cc[1]) : off[2], float(cc[0])));
}

// Sort of a freshly loaded single run, whose particles arrive in input order
// rather than cell order: the same counting sort and the same cell order, but
// the scatter stores each particle's whole payload as one record of 16-byte
// chunks at its slot, so the gather reads only records in slot order.  A
// record fills whole 32-byte sectors, which the scattered stores of an
// unsorted input then write without a read (the sort keys plus a separate
// payload read through the permutation cost more there; in steady state,
// where the slots barely move, the opposite holds).  Eight-byte lanes:
//   0: x   1: id | cell << 32   2..DIM: the other axes   DIM + 1: mass
//   then DIM position tangents (TANGENT)
template <int DIM, bool TANGENT>
struct SortRec {
    static constexpr int kLanes = 2 + DIM + (TANGENT ? DIM : 0);
    static constexpr int kChunks = (kLanes + 1) / 2;
    static constexpr int kTan = DIM + 2;
};

template <int DIM, bool TANGENT>
__global__ void __launch_bounds__(kBlock)
k_scatter_rec(int n, int64_t stride, const uint32_t* key,
              const uint32_t* start, uint32_t* __restrict__ count,
              const double* pos, const double* mass,
              const uint32_t* id, const double* tan,
              double2* __restrict__ recs) {
    using R = SortRec<DIM, TANGENT>;
    const int i = int(ordered_index());
    if (i >= n) return;
    const uint32_t c = key[i];
    double lane[2 * R::kChunks];
    lane[0] = pos[i];
    lane[1] = __longlong_as_double((long long)(uint64_t(id[i]) | (uint64_t(c) << 32)));
#pragma unroll
    for (int a = 1; a < DIM; ++a) lane[1 + a] = pos[a * stride + i];
    lane[DIM + 1] = mass[i];
    if constexpr (TANGENT) {
#pragma unroll
        for (int a = 0; a < DIM; ++a) lane[R::kTan + a] = tan[a * stride + i];
    }
    if constexpr (R::kLanes % 2 == 1) lane[R::kLanes] = 0.0;
    const uint32_t left = atomicSub(&count[c], 1u);
    const uint32_t slot = start[c] + left - 1u;
    if (!check(left >= 1u && slot < uint32_t(n), kChkSlot)) return;
    double2* r = recs + size_t(slot) * R::kChunks;
#pragma unroll
    for (int k = 0; k < R::kChunks; ++k) r[k] = make_double2(lane[2 * k], lane[2 * k + 1]);
}

// Gather from the records: the rank inside the cell by (x order key, id)
// reads chunk 0 of the cell's records; outputs as k_gather's.
template <int DIM, bool TANGENT>
__global__ void __launch_bounds__(kBlock)
k_gather_rec(int n, int64_t stride, const double2* recs,
             const uint32_t* start, uint32_t* __restrict__ id_out,
             double* __restrict__ pos_out, double* __restrict__ mass_out,
             uint32_t* __restrict__ cell_out, float* __restrict__ rec_out,
             const float2* __restrict__ corners,
             const __grid_constant__ SingleView v, double* __restrict__ tan_out,
             uint64_t* __restrict__ image_out) {
    using R = SortRec<DIM, TANGENT>;
    const int s = int(ordered_index());
    if (s >= n) return;
    double lane[2 * R::kChunks];
    const double2* me = recs + size_t(s) * R::kChunks;
#pragma unroll
    for (int k = 0; k < R::kChunks; ++k) {
        const double2 q = me[k];
        lane[2 * k] = q.x;
        lane[2 * k + 1] = q.y;
    }
    const unsigned long long idc = (unsigned long long)__double_as_longlong(lane[1]);
    const uint32_t my_id = uint32_t(idc), c = uint32_t(idc >> 32);
    const uint32_t b = start[c], e = start[c + 1];
    if (!check(b <= uint32_t(s) && uint32_t(s) < e && e <= uint32_t(n), kChkGather)) return;
    const long long my_x = order_key(lane[0]);
    const uint32_t my_rank_id = my_id & ~kGhostBit;   // ghosts rank by their own id
    uint32_t rank = 0;
    for (uint32_t k = b; k < e; ++k) {
        const double2 q = recs[size_t(k) * R::kChunks];
        const long long xo = order_key(q.x);
        const uint32_t ido = uint32_t(__double_as_longlong(q.y)) & ~kGhostBit;
        rank += (xo < my_x || (xo == my_x && ido < my_rank_id)) ? 1u : 0u;
    }
    const uint32_t dst = b + rank;
    if (!check(dst < e, kChkGather)) return;
    id_out[dst] = my_id;
    if constexpr (DIM == 3) cell_out[dst] = c;   // only the 3-d searches read it
    const RealParams& P = v.p;
    const double m = lane[DIM + 1];
    mass_out[dst] = m;
    float off[3] = {0.0f, 0.0f, 0.0f};
    int cc[3];
    cell_coords_of<DIM>(c - P.cell_base, P.g, cc);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const uint32_t ca = uint32_t(cc[a]);
        const double x = lane[a == 0 ? 0 : 1 + a];
        pos_out[a * stride + dst] = x;
        if constexpr (TANGENT) tan_out[a * stride + dst] = lane[R::kTan + a];
        if (image_out) image_out[a * stride + dst] = x_image(x, P.pp.kc.x_shift);
        if (P.transfer) {
            float xh, xlo;
            split_double(x, &xh, &xlo);
            const float2 cr = __ldg(corners + P.g.corner_off[a] + ca);
            off[a] = __fadd_rn(__fsub_rn(xh, cr.x), __fsub_rn(xlo, cr.y));
        }
    }
    store_rec(rec_out, dst,
              make_float4(off[0], off[1], DIM == 2 ? float(cc[1]) : off[2], float(cc[0])));
}

// ---------------------------------------------------------------------------
// Steps 2-5: neighbour visits.  For particle s (cell order) the candidates
// are the particles of the 3^DIM surrounding cells, s itself included, each
// neighbour row cut to the window of x that can reach the cutoff (see
// for_each_row).  The
// binary32 squared distance from the cell offsets decides every candidate
// outside a narrow band around psi^2; inside the band the exact binary64 test
// dx*dx + dy*dy (+ dz*dz) <= psi^2 (no fma, dx = x_i - x_j) decides.  The
// band half-width is set on the host from an error bound of the binary32
// evaluation, so the accepted set equals the exact binary64 pair set.
//
// The binary32 difference is (off_j - off_s) + shift, which changes sign
// exactly when s and j swap, so d2f(s, j) == d2f(j, s) bit for bit and every
// quantity derived from it is symmetric in the pair.  The self pair has
// d2f = 0, K = 1 exactly: it supplies the self term of the row sum and a zero
// flux, so no candidate is skipped.
// ---------------------------------------------------------------------------
template <int DIM>
__device__ __forceinline__ double exact_d2(const double* pos, int64_t stride,
                                           uint32_t i, uint32_t j) {
    double d2 = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const double d = __dsub_rn(ld_global(pos + a * stride + i), ld_global(pos + a * stride + j));
        const double sq = __dmul_rn(d, d);
        d2 = (a == 0) ? sq : __dadd_rn(d2, sq);
    }
    return d2;
}

// Kernel value of an accepted pair from the particles' fixed-point images (see
// expneg.cuh).  Symmetric in (i, j) bit for bit.
template <int DIM>
__device__ __forceinline__ double pair_kernel(const uint64_t* image, int64_t stride,
                                              uint32_t i, uint32_t j, const double* table,
                                              const KernelConsts& kc) {
    uint64_t d2h = 0;
#pragma unroll
    for (int a = 0; a < DIM; ++a)
        d2h += axis_square(ld_global(image + a * stride + i), ld_global(image + a * stride + j));
    return gauss_fixed(d2h, table, kc);
}

// Hardware square root approximation (relative error far below the
// windows' slack trim_eps, which covers it).
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Binary32 x difference of candidate o from particle me (cells cx_o - cx_me
// apart, |cx_o - cx_me| <= reach <= 2, so the shift is a power-of-two multiple
// of wx and exact, and one fused multiply-add rounds exactly as the sum of the
// rounded offset difference and the shift would): changes sign exactly when
// the pair swaps.
__device__ __forceinline__ float dx_f32(const float4& me, const float4& o, float wx) {
    return __fmaf_rn(__fsub_rn(o.w, me.w), wx, __fsub_rn(o.x, me.x));
}

// The same of the candidate with index j.
__device__ __forceinline__ float dx_of(const float4& me, const float* rec, uint32_t j,
                                       float wx) {
    const float* q = rec + rec_at(j);
    return __fmaf_rn(__fsub_rn(ld_global(q + 2), me.w), wx, __fsub_rn(ld_global(q), me.x));
}

template <int DIM>
__device__ __forceinline__ float d2_f32(float dx, const float4& me, const float4& o, float sy,
                                        float sz) {
    if (DIM == 1) return __fmul_rn(dx, dx);
    const float dy = __fadd_rn(__fsub_rn(o.y, me.y), sy);
    if (DIM == 2) return __fmaf_rn(dx, dx, __fmul_rn(dy, dy));
    const float dz = __fadd_rn(__fsub_rn(o.z, me.z), sz);
    return __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, __fmul_rn(dz, dz)));
}

// Lower bound of |dy_f| over the particles of the row `d` cells away along an
// axis (d = 0: the particle's own row, bound 0): the rows below hold offsets
// up to w from their cells' corners, those above offsets from 0, so the gap
// is the particle's own offset (or w minus it) plus |d| - 1 whole cells, less
// the slack that covers the roundings.
__device__ __forceinline__ float row_gap(int d, float off, float w, float eps) {
    if (d == 0) return 0.0f;
    const float near = d < 0 ? off : __fsub_rn(w, off);
    const int far = d < 0 ? -d - 1 : d - 1;
    const float gap = far == 0 ? near : __fmaf_rn(float(far), w, near);
    return fmaxf(__fsub_rn(gap, eps), 0.0f);
}

// Per-row candidate windows.  Row (dy, dz) of particle s is the particle
// range [j0, j3) of cells cx-R..cx+R at y index cy+dy (z index cz+dz), R the
// grid's reach (|dy|, |dz| <= R); the
// gather sorts it by x up to a slack.  Every accepted candidate has
// d2f <= band_hi, so with g a lower bound of |dy_f| (and |dz_f|) over the row
// its binary32 dx satisfies dx^2 <= reach2 - g^2 (reach2 carries the
// roundings).  The row is skipped when that is negative; otherwise
//   rx = sqrt(reach2 - g^2) + trim_eps
// where trim_eps (host) bounds the sqrt rounding plus the row's departure from
// x order (two dx errors and twice the cell-index error dc w).  A bisection
// finds the first j with dx_j >= -rx: every earlier candidate then has
// dx < -rx + trim_eps, too far left.  The caller's loop stops at the first
// dx_j > rx: every later one has dx > rx - trim_eps.  Neither bound drops a
// neighbour, so the accepted set is the exact binary64 one as before.
// row(j0, j3, rx, sy, sz) is called for every row that can hold a neighbour.
template <int DIM, class Row>
__device__ __forceinline__ void for_each_row(uint32_t cell, const float4 me,
                                             const float* rec,
                                             const uint32_t* start,
                                             const RealParams& P, Row&& row) {
    const Grid& g = P.g;
    const PairParams& pp = P.pp;
    int c[3];
    cell_coords_rec<DIM>(cell, me, P, c);
    const int R = g.reach;
    const int xlo = max(c[0] - R, 0);
    const int xhi = min(c[0] + R, g.n[0] - 1);
    const int zlo = DIM == 3 ? max(-R, -c[2]) : 0;
    const int zhi = DIM == 3 ? min(R, g.n[2] - 1 - c[2]) : 0;
    const int ylo = DIM >= 2 ? max(-R, -c[1]) : 0;
    const int yhi = DIM >= 2 ? min(R, g.n[1] - 1 - c[1]) : 0;
    const float eps = pp.trim_eps;
    const float wx = g.wf[0];
    for (int dz = zlo; dz <= zhi; ++dz) {
        const float sz = DIM == 3 ? float(dz) * g.wf[2] : 0.0f;
        const float gz = DIM == 3 ? row_gap(dz, me.z, g.wf[2], eps) : 0.0f;
        for (int dy = ylo; dy <= yhi; ++dy) {
            const float sy = DIM >= 2 ? float(dy) * g.wf[1] : 0.0f;
            const float gy = DIM >= 2 ? row_gap(dy, me.y, g.wf[1], eps) : 0.0f;
            const float r2 = __fsub_rn(pp.reach2, __fmaf_rn(gy, gy, __fmul_rn(gz, gz)));
            if (r2 < 0.0f) continue;
            const float rx = __fadd_rn(sqrt_approx(r2), eps);
            const uint32_t rowc = P.cell_base + (uint32_t(c[2] + dz) * uint32_t(g.n[1]) +
                                                 uint32_t(c[1] + dy)) * uint32_t(g.n[0]);
            if (!check(rowc + uint32_t(xhi) + 1u - P.cell_base <=
                           uint32_t(g.n[0]) * uint32_t(g.n[1]) * uint32_t(g.n[2]), kChkRow))
                continue;
            uint32_t lo = ld_global(start + rowc + xlo);
            uint32_t hi = ld_global(start + rowc + xhi + 1);
            const uint32_t j3 = hi;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (dx_of(me, rec, mid, wx) < -rx) lo = mid + 1;
                else hi = mid;
            }
            row(lo, j3, rx, sy, sz);
        }
    }
}

// visit(j, d2f, rec_j) is called for every neighbour j of s (s included).
template <int DIM, class Visit>
__device__ __forceinline__ void visit_neighbours(uint32_t s, uint32_t cell, int64_t stride,
                                                 const float* rec,
                                                 const double* pos,
                                                 const uint32_t* start,
                                                 const RealParams& P, Visit&& visit) {
    const PairParams& pp = P.pp;
    const float4 me = load_rec(rec, s);
    const float wx = P.g.wf[0];
    for_each_row<DIM>(cell, me, rec, start, P,
                      [&](uint32_t j0, uint32_t j3, float rx, float sy, float sz) {
#pragma unroll 2
        for (uint32_t j = j0; j < j3; ++j) {
            const float4 o = load_rec(rec, j);
            const float dx = dx_f32(me, o, wx);
            if (dx > rx) break;
            const float d2f = d2_f32<DIM>(dx, me, o, sy, sz);
            if (d2f > pp.band_hi) continue;
            if (d2f >= pp.band_lo && exact_d2<DIM>(pos, stride, s, j) > pp.psi2) continue;
            visit(j, d2f, o);
        }
    });
}

// The exact binary64 test as a real call, so the compiler cannot if-convert
// it into every candidate's path (it runs only inside the narrow band).
template <int DIM>
__device__ __noinline__ bool exact_within(const double* pos, int64_t stride,
                                          uint32_t s, uint32_t j, double psi2) {
    return exact_d2<DIM>(pos, stride, s, j) <= psi2;
}

// The candidates inside the narrow band around the cutoff that the exact test
// accepts: visit(j, d2f) in candidate order.
template <int DIM, class Visit>
__device__ __forceinline__ void scan_band(uint32_t s, uint32_t cell, int64_t stride,
                                          const float* rec,
                                          const double* pos,
                                          const uint32_t* start, const RealParams& P,
                                          Visit&& visit) {
    const PairParams& pp = P.pp;
    const float4 me = load_rec(rec, s);
    const float wx = P.g.wf[0];
    for_each_row<DIM>(cell, me, rec, start, P,
                      [&](uint32_t j0, uint32_t j3, float rx, float sy, float sz) {
        for (uint32_t j = j0; j < j3; ++j) {
            const float4 o = load_rec(rec, j);
            const float dx = dx_f32(me, o, wx);
            if (dx > rx) break;
            const float d2f = d2_f32<DIM>(dx, me, o, sy, sz);
            if (d2f >= pp.band_lo && d2f <= pp.band_hi &&
                exact_within<DIM>(pos, stride, s, j, pp.psi2))
                visit(j, d2f);
        }
    });
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Compensated summation of mixed-sign terms (Kahan-Babuska / Neumaier):
// s + c carries the sum to about twice binary32 precision whatever the order
// of magnitudes.  Used for the flux sums.
__device__ __forceinline__ void neumaier_add(float& s, float& c, float x) {
    const float t = __fadd_rn(s, x);
    const bool s_big = fabsf(s) >= fabsf(x);
    const float big = s_big ? s : x;
    const float small = s_big ? x : s;
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(big, t), small));
    s = t;
}

__device__ __forceinline__ void add_pair_count(uint32_t cnt, unsigned long long* counter) {
    const uint32_t warp_total = __reduce_add_sync(0xffffffffu, cnt);
    if ((threadIdx.x & 31) == 0 && warp_total) atomicAdd(counter, (unsigned long long)warp_total);
}

// ---------------------------------------------------------------------------
// What pass 1 keeps of its search for pass 2: accept masks.  A word {base,
// bits} holds 32 consecutive candidates of one neighbour row: bit k is set when
// candidate base + k is an accepted neighbour j != s.  Plane w (entry w * stride
// + s) holds s's w-th word with a bit set, in candidate order; a particle's
// list word is their number and the number of neighbours (mask_word), or
// kMaskOver for a particle that needs more than `cap` words: it searches again.
// With `pad` > 0 every row is filled up to `pad` words with empty ones, so
// that a warp's lanes have the same row in the same plane.
// (The precision form's 3-d runs keep lists in the same planes: plane k holds
// s's k-th accepted neighbour with its binary32 kernel value, {j, K bits}; the
// list word is the full number, and a particle with more than `cap` searches.)
// ---------------------------------------------------------------------------
struct NbPlanes {
    uint2* e;
    int cap;           // planes (masks: at most 255); 0: nothing kept
    int pad;           // words every row has at least (masks; see setup_grids)
};
constexpr uint32_t kMaskOver = 0xffffffffu;
__device__ __forceinline__ uint32_t mask_word(uint32_t words, uint32_t neighbours, int cap) {
    return words <= uint32_t(cap) && neighbours < (1u << 24) - 1u ? neighbours << 8 | words : kMaskOver;
}

// The search of one particle, its windows row by row, two candidates (one
// block of records) at a time: one 32-byte load, the distances as packed
// binary32 operations, the tests on the distances' bits (ordered like the
// values, as neither a distance nor band_lo has a sign bit).  A window starts
// at an even index and may end at an odd one, so candidates outside it are
// masked off.  With WORDS, the accepted neighbours j != s go to the sink, as mask
// words {base, bits} in candidate order: those below the narrow band around the
// cutoff, and, with EXACT, those inside it that the exact test accepts.  EACH
// calls cand(j, d2, accept, accept1) for every two candidates j and j + 1 (d2 their
// binary32 distances squared), the self pair included.
// Without EXACT returns whether any candidate was inside the band.  A search for
// words alone ends when the sink is full.
//
// Bound by instruction issue: singly, a candidate took about 20 instructions
// of which the pair shares or packs all but three.  The bisection to a
// window's first candidate pays only in long rows: of up to kBisectFrom
// candidates the loop takes those on the left too (never accepted), two at a
// time.  Pass 1 of the precision form: 175 -> 158 us by pairs and 142 without
// the bisection (4e6 particles in 2-d, three cells hold 5.4), 191 -> 187 (2e6 in
// 3-d, 2.6); at density 10 (54 candidates a row) 1.55 -> 1.18 ms by pairs, with
// the bisection (1.31 without).  With ordinary loads in place of read-only ones
// 144 and 186 us and 1.22 ms.
constexpr uint32_t kBisectFrom = 24;
template <int DIM, bool WORDS, bool EACH, bool EXACT, class Cand, class Sink>
__device__ __forceinline__ bool search_rows(uint32_t s, uint32_t cell, const float4 me,
                                            int64_t stride, const double* pos, const float* rec,
                                            const uint32_t* start, const RealParams& P,
                                            Cand&& cand, Sink&& sink) {
    const PairParams& pp = P.pp;
    const Grid& g = P.g;
    int c[3];
    cell_coords_rec<DIM>(cell, me, P, c);
    const float wx = g.wf[0], eps = pp.trim_eps;
    const int R = g.reach, xlo = max(c[0] - R, 0), xhi = min(c[0] + R, g.n[0] - 1);
    const uint32_t lo_bits = __float_as_uint(pp.band_lo);
    // (read where it is used: a batch's parameters are in memory)
    auto band_span = [&]() { return __float_as_uint(pp.band_hi) - lo_bits; };
    uint32_t nearest = 0xffffffffu;    // least (bits of d2f) - lo_bits, unsigned
    // one row's window and candidates: an empty window where the row is outside
    // the grid or beyond the cutoff (for_each_row has the windows' derivation)
    auto row = [&](int dy, int dz) {
        const float sy = DIM >= 2 ? float(dy) * g.wf[1] : 0.0f;
        const float sz = DIM == 3 ? float(dz) * g.wf[2] : 0.0f;
        const float gy = DIM >= 2 ? row_gap(dy, me.y, g.wf[1], eps) : 0.0f;
        const float gz = DIM == 3 ? row_gap(dz, me.z, g.wf[2], eps) : 0.0f;
        const float r2 = __fsub_rn(pp.reach2, __fmaf_rn(gy, gy, __fmul_rn(gz, gz)));
        const bool in_grid = (DIM < 2 || (c[1] + dy >= 0 && c[1] + dy < g.n[1])) &&
                             (DIM < 3 || (c[2] + dz >= 0 && c[2] + dz < g.n[2]));
        uint32_t j = 0, j3 = 0;
        float rx = 0.0f;
        bool wanted = in_grid && r2 >= 0.0f;
        if constexpr (WORDS && !EACH) wanted = wanted && !sink.full();
        if (wanted) {
            rx = __fadd_rn(sqrt_approx(r2), eps);
            const uint32_t rowc = P.cell_base + (uint32_t(c[2] + dz) * uint32_t(g.n[1]) +
                                                 uint32_t(c[1] + dy)) * uint32_t(g.n[0]);
            if (check(rowc + uint32_t(xhi) + 1u - P.cell_base <=
                          uint32_t(g.n[0]) * uint32_t(g.n[1]) * uint32_t(g.n[2]), kChkRow)) {
                j = ld_global(start + rowc + xlo);
                j3 = ld_global(start + rowc + xhi + 1);
                if (j3 - j > kBisectFrom) {
                    uint32_t hi = j3;
                    while (hi - j > 2u) {
                        const uint32_t mid = (j + hi) >> 1;
                        if (dx_of(me, rec, mid, wx) < -rx) j = mid + 1;
                        else hi = mid;
                    }
                }
            }
        }
        if constexpr (WORDS) sink.begin_row();
        const uint32_t first = j;
        uint32_t b = j & ~1u;
        // one block of two candidates; false past the window's right end: in x
        // order, every later candidate lies farther right still (a second
        // candidate outside the window is the row's last)
        uint32_t bits = 0;                 // accepted, latest candidate lowest
        auto block = [&]() {
            const RecPair o = load_rec_pair(rec, b);
            const uint64_t dx = fma2(sub2(o.w, pack2(me.w, me.w)), pack2(wx, wx),
                                     sub2(o.x, pack2(me.x, me.x)));
            uint64_t d2 = mul2(dx, dx);
            if constexpr (DIM >= 2) {
                const uint64_t ey = add2(sub2(o.y, pack2(me.y, me.y)), pack2(sy, sy));
                if constexpr (DIM == 2) {
                    d2 = fma2(dx, dx, mul2(ey, ey));
                } else {
                    const uint64_t ez = add2(sub2(o.z, pack2(me.z, me.z)), pack2(sz, sz));
                    d2 = fma2(dx, dx, fma2(ey, ey, mul2(ez, ez)));
                }
            }
            const float2 d = unpack2(d2);
            const uint32_t t0 = __float_as_uint(d.x) - lo_bits, t1 = __float_as_uint(d.y) - lo_bits;
            nearest = min(nearest, min(t0, t1));
            if constexpr (WORDS) {
                bits = __funnelshift_l(t0, bits, 1);   // the sign: below the band
                bits = __funnelshift_l(t1, bits, 1);
            }
            if constexpr (EACH) {
                bool a0 = int32_t(t0) < 0 && b >= first, a1 = int32_t(t1) < 0 && b + 1u < j3;
                if constexpr (EXACT) {
                    if (min(t0, t1) <= band_span()) {
                        a0 |= t0 <= band_span() && b >= first &&
                              exact_within<DIM>(pos, stride, s, b, pp.psi2);
                        a1 |= t1 <= band_span() && b + 1u < j3 &&
                              exact_within<DIM>(pos, stride, s, b + 1u, pp.psi2);
                    }
                }
                cand(b, d, a0, a1);
            }
            b += 2u;
            return !(unpack2(dx).y > rx);
        };
        if constexpr (!WORDS) {
            while (b < j3 && block()) {}
        } else {
            while (b < j3) {
                const uint32_t base = b, end = min(j3, base + 32u);
                bits = 0;
                bool more = true;
                do {
                    more = block();
                } while (more && b < end);
                bits = __brev(bits) >> (32u - (b - base));
                if (base < first) bits &= ~1u;
                if (j3 - base < 32u) bits &= (1u << (j3 - base)) - 1u;
                if constexpr (EXACT && !EACH) {
                    if (nearest <= band_span()) {
                        for (uint32_t k = max(base, first); k < min(b, j3); ++k) {
                            const float4 o = load_rec(rec, k);
                            const float d2f = d2_f32<DIM>(dx_f32(me, o, wx), me, o, sy, sz);
                            if (d2f >= pp.band_lo && d2f <= pp.band_hi &&
                                exact_within<DIM>(pos, stride, s, k, pp.psi2))
                                bits |= 1u << (k - base);
                        }
                        nearest = 0xffffffffu;
                    }
                }
                if (s - base < 32u) bits &= ~(1u << (s - base));   // the self pair is no neighbour
                if (bits) sink.word(base, bits);
                if constexpr (WORDS && !EACH) more = more && !sink.full();
                if (!more) break;
            }
        }
        if constexpr (WORDS) sink.end_row();
    };
    // rows in a fixed order for the whole warp
    if constexpr (DIM == 1) {
        row(0, 0);
    } else if constexpr (DIM == 2) {
#pragma unroll 1
        for (int dy = -R; dy <= R; ++dy) row(dy, 0);
    } else {
#pragma unroll 1
        for (int dz = -R; dz <= R; ++dz)
#pragma unroll 1
            for (int dy = -R; dy <= R; ++dy) row(dy, dz);
    }
    return nearest <= band_span();
}

// Sinks of search_rows: the planes, with their padding ...
struct PlaneSink {
    const NbPlanes& nb;
    const int64_t& stride;
    uint2* wp;                         // next mask word
    uint32_t nw = 0, cnt = 0, padded = 0;   // words written or wanted, neighbours
    __device__ __forceinline__ PlaneSink(const NbPlanes& planes, uint32_t s, const int64_t& st)
        : nb(planes), stride(st), wp(planes.e + s) {}
    __device__ __forceinline__ void begin_row() { padded = nw + uint32_t(nb.pad); }
    __device__ __forceinline__ void put(uint2 w) {
        if (nw < uint32_t(nb.cap)) *wp = w;
        wp += stride;
        ++nw;
    }
    __device__ __forceinline__ void word(uint32_t base, uint32_t bits) {
        cnt += uint32_t(__popc(bits));
        put(make_uint2(base, bits));
    }
    __device__ __forceinline__ void end_row() {
        while (nw < padded) put(make_uint2(0u, 0u));
    }
    __device__ __forceinline__ bool full() const { return nw > uint32_t(nb.cap); }
};
// ... none ...
struct NoSink {};
// ... and a call pair(j0, j1, two) for every two neighbours of a word (j1 = j0
// and `two` false for the last of an odd number).
template <class Pair>
struct PairSink {
    Pair pair;
    uint32_t cnt = 0;
    __device__ __forceinline__ void begin_row() {}
    __device__ __forceinline__ void word(uint32_t base, uint32_t bits) {
        cnt += uint32_t(__popc(bits));
        while (bits) {
            const uint32_t j0 = base + uint32_t(__ffs(int(bits)) - 1);
            bits &= bits - 1u;
            const bool two = bits != 0u;
            const uint32_t j1 = two ? base + uint32_t(__ffs(int(bits)) - 1) : j0;
            bits &= bits - 1u;
            pair(j0, j1, two);
        }
    }
    __device__ __forceinline__ void end_row() {}
    __device__ __forceinline__ bool full() const { return false; }
};
// Every neighbour of s, two at a time, in the order of its mask words, for a
// particle whose words are not kept, in binary64: returns their number.  The search
// and the pair terms are apart (a word's candidates, then its neighbours), so the
// lanes meet again in the expensive terms: the no-allocation step of 65,536
// particles in 3-d, which has no room for words, took 1072 us at density 8 with each
// neighbour evaluated where a loop over single records met it, 694 so.
template <int DIM, class Pair>
__device__ __forceinline__ uint32_t each_pair(uint32_t s, const uint32_t* cell, int64_t stride,
                                              const double* pos, const float* rec,
                                              const uint32_t* start, const RealParams& P,
                                              Pair&& pair) {
    PairSink<Pair&> sink{pair};
    search_rows<DIM, true, false, true>(s, cell_arg<DIM>(cell, s), load_rec(rec, s), stride, pos, rec,
                                        start, P, [](uint32_t, float2, bool, bool) {}, sink);
    return sink.cnt;
}

// The mask words of a particle that met candidates inside the band (about 1e-5
// of all candidates): walks its windows again with the exact test and writes
// all its words anew (without padding).  SUM (the precision form's pass 1):
// also adds the kernel values of those it accepts to the row sum {rsum, rc}.
// Returns {rsum, rc, words (bits), neighbours (bits)}.  A real call, so its
// registers do not weigh on the candidate loop.
template <int DIM, bool SUM, class View>
__device__ __noinline__ float4 band_words(uint32_t s, const uint32_t* cell, int64_t stride,
                                          const double* pos,
                                          const float* rec,
                                          const uint32_t* start, const View& v,
                                          const NbPlanes& nb, float rsum, float rc) {
    const RealParams& P = v.of_sorted(s);
    const PairParams& pp = P.pp;
    const float4 me = load_rec(rec, s);
    uint32_t cnt = 0, nw = 0;
    for_each_row<DIM>(cell_arg<DIM>(cell, s), me, rec, start, P,
                      [&](uint32_t j, uint32_t j3, float rx, float sy, float sz) {
        while (j < j3) {
            const uint32_t base = j, end = min(j3, base + 32u);
            uint32_t bits = 0;
            for (; j < end; ++j) {
                const float4 o = load_rec(rec, j);
                const float dx = dx_f32(me, o, P.g.wf[0]);
                if (dx > rx) {
                    j3 = j;
                    break;
                }
                const float d2f = d2_f32<DIM>(dx, me, o, sy, sz);
                if (d2f > pp.band_hi) continue;
                if (d2f >= pp.band_lo) {
                    if (!exact_within<DIM>(pos, stride, s, j, pp.psi2)) continue;
                    if constexpr (SUM) {
                        const float y = __fsub_rn(ex2_approx(-pp.a_log2e * d2f), rc);
                        const float t = __fadd_rn(rsum, y);
                        rc = __fsub_rn(__fsub_rn(t, rsum), y);
                        rsum = t;
                    }
                }
                if (j != s) bits |= 1u << (j - base);
            }
            if (bits) {
                cnt += uint32_t(__popc(bits));
                if (nw < uint32_t(nb.cap)) nb.e[int64_t(nw) * stride + s] = make_uint2(base, bits);
                ++nw;
            }
        }
    });
    return make_float4(rsum, rc, __uint_as_float(nw), __uint_as_float(cnt));
}

// ---------------------------------------------------------------------------
// Binary64 pair passes.  The binary64 form's two passes are a thread per
// particle throughout: its pair terms are integer arithmetic (expneg.cuh), and
// a warp that takes its particles' k-th neighbours together stores and reads
// their kernel values in whole rows.  (Evaluating the warp's neighbours one a
// lane, as below, saves the lanes idle in the longest particle's tail but
// spends as many instructions on handing them out: when both were built, with
// candidates taken singly, pass 1 took 405 us that way instead of 381, pass 2 with
// the walk 389 instead of 322, 4e6 particles in 2-d.)
// The adjoint's pair terms keep seven or eight binary64 operations, which cost the
// same however many lanes are active (a thread per particle took 45 and 51 us a
// pass where this takes 36 and 40), so there a warp works in two parts: each lane
// searches its particle and leaves mask words; then the warp takes the words'
// neighbours in lane-major order, kChunk at a time: the lanes write out their
// neighbours' indexes (shared memory), all 32 evaluate one each until the chunk
// is done, and each lane adds its own results in candidate order.
// Either way every sum runs in candidate order and repeats bit for bit.
// ---------------------------------------------------------------------------
constexpr int kWarpsPerBlock = kBlock / 32;
constexpr int kChunk = 128;                // neighbours of a warp evaluated at a time

__device__ __forceinline__ uint32_t warp_exclusive_scan(uint32_t v, uint32_t* total) {
    const int lane = threadIdx.x & 31;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    *total = __shfl_sync(0xffffffffu, inc, 31);
    return inc - v;
}

// Shared state of one block's warps.  V: type of the pair terms.
template <class V>
struct ChunkShared {
    V v[kWarpsPerBlock][kChunk];               // pair terms
    uint32_t j[kWarpsPerBlock][kChunk];        // neighbour indexes
    uint8_t owner[kWarpsPerBlock][kChunk];     // lane of each
};

// Kernel values that pass 1 of the binary64 form leaves for pass 2: plane k
// holds s's k-th neighbour's, k < cap - 1 (pass 2 evaluates the others again).
struct PairValues {
    double* v;
    int cap;           // 0: none kept
};

// The adjoint's (K, dK): the e-th neighbour of a warp (lane-major) at
// first + e, for warps with at most 32 * cap neighbours.
struct AdjValues {
    double2* v;
    int cap;
    __device__ __forceinline__ double2* of_warp(uint32_t warp_s0, uint32_t total) const {
        return total <= 32u * uint32_t(cap) ? v + size_t(warp_s0) * size_t(cap) : nullptr;
    }
};

// Neighbour indexes out of kept words and lists.  The checked build takes the
// particle itself, whose flux is zero, in place of an index that an empty word or
// one beyond the particles would give.
struct KeptIndex {
#ifdef MTPT_CHECKED
    uint32_t n, self;
    __device__ __forceinline__ KeptIndex(uint32_t particles, uint32_t s) : n(particles), self(s) {}
    __device__ __forceinline__ uint32_t of_list(uint32_t j) const {
        return check(j < n, kChkSegment) ? j : self;
    }
    __device__ __forceinline__ uint32_t of_word(uint32_t base, uint32_t bits) const {
        return check(bits != 0u, kChkSegment) ? of_list(base + uint32_t(__ffs(int(bits)) - 1)) : self;
    }
#else
    __device__ __forceinline__ KeptIndex(uint32_t, uint32_t) {}
    __device__ __forceinline__ uint32_t of_list(uint32_t j) const { return j; }
    __device__ __forceinline__ uint32_t of_word(uint32_t base, uint32_t bits) const {
        return base + uint32_t(__ffs(int(bits)) - 1);
    }
#endif
};

// A particle's neighbours from its mask words (without padding), in order; the
// word after the current one is loaded ahead.
struct WordStream {
    const uint2* e;
    int64_t stride;
    uint32_t left;               // words after `ahead`
    uint2 cur, ahead;
    KeptIndex index;
    __device__ __forceinline__ WordStream(const uint2* first, int64_t st, uint32_t words,
                                          const KeptIndex& kept)
        : e(first), stride(st), left(words > 0u ? words - 1u : 0u), cur(make_uint2(0u, 0u)),
          ahead(words > 0u ? *first : make_uint2(0u, 0u)), index(kept) {}
    __device__ __forceinline__ uint32_t next() {
        if (cur.y == 0u) {
            cur = ahead;
            if (left > 0u) {
                ahead = *(e += stride);
                --left;
            }
        }
        const uint32_t j = index.of_word(cur.x, cur.y);
        cur.y &= cur.y - 1u;
        return j;
    }
};

// The dense part for the calling warp (all its lanes): listed is the lane's
// list word (0 for a lane without a particle, kMaskOver for one that searches
// on its own: both add nothing here).  eval(e, owner_s, j) returns the pair
// term of the warp's neighbour e, add(term) is called by each lane for its
// own, in order; begin(total) comes first.
template <class V, class Begin, class Eval, class Add>
__device__ __forceinline__ void dense_words(uint32_t s, uint32_t n, uint32_t listed, int64_t stride,
                                            const uint2* e, ChunkShared<V>& S, Begin&& begin,
                                            Eval&& eval, Add&& add) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, warp_s0 = s - lane;
    if (listed == kMaskOver) listed = 0;
    const uint32_t cnt = listed >> 8, words = listed & 255u;
    uint32_t total;
    const uint32_t off = warp_exclusive_scan(cnt, &total), end = off + cnt;
    begin(total);
    WordStream stream(e + s, stride, words, KeptIndex{n, s});
    uint32_t pos = off;
    for (uint32_t c0 = 0; c0 < total; c0 += kChunk) {
        const uint32_t m = min(total - c0, uint32_t(kChunk)), stop = min(end, c0 + m);
        for (; pos < stop; ++pos) {
            S.j[warp][pos - c0] = stream.next();
            S.owner[warp][pos - c0] = uint8_t(lane);
        }
        __syncwarp();
        for (uint32_t k = lane; k < m; k += 32)
            S.v[warp][k] = eval(c0 + k, warp_s0 + S.owner[warp][k], S.j[warp][k]);
        __syncwarp();
        for (uint32_t q = max(off, c0); q < stop; ++q) add(S.v[warp][q - c0]);
        __syncwarp();
    }
}

// Search of one particle of a binary64 pass: its list word, neighbour count in cnt
// (kMaskOver as soon as its words do not fit: the caller's search counts).
template <int DIM, class View>
__device__ __forceinline__ uint32_t search_listed(uint32_t s, int64_t stride,
                                                  const double* pos,
                                                  const float* rec,
                                                  const uint32_t* cell,
                                                  const uint32_t* start, const View& v,
                                                  const RealParams& P, const NbPlanes& nb,
                                                  uint32_t& cnt) {
    cnt = 0;
    if (nb.cap == 0) return kMaskOver;
    PlaneSink sink(nb, s, stride);
    const bool band = search_rows<DIM, true, false, false>(s, cell_arg<DIM>(cell, s), load_rec(rec, s),
                                                           stride, pos, rec, start, P,
                                                           [](uint32_t, float2, bool, bool) {}, sink);
    if (sink.full()) return kMaskOver;
    uint32_t nw = sink.nw;
    cnt = sink.cnt;
    if (band) {
        const float4 b = band_words<DIM, false>(s, cell, stride, pos, rec, start, v, nb, 0.0f, 0.0f);
        nw = __float_as_uint(b.z);
        cnt = __float_as_uint(b.w);
    }
    return mask_word(nw, cnt, nb.cap);
}

// Pass 1 of one particle whose neighbours the words do not hold: its row sum and,
// in .y's bits, its neighbours.
template <int DIM, class View>
__device__ __noinline__ double2 search_rowsum(uint32_t s, int64_t stride, const double* pos,
                                              const uint64_t* image, const float* rec,
                                              const uint32_t* cell, const uint32_t* start,
                                              const double* table, const View& v) {
    const RealParams& P = v.of_sorted(s);
    RowSum r;
    const uint32_t cnt = each_pair<DIM>(
        s, cell, stride, pos, rec, start, P, [&](uint32_t j0, uint32_t j1, bool two) {
            const double K0 = pair_kernel<DIM>(image, stride, s, j0, table, P.pp.kc);
            const double K1 = pair_kernel<DIM>(image, stride, s, j1, table, P.pp.kc);
            r.add(unit_of(K0));
            r.add(two ? unit_of(K1) : 0u);
        });
    return make_double2(r.value(), __longlong_as_double((long long)cnt));
}

// Pass 1, binary64 form: r_s = 1 + sum_{j != s} exp(-a d2_sj) (the kernel
// without its constant factor, which cancels in W; the self term is 1), and
// the ordered pair count.  The kernel values and their sum are fixed-point
// (expneg.cuh): no binary64 instruction, and the sum is exact whatever its
// order.  With binary64 operations the pass was bound by that unit (86 % busy):
// 732 us at 4e6 particles in 2-d with 5.7 neighbours each, 341 now, bound by
// instruction issue (72 %).  Two neighbours at a time (their loads and integer
// chains overlap); 40 registers, 48 in 3-d (four more blocks an SM do not help
// there: 54 instead of 52 us at 250,007).
template <int DIM, class View>
__global__ void __launch_bounds__(kBlock, DIM == 3 ? 5 : 6)
k_rowsum_f64(int n, int64_t stride, const double* pos,
             const uint64_t* image, const float* rec,
             const uint32_t* cell, const uint32_t* start,
             const double* __restrict__ exp_table, const __grid_constant__ View v,
             const double* mass, double2* __restrict__ rm,
             unsigned long long* __restrict__ pair_counter, const __grid_constant__ NbPlanes nb,
             uint32_t* __restrict__ listed_out, PairValues kv,
             const uint32_t* ghost_id) {
    __shared__ double table[kExpTable];
    // Ahead of the wait, here and in pass 2: a copy from the host wrote the table,
    // never a kernel, and it overlaps the kernel before (100 steps of 1e4
    // particles: 3.15 -> 3.06 ms; nothing at 4e6).  Without the table in shared
    // memory pass 2's dense runs took 1 % longer.
    for (int t = threadIdx.x; t < kExpTable; t += blockDim.x) table[t] = exp_table[t];
    const uint32_t s = ordered_index();
    __syncthreads();
    uint32_t cnt = 0;
    if (s < uint32_t(n)) {
        const RealParams& P = v.of_sorted(s);
        uint32_t listed = 0;
        double r = 1.0;
        if (P.transfer) {
            listed = search_listed<DIM>(s, stride, pos, rec, cell, start, v, P, nb, cnt);
            if (listed == kMaskOver) {
                const double2 rc = search_rowsum<DIM>(s, stride, pos, image, rec, cell, start, table, v);
                r = rc.x;
                cnt = uint32_t(__double_as_longlong(rc.y));
            } else {
                uint64_t xs[DIM];
#pragma unroll
                for (int a = 0; a < DIM; ++a) xs[a] = image[a * stride + s];
                RowSum sum;
                WordStream stream(nb.e + s, stride, listed & 255u, KeptIndex{uint32_t(n), s});
                auto kernel = [&](uint32_t j) {
                    uint64_t d2h = 0;
#pragma unroll
                    for (int a = 0; a < DIM; ++a) d2h += axis_square(xs[a], ld_global(image + a * stride + j));
                    return gauss_fixed(d2h, table, P.pp.kc);
                };
                double* keep = kv.v + s;
                uint32_t k = 0;
                for (; k + 2 <= cnt; k += 2) {
                    const uint32_t j0 = stream.next(), j1 = stream.next();
                    const double K0 = kernel(j0), K1 = kernel(j1);
                    if (k + 1u < uint32_t(kv.cap)) {
                        keep[0] = K0;
                        keep[stride] = K1;
                        keep += 2 * stride;
                    }
                    sum.add(unit_of(K0));
                    sum.add(unit_of(K1));
                }
                if (k < cnt) {
                    const double K = kernel(stream.next());
                    if (k + 1u < uint32_t(kv.cap)) *keep = K;
                    sum.add(unit_of(K));
                }
                r = sum.value();
            }
        }
        rm[s] = make_double2(r, mass[s]);
        if (listed_out) listed_out[s] = listed;
        // with ghost_id (a tile), pairs are counted for the tile's own particles only
        if (ghost_id && (ghost_id[s] & kGhostBit)) cnt = 0;
    }
    add_pair_count(cnt, pair_counter);
}

// Species B of a binary64 reaction run: its masses in place of A's in the
// records {r, m} that pass 2 reads.
__global__ void __launch_bounds__(kBlock)
k_record_mass(int n, const double* mass_b, double2* __restrict__ rm) {
    const int s = int(ordered_index());
    if (s < n) rm[s].y = mass_b[s];
}

// The next step's walk done at the end of pass 2 (walk-ahead, for the steps of
// one call that another step follows): particle s of this step's cell order
// keeps its index, and its walked position, its id, cell key and cell count
// go to the other buffer pair, which the next step's sort then reads as its
// input order.  The walk is latency-tolerant arithmetic (binary64 pipe,
// generator) and pass 2 waits on memory, so the two overlap in one kernel.
struct WalkAhead {
    const uint32_t* id_in;              // this step's ids (cell order)
    double* pos_next;                   // walked positions, same index
    uint32_t* id_next;                  // the ids, same index
    uint32_t* key;                      // cell keys of the next sort
    uint32_t* count;                    // cell counts of the next sort
    uint32_t* status;
    const unsigned long long* step_dev; // the walk's step counter, already advanced
    const uint32_t* rid_in = nullptr;   // a batch: realisation of each particle (cell order)
    uint32_t* rid_next = nullptr;       // a batch: the same, same index
};

// WALK selects the walk-ahead instance of a pass-2 kernel: 0 none, 1 the
// walk, 2 the walk with the advection term.
template <int DIM, int WALK>
__device__ __forceinline__ void walk_ahead(const RealParams& P, int s, int64_t stride,
                                           const double* pos, const WalkAhead& wa) {
    double x[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) x[a] = pos[a * stride + s];
    const uint32_t idv = wa.id_in[s];
    if (P.walk)
        walk_particle<DIM, false, WALK == 2>(P, idv - P.id_offset, *wa.step_dev, x, nullptr, stride, s);
#pragma unroll
    for (int a = 0; a < DIM; ++a) wa.pos_next[a * stride + s] = x[a];
    wa.id_next[s] = idv;
    if (wa.rid_next) wa.rid_next[s] = wa.rid_in[s];
    key_particle<DIM>(P, x, wa.status, wa.key + s, wa.count);
}

// Pass 2, binary64 form: M'_s = M_s + beta sum_j (M_j - M_s) 2 K_sj / (r_s + r_j).
// Weight, flux and sum are integer arithmetic (expneg.cuh), which leaves the
// binary64 unit the mass difference, one operation a pair of nine: 543 -> 283 us
// (4e6 particles, 2-d), 593 -> 336 with the next walk.
// Pass 2 of one particle whose neighbours the words do not hold.
template <int DIM, class View>
__device__ __noinline__ double search_flux_f64(uint32_t s, int64_t stride,
                                               const double* pos,
                                               const uint64_t* image,
                                               const float* rec,
                                               const uint32_t* cell,
                                               const uint32_t* start,
                                               const double* table, const View& v,
                                               const double2* rm) {
    const RealParams& P = v.of_sorted(s);
    const double2 me = rm[s];
    FluxSum64 sum;
    each_pair<DIM>(s, cell, stride, pos, rec, start, P, [&](uint32_t j0, uint32_t j1, bool two) {
        const double K0 = pair_kernel<DIM>(image, stride, s, j0, table, P.pp.kc);
        const double K1 = pair_kernel<DIM>(image, stride, s, j1, table, P.pp.kc);
        const double2 q0 = ld_global(rm + j0), q1 = ld_global(rm + j1);
        sum.add(__dsub_rn(q0.y, me.y), weight_fixed(K0, me.x, q0.x));
        if (two) sum.add(__dsub_rn(q1.y, me.y), weight_fixed(K1, me.x, q1.x));
    });
    return sum.value();
}

template <int DIM, class View, int WALK = 0>
__global__ void __launch_bounds__(kBlock, 5)
k_exchange_f64(int n, int64_t stride, const double* pos,
               const uint64_t* image, const float* rec,
               const uint32_t* cell, const uint32_t* start,
               const double* __restrict__ exp_table, const __grid_constant__ View v,
               const double2* rm, double* __restrict__ mass_out, NbPlanes nb,
               const uint32_t* listed_in, PairValues kv,
               const WalkAhead wa = WalkAhead{}) {
    __shared__ double table[kExpTable];   // of use to the particles that search or evaluate again
    for (int t = threadIdx.x; t < kExpTable; t += blockDim.x) table[t] = exp_table[t];
    const uint32_t s = ordered_index();   // (the table ahead of the wait, as in pass 1)
    __syncthreads();
    if (s >= uint32_t(n)) return;
    const RealParams& P = v.of_sorted(s);
    const double2 me = ld_global(rm + s);
    double m = me.y;
    if (P.transfer) {
        const uint32_t listed = listed_in ? listed_in[s] : kMaskOver;
        double flux;
        if (listed == kMaskOver) {
            flux = search_flux_f64<DIM>(s, stride, pos, image, rec, cell, start, table, v, rm);
        } else {
            const uint32_t cnt = listed >> 8;
            // pass 1's kernel values: whole pairs below the capacity
            const uint32_t kept = kv.cap > 0 ? min(cnt, uint32_t(kv.cap - 1) & ~1u) : 0u;
            const uint32_t listed_k = cnt < uint32_t(kv.cap) ? cnt : kept;
            FluxSum64 sum;
            WordStream stream(nb.e + s, stride, listed & 255u, KeptIndex{uint32_t(n), s});
            const double* keep = kv.v + s;
            uint32_t k = 0;
            for (; k + 2 <= listed_k; k += 2, keep += 2 * stride) {
                const uint32_t j0 = stream.next(), j1 = stream.next();
                const double K0 = ld_global(keep), K1 = ld_global(keep + stride);
                const double2 q0 = ld_global(rm + j0), q1 = ld_global(rm + j1);
                sum.add(__dsub_rn(q0.y, me.y), weight_fixed(K0, me.x, q0.x));
                sum.add(__dsub_rn(q1.y, me.y), weight_fixed(K1, me.x, q1.x));
            }
            for (; k < cnt; ++k) {
                const uint32_t j = stream.next();
                const double K = k < listed_k ? ld_global(keep)
                                              : pair_kernel<DIM>(image, stride, s, j, table, P.pp.kc);
                const double2 q = ld_global(rm + j);
                sum.add(__dsub_rn(q.y, me.y), weight_fixed(K, me.x, q.x));
            }
            flux = sum.value();
        }
        m = __dadd_rn(m, __dmul_rn(P.pp.beta, flux));
    }
    mass_out[s] = m;
    if constexpr (WALK > 0) walk_ahead<DIM, WALK>(P, int(s), stride, pos, wa);
}

// The particle's record that pass 2 reads per neighbour, written whole by pass
// 1: m = {m_hi, m_lo, r, list word (bits, see NbPlanes; of use to the particle
// itself only)}, the mass's binary32 head/tail split and the row sum.  Below
// 3-d it is preceded by a copy of the particle's rec, so that all of a
// neighbour's 32 bytes (from which pass 2 also forms K again) are one sector
// and one 32-byte load.
template <int DIM>
struct ExRec {
    static constexpr int kVec = DIM == 3 ? 1 : 2;   // float4 per particle
};
struct PairRec {
    float4 rec, m;
};
__device__ __forceinline__ PairRec load_pair_rec(const float4* ex, uint32_t j) {
    PairRec q;
    asm("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(q.rec.x), "=f"(q.rec.y), "=f"(q.rec.z), "=f"(q.rec.w), "=f"(q.m.x), "=f"(q.m.y),
          "=f"(q.m.z), "=f"(q.m.w)
        : "l"(ex + 2 * size_t(j)));
    return q;
}
__device__ __forceinline__ void store_pair_rec(float4* __restrict__ ex, uint32_t s, const float4& rec,
                                               const float4& m) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(ex + 2 * size_t(s)),
                 "f"(rec.x), "f"(rec.y), "f"(rec.z), "f"(rec.w), "f"(m.x), "f"(m.y), "f"(m.z), "f"(m.w)
                 : "memory");
}
template <int DIM>
__device__ __forceinline__ float4 load_ex(const float4* ex, uint32_t j) {
    return ld_global(ex + size_t(ExRec<DIM>::kVec) * j + (ExRec<DIM>::kVec - 1));
}

// Pass 1, precision form: binary32 kernel exp2(-a log2(e) d2f) with the
// hardware ex2, compensated binary32 row sum, rounded to binary32; written
// in the particle's record ex (ExRec); with nb.cap > 0 also what pass 2 needs
// of the search (NbPlanes).  Bound by instruction issue and the candidate loads'
// latency.  In 1-d and 2-d the accepted neighbours leave as mask words, one
// 8-byte store a row next to the other lanes' stores: a {j, K} list entry per
// neighbour was a partly written sector each, and those writes bounded the
// pass (2-d, 4e6 particles with 5.7 neighbours each: 218 us with lists, 170
// with masks; 1e7 with 57 each: 6.5 and 1.5 ms).  In 3-d (3.6 neighbours over
// nine rows) the list is the shorter of the two.
template <int DIM, class View>
__global__ void __launch_bounds__(kBlock, (DIM == 3 || View::kBatch ? 1536 : 2048) / kBlock)
k_rowsum_f32(int n, int64_t stride, const double* pos, const float* rec,
             const uint32_t* cell, const uint32_t* start,
             const __grid_constant__ View v, const double* mass,
             float4* __restrict__ ex, unsigned long long* __restrict__ pair_counter,
             const uint32_t* ghost_id, const __grid_constant__ NbPlanes nb,
             const double* mass_b, float2* __restrict__ exb) {
    const int s = int(ordered_index());
    uint32_t cnt = 0;
    if (s < n) {
        const RealParams& P = v.of_sorted(uint32_t(s));
        float rsum = 0.0f, rc = 0.0f;
        uint32_t list_word = 0;
        // compensated (Kahan) step for positive terms: rsum - rc carries the
        // sum; kept only for accepted pairs
        auto add = [&](float K, bool accept) {
            const float y = __fsub_rn(K, rc);
            const float t = __fadd_rn(rsum, y);
            const float cn = __fsub_rn(__fsub_rn(t, rsum), y);
            rsum = accept ? t : rsum;
            rc = accept ? cn : rc;
        };
        if (!P.transfer) {
            rsum = 1.0f;
        } else if constexpr (DIM == 3) {
            const float na = -P.pp.a_log2e;
            const uint32_t cap = uint32_t(nb.cap);
            uint2* lp = nb.e + s;          // slot `cnt` of s
            bool band;
            auto visit = [&](uint32_t j, float d2f, bool accept) {
                const float K = ex2_approx(na * d2f);
                add(K, accept);
                const bool keep = accept && j != uint32_t(s);
                if (keep && cnt < cap) *lp = make_uint2(j, __float_as_uint(K));
                if (keep) lp += stride;
                cnt += keep ? 1u : 0u;
            };
            NoSink none;
            band = search_rows<DIM, false, true, false>(uint32_t(s), cell[s], load_rec(rec, uint32_t(s)),
                                                        stride, pos, rec, start, P,
                                                        [&](uint32_t j, float2 d2, bool a0, bool a1) {
                                                            visit(j, d2.x, a0);
                                                            visit(j + 1u, d2.y, a1);
                                                        }, none);
            // the band's exact accepts come last
            if (band)
                scan_band<DIM>(uint32_t(s), cell[s], stride, rec, pos, start, P,
                               [&](uint32_t j, float d2f) { visit(j, d2f, true); });
            list_word = cnt;
        } else {
            const float na = -P.pp.a_log2e;
            PlaneSink sink(nb, uint32_t(s), stride);
            const bool band = search_rows<DIM, true, true, false>(
                uint32_t(s), 0u, load_rec(rec, uint32_t(s)), stride, pos, rec, start, P,
                [&](uint32_t, float2 d2, bool a0, bool a1) {
                    add(ex2_approx(na * d2.x), a0);
                    add(ex2_approx(na * d2.y), a1);
                }, sink);
            uint32_t nw = sink.nw;
            cnt = sink.cnt;
            if (band) {
                const float4 b = band_words<DIM, true>(uint32_t(s), cell, stride, pos, rec, start, v,
                                                       nb, rsum, rc);
                rsum = b.x;
                rc = b.y;
                nw = __float_as_uint(b.z);
                cnt = __float_as_uint(b.w);
            }
            list_word = mask_word(nw, cnt, nb.cap);
        }
        float mhi, mlo;
        split_double(mass[s], &mhi, &mlo);
        const float4 m = make_float4(mhi, mlo, __fsub_rn(rsum, rc), __uint_as_float(list_word));
        if constexpr (DIM == 3) ex[s] = m;
        else store_pair_rec(ex, uint32_t(s), load_rec(rec, uint32_t(s)), m);
        if (mass_b) {                      // a reaction: species B's split for pass 2
            split_double(mass_b[s], &mhi, &mlo);
            exb[s] = make_float2(mhi, mlo);
        }
        // with ghost_id (a tile), pairs are counted for the tile's own particles only
        if (ghost_id && (ghost_id[s] & kGhostBit)) cnt = 0;
    }
    add_pair_count(cnt, pair_counter);
}

// The flux sum of pass 2, precision form: W = 2 beta K / (r_s + r_j) in
// binary32 (symmetric bit for bit), the mass difference from the binary32
// head/tail split (exactly antisymmetric), compensated accumulation, and the
// update in binary64.  Each particle's record ex = {m_hi, m_lo, r, count} is one
// 16-byte load per neighbour.
struct FluxSum {
    float rs, two_beta;
    float2 ms;
    float acc = 0.0f, comp = 0.0f;
    // the pair's weight (shared by both species of a reaction run)
    __device__ __forceinline__ float weight(const float4& xj, float K) const {
        return __fdividef(two_beta * K, __fadd_rn(rs, xj.z));
    }
    // the flux of neighbour mass split mj under weight W
    __device__ __forceinline__ void add_w(float2 mj, float W, bool accept = true) {
        const float dm = __fadd_rn(__fsub_rn(mj.x, ms.x), __fsub_rn(mj.y, ms.y));
        // a rejected candidate (and the self pair) adds an exact zero
        neumaier_add(acc, comp, accept ? __fmul_rn(dm, W) : 0.0f);
    }
    __device__ __forceinline__ void add(const float4& xj, float K, bool accept = true) {
        add_w(make_float2(xj.x, xj.y), weight(xj, K), accept);
    }
    // two binary64 additions per particle: acc + comp is exact in binary64
    __device__ __forceinline__ double delta() const {
        return __dadd_rn(f32_to_f64(acc), f32_to_f64(comp));
    }
};

// ---------------------------------------------------------------------------
// Bimolecular reaction A + B -> 0 (the extension Sec. 8 names; the model is
// this library's reading).  After the transfer of both species with the same
// weights, each particle reacts well mixed over dt: with concentrations
// C = N M / V the rate law dC_A/dt = dC_B/dt = -k C_A C_B is
// da/dt = db/dt = -kp a b on its masses, kp = k N / V, solved exactly over
// dt.  With `big` the larger of a and b, x = kp (big - small) dt,
// phi(x) = (1 - e^-x) / x (phi(0) = 1) and q = 1 + kp small dt phi(x):
//   big' = big / q,   small' = small e^-x / q
// (the closed form a(t) = D a / (a - b e^-kpDt), D = a - b, rearranged so
// that neither D -> 0 nor the species in deficit loses digits).  A particle
// with a negative mass of either species (sign bit set) does not react.
// ---------------------------------------------------------------------------

// F64: binary64 throughout (exp, expm1 and IEEE division).  Otherwise (the
// precision form) the two factors 1/q and e^-x / q in binary32 from the
// binary32 heads of the masses (kpdt_f = kp dt rounded to binary32), each
// applied to its binary64 mass with one binary64 multiply.
template <bool F64>
__device__ __forceinline__ void react_masses(double& ma, double& mb, double kp, double dt,
                                             float kpdt_f) {
    const double a = ma, b = mb;
    const long long ka = __double_as_longlong(a), kb = __double_as_longlong(b);
    if ((ka | kb) < 0) return;                       // a negative mass: no reaction
    const bool a_big = ka >= kb;                     // non-negative values order by their bits
    const double big = a_big ? a : b, small = a_big ? b : a;
    double nbig, nsmall;
    if constexpr (F64) {
        const double x = __dmul_rn(__dmul_rn(kp, __dsub_rn(big, small)), dt);
        const double phi = x > 0.0 ? -expm1(-x) / x : 1.0;
        const double q = __dadd_rn(1.0, __dmul_rn(__dmul_rn(__dmul_rn(kp, small), dt), phi));
        nbig = big / q;
        nsmall = __dmul_rn(small, exp(-x)) / q;
    } else {
        float bh, bl, sh, sl;
        split_double(big, &bh, &bl);
        split_double(small, &sh, &sl);
        const float x = __fmul_rn(kpdt_f, __fsub_rn(bh, sh));
        const float phi = x > 0.0f ? __fdiv_rn(-expm1f(-x), x) : 1.0f;
        const float rq = __frcp_rn(__fmaf_rn(__fmul_rn(kpdt_f, sh), phi, 1.0f));
        nbig = __dmul_rn(big, f32_to_f64(rq));
        nsmall = __dmul_rn(small, f32_to_f64(__fmul_rn(expf(-x), rq)));
    }
    ma = a_big ? nbig : nsmall;
    mb = a_big ? nsmall : nbig;
}

template <bool F64>
__global__ void __launch_bounds__(kBlock)
k_react(int n, double* __restrict__ ma, double* __restrict__ mb, double kp, double dt,
        float kpdt_f) {
    const int s = int(ordered_index());
    if (s >= n) return;
    double a = ma[s], b = mb[s];
    react_masses<F64>(a, b, kp, dt, kpdt_f);
    ma[s] = a;
    mb[s] = b;
}

// The 32-byte records of neighbours j0 and, with `two`, j1 (both gathers in
// flight), their kernel formed by pass 1's operations from the same values,
// and their fluxes.
// WIDE: one 32-byte load a record (not in real calls: ptxas 13.0 crashes on
// it there), otherwise two of 16 bytes.
template <int DIM, bool TWO, bool WIDE>
struct PairFlux {
    const float4* ex;
    const float2* exb;
    float4 me;
    float na, wx, wy;
    KeptIndex index;
    __device__ __forceinline__ float kernel(const float4& o) const {
        const float sy = DIM == 2 ? __fmul_rn(__fsub_rn(o.z, me.z), wy) : 0.0f;
        return ex2_approx(na * d2_f32<DIM>(dx_f32(me, o, wx), me, o, sy, 0.0f));
    }
    __device__ __forceinline__ PairRec load(uint32_t j) const {
        if constexpr (WIDE) return load_pair_rec(ex, j);
        else return PairRec{ld_global(ex + 2 * size_t(j)), ld_global(ex + 2 * size_t(j) + 1)};
    }
    __device__ __forceinline__ void add(FluxSum& f, FluxSum& g, uint32_t j0, uint32_t j1,
                                        bool two) const {
        const PairRec q0 = load(j0), q1 = load(j1);
        if constexpr (TWO) {
            const float2 b0 = ld_global(exb + j0), b1 = ld_global(exb + j1);
            const float w0 = f.weight(q0.m, kernel(q0.rec)), w1 = f.weight(q1.m, kernel(q1.rec));
            f.add_w(make_float2(q0.m.x, q0.m.y), w0);
            g.add_w(b0, w0);
            f.add_w(make_float2(q1.m.x, q1.m.y), w1, two);
            g.add_w(b1, w1, two);
        } else {
            f.add(q0.m, kernel(q0.rec));
            f.add(q1.m, kernel(q1.rec), two);
        }
    }
};

// Pass 2 of a particle's mask words (padding included) word by word, the next
// word loaded ahead.
template <int DIM, bool TWO, bool WIDE>
__device__ __forceinline__ void add_words(const uint2* e, int64_t stride, uint32_t words,
                                          const PairFlux<DIM, TWO, WIDE>& pf, FluxSum& f, FluxSum& g) {
    uint2 ahead = ld_global(e);
    for (uint32_t w = 1; w <= words; ++w) {
        const uint32_t base = ahead.x;
        uint32_t bits = ahead.y;
        if (w < words) ahead = ld_global(e += stride);
        while (bits) {
            const uint32_t j0 = pf.index.of_word(base, bits);
            bits &= bits - 1u;
            const bool two = bits != 0u;
            const uint32_t j1 = two ? pf.index.of_word(base, bits) : j0;
            bits &= bits - 1u;
            pf.add(f, g, j0, j1, two);
        }
    }
}

// The same as a real call, for the few particles with more than three words of
// a run whose windows are short: its registers do not weigh on their loop.
// {acc_A, comp_A, acc_B, comp_B}.
template <int DIM, bool TWO>
__device__ __noinline__ float4 words_flux(const uint2* e, int64_t stride,
                                          uint32_t words, const float4* ex,
                                          const float2* exb, float4 me, float na,
                                          float wx, float wy, float rs, float two_beta, float2 ms,
                                          float2 msb, KeptIndex index) {
    const PairFlux<DIM, TWO, false> pf{ex, exb, me, na, wx, wy, index};
    FluxSum f{rs, two_beta, ms}, g{rs, two_beta, msb};
    add_words<DIM, TWO>(e, stride, words, pf, f, g);
    return make_float4(f.acc, f.comp, g.acc, g.comp);
}

// Pass 2 of one particle by search, in the order in which its list or masks
// hold its neighbours (3-d: the band's exact accepts last), for a particle
// they do not cover or when there are none; TWO: for both species of a reaction
// run (species B's mass split in exb).  Two candidates at a time, as in pass 1:
// 3-d, 300,007 particles with some 300 neighbours, beyond their lists: 2001 -> 1564
// us for two steps.  A real call, with few arguments, so its registers do not weigh
// on the list loop.  {acc_A, comp_A, acc_B, comp_B}.
template <int DIM, bool TWO, class View>
__device__ __noinline__ float4 search_flux(uint32_t s, int64_t stride, const double* pos,
                                           const float* rec, const uint32_t* cell,
                                           const uint32_t* start, const View& v, const float4* ex,
                                           const float2* exb) {
    const RealParams& P = v.of_sorted(s);
    const float na = -P.pp.a_log2e;
    const float4 xs = load_ex<DIM>(ex, s);
    FluxSum f{xs.z, float(2.0 * P.pp.beta), make_float2(xs.x, xs.y)};
    FluxSum g{xs.z, f.two_beta, TWO ? ld_global(exb + s) : make_float2(0.0f, 0.0f)};
    auto add = [&](uint32_t j, const float4& x, float d2f, bool accept) {
        const float w = f.weight(x, ex2_approx(na * d2f));
        f.add_w(make_float2(x.x, x.y), w, accept);
        if constexpr (TWO) g.add_w(ld_global(exb + j), w, accept);
    };
    const uint32_t c = cell_arg<DIM>(cell, s);
    NoSink none;
    const bool band = search_rows<DIM, false, true, DIM != 3>(
        s, c, load_rec(rec, s), stride, pos, rec, start, P,
        [&](uint32_t j, float2 d2, bool a0, bool a1) {
            if (!a0 && !a1) return;
            const uint32_t j1 = a1 ? j + 1u : j;       // (j + 1 may lie past the last particle)
            const float4 x0 = load_ex<DIM>(ex, j), x1 = load_ex<DIM>(ex, j1);
            add(j, x0, d2.x, a0);
            add(j1, x1, d2.y, a1);
        }, none);
    if (DIM == 3 && band)
        scan_band<DIM>(s, c, stride, rec, pos, start, P,
                       [&](uint32_t j, float d2f) { add(j, load_ex<DIM>(ex, j), d2f, true); });
    return make_float4(f.acc, f.comp, g.acc, g.comp);
}

// Pass 2, precision form: each particle walks the neighbours that pass 1 kept
// (3-d: its list, with pass 1's K; 1-d and 2-d: its mask words, with K formed
// again from the two records as pass 1 formed it), two at a time so two
// gathers are in flight, or searches when it has none or they do not cover
// it.  Both add the same terms in the same order.  Bound by the gathers'
// latency.  Masks in place of lists move 24 instead of 45 bytes a particle for
// eight more operations a neighbour: 104 us at 4e6 particles in 2-d (100 with
// lists), 1.3 ms at 1e7 with 57 neighbours (2.0).  Registers: 32 keep all 2048
// threads of an SM (four more would cost 4 us); both species need 40 (62 and 58
// us at 32 and 40 for the reaction at 1e6), a batch's view 36 (1.23, 1.15 and 1.19
// ms at 32, 36 and 40 for the 512-member ensemble).
// The bounds hold for blocks of 128 too (the tuning's other block size).
// LONG: for runs with long windows (padded words) or half-width cells, whose
// particles all go word by word, inline and with 32-byte loads (1.59 -> 1.39 ms at 1e7 particles with
// 57 neighbours, the next walk included).
template <int DIM, class View, bool TWO = false, int WALK = 0, bool LONG = false>
__global__ void __launch_bounds__(kBlock, (TWO ? 1536 : (View::kBatch || LONG ? 1792 : 2048)) / kBlock)
k_exchange_f32(int n, int64_t stride, const double* pos, const float* rec,
               const uint32_t* cell, const uint32_t* start,
               const __grid_constant__ View v, const float4* ex,
               const double* mass, double* __restrict__ mass_out, NbPlanes nb,
               const float2* exb = nullptr, const double* mass_b = nullptr,
               double* __restrict__ mass_b_out = nullptr, double kp = 0.0, double dt = 0.0,
               float kpdt_f = 0.0f, const WalkAhead wa = WalkAhead{}) {
    const int s = int(ordered_index());
    if (s >= n) return;
    const RealParams& P = v.of_sorted(uint32_t(s));
    if (!P.transfer) {
        if constexpr (TWO) {
            double a = mass[s], b = mass_b[s];
            react_masses<false>(a, b, kp, dt, kpdt_f);
            mass_out[s] = a;
            mass_b_out[s] = b;
        } else {
            mass_out[s] = mass[s];
        }
        if constexpr (WALK > 0) walk_ahead<DIM, WALK>(P, s, stride, pos, wa);
        return;
    }
    const float4 xs = load_ex<DIM>(ex, uint32_t(s));
    FluxSum f{xs.z, float(2.0 * P.pp.beta), make_float2(xs.x, xs.y)};   // beta folded into W
    FluxSum g{xs.z, f.two_beta, TWO ? ld_global(exb + s) : make_float2(0.0f, 0.0f)};
    const uint32_t listed = __float_as_uint(xs.w);   // see NbPlanes
    if (nb.cap > 0 && (DIM == 3 ? listed <= uint32_t(nb.cap) : listed != kMaskOver)) {
        const KeptIndex index{uint32_t(n), uint32_t(s)};
        if constexpr (DIM < 3) {
            const PairFlux<DIM, TWO, true> pf{ex, exb, ld_global(ex + 2 * size_t(s)), -P.pp.a_log2e,
                                              P.g.wf[0], P.g.wf[1], index};
            const uint2* e = nb.e + s;
            const uint32_t words = listed & 255u;
            if constexpr (LONG) {
                if (words) add_words<DIM, TWO>(e, stride, words, pf, f, g);
            } else if (words <= 3u) {
                // up to three words (a row each, at the densities where a row's
                // window stays below 32 candidates): one stream of neighbours
                // over them, so a warp runs as long as its longest particle's
                // count and not its rows'
                const uint2 none = make_uint2(0u, 0u);
                uint2 w0 = words > 0u ? ld_global(e) : none;
                uint2 w1 = words > 1u ? ld_global(e + stride) : none;
                const uint2 w2 = words > 2u ? ld_global(e + 2 * stride) : none;
                auto next = [&]() {
                    const bool shift = w0.y == 0u;
                    w0 = shift ? w1 : w0;
                    w1 = shift ? w2 : w1;
                    const uint32_t j = index.of_word(w0.x, w0.y);
                    w0.y &= w0.y - 1u;
                    return j;
                };
                uint32_t left = listed >> 8;
                for (; left >= 2u; left -= 2u) {
                    const uint32_t j0 = next();
                    pf.add(f, g, j0, next(), true);
                }
                if (left) {
                    const uint32_t j = next();
                    pf.add(f, g, j, j, false);
                }
            } else {
                const float4 sum = words_flux<DIM, TWO>(e, stride, words, ex, exb, pf.me, pf.na, pf.wx,
                                                        pf.wy, f.rs, f.two_beta, f.ms, g.ms, index);
                f.acc = sum.x;
                f.comp = sum.y;
                g.acc = sum.z;
                g.comp = sum.w;
            }
        } else {
            const uint2* e = nb.e + s;
            uint32_t k = 0;
            auto entry = [&](const uint2* p) {
                const uint2 q = ld_global(p);
                return make_uint2(index.of_list(q.x), q.y);
            };
            if constexpr (TWO) {
                for (; k + 2 <= listed; k += 2, e += 2 * stride) {
                    const uint2 q0 = entry(e), q1 = entry(e + stride);
                    const float4 x0 = ld_global(ex + q0.x), x1 = ld_global(ex + q1.x);
                    const float2 b0 = ld_global(exb + q0.x), b1 = ld_global(exb + q1.x);
                    const float w0 = f.weight(x0, __uint_as_float(q0.y));
                    f.add_w(make_float2(x0.x, x0.y), w0);
                    g.add_w(b0, w0);
                    const float w1 = f.weight(x1, __uint_as_float(q1.y));
                    f.add_w(make_float2(x1.x, x1.y), w1);
                    g.add_w(b1, w1);
                }
                if (k < listed) {
                    const uint2 q = entry(e);
                    const float4 x = ld_global(ex + q.x);
                    const float w = f.weight(x, __uint_as_float(q.y));
                    f.add_w(make_float2(x.x, x.y), w);
                    g.add_w(ld_global(exb + q.x), w);
                }
            } else {
                // two entries per iteration, the next two list entries loaded
                // while this pair's neighbour records are in flight
                uint2 p0 = listed > 0u ? entry(e) : make_uint2(uint32_t(s), 0u);
                uint2 p1 = listed > 1u ? entry(e + stride) : p0;
                for (; k + 2 <= listed; k += 2, e += 2 * stride) {
                    const uint2 q0 = p0, q1 = p1;
                    const float4 x0 = ld_global(ex + q0.x), x1 = ld_global(ex + q1.x);
                    p0 = k + 2 < listed ? entry(e + 2 * stride) : q0;
                    p1 = k + 3 < listed ? entry(e + 3 * stride) : q1;
                    f.add(x0, __uint_as_float(q0.y));
                    f.add(x1, __uint_as_float(q1.y));
                }
                if (k < listed) f.add(ld_global(ex + p0.x), __uint_as_float(p0.y));   // p0 = entry k
            }
        }
    } else {
        const float4 sum = search_flux<DIM, TWO>(uint32_t(s), stride, pos, rec, cell, start, v, ex, exb);
        f.acc = sum.x;
        f.comp = sum.y;
        g.acc = sum.z;
        g.comp = sum.w;
    }
    if constexpr (TWO) {
        // both species' transfer, then the reaction on this particle
        double a = __dadd_rn(mass[s], f.delta()), b = __dadd_rn(mass_b[s], g.delta());
        react_masses<false>(a, b, kp, dt, kpdt_f);
        mass_out[s] = a;
        mass_b_out[s] = b;
    } else {
        mass_out[s] = __dadd_rn(mass[s], f.delta());
    }
    if constexpr (WALK > 0) walk_ahead<DIM, WALK>(P, s, stride, pos, wa);
}

// Test support: every accepted ordered pair j != s as (id_s, id_j).
template <int DIM, class View>
__global__ void __launch_bounds__(kBlock)
k_emit_pairs(int n, int64_t stride, const double* __restrict__ pos, const float* __restrict__ rec,
             const uint32_t* __restrict__ cell, const uint32_t* __restrict__ start,
             const uint32_t* __restrict__ id, const __grid_constant__ View v,
             unsigned long long cap, unsigned long long* __restrict__ counter,
             uint32_t* __restrict__ out_i, uint32_t* __restrict__ out_j) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const RealParams& P = v.of_sorted(uint32_t(s));
    if (!P.transfer) return;
    const uint32_t ids = id[s];
    visit_neighbours<DIM>(uint32_t(s), cell_arg<DIM>(cell, s), stride, rec, pos, start, P,
                          [&](uint32_t j, float, const float4&) {
                              if (j == uint32_t(s)) return;
                              const unsigned long long k = atomicAdd(counter, 1ull);
                              if (k < cap) {
                                  out_i[k] = ids;
                                  out_j[k] = id[j];
                              }
                          });
}

// ---------------------------------------------------------------------------
// Adjoint of the step (binary64).  The mass update is M' = A M with
// A = I + beta (W - diag(W 1)) symmetric, so the mass adjoint is
// lambda_t = A lambda_{t+1}, the same pair sum with lambda in place of M.  The
// derivative with respect to D follows the positions' pathwise tangents
// (tan = dX/dD) and h^2 = 2 D_MT dt / beta (dh^2/dD = h^2 / D):
//   dK_ij/dD = K_ij (-(x_i - x_j).(t_i - t_j) + d2_ij / (2 D)) / h^2,
//   dr_i = sum_j dK_ij,
//   dW_ij = 2 dK_ij / (r_i + r_j) - 2 K_ij (dr_i + dr_j) / (r_i + r_j)^2,
// and step t adds beta sum_i lambda_{t+1,i} sum_j dW_ij (M_j - M_i) to dL/dD.
// Pair-set and bin changes contribute zero almost everywhere.
// ---------------------------------------------------------------------------
// The positions enter through their fixed-point images: distances, d2 and K are
// integer work, and the binary64 unit keeps seven operations a pair (the
// tangents' differences and products, K's last product, dK).  Returns K and
// h^2 dK/dD: the passes carry dK and dr times h^2, and pass B divides its sum.
template <int DIM>
__device__ __forceinline__ double2 pair_terms(const uint64_t* image,
                                              const double* tan, int64_t stride,
                                              uint32_t s, uint32_t j, const RealParams& P,
                                              const double* table) {
    const KernelConsts& kc = P.pp.kc;
    uint64_t d2h = 0;
    double dot = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const uint64_t xi = ld_global(image + a * stride + s), xj = ld_global(image + a * stride + j);
        const uint64_t d = axis_distance(xi, xj);
        d2h += square_hi(d);
        const double sign_d = double_of(bits_of(scaled(d, -kc.x_shift)) |
                                        ((xi - xj) & 0x8000000000000000ull));
        const double dt = __dsub_rn(ld_global(tan + a * stride + s), ld_global(tan + a * stride + j));
        dot = a == 0 ? __dmul_rn(sign_d, dt) : __fma_rn(sign_d, dt, dot);
    }
    const double K = gauss_fixed(d2h, table, kc);
    const double d2 = scaled(d2h, 64 - 2 * kc.x_shift);
    return make_double2(K, __dmul_rn(K, __fma_rn(d2, P.inv_2D, -dot)));
}

// The sums of pass A: the row sum exactly, its derivative in 64-bit integers.
struct AdjRowSum {
    RowSum r;
    AdjSum64 dr;
    __device__ __forceinline__ void add(double2 kd) {
        r.add(unit_of(kd.x));
        dr.add(kd.y);
    }
    __device__ __forceinline__ double2 value() const { return make_double2(r.value(), dr.value()); }
};
// The two passes of one particle whose neighbours the words do not hold.
template <int DIM, class View>
__device__ __noinline__ double2 adj_search_rowsum(uint32_t s, int64_t stride,
                                                  const double* pos,
                                                  const uint64_t* image,
                                                  const double* tan,
                                                  const float* rec,
                                                  const uint32_t* cell,
                                                  const uint32_t* start,
                                                  const double* table, const View& v) {
    const RealParams& P = v.of_sorted(s);
    AdjRowSum sum;
    each_pair<DIM>(s, cell, stride, pos, rec, start, P, [&](uint32_t j0, uint32_t j1, bool) {
        for (uint32_t j = j0;; j = j1) {
            sum.add(pair_terms<DIM>(image, tan, stride, s, j, P, table));
            if (j == j1) break;
        }
    });
    return sum.value();
}

// What pass B reads of a particle: {r, h^2 dr, M, lambda} as one 32-byte record.
struct AdjRec {
    double r, dr, mass, lam;
};
__device__ __forceinline__ AdjRec load_adj_rec(const double* rec4, uint32_t j) {
    AdjRec q;
    asm("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
        : "=d"(q.r), "=d"(q.dr), "=d"(q.mass), "=d"(q.lam)
        : "l"(rec4 + 4 * size_t(j)));
    return q;
}
__global__ void __launch_bounds__(kBlock)
k_adj_records(int n, const double* r, const double* dr,
              const double* mass, const uint32_t* id,
              const double* lam_in, double* __restrict__ rec4) {
    const int s = int(ordered_index());
    if (s >= n) return;
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(rec4 + 4 * size_t(s)), "d"(r[s]),
                 "d"(dr[s]), "d"(mass[s]), "d"(lam_in[id[s]])
                 : "memory");
}

// Half of one pair's terms of pass B, {W (lambda_j - lambda_s), h^2 dW (M_j - M_s)} / 2:
// with h = K / (r_s + r_j), W = 2 h and dW = 2 (dK - h (dr_s + dr_j)) / (r_s + r_j).
// The reciprocal is integer work, which leaves eight binary64 operations of
// nineteen.
__device__ __forceinline__ double2 adj_flux(double2 kd, const AdjRec& me, const AdjRec& o) {
    const double inv = Reciprocal(me.r, o.r).inverse().value();
    const double h = __dmul_rn(kd.x, inv);
    const double dh = __dmul_rn(inv, __fma_rn(-h, __dadd_rn(me.dr, o.dr), kd.y));
    return make_double2(__dmul_rn(h, __dsub_rn(o.lam, me.lam)),
                        __dmul_rn(dh, __dsub_rn(o.mass, me.mass)));
}
struct AdjFluxSum {
    AdjSum64 lam, gD;
    __device__ __forceinline__ void add(double2 t) {
        lam.add(t.x);
        gD.add(t.y);
    }
    __device__ __forceinline__ double2 value() const {
        return make_double2(lam.value(), gD.value());
    }
};

template <int DIM, class View>
__device__ __noinline__ double2 adj_search_flux(uint32_t s, int64_t stride,
                                                const double* pos,
                                                const uint64_t* image,
                                                const double* tan,
                                                const float* rec,
                                                const uint32_t* cell,
                                                const uint32_t* start,
                                                const double* table, const View& v,
                                                const double* rec4) {
    const RealParams& P = v.of_sorted(s);
    const double* mine = rec4 + 4 * size_t(s);
    const AdjRec me{mine[0], mine[1], mine[2], mine[3]};
    AdjFluxSum sum;
    each_pair<DIM>(s, cell, stride, pos, rec, start, P, [&](uint32_t j0, uint32_t j1, bool) {
        for (uint32_t j = j0;; j = j1) {
            sum.add(adj_flux(pair_terms<DIM>(image, tan, stride, s, j, P, table), me,
                             load_adj_rec(rec4, j)));
            if (j == j1) break;
        }
    });
    return sum.value();
}

// What one step leaves on the adjoint's tape beside its mask words and (K, dK)
// (see mtpt_adjoint_backward): with these, and none of the step's positions,
// cells or tangents, pass B runs.
struct TapeOut {
    const double* mass;          // masses entering the step, ids: cell order
    const uint32_t* id;
    double* mass_out;
    uint32_t* id_out;
    uint32_t* incomplete;        // set when a particle's words or a warp's values did not fit
};

// Pass A: r_s = sum_j K_sj (self included) and h^2 sum_j dK_sj / dD; with
// tape.mass_out also the rest of the step's tape.
template <int DIM, class View>
__global__ void __launch_bounds__(kBlock, 4)
k_adj_rowsum(int n, int64_t stride, const double* pos,
             const uint64_t* image, const double* tan,
             const float* rec, const uint32_t* cell,
             const uint32_t* start, const double* __restrict__ exp_table,
             const __grid_constant__ View v, double* __restrict__ r_out,
             double* __restrict__ dr_out, NbPlanes nb, uint32_t* __restrict__ listed_out,
             AdjValues kv, TapeOut tape) {
    __shared__ double table[kExpTable];
    __shared__ ChunkShared<double2> chunk;
    const uint32_t s = ordered_index();
    for (int t = threadIdx.x; t < kExpTable; t += blockDim.x) table[t] = exp_table[t];
    __syncthreads();
    const RealParams& P = v.of_sorted(s < uint32_t(n) ? s : 0u);
    const bool valid = s < uint32_t(n) && P.transfer;
    uint32_t listed = 0, cnt = 0;
    if (valid) listed = search_listed<DIM>(s, stride, pos, rec, cell, start, v, P, nb, cnt);
    AdjRowSum rows;
    double2* keep = nullptr;
    dense_words(
        s, uint32_t(n), listed, stride, nb.e, chunk,
        [&](uint32_t total) { keep = kv.of_warp(s - (threadIdx.x & 31u), total); },
        [&](uint32_t e, uint32_t so, uint32_t j) {
            const double2 kd = pair_terms<DIM>(image, tan, stride, so, j, v.of_sorted(so), table);
            if (keep) keep[e] = kd;
            return kd;
        },
        [&](double2 kd) { rows.add(kd); });
    if (s < uint32_t(n)) {
        double2 sum = rows.value();
        if (listed == kMaskOver)
            sum = adj_search_rowsum<DIM>(s, stride, pos, image, tan, rec, cell, start, table, v);
        r_out[s] = sum.x;
        dr_out[s] = sum.y;
        listed_out[s] = listed;
        if (tape.mass_out) {
            tape.mass_out[s] = tape.mass[s];
            tape.id_out[s] = tape.id[s];
            if (listed == kMaskOver || !keep) atomicOr(tape.incomplete, 1u);
        }
    }
}

// Pass B: lambda_t,s = lambda_s + beta sum_j W_sj (lambda_j - lambda_s) and the
// step's D-gradient terms g_s = beta lambda_s sum_j dW_sj (M_j - M_s), with M the
// masses entering the step, summed over the block in a fixed tree.
// Lambda goes back to input order at once.
//
// Both passes are bound by the binary64 unit and its latency together: 44 -> 36 us
// (A) and 54 -> 40 us (B) at 250,000 particles with 2.8 neighbours each when K,
// reciprocals and sums became integer work and the neighbour's four values one
// load (34 and 36 us of kernel time alone now); four blocks an SM (three and six: 7
// and 4 % slower sweeps).
template <int DIM, class View>
__global__ void __launch_bounds__(kBlock, 4)
k_adj_exchange(int n, int64_t stride, const double* pos,
               const uint64_t* image, const double* tan,
               const float* rec, const uint32_t* cell,
               const uint32_t* start, const double* __restrict__ exp_table,
               const __grid_constant__ View v, const double* rec4,
               const uint32_t* id, double* __restrict__ lam_out,
               double* __restrict__ gD_block, NbPlanes nb,
               const uint32_t* listed_in, AdjValues kv) {
    __shared__ double table[kExpTable];
    __shared__ ChunkShared<double2> chunk;
    const uint32_t s = ordered_index();
    for (int t = threadIdx.x; t < kExpTable; t += blockDim.x) table[t] = exp_table[t];
    __syncthreads();
    const RealParams& P = v.of_sorted(s < uint32_t(n) ? s : 0u);
    const bool valid = s < uint32_t(n) && P.transfer;
    const uint32_t listed = valid ? listed_in[s] : 0u;
    AdjFluxSum sums;
    double g = 0.0;
    const double2* keep = nullptr;
    dense_words(
        s, uint32_t(n), listed, stride, nb.e, chunk,
        [&](uint32_t total) { keep = kv.of_warp(s - (threadIdx.x & 31u), total); },
        [&](uint32_t e, uint32_t so, uint32_t j) {
            const AdjRec me = load_adj_rec(rec4, so), o = load_adj_rec(rec4, j);
            const double2 kd = keep ? ld_global(keep + e)
                                    : pair_terms<DIM>(image, tan, stride, so, j, v.of_sorted(so), table);
            return adj_flux(kd, me, o);
        },
        [&](double2 t) { sums.add(t); });
    if (s < uint32_t(n)) {
        double2 acc = sums.value();      // halves of the sums
        if (listed == kMaskOver)
            acc = adj_search_flux<DIM>(s, stride, pos, image, tan, rec, cell, start, table, v, rec4);
        const double ls = rec4[4 * size_t(s) + 3], two_beta = 2.0 * P.pp.beta;
        lam_out[id[s]] = valid ? __fma_rn(two_beta, acc.x, ls) : ls;
        if (valid) g = __dmul_rn(__dmul_rn(__dmul_rn(two_beta, P.inv_h2), ls), acc.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) g = __dadd_rn(g, __shfl_xor_sync(0xffffffffu, g, o));
    __shared__ double warp_g[kWarpsPerBlock];
    if ((threadIdx.x & 31) == 0) warp_g[threadIdx.x >> 5] = g;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kWarpsPerBlock; ++w) g = __dadd_rn(g, warp_g[w]);
        gD_block[blockIdx.x] = g;
    }
}

constexpr int kReduceThreads = 512;

// Deterministic sum of a step's (or a segment's) block sums.
// One block: thread t adds partial[t], partial[t + T], ... in order, then a
// fixed tree over the threads; the result is added to *acc.
__global__ void __launch_bounds__(kReduceThreads)
k_sum_into(int nparts, const double* partial, double* __restrict__ acc) {
    __shared__ double buf[kReduceThreads];
    double s = 0.0;
    for (int k = int(ordered_index()); k < nparts; k += kReduceThreads) s = __dadd_rn(s, partial[k]);
    buf[threadIdx.x] = s;
    __syncthreads();
    for (int w = kReduceThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) buf[threadIdx.x] = __dadd_rn(buf[threadIdx.x], buf[threadIdx.x + w]);
        __syncthreads();
    }
    if (threadIdx.x == 0) *acc = __dadd_rn(*acc, buf[0]);
}

// A per-particle binary64 array from input order into cell order.
__global__ void k_take_by_id(int n, const uint32_t* __restrict__ id, const double* __restrict__ src,
                             double* __restrict__ dst) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < n) dst[s] = src[id[s]];
}

// Row sums in input order and in the paper's units:
// out[id[s]] = r_s * kernel_norm of the particle's realisation.
template <typename T, class View>
__global__ void k_row_sums_out(int n, const uint32_t* __restrict__ id, const T* __restrict__ src,
                               int src_step, const __grid_constant__ View v,
                               double* __restrict__ out) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const RealParams& P = v.of_sorted(uint32_t(s));
    out[id[s]] = __dmul_rn(double(src[int64_t(s) * src_step]), P.kernel_norm);
}

// Outputs in input order: out[a * n + id[s]] = src[a * stride + s] * scale
// (binary32 sources widened exactly by integer operations; no multiply when
// scale is 1).
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) { return f32_to_f64(x); }

template <typename T>
__global__ void k_unpermute(int n, int64_t stride, int naxes, const uint32_t* id,
                            const T* src, int src_step, double scale,
                            double* __restrict__ out) {
    const int s = int(ordered_index());
    if (s >= n) return;
    const uint32_t k = id[s];
    if (!check(k < uint32_t(n), kChkOutput)) return;
    for (int a = 0; a < naxes; ++a) {
        const double x = widen(src[(a * stride + s) * src_step]);
        out[int64_t(a) * n + k] = scale == 1.0 ? x : __dmul_rn(x, scale);
    }
}

}  // namespace mtpt
