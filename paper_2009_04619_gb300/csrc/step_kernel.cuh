// Fused 25-point wave step with in-launch PML (sm_103a), templated on the
// wavefield storage type: fp32, fp16 with a per-field power-of-two scale, or
// bf16; the arithmetic is fp32 in every case.
//
// What it computes (arXiv 2009.04619, section III-A): one leapfrog step of
// Eq. 2, u^{n+1} = 2u^n - u^{n-1} + m L u^n with m = V^2 dt^2 and L the
// 25-point star Laplacian of Eq. 3, at every computed point of the inner
// region; a PML update at the points outside it (the paper names a PML and a
// 7-point stencil on an eta array but prints no formulas; the reading used
// is the single-stretch PML
//     u^{n+1} (1 + e) = (2 - e^2) u^n - (1 - e) u^{n-1} + m (L u^n + phi^n)
//     phi^{n+1} (1 + e) = phi^n - dt grad(eta) . grad(u^n)
// with e = eta dt, eta = eta_x(i) + eta_y(j) + eta_z(k), eta_a = eta_max
// (d_a / nb)^2 and 2nd-order central differences for both gradients); the
// point source of Eq. 2's right-hand side (Algorithm 1).
//
// How (a GB300 design; the paper's 2.5D register-streaming kernels of
// section IV are the starting idea, not the blueprint):
//  - one CTA owns a BX x BY tile of the x-y plane and streams a chunk of z
//    (2.5D blocking);
//  - planes of u^n arrive by TMA, with their radius-4 x-y halo, into an
//    NU-stage shared-memory ring (the 4 planes below and above a z-chunk are
//    only needed for the z-neighbours of the chunk's own points, so they come
//    without the halo, with an L2 evict-last hint for the neighbouring chunk
//    that reads them again); u^{n-1}, m and (PML planes only) phi tiles
//    into an NP-stage ring, with no evict-first hint because u^{n-1} and phi
//    are rewritten in place a few planes later; phi comes in 32-column blocks,
//    and a tile that touches only the x-PML loads only the blocks holding PML
//    columns outside the z-PML; one lane of a dedicated producer warp issues the
//    copies in the order the consumers need them, as far ahead as the rings
//    allow; "full" mbarriers carry copy completion to the consumer warps and
//    "empty" mbarriers (one arrival per consumer warp) carry slot release back
//    to the producer, so there is no block-wide barrier in the z loop;
//  - each thread owns 4 consecutive x points (128-bit accesses) in TY rows;
//    the z-neighbours of its points sit in a register queue (the paper's
//    register-streaming idea, section IV) that moves by one place per plane.
//    Full 9-fold unrolling (the paper's st_reg_fixed form, no moves at all)
//    measured slower on GB300: its code no longer fits the instruction cache.
//    Partial sums that move with each multiply-add need no moves either, but
//    lengthen the start of every chunk and spill in the PML planes;
//  - whether a plane takes the PML path depends only on the tile and k, so
//    the branch is uniform across the CTA: the z range of a tile splits into
//    segments of three plane kinds (interior; PML path outside the z-PML, where
//    1/(1+e) and 1-e come from per-thread tables; z-PML), each a separately
//    compiled loop, and compiled once; inside a PML-path plane, inner points select the Eq. 2
//    result computed by the same instructions as the interior path, bit for bit;
//  - what bounds it: two warps per scheduler run a plane's chain of about 330
//    (interior) to 450 (PML) instructions each, DRAM at 84-92% of the measured
//    copy rate beside them, so instructions count: ring positions are running
//    offsets with the barriers at a fixed place in each slot, what a thread has
//    to know about its points is one word of flags, both waits of a plane are
//    polled at once, the x taps and the PML update are packed pairs, and each
//    plane kind is compiled once (83 -> 46 KB of code).  Per step, before and
//    after: 512^3 + PML 32 411 -> 403 us, 256^3 + PML 16 63.1 -> 61.5 us, 96^3
//    7.6 -> 7.2 us; bf16 at 512^3 427 -> 362 us and fp16 at 384 x 384 x 256 143 -> 126
//    us, with bf16 pairs unpacked by shift and mask (-13 us), no spilled values
//    (-10 us) and 32 x 32 tiles (-11 us), the bf16 figures.  No register may spill:
//    beside 2 x 113 KB of shared memory the L1 holds
//    a few KB, and a spilled value read in the z loop comes from L2 (80 bytes of
//    spills took 256^3 from 65 to 95 us);
//  - eta and its central differences are evaluated in closed form from the
//    integer depth into the layer: no eta array is read;
//  - every mbarrier wait is bounded (2 s); on timeout the CTA records
//    DEV_ERR_TIMEOUT, drains its own copies (bounded) and exits;
//  - 16-bit storage keeps only the two wavefields in 16 bits (m and phi stay
//    fp32).  The Laplacian is accumulated on the stored values and multiplied
//    by the field's scale once.  The fp16 scale of u^{n+1} is a power of two
//    chosen in the kernel from max|u^n|, max|u^{n-1}| and the injected
//    amplitude, so that |u^{n+1}| / scale < 2^14 (fp16 max 65504); every CTA
//    also contributes max|u^{n+1}| (warp max + atomicMax) for the next step.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "ptx.cuh"

namespace sgb {

constexpr int R = 4;          // stencil radius (half the spatial order)
constexpr int HALO_LO_X = 8;  // zero points before computed x = 0 (16-byte aligned origin)
constexpr int HALO = 4;       // zero points before y = 0, z = 0 and after every axis

enum : int { DEV_ERR_TIMEOUT = 1, DEV_ERR_NONFINITE = 2, DEV_ERR_RANGE = 4 };

// Kernel modes: the forward step; the forward step that also stores its
// acceleration term g^n = L u^n + phi^n + f^n (recomputation for the adjoint);
// the adjoint step (see adjoint notes below).
// MODE_DIFF: the forward step in difference form. The state is (u^n, d^n) with
// d^n = u^n - u^{n-1} instead of (u^n, u^{n-1}): the same scheme in exact
// arithmetic, but a rounding error stored in u no longer also enters the time
// difference, so stored 16-bit values lose far less (each field keeps its own
// relative precision). d is read through the u^{n-1} tile map and updated in
// place through d_io; u^{n+1} goes to u_out.
enum : int { MODE_FWD = 0, MODE_FWD_ACC = 1, MODE_ADJ = 2, MODE_DIFF = 3 };

// Plane kinds of a work unit (compile-time paths of the plane body).
enum : int { PLANE_INTERIOR = 0, PLANE_XY = 1, PLANE_Z = 2 };

// Scale state of a 16-bit wavefield pair (device memory): s[k & 3] is the
// scale of u^k (stored value = u^k / s), mx[k & 3] is max |u^k|.
struct ScaleState {
    float s[4];
    float mx[4];
};

struct StepArgs {
    void *u_out;           // padded base: holds u^{n-1} on entry, u^{n+1} on exit
    void *d_io;            // MODE_DIFF: padded base of d^n on entry, d^{n+1} on exit
    const void *u_cur;     // padded base of u^n (receiver pre-sampling only)
    float *phi;            // padded base of phi (PML auxiliary field, fp32)
    int Nx, Ny, Nz;        // computed extents
    int nb, nx, ny, nz;    // PML width, inner extents
    long long sx, sxy;     // element strides of y and z
    long long origin;      // element offset of computed (0, 0, 0)
    float c0;              // centre coefficient of Eq. 3
    float cx[4], cy[4], cz[4];
    float ax, ay, az;      // eta_a dt = a * d^2
    float kx, ky, kz;      // dt d(eta)/da d(u)/da = k (d(+1)^2 - d(-1)^2) (u(+1) - u(-1))
    int si, sj, sk;        // source point (sk < 0: none)
    const float *wavelet;  // w(n dt) samples
    const float *m_src;    // m at the source point (fp16 scale bound)
    float inv_vol;         // 1 / (dx dy dz)
    const int *step_ptr;   // device step counter (graph replays) or null
    int step_add;          // n = *step_ptr + step_add
    int nrec;              // receivers sampled from u^n into row n - 1 - rec_n0 (n > rec_n0)
    int rec_n0;            // first step of the traces buffer (a shot segment's first step)
    const long long *rec_off;
    float *traces;
    ScaleState *scale;     // fp16 storage only
    ScaleState *scale_d;   // fp16 storage in MODE_DIFF: scales and maxima of d
    float *acc_out;        // MODE_FWD_ACC: g = L u^n + phi^n + f^n (padded fp32)
    float *gsum;           // MODE_ADJ: fp32 partial sum of w^k g^{k-1} (padded)
    const float *mu_in;    // MODE_ADJ: mu^{k+1} (padded); phi is mu^k
    // MODE_ADJ: the residual of step k - 1 enters w^k at the receivers. rec_off
    // then lists them grouped by the work unit that computes them: those of unit
    // u are rec_start[u] .. rec_start[u + 1] - 1, in the order of their offsets,
    // receiver rec_idx[q] of the rows (rec_lo, rec_hi: the box they lie in, inclusive)
    const int *rec_start, *rec_idx;
    const float *tr_row, *obs_row;  // traces and observed samples of step k - 1
    const float *m_all, *acc_in;    // m and g^{k-1} (padded)
    int rec_lo[3], rec_hi[3];
    int *err;              // device error word
    int tiles_x, tiles_y, zc;
    // shell launches of a temporally blocked pair: work units (x0, y0, z0, z1)
    // from a table, and no store inside the box [bx0,bx1) x [by0,by1) x
    // [bz0,bz1), which the two-step kernel writes
    const int4 *units;
    int bx0, bx1, by0, by1, bz0, bz1;
};

// Counter-based hash (Murmur3 finaliser) of a point index and a step: the random
// bits of stochastic rounding, reproducible run to run.  One hash is drawn per
// thread and plane; the other 32-bit words that thread needs for the plane come
// from it by an odd multiply (a bijection of 2^32, so each word is uniform when
// the hash is, and its low half is a permutation of the hash's low half): see
// next_bits and Elem<T>::st.
__device__ __forceinline__ uint32_t hash_bits(uint32_t a, uint32_t b)
{
    uint32_t h = a * 0x9E3779B1u ^ (b + 0x7F4A7C15u);
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    return h;
}

// Next random word of the same thread and plane (another row's quad).
__device__ __forceinline__ uint32_t next_bits(uint32_t h)
{
    return (h ^ (h >> 16)) * 0x45D9F3Bu;
}

// Stochastic rounding of an fp32 pair to 16 bits in the conversion itself
// (the cvt.rs form of sm_100-family GPUs, fed 32 random bits): each value
// rounds up with probability equal to its distance from the lower neighbour.
// With round-to-nearest, the rounding errors of a smooth field repeat from
// step to step and add up coherently over a run; stochastic rounding makes
// them uncorrelated (zero mean), so they grow like a random walk instead.
// The first source operand of the pair conversion lands in the upper half.
__device__ __forceinline__ uint32_t cvt_rs_f16x2(float lo, float hi, uint32_t rnd)
{
    uint32_t d;
    asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(rnd));
    return d;
}

__device__ __forceinline__ uint32_t cvt_rs_bf16x2(float lo, float hi, uint32_t rnd)
{
    uint32_t d;
    asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(rnd));
    return d;
}

// The first n (1..3) of four fp32 values: the quad that crosses the grid's last
// column. Straight-line predicated stores: a loop over n here made the tiles at
// a ragged edge the slowest of the grid (343 columns: 81 us a step, 344: 62).
__device__ __forceinline__ void st_part(float *p, const float4 &v, int n)
{
    if (n > 0) p[0] = v.x;
    if (n > 1) p[1] = v.y;
    if (n > 2) p[2] = v.z;
}
// The same of two words of packed 16-bit pairs.
__device__ __forceinline__ void st_part16(void *p, const uint2 &r, int n)
{
    uint16_t *q = static_cast<uint16_t *>(p);
    if (n > 0) q[0] = (uint16_t)r.x;
    if (n > 1) q[1] = (uint16_t)(r.x >> 16);
    if (n > 2) q[2] = (uint16_t)r.y;
}

// Storage traits: TMA x margin (16 bytes), 4-wide loads from shared memory and
// stores to global memory (rnd: random bits for stochastic rounding; FULL: all
// four values, else the first n), scalar reads.
template <class T>
struct Elem;

template <>
struct Elem<float> {
    static constexpr int HX = 4;
    static constexpr bool SCALED = false;
    __device__ static __forceinline__ float4 ld(const float *p) { return lds128(p); }
    template <bool FULL>
    __device__ static __forceinline__ void st(float *p, float4 v, uint32_t, int n)
    {
        if (FULL) stg128(p, v);
        else st_part(p, v, n);
    }
    __device__ static __forceinline__ float get(const float *p) { return *p; }
};

template <>
struct Elem<__half> {
    static constexpr int HX = 8;
    static constexpr bool SCALED = true;
    __device__ static __forceinline__ float4 ld(const __half *p)
    {
        const uint2 r = *reinterpret_cast<const uint2 *>(p);
        const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&r.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&r.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    __device__ static __forceinline__ __half2 pack(float x, float y, uint32_t rnd)
    {
#ifdef SGB_16BIT_RN
        (void)rnd;
        return __floats2half2_rn(x, y);
#else
        const uint32_t d = cvt_rs_f16x2(x, y, rnd);
        return *reinterpret_cast<const __half2 *>(&d);
#endif
    }
    template <bool FULL>
    __device__ static __forceinline__ void st(__half *p, float4 v, uint32_t rnd, int n)
    {
        // the second pair's word: an odd multiple of the first (cheap, uniform)
        __half2 a = pack(v.x, v.y, rnd), b = pack(v.z, v.w, rnd * 0x9E3779B1u);
        uint2 r;
        r.x = *reinterpret_cast<uint32_t *>(&a);
        r.y = *reinterpret_cast<uint32_t *>(&b);
        if (FULL) *reinterpret_cast<uint2 *>(p) = r;
        else st_part16(p, r, n);
    }
    __device__ static __forceinline__ float get(const __half *p) { return __half2float(*p); }
};

template <>
struct Elem<__nv_bfloat16> {
    static constexpr int HX = 8;
    static constexpr bool SCALED = false;
    __device__ static __forceinline__ float4 ld(const __nv_bfloat16 *p)
    {
        const uint2 r = *reinterpret_cast<const uint2 *>(p);
        return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u),
                           __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xffff0000u));
    }
    __device__ static __forceinline__ __nv_bfloat162 pack(float x, float y, uint32_t rnd)
    {
#ifdef SGB_16BIT_RN
        (void)rnd;
        return __floats2bfloat162_rn(x, y);
#else
        const uint32_t d = cvt_rs_bf16x2(x, y, rnd);
        return *reinterpret_cast<const __nv_bfloat162 *>(&d);
#endif
    }
    template <bool FULL>
    __device__ static __forceinline__ void st(__nv_bfloat16 *p, float4 v, uint32_t rnd, int n)
    {
        // the second pair's word: an odd multiple of the first (cheap, uniform)
        __nv_bfloat162 a = pack(v.x, v.y, rnd), b = pack(v.z, v.w, rnd * 0x9E3779B1u);
        uint2 r;
        r.x = *reinterpret_cast<uint32_t *>(&a);
        r.y = *reinterpret_cast<uint32_t *>(&b);
        if (FULL) *reinterpret_cast<uint2 *>(p) = r;
        else st_part16(p, r, n);
    }
    __device__ static __forceinline__ float get(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
};

constexpr int align128(int b) { return (b + 127) / 128 * 128; }

template <int TXT_, int TYT_, int TY_, int NU_, int NP_, int MINB_>
struct TileCfg {
    static constexpr int TXT = TXT_, TYT = TYT_, TY = TY_, NU = NU_, NP = NP_, MINB = MINB_;
    static constexpr int QN = 2 * R + 1;  // register-queue length
    static constexpr int THREADS = TXT * TYT;   // consumer (compute) threads
    static constexpr int BLOCK = THREADS + 32;  // plus one producer warp
    static constexpr int BX = 4 * TXT, BY = TY * TYT;
    static constexpr int SH = BY + 2 * R;
    static constexpr int P_TILE = BX * BY;
    static constexpr int WARPS = THREADS / 32;
    // phi (or mu) tiles travel as PHI_BW-column blocks, stored block after
    // block in shared memory, so that a tile touching only the x-PML can load
    // just the blocks that hold PML columns
    static constexpr int PHI_BW = 32, PHI_NB = BX / PHI_BW;
    static_assert(NU >= 8, "the u ring must hold the 8 planes that prime the register queue");
    static_assert(BX % PHI_BW == 0 && PHI_NB <= 8, "phi blocks");
    static_assert(TY <= 2, "flag bits of a thread's rows");
    static_assert(NP >= 2 && THREADS % 32 == 0, "ring sizes");
    static_assert(SH <= 256 && BX <= 240 && BY <= 256, "TMA box limits");
};

// Dynamic shared memory of the step kernels (no static shared memory, so the TMA
// destinations start at the aligned base).
extern __shared__ __align__(128) unsigned char step_smem[];

// Shared-memory geometry of a configuration for storage type T (bytes).
template <class C, class T, int MODE = MODE_FWD>
struct Stage {
    static constexpr int HX = Elem<T>::HX;         // x margin of the u^n box
    static constexpr int SW = C::BX + 2 * HX;      // u^n box width (elements)
    static constexpr int U_BYTES = align128(SW * C::SH * (int)sizeof(T));
    static constexpr int UP_BYTES = align128(C::P_TILE * (int)sizeof(T));
    static constexpr int F_BYTES = C::P_TILE * 4;  // one fp32 tile (m, phi, g, S)
    // the adjoint's mu^{k+1} tile carries its x-y neighbours: a (BX + 8) x (BY + 2)
    // box (x halo 4 for the TMA's 16-byte alignment, y halo 1)
    static constexpr int MBW = C::BX + 8, MBH = C::BY + 2;
    static constexpr int MU_BYTES = align128(MBW * MBH * 4);
    static constexpr int PH_BYTES = MODE == MODE_ADJ ? MU_BYTES : F_BYTES;  // phi or mu slot
    static constexpr int P_BYTES = UP_BYTES + F_BYTES + PH_BYTES + (MODE == MODE_ADJ ? 2 : 0) * F_BYTES;
    // MODE_ADJ: mu^{k+1} one plane below each thread's points, kept from plane to
    // plane in shared memory (registers are at their limit)
    static constexpr int MZ_BYTES = MODE == MODE_ADJ ? C::THREADS * C::TY * 16 : 0;
    // ring depths: 16-bit storage halves the stages' bytes, so its rings run deeper
    // (12 u^n planes and 6 tile stages in ~108 KB, still two CTAs per SM)
#ifndef SGB_NU16
#define SGB_NU16 12
#endif
#ifndef SGB_NP16
#define SGB_NP16 6
#endif
    static constexpr int NU = sizeof(T) == 2 ? SGB_NU16 : C::NU;
    static constexpr int NP = sizeof(T) == 2 ? SGB_NP16 : C::NP;
    // a slot: its tiles, then its full and empty barriers
    static constexpr int U_PITCH = U_BYTES + 128, P_PITCH = P_BYTES + 128;
    static constexpr int MZ_OFF = NU * U_PITCH + NP * P_PITCH, ABORT_OFF = MZ_OFF + MZ_BYTES;
    static constexpr size_t SMEM_BYTES = size_t(ABORT_OFF) + 8;
    static_assert(U_BYTES % 128 == 0 && F_BYTES % 128 == 0, "stage alignment");
    static_assert(SW <= 256, "TMA box limit");
};

// Depth (points) of index i into the PML along one axis; 0 in the inner range.
__device__ __forceinline__ int pml_depth(int n_inner, int nb, int i)
{
    return max(max(nb - i, i - (nb + n_inner - 1)), 0);
}

__device__ __forceinline__ float f4get(const float4 &v, int e)
{
    return e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w;
}
__device__ __forceinline__ void f4set(float4 &v, int e, float s)
{
    if (e == 0) v.x = s;
    else if (e == 1) v.y = s;
    else if (e == 2) v.z = s;
    else v.w = s;
}
// acc += c * v on a float4 as two packed f32x2 FMAs.
__device__ __forceinline__ void f4fma(float4 &acc, float c, const float4 &v)
{
    const float2 cc = make_float2(c, c);
    float2 lo = __ffma2_rn(cc, make_float2(v.x, v.y), make_float2(acc.x, acc.y));
    float2 hi = __ffma2_rn(cc, make_float2(v.z, v.w), make_float2(acc.z, acc.w));
    acc = make_float4(lo.x, lo.y, hi.x, hi.y);
}

__device__ __forceinline__ float4 f4mul(float c, const float4 &v)
{
    const float2 cc = make_float2(c, c);
    float2 lo = __fmul2_rn(cc, make_float2(v.x, v.y));
    float2 hi = __fmul2_rn(cc, make_float2(v.z, v.w));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// a * b + c, a * b, a + b and a - b element by element: packed pairs, each
// operation rounded once.
__device__ __forceinline__ float4 f4fma4(const float4 &a, const float4 &b, const float4 &c)
{
    const float2 lo = __ffma2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y), make_float2(c.x, c.y));
    const float2 hi = __ffma2_rn(make_float2(a.z, a.w), make_float2(b.z, b.w), make_float2(c.z, c.w));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ float4 f4mul4(const float4 &a, const float4 &b)
{
    const float2 lo = __fmul2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
    const float2 hi = __fmul2_rn(make_float2(a.z, a.w), make_float2(b.z, b.w));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ float4 f4add4(const float4 &a, const float4 &b)
{
    const float2 lo = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
    const float2 hi = __fadd2_rn(make_float2(a.z, a.w), make_float2(b.z, b.w));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ float4 f4sub(const float4 &a, const float4 &b)
{
    float4 r = a;
    f4fma(r, -1.0f, b);
    return r;
}
// L plus the x part of Eq. 3 at the quad c, from the quads left and right of it.
// The taps at even distance meet aligned pairs for the output pairs (0, 1) and
// (2, 3), those at odd distance for the pair (1, 2); outputs 0 and 3 take their
// odd taps one by one: 22 instructions instead of 32.
__device__ __forceinline__ float4 lap_x(const float4 &L, const float (&cx)[4], const float4 &lf,
                                        const float4 &c, const float4 &rt)
{
    const float2 l0 = make_float2(lf.x, lf.y), l1 = make_float2(lf.z, lf.w);
    const float2 c0 = make_float2(c.x, c.y), c1 = make_float2(c.z, c.w);
    const float2 r0 = make_float2(rt.x, rt.y), r1 = make_float2(rt.z, rt.w);
    const float2 k1 = make_float2(cx[0], cx[0]), k2 = make_float2(cx[1], cx[1]);
    const float2 k3 = make_float2(cx[2], cx[2]), k4 = make_float2(cx[3], cx[3]);
    float2 lo = make_float2(L.x, L.y), hi = make_float2(L.z, L.w);
    float2 mid = __fmul2_rn(k1, c0);
    lo = __ffma2_rn(k2, l1, lo);
    hi = __ffma2_rn(k2, c0, hi);
    mid = __ffma2_rn(k1, c1, mid);
    lo = __ffma2_rn(k2, c1, lo);
    hi = __ffma2_rn(k2, r0, hi);
    mid = __ffma2_rn(k3, l1, mid);
    lo = __ffma2_rn(k4, l0, lo);
    hi = __ffma2_rn(k4, l1, hi);
    mid = __ffma2_rn(k3, r0, mid);
    lo = __ffma2_rn(k4, r0, lo);
    hi = __ffma2_rn(k4, r1, hi);
    float x = fmaf(cx[0], l1.y, lo.x), w = fmaf(cx[0], c1.x, hi.y);
    x = fmaf(cx[0], c0.y, x);
    w = fmaf(cx[0], r0.x, w);
    x = fmaf(cx[2], l0.y, x);
    w = fmaf(cx[2], c0.x, w);
    x = fmaf(cx[2], c1.y, x);
    w = fmaf(cx[2], r1.x, w);
    return make_float4(x, __fadd_rn(lo.y, mid.x), __fadd_rn(hi.x, mid.y), w);
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Launch variants of the step: one launch per step over the standard units;
// the shell launches of a temporally blocked pair (units from a table, no store
// inside the two-step kernel's box); the persistent dataflow launch (CTAs take
// (step, unit) items in turn, ring slots counted across units); one launch per
// step whose output buffer is chosen on the device by the parity of the step
// (CUDA-graph replays that do not repeat with the buffer parity).
enum : int { VAR_PLAIN = 0, VAR_SHELL = 1, VAR_FLOW = 2, VAR_PARITY = 3 };

// Position in a ring of N slots of PITCH bytes: the slot's byte offset and the
// parity of the current pass over the ring.
template <int N, int PITCH>
struct RingPos {
    uint32_t off = 0, ph = 0;
    __device__ __forceinline__ void next()
    {
        off += PITCH;
        if (off == N * PITCH) {
            off = 0;
            ph ^= 1;
        }
    }
    // offset of the slot `back` places behind (back < N)
    __device__ __forceinline__ uint32_t behind(int back) const
    {
        return off >= uint32_t(back) * PITCH ? off - back * PITCH : off + (N - back) * PITCH;
    }
    // parity of the last fill of slot s, counting fills up to this position
    // (a slot that was never filled: a parity that a fresh barrier satisfies)
    __device__ __forceinline__ uint32_t last_parity(int s) const
    {
        return uint32_t(s) * PITCH < off ? ph : ph ^ 1;
    }
};

// Per-thread state of one fused-step work unit (a tile x a z-chunk).
template <class C, class T, int MODE = MODE_FWD, int VAR = VAR_PLAIN>
struct StepCta {
    static constexpr bool SHELL = VAR == VAR_SHELL, FLOW = VAR == VAR_FLOW;
    static constexpr bool OUTV = VAR == VAR_FLOW || VAR == VAR_PARITY;  // output via u_out_v
    using E = Elem<T>;
    using G = Stage<C, T, MODE>;
    // the adjoint's PML-path band is one point wider: inner points next to the
    // PML receive psi from their PML neighbours
    static constexpr int BAND = MODE == MODE_ADJ ? 1 : 0;
    static constexpr bool SCALED = E::SCALED;
    static constexpr int TXT = C::TXT, TY = C::TY, NU = G::NU, NP = G::NP;
    static constexpr int THREADS = C::THREADS, QN = C::QN, WARPS = C::WARPS;
    static constexpr int BX = C::BX, BY = C::BY, HX = G::HX, SW = G::SW;
    static constexpr int P_TILE = C::P_TILE;
    static constexpr uint64_t WAIT_NS = 2000000000ull;
    // offsets inside a tile slot: u^{n-1}, m, phi (or the haloed mu box), g^{k-1}, S
    static constexpr int M_OFF = G::UP_BYTES, PH_OFF = M_OFF + G::F_BYTES;
    static constexpr int ACC_OFF = PH_OFF + G::PH_BYTES, GS_OFF = ACC_OFF + G::F_BYTES;

    const StepArgs *pa;  // the kernel argument, in the constant parameter space
    const CUtensorMap *tm_ucur, *tm_ucur_in, *tm_uprev, *tm_m, *tm_phi, *tm_acc, *tm_gs;
    int tid, x0, y0, z0, z1, n;
    uint32_t uthr, pthr;  // byte offset of this thread's row-0 quad in a u slot; elements of it in a tile
    uint32_t toff;        // elements from the tile's corner to it in the padded field
    bool xy_inner, aborted;
    // flags of this thread's points, few enough for one register: bits 0-3 its
    // PML columns, 4 + r a PML row, 8 + 3 r the points of row r's quad inside
    // the grid (0..4), 16 + r row r's quad holds the source's x and y
    uint32_t flags;
    int phi_xmask;  // phi blocks holding x-PML columns, when the tile touches only the
                    // x-PML (planes outside the z-PML load only these); 0 otherwise

    RingPos<NU, G::U_PITCH> uf;  // front plane k + 4, four slots ahead of plane k (producer: next plane)
    RingPos<NP, G::P_PITCH> pc;  // (u^{n-1}, m, phi) plane k (producer: next plane)
    void *u_out_v;   // FLOW, PARITY: the output buffer of the current step
    const void *u_cur_v;  // PARITY: u^n of the current step
    float s_cur, s_prev, inv_s_next;  // fp16 scales (1 otherwise)
    float sd_cur, inv_sd_next;        // fp16 MODE_DIFF: scales of d^n and d^{n+1}
    float vmax, vmax_d;               // running max |u^{n+1}|, |d^{n+1}| of this thread
    // PML terms of the thread's fixed columns i = gi + e and rows j = gj0 + r:
    // eta dt = a d(i)^2, the gradient factor k (d(i+1)^2 - d(i-1)^2), the
    // adjoint's k G(i +- 1) with G(y) = d(y+1)^2 - d(y-1)^2, and PML masks
    // (x terms as quads over e; nhxm = -k G(i - 1))
    float4 pex, pgx, phxp, nhxm;
    float pey[TY], pgy[TY], phyp[TY], phym[TY];
    // 1 / (1 + e) and 1 - e of the thread's points in planes outside the z-PML
    // (e = eta dt depends on x and y only there; the adjoint, short of registers,
    // computes both in every plane)
    float4 pinv[TY], pome[TY];

    // u slot at ring offset o; tile slot at ring offset o; their barriers
    __device__ __forceinline__ unsigned char *uslot(uint32_t o) const { return step_smem + o; }
    __device__ __forceinline__ unsigned char *pslot(uint32_t o) const
    {
        return step_smem + NU * G::U_PITCH + o;
    }
    __device__ __forceinline__ uint64_t *full_u(uint32_t o) const
    {
        return reinterpret_cast<uint64_t *>(uslot(o) + G::U_BYTES);
    }
    __device__ __forceinline__ uint64_t *empty_u(uint32_t o) const { return full_u(o) + 1; }
    __device__ __forceinline__ uint64_t *full_p(uint32_t o) const
    {
        return reinterpret_cast<uint64_t *>(pslot(o) + G::P_BYTES);
    }
    __device__ __forceinline__ uint64_t *empty_p(uint32_t o) const { return full_p(o) + 1; }
    __device__ __forceinline__ volatile int *s_abort() const
    {
        return reinterpret_cast<volatile int *>(step_smem + G::ABORT_OFF);
    }
    __device__ __forceinline__ int tile_quads(int r) const { return (flags >> (8 + 3 * r)) & 7; }
    // MODE_ADJ: mu^{k+1} at this thread's row-r points one plane below, kept from
    // plane to plane in shared memory (registers are at their limit)
    __device__ __forceinline__ float4 *mz_prev(int r) const
    {
        return reinterpret_cast<float4 *>(step_smem + G::MZ_OFF) + r * THREADS + tid;
    }

    // One thread sets the barriers of both rings up (full: the producer's
    // arrival; empty: one arrival per consumer warp).
    __device__ __forceinline__ void init_rings(int abort0)
    {
        *s_abort() = abort0;
        for (int i = 0; i < NU; ++i) {
            mbar_init(full_u(i * G::U_PITCH), 1);
            mbar_init(empty_u(i * G::U_PITCH), WARPS);
        }
        for (int i = 0; i < NP; ++i) {
            mbar_init(full_p(i * G::P_PITCH), 1);
            mbar_init(empty_p(i * G::P_PITCH), WARPS);
        }
    }

    __device__ __forceinline__ void set_maps(const CUtensorMap *ucur, const CUtensorMap *ucur_in,
                                             const CUtensorMap *uprev, const CUtensorMap *m,
                                             const CUtensorMap *phi)
    {
        tm_ucur = ucur;
        tm_ucur_in = ucur_in;
        tm_uprev = uprev;
        tm_m = m;
        tm_phi = phi;
    }

    __device__ __forceinline__ void pml_axis(int n_in, int i, float ca, float ck, float &e, float &gk,
                                             float &hp, float &hm, bool &in_pml) const
    {
        const int nb = pa->nb;
        const int d = pml_depth(n_in, nb, i), dp = pml_depth(n_in, nb, i + 1);
        const int dm = pml_depth(n_in, nb, i - 1);
        const int d2p = pml_depth(n_in, nb, i + 2), d2m = pml_depth(n_in, nb, i - 2);
        e = __fmul_rn(ca, float(d * d));
        gk = __fmul_rn(ck, float(dp * dp - dm * dm));
        hp = __fmul_rn(ck, float(d2p * d2p - d * d));
        hm = __fmul_rn(ck, float(d * d - d2m * d2m));
        in_pml = d > 0;
    }

    // Every PML-path operation below has an explicit rounding (fmaf, __fmul_rn,
    // __fadd_rn): implicit contraction may differ between the kernels that
    // inline this code, and the serving kernel must reproduce run_shot to the bit.
    __device__ __forceinline__ void pml_tables()
    {
        const StepArgs &a = *pa;
        const int gi = x0 + 4 * (tid % TXT), gj0 = y0 + TY * (tid / TXT);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            bool in;
            float v[4];
            pml_axis(a.nx, gi + e, a.ax, a.kx, v[0], v[1], v[2], v[3], in);
            f4set(pex, e, v[0]);
            f4set(pgx, e, v[1]);
            f4set(phxp, e, v[2]);
            f4set(nhxm, e, -v[3]);
            flags |= uint32_t(in) << e;
        }
#pragma unroll
        for (int r = 0; r < TY; ++r) {
            bool in;
            pml_axis(a.ny, gj0 + r, a.ay, a.ky, pey[r], pgy[r], phyp[r], phym[r], in);
            flags |= uint32_t(in) << (4 + r);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float exy = __fadd_rn(f4get(pex, e), pey[r]);
                f4set(pinv[r], e, rcp_approx(__fadd_rn(1.0f, exy)));
                f4set(pome[r], e, __fsub_rn(1.0f, exy));
            }
        }
    }

    __device__ __forceinline__ bool plane_pml(int k) const
    {
        return !xy_inner || k < pa->nb + BAND || k >= pa->nb + pa->nz - BAND;
    }

    // Bounded wait of the calling thread: false (and the CTA's abort flag set)
    // after WAIT_NS, or as soon as another thread of the CTA has given up.
    __device__ __forceinline__ bool spin(uint64_t *bar, uint32_t parity)
    {
        uint64_t t0 = 0;
        for (;;) {
#pragma unroll 1
            for (int i = 0; i < 32; ++i)  // the timer read is slow: between batches of polls
                if (mbar_try_wait(bar, parity)) return true;
            if (*s_abort()) return false;
            const uint64_t t = global_timer_ns();
            if (t0 == 0) t0 = t;
            if (t - t0 > WAIT_NS) {
                *s_abort() = 1;
                atomicOr(pa->err, DEV_ERR_TIMEOUT);
                return false;
            }
        }
    }

    // ... of one thread; sets aborted when it gives up.
    __device__ __forceinline__ void wait(uint64_t *bar, uint32_t parity)
    {
        if (!mbar_try_wait(bar, parity) && !spin(bar, parity)) aborted = true;
    }

    // ... of a whole warp; aborted stays uniform over it.
    __device__ __forceinline__ void wait_warp(uint64_t *bar, uint32_t parity)
    {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return;
        const bool ok = spin(bar, parity);
        if (!__all_sync(0xffffffffu, ok)) aborted = true;
    }

    // Planes outside the chunk feed only the z-queue: they need no x-y halo (but
    // land at their place in a full slot, x margin included).
    __device__ __forceinline__ bool front_only(int p) const { return p < z0 || p >= z1; }

    // This thread's row-r quad in the u slot at ring offset o.
    __device__ __forceinline__ const T *own_ptr(uint32_t o, int r) const
    {
        return reinterpret_cast<const T *>(uslot(o) + uthr) + r * SW;
    }

    __device__ __forceinline__ void issue_u(int p)
    {
        const uint32_t o = uf.off;
        wait(empty_u(o), uf.ph ^ 1);  // previous plane of the slot released (true on the first pass)
        if (aborted) return;
        uf.next();
        if (front_only(p)) {
            mbar_arrive_expect_tx(full_u(o), SW * BY * (int)sizeof(T));
            // a neighbouring z-chunk's plane: kept in L2 for that chunk's own read
            tma_load_3d_hint(uslot(o) + R * SW * (int)sizeof(T), tm_ucur_in, full_u(o), x0 - HX, y0, p,
                             policy_evict_last());
        } else {
            mbar_arrive_expect_tx(full_u(o), SW * C::SH * (int)sizeof(T));
            tma_load_3d(uslot(o), tm_ucur, full_u(o), x0 - HX, y0 - R, p);
        }
    }

    __device__ __forceinline__ void issue_p(int k)
    {
        const uint32_t o = pc.off;
        wait(empty_p(o), pc.ph ^ 1);
        if (aborted) return;
        pc.next();
        const bool pml = plane_pml(k);
        const bool zpml = k < pa->nb || k >= pa->nb + pa->nz;
        const int phmask = !pml ? 0 : (phi_xmask && !zpml) ? phi_xmask : (1 << C::PHI_NB) - 1;
        const int ntiles = 1 + (MODE == MODE_ADJ ? 2 : 0);
        constexpr int PHB_BYTES = C::PHI_BW * C::BY * 4;
        const int ph_bytes = MODE == MODE_ADJ ? (pml ? G::MBW * G::MBH * 4 : 0)
                                              : __popc(phmask) * PHB_BYTES;
        uint64_t *full = full_p(o);
        mbar_arrive_expect_tx(full, P_TILE * (int)sizeof(T) + ntiles * G::F_BYTES + ph_bytes);
        unsigned char *d = pslot(o);
        // No evict-first hint: u^{n-1} and phi are overwritten in place (u^{n+1},
        // phi^{n+1}) a few planes later, and marking their lines first-to-go cost
        // 8% of the step at 512^3 (118 MB more DRAM read per launch).
        tma_load_3d(d, tm_uprev, full, x0, y0, k);
        tma_load_3d(d + M_OFF, tm_m, full, x0, y0, k);
        if constexpr (MODE == MODE_ADJ) {
            // mu^{k+1} with its x-y halo; g^{k-1} of the recomputation; partial sum S
            if (pml) tma_load_3d(d + PH_OFF, tm_phi, full, x0 - 4, y0 - 1, k);
            tma_load_3d(d + ACC_OFF, tm_acc, full, x0, y0, k);
            tma_load_3d(d + GS_OFF, tm_gs, full, x0, y0, k);
        } else {
#pragma unroll
            for (int b = 0; b < C::PHI_NB; ++b)
                if ((phmask >> b) & 1)
                    tma_load_3d(d + PH_OFF + b * PHB_BYTES, tm_phi, full, x0 + b * C::PHI_BW, y0, k);
        }
    }

    // Producer lane: every plane of u^n (z0-4 .. z1+3) and every (u^{n-1}, m,
    // phi) plane (z0 .. z1-1), in the order the consumers need them; each
    // refill first waits for its slot to be released.  Then waits for its own
    // copies to land, so no copy is in flight when it exits.
    __device__ __forceinline__ void produce()
    {
        produce_unit();
        drain();
    }

    __device__ __forceinline__ void produce_unit()
    {
        int nu = z0 - 4, np = z0;
        while ((nu < z1 + 4 || np < z1) && !aborted) {
            // plane nu is first needed at iteration nu - z0 - 4 (as the front
            // plane), plane np at iteration np - z0
            const bool do_u = nu < z1 + 4 && (np >= z1 || nu - z0 - 4 <= np - z0);
            if (do_u) issue_u(nu++);
            else issue_p(np++);
        }
    }

    __device__ __forceinline__ void drain()
    {
        for (int s = 0; s < NU; ++s)
            mbar_wait_bounded(full_u(s * G::U_PITCH), uf.last_parity(s), WAIT_NS);
        for (int s = 0; s < NP; ++s)
            mbar_wait_bounded(full_p(s * G::P_PITCH), pc.last_parity(s), WAIT_NS);
    }

    // One z-plane k.  The queue holds planes k-4 .. k+3 at q[0 .. 7]; the front
    // plane k+4 is loaded into q[8].
    // Queue values are the stored (scaled) values; true u = stored * s_cur.
    // KIND: PLANE_INTERIOR (no PML point in the tile's plane), PLANE_XY (PML
    // path, plane outside the z-PML: e from the thread's tables), PLANE_Z (a
    // z-PML plane).
    template <int KIND>
    __device__ __forceinline__ void plane(float4 (&q)[TY][QN], int k)
    {
        constexpr bool PML = KIND != PLANE_INTERIOR;
        constexpr bool ZP = KIND == PLANE_Z;
        const StepArgs &a = *pa;
        {
            const bool fu = mbar_try_wait(full_u(uf.off), uf.ph), fp = mbar_try_wait(full_p(pc.off), pc.ph);
            if (!__all_sync(0xffffffffu, fu && fp)) {
#pragma unroll 1
                for (int w = 0; w < 2; ++w)
                    wait_warp(w ? full_p(pc.off) : full_u(uf.off), w ? pc.ph : uf.ph);
            }
        }
#pragma unroll
        for (int r = 0; r < TY; ++r) q[r][8] = E::ld(own_ptr(uf.off, r));
        const unsigned char *pu = pslot(pc.off);
        const uint32_t uc = uf.behind(4);  // plane k
        const T *cu = own_ptr(uc, 0);

        // 25-point Laplacian (Eq. 3): centre and z part from the queue
        float4 L[TY], gy[TY];
#pragma unroll
        for (int r = 0; r < TY; ++r) {
            L[r] = f4mul(a.c0, q[r][4]);
#pragma unroll
            for (int m = 1; m <= R; ++m) {
                f4fma(L[r], a.cz[m - 1], q[r][4 - m]);
                f4fma(L[r], a.cz[m - 1], q[r][4 + m]);
            }
        }
        // y part: rows -4 .. TY+3 around the thread's first row
#pragma unroll
        for (int d = -R; d < TY + R; ++d) {
            float4 v;
            if (d >= 0 && d < TY) v = q[d][4];
            else v = E::ld(cu + d * SW);
#pragma unroll
            for (int r = 0; r < TY; ++r) {
                const int m = d > r ? d - r : r - d;
                if (m >= 1 && m <= R) f4fma(L[r], a.cy[m - 1], v);
                // gy = u(j+1) - u(j-1); row r-1 is visited before row r+1
                if (PML && d == r - 1) gy[r] = make_float4(-v.x, -v.y, -v.z, -v.w);
                if (PML && d == r + 1) f4fma(gy[r], 1.0f, v);
            }
        }
        float ez = 0.f, gzk = 0.f, hzp = 0.f, hzm = 0.f;
        bool zin = false;
        if (PML) pml_axis(a.nz, k, a.az, a.kz, ez, gzk, hzp, hzm, zin);
        // the tile's corner in the padded fields
        const long long off0 = a.origin + (long long)k * a.sxy + (long long)y0 * a.sx + x0;
        // random bits of this thread's stores in this plane (16-bit storage)
        uint32_t rnd = 0;
        if constexpr (sizeof(T) == 2) rnd = hash_bits((uint32_t)off0 + toff, (uint32_t)n);
#pragma unroll
        for (int r = 0; r < TY; ++r) {
            const T *rowp = cu + r * SW;
            const uint32_t ro = toff + r * (uint32_t)a.sx;  // this row's quad from the tile's corner
            float4 c = q[r][4];
            const float4 lf = E::ld(rowp - 4), rt = E::ld(rowp + 4);
            const float4 cs = c;  // stored values
            float4 Lr = lap_x(L[r], a.cx, lf, c, rt);
            const uint32_t pr = pthr + r * BX;
            float4 up = E::ld(reinterpret_cast<const T *>(pu) + pr);
            const float4 mm = lds128(reinterpret_cast<const float *>(pu + M_OFF) + pr);
            if constexpr (SCALED) {  // stored values -> true values
                Lr = f4mul(s_cur, Lr);
                c = f4mul(s_cur, c);
                up = f4mul(MODE == MODE_DIFF ? sd_cur : s_prev, up);
            }
            float4 un;  // MODE_DIFF: d^{n+1} until the source is added
            if constexpr (MODE == MODE_DIFF) {  // up = d^n: d^{n+1} = d^n + m L u^n
                un = f4fma4(mm, Lr, up);
            } else {
                un = f4fma4(mm, Lr, make_float4(fmaf(2.0f, c.x, -up.x), fmaf(2.0f, c.y, -up.y),
                                                fmaf(2.0f, c.z, -up.z), fmaf(2.0f, c.w, -up.w)));
            }
            float4 phn = make_float4(0.f, 0.f, 0.f, 0.f);
            float4 ph = make_float4(0.f, 0.f, 0.f, 0.f);
            int rowmask = 0;  // bit e: point e of this row is a PML point
            if constexpr (PML) {
                const float *pph = reinterpret_cast<const float *>(pu + PH_OFF);
                rowmask = (ZP || zin || ((flags >> (4 + r)) & 1)) ? 0xF : flags & 0xF;
                // 1 / (1 + e), 1 - e
                float4 inv = pinv[r], ome = pome[r];
                if constexpr (ZP || MODE == MODE_ADJ) {
                    const float eyz = ZP ? __fadd_rn(pey[r], ez) : pey[r];
                    const float4 ed = f4add4(make_float4(eyz, eyz, eyz, eyz), pex);
                    const float4 one = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
                    const float4 oe = f4add4(one, ed);
                    ome = f4sub(one, ed);
                    inv = make_float4(rcp_approx(oe.x), rcp_approx(oe.y), rcp_approx(oe.z),
                                      rcp_approx(oe.w));
                }
                float4 rhs;  // phi^n (forward) or psi (adjoint)
                if constexpr (MODE == MODE_ADJ) {
                    // psi = sum_a k_a [G_a mu](x + e_a) - [G_a mu](x - e_a) from the six
                    // neighbours of mu^{k+1} (zero outside the PML and in the halo): x and y
                    // from the haloed box, -z kept from the plane below, +z from global memory
                    const float *mb = pph + mu_off() + r * G::MBW;
                    ph = lds128(mb);
                    const float4 myp = lds128(mb + G::MBW), mym = lds128(mb - G::MBW);
                    const float4 mzm = *mz_prev(r);
                    float4 mzp = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (tile_quads(r)) mzp = ldg128(a.mu_in + (off0 + a.sxy) + ro);
                    *mz_prev(r) = ph;
                    rhs = f4mul4(nhxm, make_float4(mb[-1], ph.x, ph.y, ph.z));
                    rhs = f4fma4(phxp, make_float4(ph.y, ph.z, ph.w, mb[4]), rhs);
                    f4fma(rhs, phyp[r], myp);
                    f4fma(rhs, -phym[r], mym);
                    f4fma(rhs, hzp, mzp);
                    f4fma(rhs, -hzm, mzm);
                } else {
                    ph = lds128(pph + phi_off() + r * C::PHI_BW);
                    rhs = ph;
                }
                const float4 lr = f4add4(Lr, rhs);
                float4 upml;
                if constexpr (MODE == MODE_DIFF) {
                    // d^{n+1} = u^{n+1} - c with u^{n-1} = c - d^n:
                    //   [(1 - e) d^n + m lr - e^2 c] / (1 + e)
                    const float4 ed = f4sub(make_float4(1.0f, 1.0f, 1.0f, 1.0f), ome);
                    const float4 e2c = f4mul4(f4mul4(ed, ed), c);
                    upml = f4mul4(inv, f4fma4(mm, lr, f4fma4(ome, up, f4mul(-1.0f, e2c))));
                } else {
                    // [(2 - e^2) c - (1 - e) u^{n-1} + m lr] / (1 + e)
                    //   = (1 - e) c + [c - (1 - e) u^{n-1} + m lr] / (1 + e)
                    upml = f4fma4(inv, f4fma4(mm, lr, f4fma4(ome, f4mul(-1.0f, up), c)), f4mul4(ome, c));
                }
                if constexpr (MODE == MODE_ADJ) {
                    // psi also reaches the inner points next to the PML;
                    // mu^k = (mu^{k+1} + w^{k+1}) / (1 + e) on the PML
                    un = f4fma4(mm, lr, make_float4(fmaf(2.0f, c.x, -up.x), fmaf(2.0f, c.y, -up.y),
                                                    fmaf(2.0f, c.z, -up.z), fmaf(2.0f, c.w, -up.w)));
                    phn = f4mul4(f4add4(ph, c), inv);
                } else {
                    // dt grad(eta) . grad(u)
                    float4 gd = f4mul(gzk, f4sub(q[r][5], q[r][3]));
                    f4fma(gd, pgy[r], gy[r]);
                    gd = f4fma4(pgx, make_float4(__fsub_rn(cs.y, lf.w), __fsub_rn(cs.z, cs.x),
                                                 __fsub_rn(cs.w, cs.y), __fsub_rn(rt.x, cs.z)), gd);
                    if constexpr (SCALED) gd = f4mul(s_cur, gd);
                    phn = f4mul4(f4sub(ph, gd), inv);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const bool pt = (rowmask >> e) & 1;
                    f4set(un, e, pt ? f4get(upml, e) : f4get(un, e));
                    f4set(phn, e, pt ? f4get(phn, e) : f4get(ph, e));
                }
            }
            if constexpr (MODE == MODE_ADJ && !PML) *mz_prev(r) = make_float4(0.f, 0.f, 0.f, 0.f);
            float4 acc4 = Lr;  // MODE_FWD_ACC: g = L u^n + phi^n + f^n
            if constexpr (MODE == MODE_FWD_ACC) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if ((rowmask >> e) & 1) f4set(acc4, e, __fadd_rn(f4get(acc4, e), f4get(ph, e)));
            }
            // point source (Eq. 2 right-hand side), added by the owning thread
            if (MODE != MODE_ADJ && k == a.sk && ((flags >> (16 + r)) & 1)) {
                const int e = a.si & 3;  // tiles start at multiples of 4
                const float f = a.wavelet[n] * a.inv_vol;
                f4set(un, e, fmaf(f4get(mm, e), f, f4get(un, e)));
                if constexpr (MODE == MODE_FWD_ACC) f4set(acc4, e, __fadd_rn(f4get(acc4, e), f));
            }
            float4 dn;  // MODE_DIFF: d^{n+1}; u^{n+1} = u^n + d^{n+1}
            if constexpr (MODE == MODE_DIFF) {
                dn = un;
                un = make_float4(__fadd_rn(c.x, dn.x), __fadd_rn(c.y, dn.y), __fadd_rn(c.z, dn.z),
                                 __fadd_rn(c.w, dn.w));
            }
            // shell launches leave the box to the two-step kernel (its x bounds
            // are multiples of 4: a quad is wholly inside or outside)
            const int gi = x0 + 4 * (tid % TXT), j = y0 + TY * (tid / TXT) + r;
            const bool boxed = SHELL && gi >= a.bx0 && gi < a.bx1 && j >= a.by0 && j < a.by1 &&
                               k >= a.bz0 && k < a.bz1;
            const int nst = tile_quads(r);
            if (nst && !boxed) {
                const long long off = off0 + ro;
                if constexpr (SCALED) {
                    vmax = fmaxf(vmax, fmaxf(fmaxf(fabsf(un.x), fabsf(un.y)),
                                             fmaxf(fabsf(un.z), fabsf(un.w))));
                    un = f4mul(inv_s_next, un);
                    if constexpr (MODE == MODE_DIFF) {
                        vmax_d = fmaxf(vmax_d, fmaxf(fmaxf(fabsf(dn.x), fabsf(dn.y)),
                                                     fmaxf(fabsf(dn.z), fabsf(dn.w))));
                        dn = f4mul(inv_sd_next, dn);
                    }
                }
                T *uo = static_cast<T *>(OUTV ? u_out_v : a.u_out) + off;
                const bool wphi = PML && rowmask;  // phi^{n+1}, or mu^k in the adjoint
                // MODE_DIFF: d^{n+1} rounded with its own random word (an odd
                // multiple of u's, so uniform and distinct)
                T *dio = nullptr;
                if constexpr (MODE == MODE_DIFF) dio = static_cast<T *>(a.d_io) + off;
                const uint32_t rnd_d = rnd * 0x2C1B3C6Du;
                float4 s4 = make_float4(0.f, 0.f, 0.f, 0.f);
                if constexpr (MODE == MODE_ADJ) {
                    // S += w^k g^{k-1} (dJ/dm = sum_k w^k g^{k-1} / m; S is folded
                    // into the fp64 sum every few steps)
                    const float4 gk = lds128(reinterpret_cast<const float *>(pu + ACC_OFF) + pr);
                    s4 = lds128(reinterpret_cast<const float *>(pu + GS_OFF) + pr);
                    s4.x = fmaf(un.x, gk.x, s4.x);
                    s4.y = fmaf(un.y, gk.y, s4.y);
                    s4.z = fmaf(un.z, gk.z, s4.z);
                    s4.w = fmaf(un.w, gk.w, s4.w);
                }
                if (nst == 4) {
                    E::template st<true>(uo, un, rnd, 4);
                    if constexpr (MODE == MODE_DIFF) E::template st<true>(dio, dn, rnd_d, 4);
                    if (wphi) stg128(a.phi + off, phn);
                    if constexpr (MODE == MODE_FWD_ACC) stg128(a.acc_out + off, acc4);
                    if constexpr (MODE == MODE_ADJ) stg128(a.gsum + off, s4);
                } else {
                    E::template st<false>(uo, un, rnd, nst);
                    if constexpr (MODE == MODE_DIFF) E::template st<false>(dio, dn, rnd_d, nst);
                    if (wphi) st_part(a.phi + off, phn, nst);
                    if constexpr (MODE == MODE_FWD_ACC) st_part(a.acc_out + off, acc4, nst);
                    if constexpr (MODE == MODE_ADJ) st_part(a.gsum + off, s4, nst);
                }
                if constexpr (sizeof(T) == 2) rnd = next_bits(rnd);  // the next row's word
            }
        }
        // release the current u plane and this tile slot
        __syncwarp();
        if ((tid & 31) == 0) {
            mbar_arrive(empty_u(uc));
            mbar_arrive(empty_p(pc.off));
        }
        uf.next();
        pc.next();
    }

    // Tile-level geometry of the unit (x0, y0, z0, z1 set): whether the tile
    // touches the x-y PML band, and which phi blocks its planes need.
    __device__ __forceinline__ void unit_geometry()
    {
        const StepArgs &a = *pa;
        const int xe = min(x0 + BX, a.Nx), ye = min(y0 + BY, a.Ny);
        xy_inner = x0 >= a.nb + BAND && xe <= a.nb + a.nx - BAND && y0 >= a.nb + BAND &&
                   ye <= a.nb + a.ny - BAND;
        phi_xmask = 0;
        if (MODE != MODE_ADJ && !xy_inner && y0 >= a.nb && ye <= a.nb + a.ny) {
            // rows all y-inner: only columns in the x-PML need phi outside the z-PML
            for (int b = 0; b < C::PHI_NB; ++b) {
                const int c0 = x0 + b * C::PHI_BW, c1 = min(c0 + C::PHI_BW, a.Nx);
                if (c0 < a.Nx && (c0 < a.nb || c1 > a.nb + a.nx)) phi_xmask |= 1 << b;
            }
        }
    }

    // This consumer thread's points in the unit and their PML tables.
    __device__ __forceinline__ void thread_geometry()
    {
        const StepArgs &a = *pa;
        const int txi = tid % C::TXT, tyi = tid / C::TXT;
        const int gi = x0 + 4 * txi, gj0 = y0 + TY * tyi;
        uthr = ((R + TY * tyi) * SW + HX + 4 * txi) * (int)sizeof(T);
        pthr = (TY * tyi) * BX + 4 * txi;
        toff = (uint32_t)(TY * tyi) * (uint32_t)a.sx + 4 * txi;
        flags = 0;
#pragma unroll
        for (int r = 0; r < TY; ++r) {
            if (gj0 + r < a.Ny) flags |= uint32_t(min(max(a.Nx - gi, 0), 4)) << (8 + 3 * r);
            if (gj0 + r == a.sj && a.si >= gi && a.si < gi + 4) flags |= 1u << (16 + r);
        }
        pml_tables();
    }
    // MODE_ADJ: this thread's row-0 quad in the haloed mu box.
    __device__ __forceinline__ int mu_off() const
    {
        return (1 + TY * (tid / TXT)) * G::MBW + 4 + 4 * (tid % TXT);
    }
    // This thread's row-0 quad in the blocked phi tile.
    __device__ __forceinline__ int phi_off() const
    {
        const int c = 4 * (tid % TXT);
        return (c / C::PHI_BW) * C::PHI_BW * BY + (TY * (tid / TXT)) * C::PHI_BW + c % C::PHI_BW;
    }

    // Prime the register queue with planes z0-4 .. z0+3 and run the unit's
    // planes: z-PML planes below the inner region, then the planes outside the
    // z-PML (interior path, or the PML path for tiles touching the x-y PML band
    // and for the adjoint's band planes next to the z-PML), then the z-PML
    // planes above it.
    __device__ __forceinline__ void consume_unit(float4 (&q)[TY][QN])
    {
        const StepArgs &a = *pa;
        if constexpr (MODE == MODE_ADJ) {  // mu^{k+1} one plane below the unit
            const long long off0 = a.origin + (long long)(z0 - 1) * a.sxy + (long long)y0 * a.sx + x0;
#pragma unroll
            for (int r = 0; r < TY; ++r)
                *mz_prev(r) = tile_quads(r) ? ldg128(a.mu_in + off0 + toff + r * (uint32_t)a.sx)
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            auto ahead = uf;
#pragma unroll 1
            for (int s = 0; s < 4; ++s) {
                wait_warp(full_u(ahead.off), ahead.ph);
                ahead.next();
            }
#pragma unroll
            for (int s = 0; s < 4; ++s) {
#pragma unroll
                for (int r = 0; r < TY; ++r) q[r][4 * h + s] = E::ld(own_ptr(uf.off, r));
                uf.next();
            }
            if (h == 0) {  // planes z0-4 .. z0-1 are not needed again
                __syncwarp();
                if ((tid & 31) == 0)
#pragma unroll 1
                    for (int s = 4; s >= 1; --s) mbar_arrive(empty_u(uf.behind(s)));
            }
        }
        const int zlo = min(max(a.nb, z0), z1);
        const int zhi = min(max(a.nb + a.nz, zlo), z1);
        // The z-PML below the inner region, the planes between, the z-PML above: as a
        // loop, so that each plane kind is compiled once (the kernel's code
        // is far beyond the instruction cache of a scheduler either way).
#pragma unroll 1
        for (int part = 0; part < 3; ++part) {
            const int k0 = part == 0 ? z0 : part == 1 ? zlo : zhi;
            const int k1 = part == 0 ? zlo : part == 1 ? zhi : z1;
            if (part != 1) {
                segment<PLANE_Z>(q, k0, k1);
            } else if constexpr (MODE != MODE_ADJ) {
                if (xy_inner) segment<PLANE_INTERIOR>(q, k0, k1);
                else segment<PLANE_XY>(q, k0, k1);
            } else {  // the band planes next to the z-PML
                const int b0 = xy_inner ? min(max(a.nb + BAND, k0), k1) : k1;
                const int b1 = xy_inner ? min(max(a.nb + a.nz - BAND, b0), k1) : k1;
#pragma unroll 1
                for (int sub = 0; sub < 3; ++sub) {
                    if (sub == 1) segment<PLANE_INTERIOR>(q, b0, b1);
                    else segment<PLANE_XY>(q, sub == 0 ? k0 : b1, sub == 0 ? b0 : k1);
                }
            }
        }
    }

    // Planes [k, k_end) of one kind.
    template <int KIND>
    __device__ __forceinline__ void segment(float4 (&q)[TY][QN], int k, int k_end)
    {
#pragma unroll 1
        for (; k < k_end && !aborted; ++k) {
            plane<KIND>(q, k);
#pragma unroll
            for (int r = 0; r < TY; ++r)
#pragma unroll
                for (int j = 0; j < QN - 1; ++j) q[r][j] = q[r][j + 1];
        }
    }
};

// Power-of-two fp16 scale for a field bounded by B: B / scale < 2^14.
__device__ __forceinline__ float pow2_scale_for(float B)
{
    if (!(B > 0.0f) || !isfinite(B)) return 1.0f;
    return ldexpf(1.0f, ilogbf(B) + 1 - 14);
}

// Resident CTAs per SM asked of the compiler, also for 16-bit storage: its shared
// memory would leave room for a third CTA, but 128 registers a thread do not hold
// the z-queue (spills, 9-27% slower).
template <class C, class T>
constexpr int min_blocks()
{
#ifdef SGB_MINB16
    return sizeof(T) == 2 ? SGB_MINB16 : C::MINB;
#else
    return C::MINB;
#endif
}

// One work unit (tile x z-chunk, index `unit` of `units`) of one step.  What
// needs only the kernel's parameters -- barriers, tile and thread geometry, PML
// tables -- comes before the wait for the previous launch, so after a
// programmatic launch it runs while that one drains.  pick(st, sample_only):
// called after the wait by every thread, returns the step n and sets the tensor
// maps and, where the step's parity decides them, the buffers; with
// sample_only, only the receivers of the previous step are sampled (the extra
// launch after a shot's last step), with a negative n nothing is done.  The
// consumers sample the receivers while the first copies are in flight.
// Back-to-back steps (PML 16): 96^3 8.35 -> 7.62 us, 128^3 11.7 -> 10.6 us,
// 256^3 64.8 -> 63.1 us.
template <class C, class T, int MODE = MODE_FWD, int VAR = VAR_PLAIN, class Pick>
__device__ __forceinline__ void step_unit(const StepArgs &a, int unit, int units, Pick pick)
{
    using S = StepCta<C, T, MODE, VAR>;
    constexpr bool SHELL = VAR == VAR_SHELL;
    static_assert(MODE == MODE_FWD || MODE == MODE_DIFF || sizeof(T) == 4,
                  "the adjoint runs in fp32");
    constexpr int TY = C::TY, THREADS = C::THREADS, BX = C::BX, BY = C::BY;

    S st;
    st.pa = &a;
    const int tid = threadIdx.x;
    st.tid = tid;

    // Work unit: chunk-major so that CTAs running together share z and their
    // x-y halos meet in L2.
    if constexpr (SHELL) {
        grid_dependency_sync();  // the unit table is in global memory
        const int4 u = a.units[unit];
        st.x0 = u.x;
        st.y0 = u.y;
        st.z0 = u.z;
        st.z1 = u.w;
    } else {
        const int per_chunk = a.tiles_x * a.tiles_y;
        const int chunk = unit / per_chunk;
        const int trem = unit - chunk * per_chunk;
        const int tyl = trem / a.tiles_x, txl = trem - tyl * a.tiles_x;
        st.x0 = txl * BX;
        st.y0 = tyl * BY;
        st.z0 = chunk * a.zc;
        st.z1 = min(st.z0 + a.zc, a.Nz);
    }
    const int nit = st.z1 - st.z0;
    st.aborted = false;
    st.unit_geometry();
    // (in difference form the early tables cost more registers than the overlap
    // gives: 74.8 us against 73.0 at 256^3 in bf16)
    constexpr bool late = MODE == MODE_DIFF;
    if (tid < THREADS) {
        if (!late) st.thread_geometry();
    } else if (tid == THREADS) {
        st.init_rings(0);
        fence_barrier_init();
    }
    __syncthreads();

    grid_dependency_sync();
    bool sample_only = false;
    const int n = pick(st, sample_only);
    if (n < 0) return;  // finished: waits for retirement
    st.n = n;
    if (tid >= THREADS) {  // producer warp: one lane issues every copy
        if (tid == THREADS && !sample_only && nit > 0) st.produce();
        return;
    }

    st.s_cur = st.s_prev = st.inv_s_next = st.sd_cur = st.inv_sd_next = 1.0f;
    st.vmax = st.vmax_d = 0.0f;
    if constexpr (S::SCALED) {
        ScaleState *ss = a.scale;
        st.s_cur = ss->s[n & 3];
        st.s_prev = ss->s[(n - 1) & 3];
        const float inj = a.sk >= 0 ? fabsf(*a.m_src * a.wavelet[n] * a.inv_vol) : 0.0f;
        float B = 4.0f * fmaxf(ss->mx[n & 3], ss->mx[(n - 1) & 3]) + inj;
        if constexpr (MODE == MODE_DIFF) {
            // |m L u| <= 4 max|u| at a stable dt, so |d^{n+1}| <= 2 max|d^n| + 4 max|u^n|
            // + the injected amplitude (the factor 2 covers the PML terms), and
            // |u^{n+1}| <= max|u^n| + that
            ScaleState *sd = a.scale_d;
            st.sd_cur = sd->s[n & 3];
            const float Bd = 2.0f * sd->mx[n & 3] + 4.0f * ss->mx[n & 3] + inj;
            const float sd_next = pow2_scale_for(Bd);
            st.inv_sd_next = 1.0f / sd_next;  // exact: a power of two
            B = ss->mx[n & 3] + Bd;
            if (unit == 0 && tid == 0 && !sample_only) {
                sd->s[(n + 1) & 3] = sd_next;
                sd->mx[(n + 2) & 3] = 0.0f;
            }
        }
        const float s_next = pow2_scale_for(B);
        st.inv_s_next = 1.0f / s_next;  // exact: a power of two
        if (unit == 0 && tid == 0 && !sample_only) {
            ss->s[(n + 1) & 3] = s_next;
            ss->mx[(n + 2) & 3] = 0.0f;
        }
    }

    // Receivers of the previous step, while the first copies are on their way: u^n
    // is read-only in this launch.
    if (a.nrec > 0 && n >= 1 + a.rec_n0) {
        const T *uc = static_cast<const T *>(S::OUTV ? st.u_cur_v : a.u_cur);
        for (int r = unit * THREADS + tid; r < a.nrec; r += units * THREADS) {
            const float v = Elem<T>::get(uc + a.rec_off[r]) * st.s_cur;
            a.traces[(long long)(n - 1 - a.rec_n0) * a.nrec + r] = v;
            if (!isfinite(v)) atomicOr(a.err, DEV_ERR_NONFINITE);
        }
    }
    if (sample_only || nit <= 0) return;
    if (late) st.thread_geometry();

    float4 q[TY][C::QN];
    st.consume_unit(q);

    if constexpr (MODE == MODE_ADJ) {
        // Residuals of this unit's receivers, on top of what its threads have just
        // written: w^k += m r and its term of the gradient sum, S += (m r) g^{k-1}.
        // Receivers at one point follow one another in the list and the thread of the
        // first adds them all, in the caller's order.
        // A launch of its own for them took 3.5 us per step and stood between two
        // steps that otherwise overlap (128^3: 41 -> 37 us per step and its
        // forward and recomputation steps).
        if (st.x0 <= a.rec_hi[0] && st.x0 + BX > a.rec_lo[0] && st.y0 <= a.rec_hi[1] &&
            st.y0 + BY > a.rec_lo[1] && st.z0 <= a.rec_hi[2] && st.z1 > a.rec_lo[2]) {
            const int r0 = a.rec_start[unit], r1 = a.rec_start[unit + 1];
            consumer_barrier(THREADS);
            float *w = static_cast<float *>(a.u_out);
            for (int q = r0 + tid; q < r1; q += THREADS) {
                const long long p = a.rec_off[q];
                bool more = q + 1 < r1 && a.rec_off[q + 1] == p;
                if (q > r0 && a.rec_off[q - 1] == p) continue;
                const float m = a.m_all[p], g = a.acc_in[p];
                float wp = __ldcg(w + p), sp = __ldcg(a.gsum + p);
                for (int e = q;; ++e) {
                    const int r = a.rec_idx[e];
                    const float add = m * (a.tr_row[r] - a.obs_row[r]);
                    wp += add;
                    sp = fmaf(add, g, sp);
                    if (!more) break;
                    more = e + 2 < r1 && a.rec_off[e + 2] == p;
                }
                w[p] = wp;
                a.gsum[p] = sp;
            }
        }
    }
    if constexpr (S::SCALED) {  // max |u^{n+1}| for the next step's scale
        float v = st.vmax;
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        if ((tid & 31) == 0 && v > 0.0f) atomicMax(reinterpret_cast<int *>(&a.scale->mx[(n + 1) & 3]),
                                                 __float_as_int(v));
        if constexpr (MODE == MODE_DIFF) {  // and max |d^{n+1}|
            float vd = st.vmax_d;
            for (int o = 16; o > 0; o >>= 1) vd = fmaxf(vd, __shfl_xor_sync(0xffffffffu, vd, o));
            if ((tid & 31) == 0 && vd > 0.0f)
                atomicMax(reinterpret_cast<int *>(&a.scale_d->mx[(n + 1) & 3]), __float_as_int(vd));
        }
    }
}

// One time step of one grid: one CTA per work unit.
template <class C, class T>
__global__ void __launch_bounds__(C::BLOCK, (min_blocks<C, T>()))
    fused_step_kernel(const __grid_constant__ StepArgs a,
                      const __grid_constant__ CUtensorMap tm_ucur,
                      const __grid_constant__ CUtensorMap tm_ucur_in,
                      const __grid_constant__ CUtensorMap tm_uprev,
                      const __grid_constant__ CUtensorMap tm_m,
                      const __grid_constant__ CUtensorMap tm_phi)
{
    step_unit<C, T>(a, blockIdx.x, gridDim.x, [&](auto &st, bool &) {
        st.set_maps(&tm_ucur, &tm_ucur_in, &tm_uprev, &tm_m, &tm_phi);
        return (a.step_ptr ? *a.step_ptr : 0) + a.step_add;
    });
}

// One time step in difference form (MODE_DIFF): one CTA per work unit.
template <class C, class T>
__global__ void __launch_bounds__(C::BLOCK, (min_blocks<C, T>()))
    diff_step_kernel(const __grid_constant__ StepArgs a,
                     const __grid_constant__ CUtensorMap tm_ucur,
                     const __grid_constant__ CUtensorMap tm_ucur_in,
                     const __grid_constant__ CUtensorMap tm_d,
                     const __grid_constant__ CUtensorMap tm_m,
                     const __grid_constant__ CUtensorMap tm_phi)
{
    step_unit<C, T, MODE_DIFF>(a, blockIdx.x, gridDim.x, [&](auto &st, bool &) {
        st.set_maps(&tm_ucur, &tm_ucur_in, &tm_d, &tm_m, &tm_phi);
        return (a.step_ptr ? *a.step_ptr : 0) + a.step_add;
    });
}

// One fused step on the work units of a table, storing nothing inside the
// two-step kernel's box (the shell of a temporally blocked pair, fp32).
template <class C>
__global__ void __launch_bounds__(C::BLOCK, C::MINB)
    shell_step_kernel(const __grid_constant__ StepArgs a, const __grid_constant__ CUtensorMap tm_ucur,
                      const __grid_constant__ CUtensorMap tm_ucur_in,
                      const __grid_constant__ CUtensorMap tm_uprev,
                      const __grid_constant__ CUtensorMap tm_m,
                      const __grid_constant__ CUtensorMap tm_phi)
{
    step_unit<C, float, MODE_FWD, VAR_SHELL>(a, blockIdx.x, gridDim.x, [&](auto &st, bool &) {
        st.set_maps(&tm_ucur, &tm_ucur_in, &tm_uprev, &tm_m, &tm_phi);
        return (a.step_ptr ? *a.step_ptr : 0) + a.step_add;
    });
}

// One step of one shot in a served replay: the step n = *step_ptr +
// step_add comes from a device counter, the buffers and tensor maps of its
// parity are chosen here (so a replay of any length repeats), and launches past
// the shot's last step do nothing (n_end: the last launch, which only samples
// the receivers of step n_end - 1).
struct ShotRun {
    void *buf[2];         // step n reads buf[(n + 1) & 1] and writes buf[n & 1]
    const int *step_ptr;  // the shot's device step counter
    int step_add;
    int n_end;
};

template <class C>
__global__ void __launch_bounds__(C::BLOCK, C::MINB)
    shot_step_kernel(const __grid_constant__ StepArgs a, const __grid_constant__ ShotRun r,
                     const __grid_constant__ CUtensorMap m0_ucur,
                     const __grid_constant__ CUtensorMap m0_ucur_in,
                     const __grid_constant__ CUtensorMap m0_uprev,
                     const __grid_constant__ CUtensorMap m0_m,
                     const __grid_constant__ CUtensorMap m0_phi,
                     const __grid_constant__ CUtensorMap m1_ucur,
                     const __grid_constant__ CUtensorMap m1_ucur_in,
                     const __grid_constant__ CUtensorMap m1_uprev,
                     const __grid_constant__ CUtensorMap m1_m,
                     const __grid_constant__ CUtensorMap m1_phi)
{
    step_unit<C, float, MODE_FWD, VAR_PARITY>(a, blockIdx.x, gridDim.x, [&](auto &st, bool &sample_only) {
        const int n = *r.step_ptr + r.step_add;
        if (n & 1) st.set_maps(&m1_ucur, &m1_ucur_in, &m1_uprev, &m1_m, &m1_phi);
        else st.set_maps(&m0_ucur, &m0_ucur_in, &m0_uprev, &m0_m, &m0_phi);
        st.u_out_v = r.buf[n & 1];
        st.u_cur_v = r.buf[(n + 1) & 1];
        sample_only = n == r.n_end;
        return n > r.n_end ? -1 : n;
    });
}

// Forward step that also stores g^n = L u^n + phi^n + f^n (adjoint recomputation).
template <class C>
__global__ void __launch_bounds__(C::BLOCK, C::MINB)
    fwd_acc_kernel(const __grid_constant__ StepArgs a, const __grid_constant__ CUtensorMap tm_ucur,
                   const __grid_constant__ CUtensorMap tm_ucur_in,
                   const __grid_constant__ CUtensorMap tm_uprev,
                   const __grid_constant__ CUtensorMap tm_m,
                   const __grid_constant__ CUtensorMap tm_phi)
{
    step_unit<C, float, MODE_FWD_ACC>(a, blockIdx.x, gridDim.x, [&](auto &st, bool &) {
        st.set_maps(&tm_ucur, &tm_ucur_in, &tm_uprev, &tm_m, &tm_phi);
        return a.step_add;
    });
}

// Adjoint step k (see the adjoint notes in adjoint.cuh): reads w^{k+1} through
// the u^n maps, w^{k+2} through the u^{n-1} map (overwritten with w^k),
// mu^{k+1} through the phi map (mu^k is written to a.phi), g^{k-1} through the
// acc map and the partial gradient sum S through the gs map (updated in place).
template <class C>
__global__ void __launch_bounds__(C::BLOCK, C::MINB)
    adjoint_step_kernel(const __grid_constant__ StepArgs a,
                        const __grid_constant__ CUtensorMap tm_ucur,
                        const __grid_constant__ CUtensorMap tm_ucur_in,
                        const __grid_constant__ CUtensorMap tm_uprev,
                        const __grid_constant__ CUtensorMap tm_m,
                        const __grid_constant__ CUtensorMap tm_mu,
                        const __grid_constant__ CUtensorMap tm_acc,
                        const __grid_constant__ CUtensorMap tm_gs)
{
    step_unit<C, float, MODE_ADJ>(a, blockIdx.x, gridDim.x, [&](auto &st, bool &) {
        st.set_maps(&tm_ucur, &tm_ucur_in, &tm_uprev, &tm_m, &tm_mu);
        st.tm_acc = &tm_acc;
        st.tm_gs = &tm_gs;
        return a.step_add;
    });
}

}  // namespace sgb
