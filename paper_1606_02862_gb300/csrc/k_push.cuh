// k_push.cuh -- fused field gather, Boris push, move and Esirkepov current
// deposition for the mixed (int32 cell + FP32 offset) particle form.
//
// One CTA works on one supercell at a time (Sec. 2.1: a supercell maps to a
// block, its threads share the supercell's particles); CTAs are persistent
// and pull the supercells that hold mobile particles (a list that the frame
// maintenance writes) from a work counter, one item ahead, so boxes of any
// size and occupancy share one launch.  Per supercell:
//   1. stage the E and B tile (supercell + G guard cells below, G = 1 for
//      CIC/TSC, 2 with PCS) from HBM into shared memory with two tensor loads;
//   2. zero a shared J tile of the same extent;
//   3. every thread takes particles of the supercell's frame lists: gather
//      E, B from shared memory (CIC 2x2x2 / TSC 3x3x3 / PCS 4x4x4 weights
//      per component at its Yee position, Sec. 4; optionally one order lower
//      along the component's staggered axes, the energy-conserving variant),
//      relativistic Boris push, move, then Esirkepov deposition (Sec. 4) into
//      the shared J tile with shared atomics; the particles that stay go back
//      to the list compacted (in chunk order, so the leavers' slots close up
//      as the list is written); particles that leave the supercell collect in
//      a shared leaver buffer that the CTA hands to the move buffer at its
//      next work item (or leave through a subdomain slab's z face into a
//      migrant message, or through a y face of an open-y box out of the
//      simulation);
//   4. add the J tile to the guard-padded global J with 16-byte vector
//      atomics (neighbouring supercells overlap in their guard cells).
//
// Esirkepov (2001): with 1D shape factors S0 (old) and S1 (new) on a common
// window and DS = S1 - S0, the x current on the half node i+1/2 is
//   Jx(i+1/2, j, k) = -(q w hx / (V dt)) * sum_{i' <= i} DSx(i')
//                     * [S0y S0z + DSy S0z / 2 + S0y DSz / 2 + DSy DSz / 3](j, k)
// i.e. an outer product of a prefix sum along x and a transverse factor.
//
// Particles go through a chunk of at most 256 at a time in list order.  Every
// sort_every-th step the frame maintenance sorts the TSC and PCS lists by
// nearest node / cell, so the lanes of a warp read neighbouring field words
// (shared-memory broadcasts) and a chunk covers a few rows of nodes.  CIC lists
// are sorted here, chunk by chunk by cell, in the push of that step (a sort
// pass; see push_list).  The chunk stage is filled by an asynchronous copy while
// the previous chunk deposits (in a CIC sort pass by plain loads).
// The push writes a deposit record
// per particle; the deposit then runs in a lane order whose neighbours are
// several list positions apart (dep_log_stride), so one warp's atomics land on
// different nodes.  The current of a list accumulates in fixed point (see
// kTileTerms).  Two deposit paths, both exact forms of that formula:
//   common: on every axis the move stays on one spline piece -- the old and
//     the new position round to the same node (TSC) / stay in the same cell
//     (CIC, PCS) -- so the union of the two supports is 3 (TSC) / 2 (CIC) /
//     4 (PCS) nodes and DS has closed per-node forms in the displacement D
//     (no cancellation in FP32); 54 (TSC) / 12 (CIC) / 144 (PCS) shared
//     atomics, no branches;
//   general: the rest (a few percent of particles) are listed and deposited
//     on a 4-node (CIC, TSC) or 5-node (PCS) window: set aside (up to
//     kGenDefer per list) and deposited lane-parallel after the list's last
//     chunk with their own fixed-point scale; beyond that, with their chunk:
//     whole groups of 32 lane-parallel, the leftover moves one per warp with
//     all 32 lanes on the move's current lines.
// The shared tiles use a row pitch of 4 mod 8 floats, so that rows are
// 16-byte aligned (the E/B tile arrives by tensor loads, the J tile leaves as
// float4) and the 32 banks spread over neighbouring rows.
#pragma once

#include "pic_internal.cuh"
#include "quotients.cuh"
#include "tma.cuh"

#include <cmath>

namespace pic {

// General-window moves of a frame list deposited together after its last
// chunk (more are deposited with their own chunk).
constexpr int kGenDefer = 64;
// Particles changing supercell that a CTA collects in shared memory and hands
// to the move buffer at the start of its next work item (more go straight
// to the move buffer).
constexpr int kLeaverBuf = 48;
// Log2 of the lane stride of the deposit over a chunk of a list of n
// particles in a supercell of S cells: neighbouring lanes take list positions
// that far apart, so that one warp's atomics land on different nodes.  The
// list is sorted by node, with n / S particles on a node on average; in a bank
// model of the 8x4x4 tile a TSC atomic of 32 lanes takes 3.1 / 3.3 / 4.8
// wavefronts at stride 4 and 3.3 / 2.9 / 3.1 at stride 8 for 2 / 8 / 16
// particles per cell.
__device__ __forceinline__ int dep_log_stride(int n, int S) { return n >= 4 * S ? 3 : 2; }

// G = guard cells below the supercell (the fields' global guards match):
// 1 for CIC/TSC, 2 when a PCS species is present (its support reaches two
// nodes below the cell and, for a move across a cell face, three above).
template <int LX_, int LY_, int LZ_, int G_ = 1>
struct Tile {
    static constexpr int LX = LX_, LY = LY_, LZ = LZ_, G = G_;
    static constexpr int GO = G - 1;  // tile index of node l - 1 is l + GO
    // x: G below, 3 (CIC/TSC) / 6 (PCS) above, 16-byte rows; y, z: G below, 2 / 3 above
    static constexpr int TX = G == 1 ? LX + 4 : LX + 8;
    static constexpr int TY = G == 1 ? LY + 3 : LY + 5;
    static constexpr int TZ = G == 1 ? LZ + 3 : LZ + 5;
    // shared-memory row pitch: the first multiple of 4 at or above TX that is
    // 4 mod 8, so that rows are 16-byte aligned and consecutive rows start 12
    // (or 20) banks apart
    static constexpr int PX = (TX % 8 == 4) ? TX : (TX % 8 == 0 ? TX + 4 : ((TX + 3) / 4) * 4);
    static constexpr int N = PX * TY * TZ;  // shared floats per component
    static constexpr int S = LX * LY * LZ;
    // the B tile starts here (floats from the E tile's start): 128-byte
    // aligned, like the E tile, for its tensor load
    static constexpr int BOFF = ((3 * N + 31) / 32) * 32;
    // shared floats of the field tiles and the two current tiles
    static constexpr int TILES = BOFF + 9 * N;
    static_assert(PX % 4 == 0 && N % 4 == 0, "tile rows and components are 16-byte aligned");
};

// ------------------------------------------------------------ shape factors

// TSC (quadratic spline, Hockney & Eastwood) at distance d, branch-free.
__host__ __device__ __forceinline__ float tsc_S(float d)
{
    float a = fabsf(d);
    float t = fmaxf(1.5f - a, 0.0f);
    return a <= 0.5f ? 0.75f - a * a : 0.5f * t * t;
}

// S(d0 + D) - S(d0) for TSC without ever forming d1 = d0 + D (rounding d1
// costs ~6e-8 absolute, which is a large relative error on a DS of order D
// for slow particles).  On one spline piece the difference is factored
// through D; across a piece boundary p (|d| = 1/2 or 3/2) it is the sum of
// the two pieces' differences to p, with the exact distance d0 -> p
// (Sterbenz) and the remainder D - (p - d0).  The spline is C1 at its joins,
// so a misjudged side of p changes the result only at second order.
__host__ __device__ __forceinline__ float tsc_dS(float d0, float D)
{
    const float a0 = fabsf(d0);
    const float s0 = d0 >= 0.0f ? 1.0f : -1.0f;
    if (a0 <= 0.5f) {
        const float d1 = d0 + D;  // classification only
        if (fabsf(d1) <= 0.5f)
            return -D * (2.0f * d0 + D);                 // centre piece: d0^2 - d1^2
        const float p = d1 >= 0.0f ? 0.5f : -0.5f;
        const float u1 = p - d0;                          // exact distance to the join
        const float t = (d1 >= 0.0f ? 1.0f : -1.0f) * (D - u1);  // |d1| - 1/2 >= 0
        return -u1 * (p + d0) + t * (0.5f * t - 1.0f);   // centre to p, then outer piece
    }
    const float a1 = a0 + s0 * D;  // |d1| on this side (classification)
    if (a0 < 1.5f) {
        if (a1 <= 0.5f) {                                 // outer piece into the centre
            const float p = 0.5f * s0;
            const float t0 = a0 - 0.5f;                   // exact
            const float u2 = s0 * t0 + D;                 // d1 - p
            return t0 * (1.0f - 0.5f * t0) - u2 * (2.0f * p + u2);
        }
        if (a1 < 1.5f)                                    // outer piece
            return -0.5f * s0 * D * (3.0f - 2.0f * a0 - s0 * D);
        const float r0 = 1.5f - a0;                       // out of the support
        return -0.5f * r0 * r0;
    }
    if (a1 < 1.5f) {                                      // into the support
        const float r1 = (1.5f - a0) - s0 * D;            // 1.5 - |d1|
        return 0.5f * r1 * r1;
    }
    return 0.0f;
}

__host__ __device__ __forceinline__ float cic_S(float d) { return fmaxf(0.0f, 1.0f - fabsf(d)); }

// S(d0 + D) - S(d0) for CIC, the same way: across the node (d = 0) the
// difference is s0 (2 d0 + D); across the support edge (|d| = 1, a kink, so
// the side is decided exactly: 1 - |d0| is exact and compared with s0 D)
// it is the distance to the edge.
__host__ __device__ __forceinline__ float cic_dS(float d0, float D)
{
    const float a0 = fabsf(d0);
    const float s0 = d0 >= 0.0f ? 1.0f : -1.0f;
    if (a0 < 1.0f) {
        if (a0 >= 0.5f && s0 * D >= 1.0f - a0)
            return -(1.0f - a0);                          // out of the support
        const float d1 = d0 + D;                          // its sign is exact
        if ((d1 >= 0.0f) == (d0 >= 0.0f))
            return -s0 * D;
        return s0 * (2.0f * d0 + D);                      // across the node
    }
    if (-s0 * D > a0 - 1.0f)
        return (1.0f - a0) - s0 * D;                      // into the support: 1 - |d1|
    return 0.0f;
}

// PCS (cubic B-spline) at distance d.
__host__ __device__ __forceinline__ float pcs_S(float d)
{
    const float a = fabsf(d);
    if (a < 1.0f)
        return (4.0f - 6.0f * a * a + 3.0f * a * a * a) * (1.0f / 6.0f);
    const float t = fmaxf(2.0f - a, 0.0f);
    return t * t * t * (1.0f / 6.0f);
}

// S(d0 + D) - S(d0) on one spline piece (the piece of the segment's midpoint),
// factored through D: central piece (|d| < 1, sign s fixed)
//   D [-(d0 + d1) + s (d0^2 + d0 d1 + d1^2) / 2],
// outer piece (1 <= |d| < 2, a = 2 - s d)   -s D (a0^2 + a0 a1 + a1^2) / 6.
__host__ __device__ __forceinline__ float pcs_seg(float d0, float D)
{
    const float d1 = d0 + D;
    const float m = d0 + 0.5f * D;
    const float s = m >= 0.0f ? 1.0f : -1.0f;
    const float am = fabsf(m);
    if (am < 1.0f)
        return D * (-(d0 + d1) + 0.5f * s * (d0 * d0 + d0 * d1 + d1 * d1));
    if (am < 2.0f) {
        const float a0 = 2.0f - s * d0, a1 = 2.0f - s * d1;
        return -s * D * (a0 * a0 + a0 * a1 + a1 * a1) * (1.0f / 6.0f);
    }
    return 0.0f;
}

// S(d0 + D) - S(d0) for PCS without forming the difference of two values:
// the pieces join at the integers (the spline is C2 there), and a move of
// less than half a cell crosses at most one join p, where the difference is
// split at p with the exact distance p - d0.
__host__ __device__ __forceinline__ float pcs_dS(float d0, float D)
{
    const float d1 = d0 + D;  // classification only
    const float lo = fminf(d0, d1), hi = fmaxf(d0, d1);
    const float p = floorf(hi);
    if (p > lo && fabsf(p) <= 2.0f) {
        const float u = p - d0;
        return pcs_seg(d0, u) + pcs_seg(p, D - u);
    }
    return pcs_seg(d0, D);
}

// Gather weights along one axis for a particle at offset o in [0,1) of its
// cell; the tile coordinate of the particle's cell is l + 1.  "i" = field
// sampled at integer nodes along this axis, "h" = at half nodes.  ec: the
// energy-conserving variant, one order lower at the half nodes (CIC inside
// the TSC window, nearest node inside the CIC window).  l is the tile index of
// node (cell - 1): cell + GO.
struct AxisCic {
    int bi, bh;  // tile index of the first node
    float wi[2], wh[2];
    __device__ __forceinline__ AxisCic(int l, float o, bool ec)
    {
        bi = l + 1;
        wi[0] = 1.0f - o;
        wi[1] = o;
        const bool up = o >= 0.5f;
        const float dh = up ? o - 0.5f : o + 0.5f;
        bh = l + (up ? 1 : 0);  // half nodes bh - 1/2 .. : the cell's own is l + 1/2
        wh[0] = ec ? (up ? 1.0f : 0.0f) : 1.0f - dh;
        wh[1] = ec ? (up ? 0.0f : 1.0f) : dh;
    }
};

template <int PX, int TY>
__device__ __forceinline__ float gather_cic(const float* __restrict__ F, int bx, int by, int bz,
                                            const float* wx, const float* wy, const float* wz)
{
    float acc = 0.0f;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const float* row = F + ((bz + c) * TY + (by + b)) * PX + bx;
            float r = 0.0f;
#pragma unroll
            for (int a = 0; a < 2; ++a)
                r = fmaf(row[a], wx[a], r);
            acc = fmaf(r, wy[b] * wz[c], acc);
        }
    }
    return acc;
}

__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 swap2(float2 v) { return make_float2(v.y, v.x); }

// The same for TSC and PCS, both kinds of node at once on the packed FP32 pipe
// (two independent operations per instruction): w = (i, h) weights, or (h, i)
// with SWAP.
template <int SHAPE, bool SWAP>
struct AxisPair {
    static constexpr int NW = SHAPE + 1;
    int bi, bh;
    float2 w[NW];
    __device__ __forceinline__ AxisPair(int l, float o, bool ec)
    {
        const bool up = o >= 0.5f;
        const float2 half = dup2(0.5f), minus = dup2(-1.0f);
        if (SHAPE == 2) {
            const float di = up ? o - 1.0f : o;  // from the nearest node
            const float dh = o - 0.5f;           // from the half node l + 1/2
            bi = l + (up ? 1 : 0);
            bh = l;  // half nodes l - 1/2, l + 1/2, l + 3/2
            const float2 d = SWAP ? make_float2(dh, di) : make_float2(di, dh);
            const float2 a = __ffma2_rn(d, minus, half), c = __fadd2_rn(d, half);
            w[0] = __fmul2_rn(__fmul2_rn(half, a), a);
            // 3/4 - d^2 within 4.5e-8 (rms 1.8e-8); as one fma of d within 3.0e-8
            // (1.7e-8), which takes 0.3 % longer per step for the same error of
            // the step
            w[1] = __ffma2_rn(a, c, half);
            w[2] = __fmul2_rn(__fmul2_rn(half, c), c);
            if (ec) {
                set_h(0, up ? 0.0f : 0.5f - o);
                set_h(1, up ? 1.5f - o : 0.5f + o);
                set_h(2, up ? o - 0.5f : 0.0f);
            }
        } else {
            // integer nodes cell-1 .. cell+2; half nodes m0 .. m0+3 with
            // m0 = cell - 2 + up (the half node m + 1/2 is stored at index m);
            // f = distance from the second of them
            bi = l;
            bh = l - 1 + (up ? 1 : 0);
            const float fh = up ? o - 0.5f : o + 0.5f;
            const float2 f = SWAP ? make_float2(fh, o) : make_float2(o, fh);
            const float2 g = __ffma2_rn(f, minus, dup2(1.0f));
            const float2 f2 = __fmul2_rn(f, f), g2 = __fmul2_rn(g, g);
            const float2 sixth = dup2(1.0f / 6.0f), two3 = dup2(2.0f / 3.0f);
            w[0] = __fmul2_rn(__fmul2_rn(g2, sixth), g);
            // (4 - 6 f^2 + 3 f^3) / 6 within 8.6e-8, f^3 / 6 within 3.7e-8 (9.1e-8 and
            // 4.9e-8 with the sums of the definition times 1/6)
            w[1] = __ffma2_rn(f2, __ffma2_rn(half, f, minus), two3);
            w[2] = __ffma2_rn(g2, __ffma2_rn(half, g, minus), two3);
            w[3] = __fmul2_rn(__fmul2_rn(f2, sixth), f);
            if (ec) {  // TSC at the half nodes cell-1, cell, cell+1
                const float a = 1.0f - o, c = o, m = 0.75f - (o - 0.5f) * (o - 0.5f);
                set_h(0, up ? 0.5f * a * a : 0.0f);
                set_h(1, up ? m : 0.5f * a * a);
                set_h(2, up ? 0.5f * c * c : m);
                set_h(3, up ? 0.0f : 0.5f * c * c);
            }
        }
    }
    __device__ __forceinline__ void set_h(int k, float v)
    {
        if (SWAP)
            w[k].x = v;
        else
            w[k].y = v;
    }
};

// Two components (windows at p1 and p2; wx, wy, wz: their weights side by
// side); per lane the sums are scalar fmaf chains.
template <int NW, int PX, int TY>
__device__ __forceinline__ float2 gather_pair(const float* __restrict__ p1, const float* __restrict__ p2,
                                              const float2* wx, const float2* wy, const float2* wz)
{
    float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int c = 0; c < NW; ++c)
#pragma unroll
        for (int b = 0; b < NW; ++b) {
            const float* r1 = p1 + (c * TY + b) * PX;
            const float* r2 = p2 + (c * TY + b) * PX;
            float2 r = __fmul2_rn(make_float2(r1[0], r2[0]), wx[0]);
#pragma unroll
            for (int a = 1; a < NW; ++a)
                r = __ffma2_rn(make_float2(r1[a], r2[a]), wx[a], r);
            acc = __ffma2_rn(r, __fmul2_rn(wy[b], wz[c]), acc);
        }
    return acc;
}

// All six components in pairs whose nodes differ along every axis -- (Bx, Ex),
// (Ey, By), (Bz, Ez) -- so that each axis' weights are needed as (i, h) and (h,
// i) only and few moves line the operands up.
template <class T, int SHAPE>
__device__ __forceinline__ void gather_pairs(const float* __restrict__ sF, int lx, int ly, int lz, float ox, float oy,
                                             float oz, bool ec, float E[3], float B[3])
{
    constexpr int NW = SHAPE + 1, PX = T::PX, TY = T::TY, N = T::N;
    AxisPair<SHAPE, false> x(lx, ox, ec), z(lz, oz, ec);
    const AxisPair<SHAPE, true> y(ly, oy, ec);  // (h, i)
    const float2 EyBy = gather_pair<NW, PX, TY>(sF + N + (z.bi * TY + y.bh) * PX + x.bi,
                                                sF + T::BOFF + N + (z.bh * TY + y.bi) * PX + x.bh, x.w, y.w, z.w);
#pragma unroll
    for (int k = 0; k < NW; ++k)
        z.w[k] = swap2(z.w[k]);
    const float2 BxEx = gather_pair<NW, PX, TY>(sF + T::BOFF + (z.bh * TY + y.bh) * PX + x.bi,
                                                sF + (z.bi * TY + y.bi) * PX + x.bh, x.w, y.w, z.w);
#pragma unroll
    for (int k = 0; k < NW; ++k)
        z.w[k] = swap2(z.w[k]), x.w[k] = swap2(x.w[k]);
    const float2 BzEz = gather_pair<NW, PX, TY>(sF + T::BOFF + 2 * N + (z.bi * TY + y.bh) * PX + x.bh,
                                                sF + 2 * N + (z.bh * TY + y.bi) * PX + x.bi, x.w, y.w, z.w);
    E[0] = BxEx.y, E[1] = EyBy.x, E[2] = BzEz.y;
    B[0] = BxEx.x, B[1] = EyBy.y, B[2] = BzEz.x;
}

// Esirkepov's transverse factor S0e S0f + (DSe S0f + S0e DSf)/2 + DSe DSf / 3
// as A S0f + B DSf with A = S0e + DSe / 2, B = S0e / 2 + DSe / 3: A and B
// belong to one node of axis e, so that a line of the window takes two
// operations instead of seven (27 lines per TSC move).  CIC moves (12 lines
// in the common window) keep the form of esk_T_cic and its rounding: see the
// sort in push_list.
__device__ __forceinline__ float esk_A(float s0, float ds) { return fmaf(0.5f, ds, s0); }
__device__ __forceinline__ float esk_B(float s0, float ds) { return fmaf(0.5f, s0, (1.0f / 3.0f) * ds); }

__device__ __forceinline__ float esk_T_cic(float s0e, float dse, float s0f, float dsf)
{
    return fmaf(s0e, s0f, fmaf(0.5f, fmaf(dse, s0f, s0e * dsf), (1.0f / 3.0f) * dse * dsf));
}

template <int SHAPE>
__device__ __forceinline__ float esk_T(float s0e, float dse, float s0f, float dsf)
{
    if (SHAPE == 1)
        return esk_T_cic(s0e, dse, s0f, dsf);
    return fmaf(esk_A(s0e, dse), s0f, esk_B(s0e, dse) * dsf);
}

// ------------------------------------------------------------ fixed-point J tile
//
// The shared J tile accumulates the current in int32: shared-memory int32
// atomics are native, where FP32 shared atomics are a compare-and-swap loop.
// Each chunk's contributions are scaled by a power of two chosen from the chunk
// itself, so that every scaled term is below 2^kTermBits in magnitude: with B =
// max over its particles and axes of Tmax |jcoef_d w D_d|, |P| <= |D| and |T| <=
// Tmax = (max S)^2 bound every term of the current by B.  A particle adds one
// term at most to a node's component, so a node's sum stays below 2^31 while
// the tile holds at most kTileTerms particles at one scale: it is folded into
// an FP32 tile before more come in and before a chunk of another scale (see
// push_list).  A term keeps 2^-22 B resolution.  Scaled terms convert to
// integers with the 1.5 * 2^23 magic-number add, which takes |x| < 2^22.
constexpr int kTermBits = 21;
constexpr int kTileTerms = 1023;
// (the rounding of a term to an integer, 1/2 each, and the FP32 rounding of
// the bound fit in the one term that is left)
static_assert((long long)(kTileTerms + 1) << kTermBits <= 1LL << 31, "a node's sum fits in int32");
static_assert(kTermBits < 22, "the magic-number range");
static_assert(kGenDefer <= kTileTerms, "the moves set aside are folded once");

__device__ __forceinline__ int magic_int(float x)
{
    return __float_as_int(x + 12582912.0f) - 0x4B400000;
}

// scale = 2^(kTermBits - e) with bound < 2^e.  Bounds below 2^-105 take that
// scale, which is the largest finite one (their terms are far below anything
// FP32 fields resolve).
__device__ __forceinline__ float chunk_scale(float bound, float* inv)
{
    const int e = bound > 0.0f ? max((__float_as_int(bound) >> 23) - 126, -105) : 0;
    *inv = __int_as_float((127 + e - kTermBits) << 23);
    return __int_as_float((127 + kTermBits - e) << 23);
}

// One window line pair: the M - 1 terms P[i] T of two parallel lines (tile
// words a0 + i st and a1 + i st), converted to fixed point two at a time.
template <int M>
__device__ __forceinline__ void add_line_pair(int* a0, int* a1, int st, const float* P, float2 T)
{
    const float2 magic = dup2(12582912.0f);
#pragma unroll
    for (int i = 0; i < M - 1; ++i) {
        const float2 v = __ffma2_rn(dup2(P[i]), T, magic);
        atomicAdd(a0 + i * st, __float_as_int(v.x) - 0x4B400000);
        atomicAdd(a1 + i * st, __float_as_int(v.y) - 0x4B400000);
    }
}

// One current component on a window of M nodes per axis (M - 1 half nodes
// along the component's own axis d, whose DS are DSd): axis e carries the
// factors A, B (times the component's coefficient cf), axis f its S0 and DS.
// at: window origin of the component's tile; SD, SE, SF: word strides of the
// three axes.  For PCS (144 atomics per move) the transverse factors and the fixed-point conversions go two lines at a time through the packed
// FP32 pipe; for CIC and TSC the pairs' extra registers cost more than they
// save.
template <int SHAPE, int M, int SD, int SE, int SF>
__device__ __forceinline__ void deposit_comp(int* at, float cf, const float* DSd, const float* S0e,
                                             const float* DSe, const float* S0f, const float* DSf)
{
    constexpr bool PAIR = SHAPE == 3;
    float P[M - 1], A[M], B[M];
    P[0] = DSd[0];
#pragma unroll
    for (int i = 1; i < M - 1; ++i)
        P[i] = P[i - 1] + DSd[i];
#pragma unroll
    for (int j = 0; j < M; ++j) {
        A[j] = cf * esk_A(S0e[j], DSe[j]);
        B[j] = cf * esk_B(S0e[j], DSe[j]);
    }
#pragma unroll
    for (int k = 0; k < M; ++k) {
        int j = 0;
        if (PAIR) {
#pragma unroll
            for (; j + 1 < M; j += 2) {
                const float2 T = __ffma2_rn(make_float2(A[j], A[j + 1]), dup2(S0f[k]),
                                            __fmul2_rn(make_float2(B[j], B[j + 1]), dup2(DSf[k])));
                add_line_pair<M>(at + k * SF + j * SE, at + k * SF + (j + 1) * SE, SD, P, T);
            }
        }
#pragma unroll
        for (; j < M; ++j) {
            const float T = SHAPE == 1 ? cf * esk_T_cic(S0e[j], DSe[j], S0f[k], DSf[k])
                                       : fmaf(A[j], S0f[k], B[j] * DSf[k]);
            int* line = at + k * SF + j * SE;
#pragma unroll
            for (int i = 0; i < M - 1; ++i)
                atomicAdd(line + i * SD, magic_int(P[i] * T));
        }
    }
}

// Deposit the three current components on a window of M nodes per axis
// (M-1 half nodes along the current's own axis); node 0 of axis d sits at
// tile index b[d].  cx..cz carry jcoef_d w times the chunk scale.
template <int SHAPE, int M, int PX, int TY, int NJ>
__device__ __forceinline__ void deposit_window(int* sJi, const int b[3], const float* S0x,
                                               const float* S0y, const float* S0z, const float* DSx,
                                               const float* DSy, const float* DSz, float cx, float cy,
                                               float cz)
{
    constexpr int PY = PX * TY;
    int* at = sJi + b[2] * PY + b[1] * PX + b[0];
    deposit_comp<SHAPE, M, 1, PX, PY>(at, cx, DSx, S0y, DSy, S0z, DSz);
    deposit_comp<SHAPE, M, PX, PY, 1>(at + NJ, cy, DSy, S0z, DSz, S0x, DSx);
    deposit_comp<SHAPE, M, PY, 1, PX>(at + 2 * NJ, cz, DSz, S0x, DSx, S0y, DSy);
}

// ------------------------------------------------------------ async copies

// 16-byte global -> shared copy that bypasses the registers (completes at
// cp_async_wait_all of the issuing thread; a block barrier then publishes it).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ------------------------------------------------------------ TMA and mbarriers
//
// The E/B tile of a supercell arrives by two tensor loads (one per field, all
// three components) that complete on a shared-memory mbarrier with a byte
// count.  One thread issues and waits; a block barrier then publishes the
// tile.  The wait is bounded: after kWaitCycles SM clocks it gives up, the
// kernel reports ST_TIMEOUT and the CTA stops taking work.  (The particle
// chunks, scattered over the frames of a list, keep 16-byte asynchronous
// copies from many threads: as bulk copies issued by one thread they measured
// 5 % (TSC) and 8 % (CIC) slower.)

// ------------------------------------------------------------ warp helpers

__device__ __forceinline__ int warp_aggregated_add(int* ctr)
{
    unsigned mask = __activemask();
    int lane = threadIdx.x & 31;
    int leader = __ffs(mask) - 1;
    int base = 0;
    if (lane == leader)
        base = atomicAdd(ctr, __popc(mask));
    base = __shfl_sync(mask, base, leader);
    return base + __popc(mask & ((1u << lane) - 1u));
}

// Exclusive prefix sum of cnt[0..K) into off[0..K) by one warp (lanes take
// contiguous ranges); the caller synchronises the block around it.
__device__ __forceinline__ void warp_exclusive_scan_counts(const int* cnt, int* off, int K)
{
    const int lane = threadIdx.x & 31;
    const int per = (K + 31) / 32;
    const int b0 = lane * per;
    int local = 0;
    for (int i = 0; i < per; ++i)
        local += (b0 + i < K) ? cnt[b0 + i] : 0;
    int x = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o)
            x += y;
    }
    int run = x - local;
    for (int i = 0; i < per; ++i)
        if (b0 + i < K) {
            off[b0 + i] = run;
            run += cnt[b0 + i];
        }
}

// ------------------------------------------------------------ shared state

// Particles of one chunk of a frame list, staged in shared memory in list
// order, and, for the sort passes of CIC lists, their counting-sort
// permutation by cell.
template <int C, bool PCS, bool SORTS>
struct Stage {
    int cell[C];
    float o[3][C];
    float u[3][C];
    float w[C];
    int pid[SORTS ? C : 1];   // particle ids (sort passes, only when tracked)
    int kr[SORTS ? C : 1];    // key << 16 | rank within key
    int perm[SORTS ? C : 1];  // sorted position -> chunk position
    int brk[PCS ? C : 1];  // PCS, by push position: bank << 16 | rank within the bank
};

// Deposit inputs of the chunk's moves, by chunk position s stored at slot
// rslot(s) = s + s / 32: the deposit reads them with a stride of 4 or 8
// between lanes, and the skew puts the 32 lanes on 32 different banks.
__host__ __device__ constexpr int rslot(int s) { return s + (s >> 5); }

// PCS (144 atomics per common-window move): the chunk's moves are
// counting-sorted by the shared-memory bank of their window origin (every
// atomic of a common-window deposit lands there plus an offset shared by all
// lanes) and dealt over the deposit lanes: slot q takes bank-major position
// deal_pos(q), so the 32 lanes of a deposit group take every (C/32)-th
// position -- mostly 32 different banks.
template <int C>
__host__ __device__ constexpr int deal_slot(int p)
{
    return (p % (C / 32)) * 32 + p / (C / 32);
}
template <int C>
__host__ __device__ constexpr int deal_pos(int q)
{
    return (q & 31) * (C / 32) + (q >> 5);
}

template <int C>
struct Records {
    static constexpr int R = C + C / 32;
    int l[R];        // packed local cell lx | ly << 8 | lz << 16, bit 24: general window
    float o[3][R];   // old in-cell offsets
    float D[3][R];   // displacement in cells
    float w[R];      // weight
    int gen[C];      // chunk positions of the moves that need the general window
};

// General-window moves set aside for one lane-parallel deposit after the
// last chunk of a frame list (the few of each chunk would otherwise keep one
// warp busy while the others wait at the chunk's last barrier).
struct GenDefer {
    int l[kGenDefer];        // packed local cell, as in Records
    float o[3][kGenDefer];   // old in-cell offsets
    float D[3][kGenDefer];   // displacement in cells
    float w[kGenDefer];      // weight
};

// Particles leaving the supercell, bound for the move buffer.
struct LeaverBuf {
    int dest[kLeaverBuf];  // destination list
    int cell[kLeaverBuf];  // cell inside the destination supercell
    float o[3][kLeaverBuf];
    float u[3][kLeaverBuf];
    float w[kLeaverBuf];
    int pid[kLeaverBuf];
};

template <class T, int NT, int ONLY>
struct SharedState {
    static constexpr bool SORTS = ONLY <= 1;                // CIC lists may be among them
    static constexpr int C = 2 * NT < 256 ? 2 * NT : 256;  // chunk: at most 256 particles
    static constexpr int NQ = C / NT;                       // particles per thread and chunk
    Stage<C, T::G == 2, SORTS> st;
    Records<C> rec;
    GenDefer gd;
    LeaverBuf lv;
    int hist[SORTS ? T::S : 1];  // sort passes: particles per cell, and each cell's first sorted position
    int off[SORTS ? T::S : 1];
    unsigned long long mb_tile;    // completion of the E/B tile's tensor loads
    unsigned alive[NQ * NT / 32];  // per warp and pass: ballot of the pushed particles that stay
    int item, nlv, lv_base;
    int tile_phase;                // parity of the tile barrier's next phase
    int abort;                     // the tile wait gave up
    int ngen[2];             // general-window moves of the chunk
    unsigned bound_bits[2];  // float bits of the chunk's largest |jcoef w D|
    unsigned gd_bound_bits;  // float bits of the largest |jcoef w D| of the set-aside moves
    int bh[T::G == 2 ? 32 : 1];  // PCS: moves of the chunk per bank of their window origin
};

// Bank of the common-window origin of a PCS particle in local cell `cell`
// (up to an offset shared by all particles).
template <class T>
__device__ __forceinline__ int dep_bank(int cell)
{
    const int lx = cell % T::LX, ly = (cell / T::LX) % T::LY, lz = cell / (T::LX * T::LY);
    return ((lz * T::TY + ly) * T::PX + lx) & 31;
}

// Exclusive prefix of the per-bank counts, bank `lane` in lane `lane`.
__device__ __forceinline__ int bank_offsets(const int* bh, int lane)
{
    const int c = bh[lane];
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += t;
    }
    return incl - c;
}

// Record slot of the move at push position sidx (all 32 lanes call it).
template <int C>
__device__ __forceinline__ int dealt_slot(const int* brk, int sidx, int cn, int boff)
{
    const int br = sidx < cn ? brk[sidx] : 0;
    return deal_slot<C>(__shfl_sync(0xffffffffu, boff, br >> 16) + (br & 0xffff));
}

// Start copying the particles of list slots [base, base + cn) into the chunk stage (cell, offsets, momenta, weight;
// 16-byte pieces of whole frames, which are allocated even past the list's
// count).  The caller waits with cp_async_wait_all and a block barrier.
template <class T, int NT, int ONLY>
__device__ __forceinline__ void stage_chunk_async(const StepDev& d, SharedState<T, NT, ONLY>& sh, int L, int base,
                                                  int cn)
{
    constexpr int S = T::S;
    const int* ft = d.ftab + d.foff[L];
    const int nq = (cn + 3) >> 2;
    for (int k = threadIdx.x; k < nq; k += NT) {
        const int slot = base + 4 * k;
        const int64_t idx = (int64_t)ft[(unsigned)slot / S] * S + (unsigned)slot % S;
        cp_async16(sh.st.cell + 4 * k, d.cell + idx);
        cp_async16(sh.st.o[0] + 4 * k, d.ox + idx);
        cp_async16(sh.st.o[1] + 4 * k, d.oy + idx);
        cp_async16(sh.st.o[2] + 4 * k, d.oz + idx);
        cp_async16(sh.st.u[0] + 4 * k, d.ux + idx);
        cp_async16(sh.st.u[1] + 4 * k, d.uy + idx);
        cp_async16(sh.st.u[2] + 4 * k, d.uz + idx);
        cp_async16(sh.st.w + 4 * k, d.w + idx);
    }
}

// ------------------------------------------------------------ deposit of one record

// The TSC common window's factors at offset di from the window's middle node,
// for a displacement D: the shape S0, P (the prefix of DS along the axis: DS[0]
// and DS[0] + DS[1] = -DS[2]), DS itself, and A, B times the coefficient c of the
// component whose transverse axis "e" this is.  V is float2 (two axes at once)
// or float.
template <class V>
struct TscAxis {
    V S0[3], DS[3], A[3], B[3];
};

__device__ __forceinline__ float2 vdup(float v, float2) { return dup2(v); }
__device__ __forceinline__ float vdup(float v, float) { return v; }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }

template <class V>
__device__ __forceinline__ void tsc_axis(TscAxis<V>& t, V di, V D, V c)
{
    const V half = vdup(0.5f, di), mhalf = vdup(-0.5f, di), third = vdup(1.0f / 3.0f, di);
    const V lo = vfma(di, vdup(-1.0f, di), half), hi = vadd(di, half);
    t.S0[0] = vmul(vmul(half, lo), lo);
    t.S0[1] = vfma(lo, hi, half);  // 3/4 - di^2, as in AxisPair
    t.S0[2] = vmul(vmul(half, hi), hi);
    // DS = -D/2 (1 - d0 - d1), -D (d0 + d1), D/2 (1 + d0 + d1), d1 = d0 + D
    const V sum = vfma(vdup(2.0f, di), di, D);
    const V h = vmul(half, D), m = vmul(mhalf, D);
    t.DS[0] = vfma(h, sum, m);
    t.DS[1] = vmul(vadd(m, m), sum);
    t.DS[2] = vfma(h, sum, h);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        t.A[k] = vmul(c, vfma(half, t.DS[k], t.S0[k]));
        t.B[k] = vmul(c, vfma(half, t.S0[k], vmul(third, t.DS[k])));
    }
}

// One component's 9 lines of 2 terms: P0, P1 along its axis (word stride SD).
template <int SD, int SE, int SF>
__device__ __forceinline__ void tsc_lines(int* at, float P0, float P1, const float A[3], const float B[3],
                                          const float S0f[3], const float DSf[3])
{
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float T = fmaf(A[j], S0f[k], B[j] * DSf[k]);
            int* line = at + k * SF + j * SE;
            atomicAdd(line, magic_int(P0 * T));
            atomicAdd(line + SD, magic_int(P1 * T));
        }
}

// TSC, common window: the factors of x and y together on the packed FP32 pipe.
template <class T, int C>
__device__ __forceinline__ void deposit_common_tsc(int* sJi, const Records<C>& r, int s, const float jc[3], float scale)
{
    constexpr int PX = T::PX, PY = T::PX * T::TY, NJ = T::N;
    const int e = rslot(s);
    const int l = r.l[e];
    const float ox = r.o[0][e], oy = r.o[1][e], oz = r.o[2][e];
    const float ws = r.w[e] * scale;
    const bool ux = ox >= 0.5f, uy = oy >= 0.5f, uz = oz >= 0.5f;
    int* at = sJi + (((l >> 16) & 0xff) + (uz ? 1 : 0)) * PY + (((l >> 8) & 0xff) + (uy ? 1 : 0)) * PX + (l & 0xff) +
              (ux ? 1 : 0);
    TscAxis<float2> xy;
    TscAxis<float> z;
    // axis e of Jx is y, of Jy z, of Jz x
    tsc_axis(xy, make_float2(ux ? ox - 1.0f : ox, uy ? oy - 1.0f : oy), make_float2(r.D[0][e], r.D[1][e]),
             make_float2(jc[2] * ws, jc[0] * ws));
    tsc_axis(z, uz ? oz - 1.0f : oz, r.D[2][e], jc[1] * ws);
    const float Sx[3] = {xy.S0[0].x, xy.S0[1].x, xy.S0[2].x}, Dx[3] = {xy.DS[0].x, xy.DS[1].x, xy.DS[2].x};
    const float Ax[3] = {xy.A[0].x, xy.A[1].x, xy.A[2].x}, Bx[3] = {xy.B[0].x, xy.B[1].x, xy.B[2].x};
    const float Sy[3] = {xy.S0[0].y, xy.S0[1].y, xy.S0[2].y}, Dy[3] = {xy.DS[0].y, xy.DS[1].y, xy.DS[2].y};
    const float Ay[3] = {xy.A[0].y, xy.A[1].y, xy.A[2].y}, By[3] = {xy.B[0].y, xy.B[1].y, xy.B[2].y};
    tsc_lines<1, PX, PY>(at, Dx[0], -Dx[2], Ay, By, z.S0, z.DS);
    tsc_lines<PX, PY, 1>(at + NJ, Dy[0], -Dy[2], z.A, z.B, Sx, Dx);
    tsc_lines<PY, 1, PX>(at + 2 * NJ, z.DS[0], -z.DS[2], Ax, Bx, Sy, Dy);
}

// Common window: nodes a-1, a, a+1 (TSC, a = round(o)), 0, 1 (CIC) or -1 .. 2
// (PCS) relative to the cell on every axis; S0 is the particle's shape there
// and DS has closed forms in D.  The record's l holds cell + GO per axis.
template <class T, int SHAPE, int C>
__device__ __forceinline__ void deposit_common(int* sJi, const Records<C>& r, int s, const float jc[3],
                                               float scale)
{
    if constexpr (SHAPE == 2) {
        deposit_common_tsc<T>(sJi, r, s, jc, scale);
        return;
    }
    const int e = rslot(s);
    constexpr int NW = SHAPE == 3 ? 4 : 2;
    const int l = r.l[e];
    const int lc[3] = {l & 0xff, (l >> 8) & 0xff, (l >> 16) & 0xff};
    float S0[3][NW], DS[3][NW];
    int b[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float o = r.o[a][e], D = r.D[a][e];
        if (SHAPE == 3) {
            // nodes cell-1 .. cell+2, each on one spline piece for the whole move:
            // outer (a = 1 - o), centre (d = o), centre (d = o - 1), outer (a = o)
            b[a] = lc[a];
            const float o1 = o + D;
            const float a0 = 1.0f - o, a1 = a0 - D;
            const float d0 = o - 1.0f, d1 = o1 - 1.0f;
            S0[a][0] = a0 * a0 * a0 * (1.0f / 6.0f);
            S0[a][1] = (4.0f - 6.0f * o * o + 3.0f * o * o * o) * (1.0f / 6.0f);
            S0[a][2] = (4.0f - 6.0f * d0 * d0 - 3.0f * d0 * d0 * d0) * (1.0f / 6.0f);
            S0[a][3] = o * o * o * (1.0f / 6.0f);
            DS[a][0] = -D * (a0 * a0 + a0 * a1 + a1 * a1) * (1.0f / 6.0f);
            DS[a][1] = D * (-(o + o1) + 0.5f * (o * o + o * o1 + o1 * o1));
            DS[a][2] = D * (-(d0 + d1) - 0.5f * (d0 * d0 + d0 * d1 + d1 * d1));
            DS[a][3] = D * (o * o + o * o1 + o1 * o1) * (1.0f / 6.0f);
        } else {
            b[a] = lc[a] + 1;
            S0[a][0] = 1.0f - o;
            S0[a][1] = o;
            DS[a][0] = -D;
            DS[a][1] = D;
        }
    }
    const float ws = r.w[e] * scale;
    deposit_window<SHAPE, NW, T::PX, T::TY, T::N>(sJi, b, S0[0], S0[1], S0[2], DS[0], DS[1], DS[2], jc[0] * ws,
                                           jc[1] * ws, jc[2] * ws);
}

// Window of the general deposit: M nodes per axis; on axis a its first node
// sits at tile index lc + first_off(o, D) and node k of the window is at
// distance d0 = o - node_off(o, D, k) from the particle.
template <int SHAPE>
struct GenWin {
    static constexpr int M = SHAPE == 3 ? 5 : 4;
    // PCS: nodes cell-2+up .. cell+2+up, up = the move ends in the next cell;
    // CIC / TSC: nodes cell-1 .. cell+2
    __device__ __forceinline__ static int first(float o, float D) { return SHAPE == 3 ? (o + D >= 1.0f) - 1 : 0; }
    __device__ __forceinline__ static float d0(float o, int first, int k) { return o - (float)(k - 1 + first); }
    __device__ __forceinline__ static float S(float d) { return SHAPE == 3 ? pcs_S(d) : (SHAPE == 2 ? tsc_S(d) : cic_S(d)); }
    __device__ __forceinline__ static float dS(float d, float D)
    {
        return SHAPE == 3 ? pcs_dS(d, D) : (SHAPE == 2 ? tsc_dS(d, D) : cic_dS(d, D));
    }
};

// General window (GenWin) on every axis, for the move of packed local cell
// l, old offsets o and displacement D (in cells) of a particle of weight w.
template <class T, int SHAPE>
__device__ __forceinline__ void deposit_general_move(int* sJi, int l, const float ov[3], const float Dv[3],
                                                     float w, const float jc[3], float scale)
{
    using W = GenWin<SHAPE>;
    constexpr int M = W::M;
    const int lc[3] = {l & 0xff, (l >> 8) & 0xff, (l >> 16) & 0xff};  // node cell-1 sits at tile index lc
    float S0[3][M], DS[3][M];
    int b[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float o = ov[a], D = Dv[a];
        const int f = W::first(o, D);
        b[a] = lc[a] + f;
#pragma unroll
        for (int k = 0; k < M; ++k) {
            const float d0 = W::d0(o, f, k);
            S0[a][k] = W::S(d0);
            DS[a][k] = W::dS(d0, D);
        }
    }
    const float ws = w * scale;
    deposit_window<SHAPE, M, T::PX, T::TY, T::N>(sJi, b, S0[0], S0[1], S0[2], DS[0], DS[1], DS[2], jc[0] * ws,
                                          jc[1] * ws, jc[2] * ws);
}

// The general-window move at position s of the chunk's records.
template <class T, int SHAPE, int C>
__device__ __forceinline__ void deposit_general(int* sJi, const Records<C>& r, int s, const float jc[3],
                                                float scale)
{
    const int e = rslot(s);
    const float o[3] = {r.o[0][e], r.o[1][e], r.o[2][e]};
    const float D[3] = {r.D[0][e], r.D[1][e], r.D[2][e]};
    deposit_general_move<T, SHAPE>(sJi, r.l[e], o, D, r.w[e], jc, scale);
}

// Bound on the current terms of one move (see push_one).
template <int SHAPE>
__device__ __forceinline__ float move_bound(const float jc[3], float w, float Dx, float Dy, float Dz)
{
    const float tmax = SHAPE == 2 ? 0.5625f * 1.001f : (SHAPE == 3 ? (4.0f / 9.0f) * 1.001f : 1.0f);
    return tmax * fabsf(w) * fmaxf(fmaxf(fabsf(jc[0] * Dx), fabsf(jc[1] * Dy)), fabsf(jc[2] * Dz));
}

// General window of one move, deposited by a whole warp (all 32 lanes
// converged): lane 8a + k (k < M) evaluates S0 and DS at node k of axis a's
// window and the prefix P of DS along that axis; then the lanes take the
// window's 3 M^2 lines (a component c and its transverse nodes p, q: M - 1
// half nodes along c) in turns, reading the factors they need from the
// lanes that hold them.
template <class T, int SHAPE, int C>
__device__ __forceinline__ void deposit_general_warp(int* sJi, const Records<C>& r, int s,
                                                     const float jc[3], float scale)
{
    using W = GenWin<SHAPE>;
    constexpr int M = W::M;
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int PX = T::PX, PY = T::PX * T::TY, NJ = T::N;
    const int lane = threadIdx.x & 31;
    const int e = rslot(s);
    const int l = r.l[e];
    int f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
        f[a] = W::first(r.o[a][e], r.D[a][e]);  // same address in every lane: broadcasts
    float s0v = 0.0f, dsv = 0.0f;
    if ((lane & 7) < M && lane < 24) {
        const int a = lane >> 3, k = lane & 7;
        const float o = r.o[a][e], D = r.D[a][e];
        const float d0 = W::d0(o, a == 0 ? f[0] : (a == 1 ? f[1] : f[2]), k);
        s0v = W::S(d0);
        dsv = W::dS(d0, D);
    }
    float pv = dsv;  // inclusive prefix over k within each group of 8 lanes
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const float t = __shfl_up_sync(FULL, pv, o, 8);
        if ((lane & 7) >= o)
            pv += t;
    }
    const float ws = r.w[e] * scale;
    const int b0 = (l & 0xff) + f[0], b1 = ((l >> 8) & 0xff) + f[1], b2 = ((l >> 16) & 0xff) + f[2];
    const int base = b2 * PY + b1 * PX + b0;
    constexpr int LINES = 3 * M * M;
#pragma unroll
    for (int round = 0; round < (LINES + 31) / 32; ++round) {
        const int L = lane + 32 * round;  // c = L / M^2, p = L % M, q = (L / M) % M
        const int c = L / (M * M);
        const int ea = c == 2 ? 0 : c + 1, fa = c == 0 ? 2 : c - 1;  // transverse axes
        const int p = L % M, q = (L / M) % M;
        const int srcE = 8 * ea + p, srcF = 8 * fa + q;
        const float s0e = __shfl_sync(FULL, s0v, srcE & 31), dse = __shfl_sync(FULL, dsv, srcE & 31);
        const float s0f = __shfl_sync(FULL, s0v, srcF & 31), dsf = __shfl_sync(FULL, dsv, srcF & 31);
        float P[M - 1];
#pragma unroll
        for (int i = 0; i < M - 1; ++i)
            P[i] = __shfl_sync(FULL, pv, (8 * c + i) & 31);
        if (L < LINES) {
            const float cf = (c == 0 ? jc[0] : (c == 1 ? jc[1] : jc[2])) * ws;
            const float Tv = cf * esk_T<SHAPE>(s0e, dse, s0f, dsf);
            const int st_c = c == 0 ? 1 : (c == 1 ? PX : PY);
            const int st_e = ea == 0 ? 1 : (ea == 1 ? PX : PY);
            const int st_f = fa == 0 ? 1 : (fa == 1 ? PX : PY);
            int* at = sJi + c * NJ + base + p * st_e + q * st_f;
#pragma unroll
            for (int i = 0; i < M - 1; ++i)
                atomicAdd(at + i * st_c, magic_int(P[i] * Tv));
        }
    }
}

// ------------------------------------------------------------ one particle

// One particle in registers.
struct Part {
    int cell;
    float o[3], u[3], w;
};

// Writes a pushed particle to pool slot idx (only the cell of a leaver);
// the weight only when the particle changed slot.
__device__ __forceinline__ void store_part(const StepDev& d, int64_t idx, const Part& q, bool with_w)
{
    d.cell[idx] = q.cell;
    if (q.cell >= 0) {
        d.ox[idx] = q.o[0];
        d.oy[idx] = q.o[1];
        d.oz[idx] = q.o[2];
        d.ux[idx] = q.u[0];
        d.uy[idx] = q.u[1];
        d.uz[idx] = q.u[2];
        if (with_w)
            d.w[idx] = q.w;
    }
}

// Pushes one particle (gather, Boris, move) and writes its deposit record
// at slot `slot` of the chunk; returns its bound |jcoef_d w D_d| on the
// current terms.  A particle that stays in the supercell gets its new cell,
// offsets and momentum in q; a leaver goes to the CTA's leaver buffer (or,
// when that is full, straight to the move buffer), to a neighbouring slab's
// migrant message, or out of an open-y box; its id is `pid` when ids are
// tracked, and q.cell becomes -1.
template <class T, int SHAPE, int ONLY, int NT>
__device__ __forceinline__ float push_one(const StepDev& d, const SpeciesDev& sp, int s, const BoxDev& bx,
                                         int scx, int scy, int scz, const float* sF,
                                         SharedState<T, NT, ONLY>& sh, Part& q, int pid,
                                         int slot, int cb, unsigned& my_status)
{
    constexpr int LX = T::LX, LY = T::LY, LZ = T::LZ, N = T::N, PX = T::PX, TY = T::TY;
    constexpr int GO = T::GO;
    auto& rec = sh.rec;
    const int cell = q.cell;
    const float ox = q.o[0], oy = q.o[1], oz = q.o[2];
    float ux = q.u[0], uy = q.u[1], uz = q.u[2];
    const float w = q.w;
    const int lx = cell % LX;
    const int ly = (cell / LX) % LY;
    const int lz = cell / (LX * LY);

    // gather (Sec. 4: product of 1D weights at each Yee position); CIC (8 terms
    // a component) keeps the scalar form, which measured faster there
    const bool ec = ONLY == 0 && sp.ec != 0;
    float Ef[3], Bf[3];
    if constexpr (SHAPE != 1) {
        gather_pairs<T, SHAPE>(sF, lx + GO, ly + GO, lz + GO, ox, oy, oz, ec, Ef, Bf);
    } else {
        const AxisCic ax(lx + GO, ox, ec), ay(ly + GO, oy, ec), az(lz + GO, oz, ec);
        Ef[0] = gather_cic<PX, TY>(sF + 0 * N, ax.bh, ay.bi, az.bi, ax.wh, ay.wi, az.wi);
        Ef[1] = gather_cic<PX, TY>(sF + 1 * N, ax.bi, ay.bh, az.bi, ax.wi, ay.wh, az.wi);
        Ef[2] = gather_cic<PX, TY>(sF + 2 * N, ax.bi, ay.bi, az.bh, ax.wi, ay.wi, az.wh);
        Bf[0] = gather_cic<PX, TY>(sF + T::BOFF, ax.bi, ay.bh, az.bh, ax.wi, ay.wh, az.wh);
        Bf[1] = gather_cic<PX, TY>(sF + T::BOFF + N, ax.bh, ay.bi, az.bh, ax.wh, ay.wi, az.wh);
        Bf[2] = gather_cic<PX, TY>(sF + T::BOFF + 2 * N, ax.bh, ay.bh, az.bi, ax.wh, ay.wh, az.wi);
    }
    const float Ex = Ef[0], Ey = Ef[1], Ez = Ef[2], Bx = Bf[0], By = Bf[1], Bz = Bf[2];

    // relativistic Boris push (Boris 1970): half kick, rotation, half kick
    const float eps = sp.eps;
    const float umx = fmaf(eps, Ex, ux), umy = fmaf(eps, Ey, uy), umz = fmaf(eps, Ez, uz);
    const float ginv = rsqrt_ge1(1.0f + umx * umx + umy * umy + umz * umz);
    const float tx = eps * Bx * ginv, ty = eps * By * ginv, tz = eps * Bz * ginv;
    const float t2 = 1.0f + tx * tx + ty * ty + tz * tz;
    const float f = SHAPE == 1 ? 2.0f / t2 : two_over_ge1(t2);
    const float sx = f * tx, sy = f * ty, sz = f * tz;
    const float upx = umx + (umy * tz - umz * ty);
    const float upy = umy + (umz * tx - umx * tz);
    const float upz = umz + (umx * ty - umy * tx);
    ux = umx + (upy * sz - upz * sy) + eps * Ex;
    uy = umy + (upz * sx - upx * sz) + eps * Ey;
    uz = umz + (upx * sy - upy * sx) + eps * Ez;
    const float gi = rsqrt_ge1(1.0f + ux * ux + uy * uy + uz * uz);
    float Dx = d.move[0] * ux * gi, Dy = d.move[1] * uy * gi, Dz = d.move[2] * uz * gi;
    if (!(fabsf(Dx) < 0.5f && fabsf(Dy) < 0.5f && fabsf(Dz) < 0.5f)) {
        my_status |= ST_PARTICLE;  // non-finite or superluminal: freeze it
        Dx = Dy = Dz = 0.0f;
        ux = uy = uz = 0.0f;
    }
    const float x1 = ox + Dx, y1 = oy + Dy, z1 = oz + Dz;

    // deposit record (the current goes in afterwards, in another lane order)
    bool common;
    if (SHAPE == 2)
        common = ((ox >= 0.5f) == (x1 >= 0.5f)) && ((oy >= 0.5f) == (y1 >= 0.5f)) &&
                 ((oz >= 0.5f) == (z1 >= 0.5f));
    else
        common = x1 >= 0.0f && x1 < 1.0f && y1 >= 0.0f && y1 < 1.0f && z1 >= 0.0f && z1 < 1.0f;
    const int rs = rslot(slot);
    rec.l[rs] = (lx + GO) | ((ly + GO) << 8) | ((lz + GO) << 16) | (common ? 0 : (1 << 24));
    rec.o[0][rs] = ox;
    rec.o[1][rs] = oy;
    rec.o[2][rs] = oz;
    rec.D[0][rs] = Dx;
    rec.D[1][rs] = Dy;
    rec.D[2][rs] = Dz;
    rec.w[rs] = w;
    if (!common)
        rec.gen[atomicAdd(&sh.ngen[cb], 1)] = slot;
    // bound on every current term of this particle: |jcoef_d w P| with |P| <= |D_d|
    // (P is a difference of cumulative shape sums, whose slope is at most 1),
    // times |T| <= (max S)^2: 9/16 for TSC (S <= 3/4), 4/9 for PCS (S <= 2/3), 1 for CIC
    const float bnd = move_bound<SHAPE>(sp.jcoef, w, Dx, Dy, Dz);

    // new cell and offsets
    const float fx_ = floorf(x1), fy_ = floorf(y1), fz_ = floorf(z1);
    const float kOneMinus = 0.99999994f;  // largest float below 1
    const float nox = fminf(x1 - fx_, kOneMinus);
    const float noy = fminf(y1 - fy_, kOneMinus);
    const float noz = fminf(z1 - fz_, kOneMinus);
    const int nlx = lx + (int)fx_, nly = ly + (int)fy_, nlz = lz + (int)fz_;
    // the edges are powers of two: any bit outside them is a supercell left
    if (((nlx & ~(LX - 1)) | (nly & ~(LY - 1)) | (nlz & ~(LZ - 1))) == 0) {
        q.cell = nlx + LX * (nly + LY * nlz);
        q.o[0] = nox;
        q.o[1] = noy;
        q.o[2] = noz;
        q.u[0] = ux;
        q.u[1] = uy;
        q.u[2] = uz;
    } else {
        // leaves the supercell: into the move buffer, towards the neighbour
        // supercell (periodic within the box), or, through a y face of an
        // open-y box, out of the simulation
        const int dsx = nlx < 0 ? -1 : (nlx >= LX ? 1 : 0);
        const int dsy = nly < 0 ? -1 : (nly >= LY ? 1 : 0);
        const int dsz = nlz < 0 ? -1 : (nlz >= LZ ? 1 : 0);
        int tsx = scx + dsx, tsy = scy + dsy, tsz = scz + dsz;
        if (bx.sub_z && (tsz < 0 || tsz >= bx.nscz)) {
            // through a z face of a subdomain slab: into that face's migrant
            // message for the neighbouring slab
            tsx += tsx < 0 ? bx.nscx : (tsx >= bx.nscx ? -bx.nscx : 0);
            tsy += tsy < 0 ? bx.nscy : (tsy >= bx.nscy ? -bx.nscy : 0);
            char* msg = d.mig + (tsz < 0 ? 0 : d.mig_bytes);
            const int m = atomicAdd(&reinterpret_cast<MigHeader*>(msg)->count, 1);
            if (m < d.mig_cap) {
                MigRec r;
                r.s = s;
                r.sx = tsx;
                r.sy = tsy;
                r.cell = (nlx - dsx * LX) + LX * ((nly - dsy * LY) + LY * (nlz - dsz * LZ));
                r.ox = nox;
                r.oy = noy;
                r.oz = noz;
                r.ux = ux;
                r.uy = uy;
                r.uz = uz;
                r.w = w;
                r.pid = pid;
                int4* dst = reinterpret_cast<int4*>(msg + sizeof(MigHeader) + (int64_t)m * sizeof(MigRec));
                const int4* src = reinterpret_cast<const int4*>(&r);
                dst[0] = src[0];
                dst[1] = src[1];
                dst[2] = src[2];
            } else {
                my_status |= ST_CAPACITY;
            }
        } else if (!(bx.oy.open_y && (tsy < 0 || tsy >= bx.nscy))) {
            tsx += tsx < 0 ? bx.nscx : (tsx >= bx.nscx ? -bx.nscx : 0);
            tsy += tsy < 0 ? bx.nscy : (tsy >= bx.nscy ? -bx.nscy : 0);
            tsz += tsz < 0 ? bx.nscz : (tsz >= bx.nscz ? -bx.nscz : 0);
            const int dest_sc = bx.sc_base + (tsz * bx.nscy + tsy) * bx.nscx + tsx;
            const int dest_cell = (nlx - dsx * LX) + LX * ((nly - dsy * LY) + LY * (nlz - dsz * LZ));
            const int destL = s * d.nsc + dest_sc;
            const int k = atomicAdd(&sh.nlv, 1);
            if (k < kLeaverBuf) {
                // handed to the move buffer at the CTA's next work item, so
                // that no warp waits here for a global atomic's reply
                sh.lv.dest[k] = destL;
                sh.lv.cell[k] = dest_cell;
                sh.lv.o[0][k] = nox;
                sh.lv.o[1][k] = noy;
                sh.lv.o[2][k] = noz;
                sh.lv.u[0][k] = ux;
                sh.lv.u[1][k] = uy;
                sh.lv.u[2][k] = uz;
                sh.lv.w[k] = w;
                sh.lv.pid[k] = pid;
            } else {
                const int m = warp_aggregated_add(d.mv_count);
                if (m < d.mv_cap) {
                    d.mv_rank[m] = atomicAdd(d.narrive + destL, 1);
                    d.mv_dest[m] = destL;
                    d.mv_cell[m] = dest_cell;
                    d.mv_ox[m] = nox;
                    d.mv_oy[m] = noy;
                    d.mv_oz[m] = noz;
                    d.mv_ux[m] = ux;
                    d.mv_uy[m] = uy;
                    d.mv_uz[m] = uz;
                    d.mv_w[m] = w;
                    if (d.pid)
                        d.mv_pid[m] = pid;
                } else {
                    my_status |= ST_CAPACITY;
                }
            }
        }
        q.cell = -1;
    }
    return bnd;
}

// The CTA's collected leavers into the move buffer: one reservation, then
// every leaver's rank among the arrivals of its destination list (all
// threads converged; sh.nlv stable since the last block barrier).
template <class T, int NT, int ONLY>
__device__ __forceinline__ void flush_leavers(const StepDev& d, SharedState<T, NT, ONLY>& sh, unsigned& my_status)
{
    const int n = min(sh.nlv, kLeaverBuf);
    if (n == 0)
        return;
    if (threadIdx.x == 0)
        sh.lv_base = atomicAdd(d.mv_count, n);
    __syncthreads();
    const int base = sh.lv_base;
    for (int k = threadIdx.x; k < n; k += NT) {
        const int m = base + k;
        if (m >= d.mv_cap) {
            my_status |= ST_CAPACITY;
            continue;
        }
        const int L = sh.lv.dest[k];
        d.mv_rank[m] = atomicAdd(d.narrive + L, 1);
        d.mv_dest[m] = L;
        d.mv_cell[m] = sh.lv.cell[k];
        d.mv_ox[m] = sh.lv.o[0][k];
        d.mv_oy[m] = sh.lv.o[1][k];
        d.mv_oz[m] = sh.lv.o[2][k];
        d.mv_ux[m] = sh.lv.u[0][k];
        d.mv_uy[m] = sh.lv.u[1][k];
        d.mv_uz[m] = sh.lv.u[2][k];
        d.mv_w[m] = sh.lv.w[k];
        if (d.pid)
            d.mv_pid[m] = sh.lv.pid[k];
    }
}

// ------------------------------------------------------------ one frame list

// Add the chunk's integer tile (scaled back by inv) into the FP32 tile and
// clear it; each thread owns its entries (16-byte groups of four; N is a
// multiple of 4 and both tiles are 16-byte aligned), no atomics.
template <int N, int NT>
__device__ __forceinline__ void fold_tile(int* sJi, float* sJf, float inv)
{
    int4* qi = reinterpret_cast<int4*>(sJi);
    float4* qf = reinterpret_cast<float4*>(sJf);
    for (int v = threadIdx.x; v < 3 * N / 4; v += NT) {
        const int4 q = qi[v];
        if ((q.x | q.y | q.z | q.w) != 0) {
            float4 f = qf[v];
            f.x = fmaf((float)q.x, inv, f.x);
            f.y = fmaf((float)q.y, inv, f.y);
            f.z = fmaf((float)q.z, inv, f.z);
            f.w = fmaf((float)q.w, inv, f.w);
            qf[v] = f;
            qi[v] = make_int4(0, 0, 0, 0);
        }
    }
}

// Pushes the frame list of species s in supercell g chunk by chunk and
// deposits its current into the shared tile; returns the number of its
// particles that stay (the list's new count; they occupy its first slots).
template <class T, int SHAPE, int ONLY, int NT>
__device__ __forceinline__ int push_list(const StepDev& d, const SpeciesDev& sp, int s, int g,
                                          const BoxDev& bx, int scx, int scy, int scz,
                                          const float* sF, int* sJi, float* sJf,
                                          SharedState<T, NT, ONLY>& sh, bool sort_pass, unsigned& my_status)
{
    constexpr int S = T::S, N = T::N;
    constexpr bool SORTS = SHAPE == 1;  // sorted in the push, chunk by chunk
    constexpr int C = SharedState<T, NT, ONLY>::C;
    constexpr bool DEAL = SHAPE == 3;  // bank-dealt deposit slots (see deal_slot)
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int L = s * d.nsc + g;
    const int n = d.count[L];
    const int* ft = d.ftab + d.foff[L];
    auto gidx = [&](int slot) -> int64_t { return (int64_t)ft[(unsigned)slot / S] * S + (unsigned)slot % S; };
    constexpr int NQ = SharedState<T, NT, ONLY>::NQ, NWARP = NT / 32;
    constexpr int kLogC = C == 256 ? 8 : 7;
    static_assert(C == 1 << kLogC, "a chunk is 128 or 256 particles");
    const int ls = SORTS ? 2 : dep_log_stride(n, S);
    // the integer tile holds the current of tile_n particles (of the chunks
    // since the last fold) at the scale 1 / tile_inv: it goes on collecting while
    // the chunks' scales (powers of two) agree and kTileTerms are not passed (256
    // threads, TSC: 128^3 at 8 per cell 0.980 -> 0.968 ms, 256^3 8.37 -> 8.33;
    // 128 threads, two particles each, 1.525 -> 1.553 ms, so those fold every
    // chunk, as CIC does, whose rounding stays)
    constexpr int kTileMax = SORTS || NT < 256 ? 0 : kTileTerms;
    static_assert(C <= kTileTerms, "a chunk fits in the tile");
    float tile_inv = 0.0f;
    int tile_n = 0;
    int ndef = 0;  // general-window moves set aside in sh.gd
    int surv = 0;  // particles of the list that stay, written back so far
    // chunk c uses the bound / general-list counters cb = c & 1; the other
    // pair is cleared after the chunk's first barrier (its last readers were
    // the previous chunk's deposits, its next writers come after the next
    // chunk's last barrier)
    int cb = 0;
    for (int base = 0; base < n; base += C, cb ^= 1) {
        const int cn = min(C, n - base);
        if (tile_n > 0 && tile_n + cn > kTileMax) {  // the push below does not touch J
            fold_tile<N, NT>(sJi, sJf, tile_inv);
            tile_n = 0;
        }
        int boff = 0;
        const bool sort = SORTS && sort_pass;
        if (sort) {
            // CIC: stage the chunk (coalesced), key = cell, then a counting
            // sort; the pushed particles go back to the list in sorted order.
            // Against a sort of the whole lists by the frame maintenance (as
            // for TSC and PCS) this costs no extra pass over the particles, and
            // CIC gains little from whole-list order (128^3, 8 per cell, push +
            // maintenance: 0.842 ms this way, 0.864 ms with the lists sorted
            // there).  It also keeps the particles of every chunk together,
            // and with them the fixed-point scale of its current: the
            // energy-conserving CIC gather jumps at half a cell, where another
            // rounding now and then gives a particle another kick.
            for (int k = tid; k < S; k += NT)
                sh.hist[k] = 0;
            __syncthreads();
            for (int j = tid; j < cn; j += NT) {
                const int64_t idx = gidx(base + j);
                const int cell = d.cell[idx];
                sh.st.cell[j] = cell;
                sh.st.o[0][j] = d.ox[idx];
                sh.st.o[1][j] = d.oy[idx];
                sh.st.o[2][j] = d.oz[idx];
                sh.st.u[0][j] = d.ux[idx];
                sh.st.u[1][j] = d.uy[idx];
                sh.st.u[2][j] = d.uz[idx];
                sh.st.w[j] = d.w[idx];
                if (d.pid)
                    sh.st.pid[j] = d.pid[idx];
                sh.st.kr[j] = (cell << 16) | atomicAdd(&sh.hist[cell], 1);
            }
            __syncthreads();
            if (wid == 0)
                warp_exclusive_scan_counts(sh.hist, sh.off, S);
            __syncthreads();
            for (int j = tid; j < cn; j += NT) {
                const int kr = sh.st.kr[j];
                sh.st.perm[sh.off[kr >> 16] + (kr & 0xffff)] = j;
            }
            __syncthreads();
        }
        if (DEAL) {
            for (int j = tid; j < cn; j += NT) {
                const int bk = dep_bank<T>(sh.st.cell[j]);
                sh.st.brk[j] = (bk << 16) | atomicAdd(&sh.bh[bk], 1);
            }
            __syncthreads();
            boff = bank_offsets(sh.bh, lane);
        }
        // push, from the stage that an async copy filled while the previous
        // chunk deposited.
        // Every read of the chunk's list slots happens before the barrier
        // below, every write after it.
        Part qs[NQ];
        int pids[NQ];
        unsigned stays[NQ];
#pragma unroll
        for (int r = 0; r < NQ; ++r) {
            const int sidx = r * NT + tid;
            const int slot = DEAL ? dealt_slot<C>(sh.st.brk, sidx, cn, boff) : sidx;
            float bnd = 0.0f;
            qs[r].cell = -1;
            if (sidx < cn) {
                const int j = sort ? sh.st.perm[sidx] : sidx;
                Part& q = qs[r];
                q.cell = sh.st.cell[j];
                q.o[0] = sh.st.o[0][j];
                q.o[1] = sh.st.o[1][j];
                q.o[2] = sh.st.o[2][j];
                q.u[0] = sh.st.u[0][j];
                q.u[1] = sh.st.u[1][j];
                q.u[2] = sh.st.u[2][j];
                q.w = sh.st.w[j];
                pids[r] = !d.pid ? 0 : (sort ? sh.st.pid[j] : d.pid[gidx(base + sidx)]);
                bnd = push_one<T, SHAPE, ONLY, NT>(d, sp, s, bx, scx, scy, scz, sF, sh, q, pids[r], slot, cb,
                                             my_status);
            }
            stays[r] = __ballot_sync(0xffffffffu, qs[r].cell >= 0);
            const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(bnd));
            if (lane == 0) {
                sh.alive[r * NWARP + wid] = stays[r];
                atomicMax(&sh.bound_bits[cb], m);
            }
        }
        __syncthreads();
        // the particles that stay go back to the list compacted, in chunk
        // order (the leavers' slots close up; sorted lists stay nearly sorted)
        {
            static_assert(NQ * NWARP <= 32, "a lane per ballot");
            const int stay_n = lane < NQ * NWARP ? __popc(sh.alive[lane]) : 0;
            const int run = __reduce_add_sync(0xffffffffu, stay_n);
            int pre[NQ];
#pragma unroll
            for (int r = 0; r < NQ; ++r)
                pre[r] = __reduce_add_sync(0xffffffffu, lane < r * NWARP + wid ? stay_n : 0);
#pragma unroll
            for (int r = 0; r < NQ; ++r) {
                if (qs[r].cell < 0)
                    continue;
                const int src = base + r * NT + tid;
                const int dst = surv + pre[r] + __popc(stays[r] & ((1u << lane) - 1u));
                const bool moved = sort || dst != src;
                const int64_t idx = gidx(dst);
                store_part(d, idx, qs[r], moved);
                if (d.pid && moved)
                    d.pid[idx] = pids[r];
            }
            surv += run;
        }
        if (tid == 0) {
            sh.ngen[cb ^ 1] = 0;
            sh.bound_bits[cb ^ 1] = 0u;
        }
        if (DEAL && T::G == 2 && tid < 32)
            sh.bh[tid] = 0;  // every warp read it before the barrier above; next written after the chunk
        if (!sort && base + C < n)  // the stage is free: the next chunk flies during the deposit
            stage_chunk_async<T, NT, ONLY>(d, sh, L, base + C, min(C, n - base - C));
        // deposit: neighbouring lanes take chunk positions 1 << ls apart (the
        // list is sorted by node, so one warp's atomics land on different nodes
        // and mostly different banks); then the general-window moves
        float inv;
        const float scale = chunk_scale(__uint_as_float(sh.bound_bits[cb]), &inv);
        if (tile_n > 0 && inv != tile_inv) {
            fold_tile<N, NT>(sJi, sJf, tile_inv);
            tile_n = 0;
            __syncthreads();
        }
        tile_inv = inv;
        tile_n += cn;
        for (int r = 0; r < C / NT; ++r) {
            const int q = r * NT + tid;
            const int e = DEAL ? q : ((q << ls) & (C - 1)) + (q >> (kLogC - ls));
            if ((DEAL ? deal_pos<C>(q) : e) < cn && !(sh.rec.l[rslot(e)] >> 24))
                deposit_common<T, SHAPE, C>(sJi, sh.rec, e, sp.jcoef, scale);
        }
        // general-window moves: set aside for the list's end while they fit
        // (ngen and ndef are the same in every thread); otherwise whole groups
        // of 32 lane-parallel, one group per warp, and the rest one move per
        // warp, all lanes on it
        const int ngen = sh.ngen[cb];
        if (ndef + ngen <= kGenDefer) {
            for (int q = tid; q < ngen; q += NT) {
                const int e = rslot(sh.rec.gen[q]);
                const int k = ndef + q;
                const float Dx = sh.rec.D[0][e], Dy = sh.rec.D[1][e], Dz = sh.rec.D[2][e], w = sh.rec.w[e];
                sh.gd.l[k] = sh.rec.l[e];
                sh.gd.o[0][k] = sh.rec.o[0][e];
                sh.gd.o[1][k] = sh.rec.o[1][e];
                sh.gd.o[2][k] = sh.rec.o[2][e];
                sh.gd.D[0][k] = Dx;
                sh.gd.D[1][k] = Dy;
                sh.gd.D[2][k] = Dz;
                sh.gd.w[k] = w;
                atomicMax(&sh.gd_bound_bits, __float_as_uint(move_bound<SHAPE>(sp.jcoef, w, Dx, Dy, Dz)));
            }
            ndef += ngen;
        } else {
            const int nfull = ngen & ~31;
            for (int q = tid; q < nfull; q += NT)
                deposit_general<T, SHAPE, C>(sJi, sh.rec, sh.rec.gen[q], sp.jcoef, scale);
            const int rem = ngen - nfull;
            for (int t = ((wid - (nfull >> 5)) % NWARP + NWARP) % NWARP; t < rem; t += NWARP)
                deposit_general_warp<T, SHAPE, C>(sJi, sh.rec, sh.rec.gen[nfull + t], sp.jcoef, scale);
        }
        cp_async_wait_all();
        __syncthreads();
    }
    if (tile_n > 0)
        fold_tile<N, NT>(sJi, sJf, tile_inv);
    if (ndef > 0) {
        // the set-aside general-window moves, one per thread, with their own
        // fixed-point scale (at most kGenDefer terms per node)
        __syncthreads();
        float inv;
        const float scale = chunk_scale(__uint_as_float(sh.gd_bound_bits), &inv);
        for (int k = tid; k < ndef; k += NT) {
            const float o[3] = {sh.gd.o[0][k], sh.gd.o[1][k], sh.gd.o[2][k]};
            const float D[3] = {sh.gd.D[0][k], sh.gd.D[1][k], sh.gd.D[2][k]};
            deposit_general_move<T, SHAPE>(sJi, sh.gd.l[k], o, D, sh.gd.w[k], sp.jcoef, scale);
        }
        __syncthreads();
        fold_tile<N, NT>(sJi, sJf, inv);
    }
    // the caller synchronises before the flush
    return surv;
}

// ------------------------------------------------------------ the kernel

// Resident CTAs the registers are allocated for: 1024 threads per SM (64
// registers each; with the PCS guards 512), or fewer CTAs where shared memory
// holds no more, so that their warps get the registers instead (128 threads:
// 4 CTAs at 128 registers; at 64 they spilled, 128^3 TSC 4x4x4 1.78 -> 1.55 ms).
template <class T, int NT, int ONLY>
constexpr int push_blocks()
{
    constexpr int by_threads = (T::G == 1 ? 1024 : 512) / NT;
    constexpr int by_smem = (int)(233472 / (sizeof(float) * T::TILES + sizeof(SharedState<T, NT, ONLY>) + 1024));
    return by_smem < 1 ? 1 : (by_smem < by_threads ? by_smem : by_threads);
}

// ONLY 1, 2, 3: every mobile species has that shape and the momentum-conserving
// gather, and the kernel holds that code alone; 0: any mix.
template <class T, int NT, int ONLY>
__global__ void __launch_bounds__(NT, (push_blocks<T, NT, ONLY>())) k_push_deposit(const StepDev d)
{
    constexpr int TX = T::TX, TY = T::TY, TZ = T::TZ, PX = T::PX, N = T::N;
    constexpr int LX = T::LX, LY = T::LY, LZ = T::LZ;
    extern __shared__ __align__(128) float smem[];
    // layout (dyn_smem): [3N E floats, padded to BOFF][3N B floats][3N int current][3N float current]
    // [SharedState]
    float* sF = smem;  // [3][TZ][TY][PX] Ex Ey Ez at sF, Bx By Bz at sF + BOFF
    int* sJi = reinterpret_cast<int*>(smem + T::BOFF + 3 * N);  // [3][TZ][TY][PX] chunk accumulator
    float* sJf = smem + T::BOFF + 6 * N;                        // [3][TZ][TY][PX] supercell current
    SharedState<T, NT, ONLY>& sh = *reinterpret_cast<SharedState<T, NT, ONLY>*>(smem + T::TILES);

    const int tid = threadIdx.x;
    unsigned my_status = 0;
    // every sort_every-th step reorders the lists; CIC lists here (the counter
    // only changes between launches, so all CTAs agree)
    const bool sort_pass = SharedState<T, NT, ONLY>::SORTS && *d.step_ctr % d.sort_every == 0;
    // work items: tid 0 asks for the next one while the block works on the
    // current one, and publishes it at the end of the item
    if (tid == 0) {
        sh.item = atomicAdd(d.work_counter, 1);
        sh.nlv = 0;
        mbar_init(&sh.mb_tile, 1);
        fence_mbar_init();
        sh.tile_phase = 0;
        sh.abort = 0;
    }
    if (T::G == 2 && tid < 32)
        sh.bh[tid] = 0;  // each chunk clears it after use
    __syncthreads();
    const int nitems = *d.nitems;
    for (;;) {
        const int item = sh.item;
        if (item >= nitems)
            break;
        int next_item = 0;
        if (tid == 0)
            next_item = atomicAdd(d.work_counter, 1);
        // the previous item's leavers into the move buffer (their global
        // atomics' replies come back while this item starts)
        flush_leavers<T, NT, ONLY>(d, sh, my_status);
        const int g = d.items[item];
        const BoxDev bx = d.boxes[d.sc_box[g]];
        const int loc = g - bx.sc_base;
        const int scx = loc % bx.nscx;
        const int scy = (loc / bx.nscx) % bx.nscy;
        const int scz = loc / (bx.nscx * bx.nscy);

        if (tid == 0)
            sh.nlv = 0;  // every thread read it in flush_leavers (before its barrier, if it had one)

        // ---- 1. the E/B tile by two tensor loads (TMA); the first chunk of
        // the first mobile list is copied meanwhile; the next work item's tile
        // is prefetched into L2; the J tiles are zeroed
        int pre_s = -1;
        for (int s = 0; s < d.nspecies && pre_s < 0; ++s) {
            const int n = d.count[s * d.nsc + g];
            if (d.sp[s].mobile && n > 0) {
                pre_s = s;
                if (!(sort_pass && d.sp[s].shape == 1))
                    stage_chunk_async<T, NT, ONLY>(d, sh, s * d.nsc + g, 0, min(SharedState<T, NT, ONLY>::C, n));
            }
        }
        if (tid == 0) {
            fence_proxy_async();
            mbar_expect_tx(&sh.mb_tile, 6u * 4u * (unsigned)N);
            const CUtensorMap* tm = d.tmaps + 2 * d.sc_box[g];
            tma_load_tile(sF, tm, scx * LX, scy * LY, scz * LZ, &sh.mb_tile);
            tma_load_tile(sF + T::BOFF, tm + 1, scx * LX, scy * LY, scz * LZ, &sh.mb_tile);
            if (next_item < nitems) {
                const int gn = d.items[next_item];
                const int bn = d.sc_box[gn];
                const BoxDev& bxn = d.boxes[bn];
                const int ln = gn - bxn.sc_base;
                const int xn = (ln % bxn.nscx) * LX, yn = ((ln / bxn.nscx) % bxn.nscy) * LY,
                          zn = (ln / (bxn.nscx * bxn.nscy)) * LZ;
                tma_prefetch_tile(d.tmaps + 2 * bn, xn, yn, zn);
                tma_prefetch_tile(d.tmaps + 2 * bn + 1, xn, yn, zn);
            }
        }
        for (int v = tid; v < 6 * N / 4; v += NT)  // int and float current tiles, contiguous; 0 bits = 0.0f
            reinterpret_cast<int4*>(sJi)[v] = make_int4(0, 0, 0, 0);
        if (tid == 0) {
            if (mbar_wait(&sh.mb_tile, (unsigned)sh.tile_phase)) {
                sh.tile_phase ^= 1;
            } else {
                sh.abort = 1;
                my_status |= ST_TIMEOUT;
            }
        }
        __syncthreads();
        if (sh.abort)
            break;

        // ---- 2. particles of every mobile species, 3. compaction
        for (int s = 0; s < d.nspecies; ++s) {
            const SpeciesDev sp = d.sp[s];
            const int L = s * d.nsc + g;
            const int n = d.count[L];
            if (!sp.mobile || n == 0)
                continue;
            if (tid == 0) {
                sh.ngen[0] = 0;
                sh.bound_bits[0] = 0u;
                sh.gd_bound_bits = 0u;
            }
            if (s != pre_s && !(sort_pass && sp.shape == 1))
                stage_chunk_async<T, NT, ONLY>(d, sh, L, 0, min(SharedState<T, NT, ONLY>::C, n));
            cp_async_wait_all();
            __syncthreads();
            int stay;
            if (ONLY == 2 || (ONLY == 0 && sp.shape == 2))
                stay = push_list<T, 2, ONLY, NT>(d, sp, s, g, bx, scx, scy, scz, sF, sJi, sJf, sh, sort_pass,
                                                 my_status);
            else if (T::G == 2 && (ONLY == 3 || (ONLY == 0 && sp.shape == 3)))
                stay = push_list<T, T::G == 2 ? 3 : 1, ONLY, NT>(d, sp, s, g, bx, scx, scy, scz, sF, sJi, sJf, sh,
                                                                sort_pass, my_status);
            else
                stay = push_list<T, 1, ONLY, NT>(d, sp, s, g, bx, scx, scy, scz, sF, sJi, sJf, sh, sort_pass,
                                                 my_status);
            if (tid == 0 && stay != n)
                d.count[L] = stay;  // the particles that stay fill the list's first slots
            __syncthreads();
        }

        // ---- 4. add the J tile to global J
        const int64_t pcell = padded_cells(bx);
        const int64_t start = ((int64_t)(scz * LZ) * bx.py + scy * LY) * bx.px + scx * LX;
        constexpr int ROW4 = TX / 4;
        constexpr int NJ4 = 3 * TZ * TY * ROW4;
        for (int v = tid; v < NJ4; v += NT) {
            const int r4 = v % ROW4;
            const int row = v / ROW4;
            const float4 val = *reinterpret_cast<const float4*>(sJf + row * PX + 4 * r4);
            if (val.x != 0.f || val.y != 0.f || val.z != 0.f || val.w != 0.f) {
                const int ty = row % TY;
                const int tz = (row / TY) % TZ;
                const int c = row / (TY * TZ);
                float* dst = bx.J + c * pcell + start + ((int64_t)tz * bx.py + ty) * bx.px + 4 * r4;
                atomicAdd(reinterpret_cast<float4*>(dst), val);
            }
        }
        if (tid == 0)
            sh.item = next_item;
        __syncthreads();
    }
    if (sh.abort) {
        // the tile wait gave up: give the loads in flight the same time once
        // more before the CTA's shared memory is released
        if (tid == 0)
            mbar_wait(&sh.mb_tile, (unsigned)sh.tile_phase);
    } else {
        flush_leavers<T, NT, ONLY>(d, sh, my_status);
    }
    if (my_status)
        atomicOr(d.status, my_status);
}

// ------------------------------------------------------------ dispatch

template <class T, int NT, int ONLY>
static size_t dyn_smem()
{
    // field tile (6 N floats) + int and float current tiles (3 N each) + shared state
    return sizeof(float) * T::TILES + sizeof(SharedState<T, NT, ONLY>);
}

// Sets the kernel's shared-memory limit and returns its resident CTAs per SM
// (call once, outside stream capture).
template <class T, int NT, int ONLY>
static cudaError_t configure_one(int* per_sm)
{
    auto kern = k_push_deposit<T, NT, ONLY>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)dyn_smem<T, NT, ONLY>());
    if (e != cudaSuccess)
        return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, NT, dyn_smem<T, NT, ONLY>());
}

template <class T, int NT, int ONLY>
static cudaError_t launch_one(const StepDev& d, int grid, cudaStream_t st)
{
    grid = min(max(grid, 1), max(1, d.nsc));
    k_push_deposit<T, NT, ONLY><<<grid, NT, dyn_smem<T, NT, ONLY>(), st>>>(d);
    return cudaGetLastError();
}

// (supercell edges, threads, guard): guard 1 for CIC/TSC contexts, 2 for
// contexts with a PCS species
#define PIC_PUSH_CASES_G1(X) \
    X(4, 4, 4, 64, 1)        \
    X(4, 4, 4, 128, 1)       \
    X(4, 4, 4, 256, 1)       \
    X(8, 4, 4, 128, 1)       \
    X(8, 4, 4, 256, 1)       \
    X(8, 8, 4, 128, 1)       \
    X(8, 8, 4, 256, 1)       \
    X(8, 8, 8, 256, 1)
#define PIC_PUSH_CASES_G2(X) \
    X(4, 4, 4, 128, 2)       \
    X(8, 4, 4, 256, 2)
#define PIC_PUSH_CASES(X) PIC_PUSH_CASES_G1(X) PIC_PUSH_CASES_G2(X)

// One translation unit per ONLY holds its kernels (they compile in parallel).
template <int ONLY>
cudaError_t configure_push_only(int LX, int LY, int LZ, int threads, int guard, int* per_sm);
template <int ONLY>
cudaError_t launch_push_only(const StepDev& d, int threads, int grid, cudaStream_t st);

#define PIC_PUSH_DEFINE(ONLY, CASES)                                                                          \
    template <>                                                                                               \
    cudaError_t configure_push_only<ONLY>(int LX, int LY, int LZ, int threads, int guard, int* per_sm)        \
    {                                                                                                         \
        CASES(PIC_PUSH_CONFIGURE_##ONLY) return cudaErrorInvalidValue;                                        \
    }                                                                                                         \
    template <>                                                                                               \
    cudaError_t launch_push_only<ONLY>(const StepDev& d, int threads, int grid, cudaStream_t st)              \
    {                                                                                                         \
        CASES(PIC_PUSH_LAUNCH_##ONLY) return cudaErrorInvalidValue;                                           \
    }
#define PIC_PUSH_CONFIGURE(ONLY, a, b, c, t, g)                      \
    if (LX == a && LY == b && LZ == c && threads == t && guard == g) \
        return configure_one<Tile<a, b, c, g>, t, ONLY>(per_sm);
#define PIC_PUSH_LAUNCH(ONLY, a, b, c, t, g)                                 \
    if (d.LX == a && d.LY == b && d.LZ == c && threads == t && d.guard == g) \
        return launch_one<Tile<a, b, c, g>, t, ONLY>(d, grid, st);
#define PIC_PUSH_CONFIGURE_0(...) PIC_PUSH_CONFIGURE(0, __VA_ARGS__)
#define PIC_PUSH_CONFIGURE_1(...) PIC_PUSH_CONFIGURE(1, __VA_ARGS__)
#define PIC_PUSH_CONFIGURE_2(...) PIC_PUSH_CONFIGURE(2, __VA_ARGS__)
#define PIC_PUSH_CONFIGURE_3(...) PIC_PUSH_CONFIGURE(3, __VA_ARGS__)
#define PIC_PUSH_LAUNCH_0(...) PIC_PUSH_LAUNCH(0, __VA_ARGS__)
#define PIC_PUSH_LAUNCH_1(...) PIC_PUSH_LAUNCH(1, __VA_ARGS__)
#define PIC_PUSH_LAUNCH_2(...) PIC_PUSH_LAUNCH(2, __VA_ARGS__)
#define PIC_PUSH_LAUNCH_3(...) PIC_PUSH_LAUNCH(3, __VA_ARGS__)

}  // namespace pic
