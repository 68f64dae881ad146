// k_fields.cu -- Yee FDTD update (Yee 1966, the "Yee field solver" of Sec. 4)
// for the mixed form's guard-padded FP32 fields, field import/export, and
// the FP64 diagnostics reductions.
//
// Staggering: Ex(i+1/2,j,k) Ey(i,j+1/2,k) Ez(i,j,k+1/2), Bx(i,j+1/2,k+1/2)
// By(i+1/2,j,k+1/2) Bz(i+1/2,j+1/2,k); J with E.  One step of the field
// half of the cycle:
//   B^{n+1/2} = B^n - dt/2 curl E^n
//   E^{n+1}   = E^n + dt (curl B^{n+1/2} - J^{n+1/2})
//   B^{n+1}   = B^{n+1/2} - dt/2 curl E^{n+1}
// Every kernel writes each updated interior value also into its periodic
// guard images, so the next kernel (and the next push's tile loads) read
// guards without a separate exchange.  The E kernel folds the J guard
// images (deposits that spilled over the periodic seam) into the current of
// each interior cell as it reads it; J itself stays as deposited (the step
// zeroes it before the push, and a read of J folds the same way).
//
// One launch covers all boxes: blocks of 32 x 8 cells in x-y, each thread
// kYeeZ cells along z, box found from a per-box block offset table.
#include "pic_internal.cuh"
#include "tma.cuh"

#include <algorithm>
#include <cmath>

namespace pic {

constexpr int kYeeZ = kYeeCellsZ;  // box edges are multiples of the supercell edge, >= 4

struct YeeArgs {
    const BoxDev* boxes;
    const int* blk_off;  // [nboxes + 1]
    int nboxes;
    float tau;           // dt/2 for the B halves, dt for E
    float ih[3];         // 1 / h_d
    const long long* step_no;
    double dt_d;
    double dx_d[3];
};

__device__ __forceinline__ int find_box(const int* off, int n, int blk)
{
    int lo = 0, hi = n;  // off[lo] <= blk < off[hi]
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (off[mid] <= blk)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

struct CellAt {
    int x, y, z;
    bool ok;
};

__device__ __forceinline__ CellAt yee_cell(const YeeArgs& a, const BoxDev*& bp)
{
    const int box = find_box(a.blk_off, a.nboxes, blockIdx.x);
    bp = a.boxes + box;  // fields read through the pointer as used, not copied
    const BoxDev& b = *bp;
    const int local = blockIdx.x - a.blk_off[box];
    const int nbx = (b.nx + 31) >> 5, nby = (b.ny + 7) >> 3;
    CellAt c;
    c.x = (local % nbx) * 32 + threadIdx.x;
    c.y = ((local / nbx) % nby) * 8 + threadIdx.y;
    c.z = local / (nbx * nby);
    c.ok = c.x < b.nx && c.y < b.ny;
    return c;
}

// Periodic images of an interior coordinate v in [0, n) inside the padded
// range [-lo, n + hi): v itself, and v + n when v < hi or v - n when
// v >= n - lo.  Boxes are at least lo + hi cells long (4 for CIC/TSC
// guards, 8 with the PCS guards), so at most one of the two applies.
// Returns the count (1 or 2), [0] = v.
__device__ __forceinline__ int images(int v, int n, int lo, int hi, int* out)
{
    out[0] = v;
    if (v < hi) {
        out[1] = v + n;
        return 2;
    }
    if (v >= n - lo) {
        out[1] = v - n;
        return 2;
    }
    return 1;
}

__device__ __forceinline__ int images_x(const BoxDev& b, int v, int* out)
{
    return images(v, b.nx, b.gx, b.px - b.nx - b.gx, out);
}
__device__ __forceinline__ int images_y(const BoxDev& b, int v, int* out)
{
    return images(v, b.ny, b.gy, b.py - b.ny - b.gy, out);
}
__device__ __forceinline__ int images_z(const BoxDev& b, int v, int* out)
{
    return images(v, b.nz, b.gz, b.pz - b.nz - b.gz, out);
}

__device__ __forceinline__ void store_with_images(const BoxDev& b, float* F, const CellAt& c,
                                                  float v)
{
    int ix[2], iy[2], iz[2];
    int nx = images_x(b, c.x, ix), ny = images_y(b, c.y, iy), nz = images_z(b, c.z, iz);
    for (int k = 0; k < nz; ++k)
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i)
                F[padded_index(b, ix[i], iy[j], iz[k])] = v;
}

// The Yee kernels take the guard layout as a template constant (G = 1:
// CIC/TSC contexts, 2: PCS), so that the image arithmetic of every cell is
// immediate.
template <int G>
struct GuardsOf {
    static constexpr int hx = G == 1 ? 3 : 6, hyz = G == 1 ? 2 : 3;
};

template <int G>
__device__ __forceinline__ int64_t pidx(const BoxDev& b, int x, int y, int z)
{
    return ((int64_t)(z + G) * b.py + (y + G)) * b.px + (x + G);
}

template <int G>
__device__ __forceinline__ void store_images_g(const BoxDev& b, float* F, const CellAt& c, float v)
{
    int ix[2], iy[2], iz[2];
    const int nx = images(c.x, b.nx, G, GuardsOf<G>::hx, ix);
    const int ny = images(c.y, b.ny, G, GuardsOf<G>::hyz, iy);
    const int nz = images(c.z, b.nz, G, GuardsOf<G>::hyz, iz);
    for (int k = 0; k < nz; ++k)
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i)
                F[pidx<G>(b, ix[i], iy[j], iz[k])] = v;
}

// Each thread updates kYeeZ cells stacked in z: all loads first, then the
// arithmetic and the stores, so that a warp keeps kYeeZ times the bytes in
// flight (the update is bound by DRAM latency with one cell per thread).
template <int G>
__global__ void __launch_bounds__(256) k_yee_b(const YeeArgs a)
{
    const BoxDev* bp;
    CellAt c = yee_cell(a, bp);
    if (!c.ok)
        return;
    const BoxDev& b = *bp;
    const int64_t pc = padded_cells(b);
    const int64_t sx = 1, sy = b.px, sz = (int64_t)b.px * b.py;
    const float* __restrict__ Ex = b.E;
    const float* __restrict__ Ey = b.E + pc;
    const float* __restrict__ Ez = b.E + 2 * pc;
    float* __restrict__ Bx = b.B;
    float* __restrict__ By = b.B + pc;
    float* __restrict__ Bz = b.B + 2 * pc;
    const int z0 = c.z * kYeeZ;
    float cx[kYeeZ], cy[kYeeZ], cz[kYeeZ], bx[kYeeZ], by[kYeeZ], bz[kYeeZ];
    // Ex, Ey one plane up are the next cell's own values (the thread's cells
    // are stacked in z): kYeeZ + 1 planes of them, loaded once
    float exs[kYeeZ + 1], eys[kYeeZ + 1];
#pragma unroll
    for (int q = 0; q <= kYeeZ; ++q) {
        const int64_t i = pidx<G>(b, c.x, c.y, z0 + q);
        exs[q] = __ldg(Ex + i);
        eys[q] = __ldg(Ey + i);
    }
#pragma unroll
    for (int q = 0; q < kYeeZ; ++q) {
        const int64_t i = pidx<G>(b, c.x, c.y, z0 + q);
        const float ex = exs[q], ey = eys[q], ez = __ldg(Ez + i);
        cx[q] = (__ldg(Ez + i + sy) - ez) * a.ih[1] - (eys[q + 1] - ey) * a.ih[2];
        cy[q] = (exs[q + 1] - ex) * a.ih[2] - (__ldg(Ez + i + sx) - ez) * a.ih[0];
        cz[q] = (__ldg(Ey + i + sx) - ey) * a.ih[0] - (__ldg(Ex + i + sy) - ex) * a.ih[1];
        bx[q] = Bx[i];
        by[q] = By[i];
        bz[q] = Bz[i];
    }
#pragma unroll
    for (int q = 0; q < kYeeZ; ++q) {
        c.z = z0 + q;
        store_images_g<G>(b, Bx, c, bx[q] - a.tau * cx[q]);
        store_images_g<G>(b, By, c, by[q] - a.tau * cy[q]);
        store_images_g<G>(b, Bz, c, bz[q] - a.tau * cz[q]);
    }
}

// Laser antenna: adds the sheet current at the Ex positions
// (x+1/2, ant_j, z) of every box with an antenna into J, at the time of this
// step's current, t = (n + 1/2) dt, n = steps taken before it (step_no was
// advanced earlier in the step).  Runs before the E update, which folds it
// in with the deposits.  FP64 throughout: omega t reaches thousands of
// radians.  One thread per (box, x, z), grid-stride.  The FP64 pipe bounds it,
// so the two factors of the time alone are formed once per block (by two of
// its warps) and the points are spread over every SM.
constexpr int kAntThreads = 128, kAntBlocks = 304;

__global__ void __launch_bounds__(kAntThreads) k_antenna(const YeeArgs a)
{
    __shared__ double time_factor[2];
    for (int box = 0; box < a.nboxes; ++box) {
        const BoxDev& b = a.boxes[box];
        const OpenYDev o = b.oy;
        const int j = o.ant_j;
        const int64_t n = (int64_t)b.nx * b.nz;
        const int64_t t0 = blockIdx.x * (int64_t)kAntThreads;
        if (j < 0 || t0 >= n)
            continue;
        if ((threadIdx.x & 31) == 0 && threadIdx.x < 64) {
            const double t = ((double)(*a.step_no) - 0.5) * a.dt_d;
            if (threadIdx.x == 0)
                time_factor[0] = o.ant_tau > 0.0 ? exp(-((t - o.ant_t0) / o.ant_tau) * ((t - o.ant_t0) / o.ant_tau)) : 1.0;
            else
                time_factor[1] = cos(o.ant_omega * (t - o.ant_t0));
        }
        __syncthreads();
        const double T = time_factor[0], C = time_factor[1];
        for (int64_t t = t0 + threadIdx.x; t < n; t += (int64_t)kAntBlocks * kAntThreads) {
            const int x = (int)(t % b.nx), z = (int)(t / b.nx);
            double G = 1.0;
            if (o.ant_w0 > 0.0) {
                const double px = ((double)x + 0.5) * a.dx_d[0] - o.ant_xc;
                const double pz = (double)z * a.dx_d[2] - o.ant_zc;
                G = exp(-(px * px + pz * pz) / (o.ant_w0 * o.ant_w0));
            }
            b.J[padded_index(b, x, j, z)] += (float)(o.ant_J0 * G * T * C);
        }
        __syncthreads();  // time_factor is free for the next box
    }
}

// FOLD_Z false: the boxes are subdomain slabs, whose z guards went to their
// neighbours (and theirs came in as additions): no z images to fold.
template <int G, bool FOLD_Z>
__global__ void __launch_bounds__(256, 4) k_yee_e(const YeeArgs a)
{
    const BoxDev* bp;
    CellAt c = yee_cell(a, bp);
    if (!c.ok)
        return;
    const BoxDev& b = *bp;
    const int64_t pc = padded_cells(b);
    const int64_t sx = 1, sy = b.px, sz = (int64_t)b.px * b.py;
    const float* __restrict__ Bx = b.B;
    const float* __restrict__ By = b.B + pc;
    const float* __restrict__ Bz = b.B + 2 * pc;
    float* __restrict__ Ex = b.E;
    float* __restrict__ Ey = b.E + pc;
    float* __restrict__ Ez = b.E + 2 * pc;
    const float* __restrict__ J = b.J;
    const int z0 = c.z * kYeeZ;
    int ix[2], iy[2];
    const int nx = images(c.x, b.nx, G, GuardsOf<G>::hx, ix);
    const int ny = images(c.y, b.ny, G, GuardsOf<G>::hyz, iy);
    float jx[kYeeZ], jy[kYeeZ], jz[kYeeZ], cx[kYeeZ], cy[kYeeZ], cz[kYeeZ], ex[kYeeZ], ey[kYeeZ], ez[kYeeZ];
    float bxs[kYeeZ + 1], bys[kYeeZ + 1];
    {
        const int64_t i0 = pidx<G>(b, c.x, c.y, z0 - 1);
        bxs[0] = __ldg(Bx + i0);
        bys[0] = __ldg(By + i0);
    }
#pragma unroll
    for (int q = 0; q < kYeeZ; ++q) {
        const int64_t i = pidx<G>(b, c.x, c.y, z0 + q);
        int iz[2];
        const int nz = FOLD_Z ? images(z0 + q, b.nz, G, GuardsOf<G>::hyz, iz) : (iz[0] = z0 + q, 1);
        // fold the J guard images into the interior
        jx[q] = 0.f;
        jy[q] = 0.f;
        jz[q] = 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    if (k < nz && j < ny && r < nx) {
                        const int64_t g = pidx<G>(b, ix[r], iy[j], iz[k]);
                        jx[q] += J[g];
                        jy[q] += J[pc + g];
                        jz[q] += J[2 * pc + g];
                    }
        // Bx, By one plane down: the previous cell's own values (cells stacked in z)
        bxs[q + 1] = __ldg(Bx + i);
        bys[q + 1] = __ldg(By + i);
        const float bxv = bxs[q + 1], byv = bys[q + 1], bzv = __ldg(Bz + i);
        cx[q] = (bzv - __ldg(Bz + i - sy)) * a.ih[1] - (byv - bys[q]) * a.ih[2];
        cy[q] = (bxv - bxs[q]) * a.ih[2] - (bzv - __ldg(Bz + i - sx)) * a.ih[0];
        cz[q] = (byv - __ldg(By + i - sx)) * a.ih[0] - (bxv - __ldg(Bx + i - sy)) * a.ih[1];
        ex[q] = Ex[i];
        ey[q] = Ey[i];
        ez[q] = Ez[i];
    }
#pragma unroll
    for (int q = 0; q < kYeeZ; ++q) {
        // J is left as deposited (the step zeroes it before the push, and a
        // read of J folds the images the same way)
        c.z = z0 + q;
        store_images_g<G>(b, Ex, c, ex[q] + a.tau * (cx[q] - jx[q]));
        store_images_g<G>(b, Ey, c, ey[q] + a.tau * (cy[q] - jy[q]));
        store_images_g<G>(b, Ez, c, ez[q] + a.tau * (cz[q] - jz[q]));
    }
}

// y absorber: every E and B value whose staggered y position lies in a
// damping layer is multiplied by exp(-sigma d^2) (d = depth in the layer, 0
// at its inner edge, 1 at the face), images included.  The fused field
// update multiplies the values as it stores them (1 outside the layers); after
// the in-place one k_absorb_y does.
__device__ __forceinline__ float absorb_factor(float y, int ny, int A, float sigma)
{
    float depth = 0.0f;
    if (y < (float)A)
        depth = ((float)A - y) / (float)A;
    else if (y > (float)(ny - A))
        depth = (y - (float)(ny - A)) / (float)A;
    depth = fminf(depth, 1.0f);
    return expf(-sigma * depth * depth);
}

// ------------------------------------------------------------ fused field update
//
// The whole field half of the cycle in one kernel, from one buffer pair into
// the other: E^n, B^n and J are read from `src`, E^{n+1} and B^{n+1} (with
// their periodic guard images) are written into `dst`, so that no value is
// overwritten while a neighbouring cell still needs it.  Each block z-marches
// an output tile of kFusedTX x kFusedTY cells through a chunk of planes, one
// thread per column of the tile and of the one-cell rim around it (a warp per
// row, the two rim columns of all rows in the last warp).  Iteration s:
//   B^{n+1/2}(s)  on the tile and its rim (E^n planes s, s+1),
//   one block barrier,
//   E^{n+1}(s)    on the tile and the rim above it in x and y
//                 (B^{n+1/2} planes s-1, s),
//   B^{n+1}(s-1)  on the tile (E^{n+1} planes s-1, s).
// A thread keeps its column's values of both planes in registers; shared
// memory holds what the four neighbouring columns need (two planes each of
// B^{n+1/2} and E^{n+1}).  Rim cells are formed again by the neighbouring
// tiles, and the first planes of a chunk by the chunk below.  The inputs of
// iteration s -- E^n(s+1), B^n(s) and J(s), each a plane tile of the three
// components -- arrive by tensor loads issued three iterations ahead on one
// mbarrier; a thread otherwise touches global memory only for its stores and
// for the few J guard images that fold into cells next to a box face (loaded
// an iteration ahead: the blocks at the faces set the pace of the others).
// HBM traffic per cell: E^n, B^n, J read and E^{n+1}, B^{n+1} written, 60 bytes
// (the three in-place kernels move 120); the rim comes from L2.  The arithmetic
// of every value is that of k_yee_b, k_yee_e, k_yee_b, to the last bit.  A block
// whose rows reach into a y absorber's layer multiplies what it stores by the
// column's two factors (a pass over the layers less: with the antenna's factors
// of time once per block, the field update of a 64x512x64 box with both 0.091 ->
// 0.077 ms).
// Measured: 256^3 0.240 ms (4.2 TB/s of the 60 bytes; in place 0.450), 192x768x192
// 0.401 ms (0.739), 128^3 0.057 ms (0.064).  With every stage's values of its own
// column in shared memory too (39 shared loads per cell instead of 20), 24
// planes per chunk and the image code in every block it took 0.400 ms, 0.698
// ms and 0.067 ms.  What bounds it now is the blocks at the box faces and the
// barrier of every iteration; tiles of 6, 12, 14 and 16 rows were no faster, and
// the absorber's factors in the march of every block cost 2 %.
constexpr int kFX = kFusedTX, kFY = kFusedTY;
constexpr int kHX = kFX + 2, kHY = kFY + 2, kHN = kHX * kHY;  // columns x0-1 .. x0+kFX, y0-1 .. y0+kFY
constexpr int kFWarps = kHY + (2 * kHY + 31) / 32;            // a warp per row, then the rim columns
constexpr int kFT = 32 * kFWarps;
constexpr int kFBlocksSM = 3;                                 // resident blocks per SM (shared memory)
// plane tiles: cells x0-G .. x0-G+35; E^n rows y0-1 .. y0+kFY+1, B^n rows y0-1 .. y0+kFY, J rows y0 .. y0+kFY
constexpr int kFEX = kFusedEX, kEC = kFusedERows * kFEX, kBC = kFusedBRows * kFEX, kJC = kFusedJRows * kFEX;
static_assert(kFusedERows == kFY + 3 && kFusedBRows == kFY + 2 && kFusedJRows == kFY + 1, "rows of the plane tiles");
constexpr int slot_floats(int comp) { return (3 * comp + 31) / 32 * 32; }  // 128-byte slots
constexpr int kFRE = 4, kFRB = 3;  // E^n slots; B^n, J slots and mbarriers
static_assert(kFX == 32 && kFEX >= kFX + 4 && kFEX % 4 == 0, "a warp per row; plane rows reach x0 + kFX + 2 from a 16-byte start");

struct FusedSmem {
    float en[kFRE][slot_floats(kEC)];  // E^n plane tiles [c][y][x]
    float bn[kFRB][slot_floats(kBC)];  // B^n plane tiles
    float jn[kFRB][slot_floats(kJC)];  // J plane tiles (as deposited; guard images folded by the reader)
    float bh[2][3][kHN];     // B^{n+1/2}, two planes [plane % 2][c][column]
    float e1[2][3][kHN];     // E^{n+1}, two planes
    unsigned long long mb[kFRB];
};

struct FusedArgs {
    const BoxDev* src;
    const BoxDev* dst;
    const CUtensorMap* maps;  // [nboxes][3]: E, B, J plane maps over src
    const int* blk_off;
    int nboxes;
    int tz;  // planes per chunk
    float dt, tau;  // tau = dt / 2
    float ih[3];
    unsigned* status;
};

int fused_blocks(int nx, int ny, int nz, int tz)
{
    return ((nx + kFX - 1) / kFX) * ((ny + kFY - 1) / kFY) * ((nz + tz - 1) / tz);
}

int fused_resident() { return kFBlocksSM; }

// The march of one block through its chunk of planes [zc0, zc1).  FACES: some
// column of the tile or its rim, or some plane, is next to a box face, where
// J gathers guard images and E, B are stored to them as well; without it (most
// blocks of a large box) none of that code is in the loop.  Returns false when
// a wait gave up.
template <int G, bool FACES, bool ABSORB>
__device__ __forceinline__ bool fused_march(const FusedArgs& a, FusedSmem& sm, int box, int x0, int y0, int zc0, int zc1)
{
    // the box's geometry and arrays in registers (stores through the field
    // pointers could otherwise alias the table and force reloads)
    const BoxDev& bt = a.src[box];
    const int nx = bt.nx, ny = bt.ny, nz = bt.nz, px = bt.px, py = bt.py;
    const int64_t plane = (int64_t)px * py;
    const int64_t pc = plane * bt.pz;
    const float* __restrict__ Jg = bt.J;
    float* __restrict__ Eo = a.dst[box].E;
    float* __restrict__ Bo = a.dst[box].B;
    constexpr int hx = GuardsOf<G>::hx, hyz = GuardsOf<G>::hyz;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const CUtensorMap* maps = a.maps + 3 * box;

    // this thread's column
    const int rim = (wid - kHY) * 32 + lane;  // >= 0: a column of the x rim
    const int ry = wid < kHY ? wid : rim % kHY;
    const int rx = wid < kHY ? lane + 1 : (rim < kHY ? 0 : kHX - 1);
    const bool doh = rim < 2 * kHY;
    const bool doe = doh && rx >= 1 && ry >= 1;
    const int x = x0 - 1 + rx, y = y0 - 1 + ry;
    const bool dob = doe && rx <= kFX && ry <= kFY && x < nx && y < ny;  // an output cell of this tile
    const int e = ry * kFEX + rx + G - 1, h = ry * kHX + rx;             // index in the plane tiles, in bh and e1
    // FACES: the cell (xc, yc) that the column is an image of (itself, but for
    // the rim beyond the upper faces), and the word offsets of its image along
    // x and y (0: none)
    const int xc = FACES && x >= nx ? x - nx : x, yc = FACES && y >= ny ? y - ny : y;
    auto image = [](int v, int n, int h) { return v < h ? n : (v >= n - G ? -n : 0); };
    const bool inside = x <= nx && y <= ny;
    const int dx = FACES && inside ? image(xc, nx, hx) : 0, dy = FACES && inside ? image(yc, ny, hyz) * px : 0;
    const bool edge = dx != 0 || dy != 0 || x >= nx || y >= ny;
    auto inner_plane = [&](int z) { return z >= hyz && z < nz - G; };
    const int64_t ccol = (int64_t)(yc + G) * px + (xc + G);
    // the absorber's factors of this column (1: none): integer and half y positions
    float fi = 1.0f, fh = 1.0f;
    if (ABSORB && dob) {
        fi = absorb_factor((float)y, ny, bt.oy.abs_cells, bt.oy.abs_sigma);
        fh = absorb_factor((float)y + 0.5f, ny, bt.oy.abs_cells, bt.oy.abs_sigma);
    }
    auto put = [&](float* p, float v0, float v1, float v2) {
        p[0] = v0;
        p[pc] = v1;
        p[2 * pc] = v2;
    };
    // the cell and its images; p: the cell's first component
    auto store3 = [&](float* p, int z, float v0, float v1, float v2) {
        put(p, v0, v1, v2);
        if (FACES && (edge || !inner_plane(z))) {
            const int dz = image(z, nz, hyz);
            for (int k = 0; k < (dz != 0 ? 2 : 1); ++k)
                for (int j = 0; j < (dy != 0 ? 2 : 1); ++j)
                    for (int i = 0; i < (dx != 0 ? 2 : 1); ++i)
                        if (i + j + k > 0)
                            put(p + k * dz * plane + j * dy + i * dx, v0, v1, v2);
        }
    };
    // FACES, J of the cell (xc, yc) in plane s: with no image it is the tile's
    // own value; with one, the two values' sum, of which the one that is not
    // this column's own is loaded an iteration ahead; with more (edges of the
    // box), all are summed from global memory in the order of k_yee_e.
    // extra_of: the number of images beside the own value, offset of the first
    auto extra_of = [&](int s, int64_t* off) {
        const int sc = s < nz ? s : s - nz;
        const int dz = image(sc, nz, hyz);
        const int n = (dx != 0 ? 2 : 1) * (dy != 0 ? 2 : 1) * (dz != 0 ? 2 : 1) - 1;
        // n == 1: the own value is the cell's or its image's, the other is wanted
        const bool own_is_image = x != xc || y != yc || s != sc;
        *off = (int64_t)(sc + G) * plane + ccol + (own_is_image ? 0 : dx + dy + dz * plane);
        return inside ? n : 0;
    };

    // bundle k (zc0 - 1 .. zc1), for iteration k: E^n(k+1), B^n(k) and, from
    // zc0 on, J(k); the first one brings E^n(zc0-1) too.  Plane p of E^n sits
    // in slot (p - zc0 + 1) % kFRE, B^n and J of bundle k in slot (k - zc0 + 1)
    // % kFRB, completing on that slot's mbarrier.
    const int k0 = zc0 - 1;
    int kiss = k0 - 1;  // tid 0: the last bundle issued
    auto issue = [&](int k) {
        kiss = k;
        const int r = (k - k0) % kFRB;
        const bool first = k == k0;
        unsigned long long* mb = &sm.mb[r];
        mbar_expect_tx(mb, 12u * (kEC + kBC + (first ? kEC : kJC)));
        tma_load_tile(sm.en[(k + 1 - k0) & (kFRE - 1)], maps + 0, x0, y0 - 1 + G, k + 1 + G, mb);
        tma_load_tile(sm.bn[r], maps + 1, x0, y0 - 1 + G, k + G, mb);
        if (first)
            tma_load_tile(sm.en[0], maps + 0, x0, y0 - 1 + G, k + G, mb);
        else
            tma_load_tile(sm.jn[r], maps + 2, x0, y0 + G, k + G, mb);
    };
    if (tid == 0) {
        for (int r = 0; r < kFRB; ++r)
            mbar_init(&sm.mb[r], 1);
        fence_mbar_init();
        for (int k = k0; k <= min(k0 + kFRB - 1, zc1); ++k)
            issue(k);
    }
    __syncthreads();  // the mbarriers are initialised

    const float ih0 = a.ih[0], ih1 = a.ih[1], ih2 = a.ih[2], dt = a.dt, tau = a.tau;
    float ex = 0.f, ey = 0.f, ez = 0.f;     // E^n(s)
    float qx = 0.f, qy = 0.f, qz = 0.f;     // B^{n+1/2}(s-1)
    float fx = 0.f, fy = 0.f, fz = 0.f;     // E^{n+1}(s-1)
    float ax = 0.f, ay = 0.f, az = 0.f;     // FACES: J(s) of this column's one image
    float* pe = Eo + (int64_t)(k0 + G) * plane + ccol;  // this column in plane s
    float* pb = Bo + (int64_t)(k0 - 1 + G) * plane + ccol;  // in plane s - 1
    bool timed_out = false;
    int r = 0, phase = 0;  // slot and parity of bundle s
    for (int s = k0; s <= zc1; ++s, pe += plane, pb += plane) {
        // the bundle of iteration s; its mbarrier was re-armed (after the
        // barrier of iteration s - 3) only after every thread had waited on
        // that mbarrier's previous bundle, s - 3
        if (!mbar_wait(&sm.mb[r], (unsigned)phase))
            timed_out = true;
        const float* E0 = sm.en[(s - k0) & (kFRE - 1)] + e;
        const float* E1 = sm.en[(s + 1 - k0) & (kFRE - 1)] + e;
        const float* Bp = sm.bn[r] + e;
        const float* Jp = sm.jn[r] + e - kFEX;
        float* H = sm.bh[s & 1][0] + h;
        if (s == k0) {
            ex = E0[0];
            ey = E0[kEC];
            ez = E0[2 * kEC];
        }
        // B^{n+1/2}(s) = B^n - tau curl E^n
        const float ex1 = E1[0], ey1 = E1[kEC], ez1 = E1[2 * kEC];
        const float bx = Bp[0] - tau * ((E0[2 * kEC + kFEX] - ez) * ih1 - (ey1 - ey) * ih2);
        const float by = Bp[kBC] - tau * ((ex1 - ex) * ih2 - (E0[2 * kEC + 1] - ez) * ih0);
        const float bz = Bp[2 * kBC] - tau * ((E0[kEC + 1] - ey) * ih0 - (E0[kFEX] - ex) * ih1);
        if (doh) {
            H[0] = bx;
            H[kHN] = by;
            H[2 * kHN] = bz;
        }
        float jx = 0.f, jy = 0.f, jz = 0.f;
        if (doe && s >= zc0) {
            jx = Jp[0];
            jy = Jp[kJC];
            jz = Jp[2 * kJC];
        }
        if (__syncthreads_or(timed_out ? 1 : 0)) {
            timed_out = true;
            break;
        }
        // every thread is past its reads of E^n(s), B^n(s) and J(s): their
        // slots take bundle s + 3
        if (tid == 0 && s + kFRB <= zc1) {
            fence_proxy_async();  // the slots being refilled were read by generic loads
            issue(s + kFRB);
        }
        // E^{n+1}(s) = E^n + dt (curl B^{n+1/2} - J)
        float nex = 0.f, ney = 0.f, nez = 0.f;
        if (s >= zc0) {
            if (doe) {
                if (FACES && (edge || !inner_plane(s))) {
                    int64_t off;
                    const int extra = extra_of(s, &off);
                    if (extra == 1) {
                        jx += ax;
                        jy += ay;
                        jz += az;
                    } else if (extra > 1) {
                        jx = jy = jz = 0.f;
                        const int sc = s < nz ? s : s - nz;
                        const int dz = image(sc, nz, hyz);
                        for (int kk = 0; kk < (dz != 0 ? 2 : 1); ++kk)
                            for (int j = 0; j < (dy != 0 ? 2 : 1); ++j)
                                for (int i = 0; i < (dx != 0 ? 2 : 1); ++i) {
                                    const float* p = Jg + (int64_t)(sc + G + kk * dz) * plane + ccol + j * dy + i * dx;
                                    jx += __ldg(p);
                                    jy += __ldg(p + pc);
                                    jz += __ldg(p + 2 * pc);
                                }
                    }
                }
                const float cx = (bz - H[2 * kHN - kHX]) * ih1 - (by - qy) * ih2;
                const float cy = (bx - qx) * ih2 - (bz - H[2 * kHN - 1]) * ih0;
                const float cz = (by - H[kHN - 1]) * ih0 - (bx - H[-kHX]) * ih1;
                nex = ex + dt * (cx - jx);
                ney = ey + dt * (cy - jy);
                nez = ez + dt * (cz - jz);
                float* X = sm.e1[s & 1][0] + h;
                X[0] = nex;
                X[kHN] = ney;
                X[2 * kHN] = nez;
            }
            if (dob) {
                if (s < zc1)
                    store3(pe, s, ABSORB ? nex * fi : nex, ABSORB ? ney * fh : ney, ABSORB ? nez * fi : nez);
                // B^{n+1}(s-1) = B^{n+1/2} - tau curl E^{n+1}
                if (s > zc0) {
                    const float* X0 = sm.e1[(s - 1) & 1][0] + h;
                    const float cx = (X0[2 * kHN + kHX] - fz) * ih1 - (ney - fy) * ih2;
                    const float cy = (nex - fx) * ih2 - (X0[2 * kHN + 1] - fz) * ih0;
                    const float cz = (X0[kHN + 1] - fy) * ih0 - (X0[kHX] - fx) * ih1;
                    {
                        const float vx = qx - tau * cx, vy = qy - tau * cy, vz = qz - tau * cz;
                        store3(pb, s - 1, ABSORB ? vx * fh : vx, ABSORB ? vy * fi : vy, ABSORB ? vz * fh : vz);
                    }
                }
            }
        }
        if (FACES && doe && s + 1 >= zc0 && s < zc1 && (edge || !inner_plane(s + 1))) {
            int64_t off;
            if (extra_of(s + 1, &off) == 1) {
                ax = __ldg(Jg + off);
                ay = __ldg(Jg + pc + off);
                az = __ldg(Jg + 2 * pc + off);
            }
        }
        ex = ex1, ey = ey1, ez = ez1;
        qx = bx, qy = by, qz = bz;
        fx = nex, fy = ney, fz = nez;
        if (++r == kFRB) {
            r = 0;
            phase ^= 1;
        }
    }
    if (timed_out && tid == 0) {
        // loads still in flight land before the block's shared memory goes
        // away: the last bundle issued on each mbarrier
        for (int k = max(k0, kiss - kFRB + 1); k <= kiss; ++k)
            mbar_wait(&sm.mb[(k - k0) % kFRB], (unsigned)(((k - k0) / kFRB) & 1));
    }
    return !timed_out;
}

template <int G>
__global__ void __launch_bounds__(kFT, kFBlocksSM) k_yee_fused(const FusedArgs a)
{
    extern __shared__ __align__(128) unsigned char fused_smem[];
    FusedSmem& sm = *reinterpret_cast<FusedSmem*>(fused_smem);
    const int box = find_box(a.blk_off, a.nboxes, blockIdx.x);
    const BoxDev& b = a.src[box];
    const int local = blockIdx.x - a.blk_off[box];
    const int ntx = (b.nx + kFX - 1) / kFX, nty = (b.ny + kFY - 1) / kFY;
    const int x0 = (local % ntx) * kFX, y0 = ((local / ntx) % nty) * kFY;
    const int zc0 = (local / (ntx * nty)) * a.tz, zc1 = min(zc0 + a.tz, b.nz);
    // columns x0 .. x0 + kFX, y0 .. y0 + kFY and planes zc0 .. zc1 take part in
    // the E update: none of them within the reach of a face's guards
    const bool faces = x0 < GuardsOf<G>::hx || x0 + kFX >= b.nx - G || y0 < GuardsOf<G>::hyz ||
                       y0 + kFY >= b.ny - G || zc0 < GuardsOf<G>::hyz || zc1 >= b.nz - G;
    // rows y0 .. y0 + kFY - 1 reach into an absorber layer
    const int A = b.oy.abs_cells;
    const bool absorb = A > 0 && (y0 < A || y0 + kFY > b.ny - A);
    const bool ok = absorb ? fused_march<G, true, true>(a, sm, box, x0, y0, zc0, zc1)
                           : (faces ? fused_march<G, true, false>(a, sm, box, x0, y0, zc0, zc1)
                                    : fused_march<G, false, false>(a, sm, box, x0, y0, zc0, zc1));
    if (!ok && threadIdx.x == 0)
        atomicOr(a.status, ST_TIMEOUT);
}

size_t fused_smem_bytes() { return sizeof(FusedSmem); }

cudaError_t configure_yee_fused()
{
    cudaError_t e = cudaFuncSetAttribute(k_yee_fused<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(FusedSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_yee_fused<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(FusedSmem));
    return e;
}

// The in-place update's absorber: a block per 32 x 8 cells (x, layer row) of
// the 2A rows j < A and j >= ny - A of a plane of each box with a layer.
int absorber_blocks(const BoxDev& b)
{
    return ((b.nx + 31) / 32) * ((2 * b.oy.abs_cells + 7) / 8) * b.nz;
}

__global__ void __launch_bounds__(256) k_absorb_y(const BoxDev* boxes, const int* off, int nboxes)
{
    const int box = find_box(off, nboxes, blockIdx.x);
    const BoxDev& b = boxes[box];
    const int A = b.oy.abs_cells, local = blockIdx.x - off[box];
    const int nbx = (b.nx + 31) / 32, nbp = (2 * A + 7) / 8;
    CellAt c;
    c.x = (local % nbx) * 32 + threadIdx.x;
    const int p = (local / nbx) % nbp * 8 + threadIdx.y;
    c.z = local / (nbx * nbp);
    c.y = p < A ? p : b.ny - 2 * A + p;
    c.ok = c.x < b.nx && p < 2 * A;
    if (!c.ok)
        return;
    const int64_t pc = padded_cells(b);
    const int64_t i = padded_index(b, c.x, c.y, c.z);
    float* __restrict__ E = b.E;
    float* __restrict__ B = b.B;
    const float ex = E[i], ey = E[pc + i], ez = E[2 * pc + i], bx = B[i], by = B[pc + i], bz = B[2 * pc + i];
    const float s = b.oy.abs_sigma;
    const float fi = absorb_factor((float)c.y, b.ny, A, s);          // Ex, Ez, By
    const float fh = absorb_factor((float)c.y + 0.5f, b.ny, A, s);   // Ey, Bx, Bz
    store_with_images(b, E, c, ex * fi);
    store_with_images(b, E + pc, c, ey * fh);
    store_with_images(b, E + 2 * pc, c, ez * fi);
    store_with_images(b, B, c, bx * fh);
    store_with_images(b, B + pc, c, by * fi);
    store_with_images(b, B + 2 * pc, c, bz * fh);
}

cudaError_t launch_yee_mixed_part(const YeePlan& p, int part, cudaStream_t st)
{
    YeeArgs a{p.boxes, p.blk_off, p.nboxes, 0.5f * p.dt, {p.ih[0], p.ih[1], p.ih[2]},
              p.step_no, p.dt_d, {p.dx_d[0], p.dx_d[1], p.dx_d[2]}};
    dim3 blk(32, 8);
    auto yb = p.guard == 2 ? k_yee_b<2> : k_yee_b<1>;
    auto ye = p.guard == 2 ? (p.sub_z ? k_yee_e<2, false> : k_yee_e<2, true>)
                           : (p.sub_z ? k_yee_e<1, false> : k_yee_e<1, true>);
    if (part == 0) {
        yb<<<p.nblocks, blk, 0, st>>>(a);
    } else if (part == 1) {
        if (p.antenna)
            k_antenna<<<kAntBlocks, kAntThreads, 0, st>>>(a);
        a.tau = p.dt;
        ye<<<p.nblocks, blk, 0, st>>>(a);
    } else {
        yb<<<p.nblocks, blk, 0, st>>>(a);
        if (p.abs_nblocks > 0)
            k_absorb_y<<<p.abs_nblocks, blk, 0, st>>>(p.boxes, p.abs_off, p.nboxes);
    }
    return cudaGetLastError();
}

cudaError_t launch_yee_mixed_plan(const YeePlan& p, cudaStream_t st)
{
    for (int part = 0; part < 3; ++part) {
        const cudaError_t e = launch_yee_mixed_part(p, part, st);
        if (e != cudaSuccess)
            return e;
    }
    return cudaSuccess;
}

cudaError_t launch_yee_fused(const YeePlan& p, const FusedPlan& f, cudaStream_t st)
{
    if (p.antenna) {
        YeeArgs ya{f.src, p.blk_off, p.nboxes, p.dt, {p.ih[0], p.ih[1], p.ih[2]},
                   p.step_no, p.dt_d, {p.dx_d[0], p.dx_d[1], p.dx_d[2]}};
        k_antenna<<<kAntBlocks, kAntThreads, 0, st>>>(ya);
    }
    FusedArgs a{f.src, f.dst, f.maps, f.blk_off, p.nboxes, f.tz, p.dt, 0.5f * p.dt, {p.ih[0], p.ih[1], p.ih[2]},
                f.status};
    if (p.guard == 2)
        k_yee_fused<2><<<f.nblocks, kFT, sizeof(FusedSmem), st>>>(a);
    else
        k_yee_fused<1><<<f.nblocks, kFT, sizeof(FusedSmem), st>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------------ subdomain halos

// Whole padded planes [p0, p0 + np) of the three components of F and a
// contiguous buffer [comp][plane][py][px]: mode 0 copies F to buf, 1 buf to
// F, 2 adds buf into F.  The planes of one component are contiguous in F
// too, so both sides are read and written in 16-byte pieces (px is a
// multiple of 4).
__global__ void k_halo_planes(const BoxDev b, float* F, int p0, int np, float* buf, int mode)
{
    const int64_t plane4 = (int64_t)b.px * b.py / 4;
    const int64_t per_comp = plane4 * np;
    const int64_t pc4 = padded_cells(b) / 4;
    float4* F4 = reinterpret_cast<float4*>(F);
    float4* B4 = reinterpret_cast<float4*>(buf);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 3 * per_comp;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int comp = (int)(t / per_comp);
        const int64_t r = t - comp * per_comp;
        const int64_t f = comp * pc4 + (int64_t)p0 * plane4 + r;
        if (mode == 0) {
            B4[t] = F4[f];
        } else if (mode == 1) {
            F4[f] = B4[t];
        } else {
            const float4 v = B4[t];
            float4 u = F4[f];
            u.x += v.x;
            u.y += v.y;
            u.z += v.z;
            u.w += v.w;
            F4[f] = u;
        }
    }
}

cudaError_t launch_halo_planes(const BoxDev& b, float* F, int p0, int np, float* buf, int mode,
                               cudaStream_t st)
{
    if (np <= 0)
        return cudaSuccess;
    const int64_t n4 = 3 * (int64_t)b.px * b.py / 4 * np;
    const int blocks = (int)std::min<int64_t>((n4 + 255) / 256, 2048);
    k_halo_planes<<<blocks, 256, 0, st>>>(b, F, p0, np, buf, mode);
    return cudaGetLastError();
}

// Moving window: F (3 components) takes the values of scratch (a copy of F)
// `cells` planes higher; the planes entering at the top are zero; images
// rewritten.
__global__ void k_shift_fields(const BoxDev b, float* F, const float* scratch, int cells)
{
    const int64_t n = (int64_t)b.nx * b.ny * b.nz;
    const int64_t pc = padded_cells(b);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 3 * n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int comp = (int)(t / n);
        const int64_t r = t - comp * n;
        CellAt c;
        c.x = (int)(r % b.nx);
        c.y = (int)((r / b.nx) % b.ny);
        c.z = (int)(r / ((int64_t)b.nx * b.ny));
        c.ok = true;
        const float v = c.y + cells < b.ny ? scratch[comp * pc + padded_index(b, c.x, c.y + cells, c.z)] : 0.0f;
        store_with_images(b, F + comp * pc, c, v);
    }
}

cudaError_t launch_shift_fields(const BoxDev& b, float* F, const float* scratch, int cells,
                                cudaStream_t st)
{
    k_shift_fields<<<1024, 256, 0, st>>>(b, F, scratch, cells);
    return cudaGetLastError();
}

// ------------------------------------------------------------ import/export

// src: FP64 [3][nz][ny][nx] on the device -> padded FP32 field with images.
__global__ void k_fields_to_padded(const BoxDev b, float* F, const double* src)
{
    const int64_t n = (int64_t)b.nx * b.ny * b.nz;
    const int64_t pc = padded_cells(b);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 3 * n;
         t += (int64_t)gridDim.x * blockDim.x) {
        int comp = (int)(t / n);
        int64_t r = t - comp * n;
        CellAt c;
        c.x = (int)(r % b.nx);
        c.y = (int)((r / b.nx) % b.ny);
        c.z = (int)(r / ((int64_t)b.nx * b.ny));
        store_with_images(b, F + comp * pc, c, (float)src[t]);
    }
}

// fold: sum the periodic images (the current, whose guards hold deposits
// that crossed the seam), in the order of the E update's fold.
__global__ void k_fields_from_padded(const BoxDev b, const float* F, double* dst, int fold)
{
    const int64_t n = (int64_t)b.nx * b.ny * b.nz;
    const int64_t pc = padded_cells(b);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 3 * n;
         t += (int64_t)gridDim.x * blockDim.x) {
        int comp = (int)(t / n);
        int64_t r = t - comp * n;
        int x = (int)(r % b.nx), y = (int)((r / b.nx) % b.ny), z = (int)(r / ((int64_t)b.nx * b.ny));
        const float* Fc = F + comp * pc;
        if (!fold) {
            dst[t] = (double)Fc[padded_index(b, x, y, z)];
            continue;
        }
        int ix[2], iy[2], iz[2];
        const int nx = images_x(b, x, ix), ny = images_y(b, y, iy);
        const int nz = b.sub_z ? (iz[0] = z, 1) : images_z(b, z, iz);
        float v = 0.0f;
        for (int k = 0; k < nz; ++k)
            for (int j = 0; j < ny; ++j)
                for (int q = 0; q < nx; ++q)
                    v += Fc[padded_index(b, ix[q], iy[j], iz[k])];
        dst[t] = (double)v;
    }
}

cudaError_t launch_fields_to_padded(const BoxDev& b, int which, const double* src, cudaStream_t st)
{
    float* F = which == 0 ? b.E : (which == 1 ? b.B : b.J);
    k_fields_to_padded<<<1024, 256, 0, st>>>(b, F, src);
    return cudaGetLastError();
}

cudaError_t launch_fields_from_padded(const BoxDev& b, int which, double* dst, cudaStream_t st)
{
    const float* F = which == 0 ? b.E : (which == 1 ? b.B : b.J);
    k_fields_from_padded<<<1024, 256, 0, st>>>(b, F, dst, which == 2);
    return cudaGetLastError();
}

// ------------------------------------------------------------ FP64 diagnostics

__device__ __forceinline__ double block_sum(double v)
{
    __shared__ double s[32];
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0)
        s[wid] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x + 31) / 32; ++i)
            r += s[i];
    __syncthreads();
    return r;
}

__global__ void k_diag_fields(const BoxDev b, double* out, double vol)
{
    const int64_t n = (int64_t)b.nx * b.ny * b.nz;
    const int64_t pc = padded_cells(b);
    double acc = 0.0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        int x = (int)(t % b.nx), y = (int)((t / b.nx) % b.ny), z = (int)(t / ((int64_t)b.nx * b.ny));
        int64_t i = padded_index(b, x, y, z);
        for (int c = 0; c < 3; ++c) {
            double e = b.E[c * pc + i], m = b.B[c * pc + i];
            acc += e * e + m * m;
        }
    }
    double s = block_sum(acc);
    if (threadIdx.x == 0)
        atomicAdd(out, 0.5 * s * vol);
}

// Nodes of the charge density along one axis, for a particle at offset o of
// its cell: the first node relative to the cell, and ORDER + 1 weights.
template <int ORDER>
__device__ __forceinline__ int node_weights64(double o, double* w)
{
    if (ORDER == 1) {
        w[0] = 1.0 - o;
        w[1] = o;
        return 0;
    }
    if (ORDER == 2) {
        const bool up = o >= 0.5;
        const double d = up ? o - 1.0 : o, lo = 0.5 - d, hi = 0.5 + d;
        w[0] = 0.5 * lo * lo;
        w[1] = 0.75 - d * d;
        w[2] = 0.5 * hi * hi;
        return up ? 0 : -1;
    }
    const double c = 1.0 - o, o2 = o * o, c2 = c * c;
    w[0] = c2 * c * (1.0 / 6.0);
    w[1] = (4.0 - 6.0 * o2 + 3.0 * o2 * o) * (1.0 / 6.0);
    w[2] = (4.0 - 6.0 * c2 + 3.0 * c2 * c) * (1.0 / 6.0);
    w[3] = o2 * o * (1.0 / 6.0);
    return -1;
}

// The charge density of one species' particles in supercell g of box b, added
// into rho (FP64 atomics), and, with ENERGY, its kinetic energy and charge.
template <int ORDER, bool ENERGY>
__device__ __forceinline__ void diag_list(const StepDev& d, const BoxDev& b, int s, int g, int scx, int scy, int scz,
                                          double* rho, double ivol, double* ekin, double* charge)
{
    constexpr int NW = ORDER + 1;
    const SpeciesDev& sp = d.sp[s];
    const int L = s * d.nsc + g;
    const int n = d.count[L];
    const int* ft = d.ftab + d.foff[L];
    const double mass = (double)sp.m, charge_q = (double)sp.q;
    const int Nd[3] = {b.nx, b.ny, b.nz};
    for (int p = threadIdx.x; p < n; p += blockDim.x) {
        const int64_t idx = (int64_t)ft[p >> d.log2S] * d.S + (p & (d.S - 1));
        const double w = d.w[idx];
        if (ENERGY) {
            const double ux = d.ux[idx], uy = d.uy[idx], uz = d.uz[idx];
            const double u2 = ux * ux + uy * uy + uz * uz;
            *ekin += w * mass * (u2 / (sqrt(1.0 + u2) + 1.0));
            *charge += charge_q * w;
        }
        const int cell = d.cell[idx];
        const int at[3] = {scx * d.LX + cell % d.LX, scy * d.LY + (cell / d.LX) % d.LY, scz * d.LZ + cell / (d.LX * d.LY)};
        const float off[3] = {d.ox[idx], d.oy[idx], d.oz[idx]};
        int node[3][NW];
        double wt[3][NW];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int first = at[a] + node_weights64<ORDER>((double)off[a], wt[a]);
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                const int v = first + k;  // in [-1, N + 2]
                node[a][k] = v < 0 ? v + Nd[a] : (v >= Nd[a] ? v - Nd[a] : v);
            }
        }
        const double qw = charge_q * w * ivol;
#pragma unroll
        for (int kz = 0; kz < NW; ++kz) {
            const double qz = qw * wt[2][kz];
#pragma unroll
            for (int ky = 0; ky < NW; ++ky) {
                const double qzy = qz * wt[1][ky];
                double* row = rho + ((int64_t)node[2][kz] * b.ny + node[1][ky]) * b.nx;
#pragma unroll
                for (int kx = 0; kx < NW; ++kx)
                    atomicAdd(row + node[0][kx], qzy * wt[0][kx]);
            }
        }
    }
}

// One CTA per supercell of the box: the charge density deposited (FP64
// atomics) into rho[nz][ny][nx] and, with ENERGY, kinetic energy and charge.
// Bound by the FP64 pipe (2 FMA per clock and SM): the weights come from each
// axis' own nodes (9 values for TSC) and the products are taken axis by axis
// (39 of them), against 12 weights and 128 products on a 4-node window before.
template <bool ENERGY>
__global__ void __launch_bounds__(128) k_diag_particles(const StepDev d, int box, double* rho, double* out, double ivol)
{
    const BoxDev& b = d.boxes[box];
    const int loc = blockIdx.x;
    const int g = b.sc_base + loc;
    const int scx = loc % b.nscx, scy = (loc / b.nscx) % b.nscy, scz = loc / (b.nscx * b.nscy);
    double ekin = 0.0, q = 0.0;
    for (int s = 0; s < d.nspecies; ++s) {
        if (d.sp[s].shape == 3)
            diag_list<3, ENERGY>(d, b, s, g, scx, scy, scz, rho, ivol, &ekin, &q);
        else if (d.sp[s].shape == 2)
            diag_list<2, ENERGY>(d, b, s, g, scx, scy, scz, rho, ivol, &ekin, &q);
        else
            diag_list<1, ENERGY>(d, b, s, g, scx, scy, scz, rho, ivol, &ekin, &q);
    }
    if (!ENERGY)
        return;
    double se = block_sum(ekin);
    double sq = block_sum(q);
    if (threadIdx.x == 0) {
        atomicAdd(out + 1, se);
        atomicAdd(out + 2, sq);
    }
}

__global__ void k_fill(double* p, int64_t n, double v)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        p[t] = v;
}

__global__ void k_diag_gauss(const BoxDev b, const double* rho, double rho_bg, double ih0, double ih1,
                             double ih2, unsigned long long* maxbits)
{
    const int64_t n = (int64_t)b.nx * b.ny * b.nz;
    const int64_t pc = padded_cells(b);
    double m = 0.0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        int x = (int)(t % b.nx), y = (int)((t / b.nx) % b.ny), z = (int)(t / ((int64_t)b.nx * b.ny));
        // a subdomain slab's charge density near its z faces misses the
        // neighbour's particles: its residual is taken 3 planes inside
        if (b.sub_z && (z < 3 || z >= b.nz - 3))
            continue;
        int64_t i = padded_index(b, x, y, z);
        double div = ((double)b.E[i] - (double)b.E[i - 1]) * ih0 +
                     ((double)b.E[pc + i] - (double)b.E[pc + i - b.px]) * ih1 +
                     ((double)b.E[2 * pc + i] - (double)b.E[2 * pc + i - (int64_t)b.px * b.py]) * ih2;
        m = fmax(m, fabs(div - rho[t] - rho_bg));
    }
    for (int o = 16; o > 0; o >>= 1)
        m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(maxbits, (unsigned long long)__double_as_longlong(m));
}

cudaError_t launch_diag_mixed(const StepDev& d, const BoxDev& hb, int box, double rho_bg,
                              double* rho_scratch, double* out, const double h[3], cudaStream_t st)
{
    const int64_t n = (int64_t)hb.nx * hb.ny * hb.nz;
    cudaError_t e = cudaMemsetAsync(rho_scratch, 0, sizeof(double) * n, st);
    if (e != cudaSuccess)
        return e;
    e = cudaMemsetAsync(out, 0, sizeof(double) * 4, st);
    if (e != cudaSuccess)
        return e;
    const double vol = h[0] * h[1] * h[2];
    k_diag_fields<<<512, 256, 0, st>>>(hb, out, vol);
    k_diag_particles<true><<<hb.nscx * hb.nscy * hb.nscz, 128, 0, st>>>(d, box, rho_scratch, out, 1.0 / vol);
    k_diag_gauss<<<512, 256, 0, st>>>(hb, rho_scratch, rho_bg, 1.0 / h[0], 1.0 / h[1], 1.0 / h[2],
                                      reinterpret_cast<unsigned long long*>(out + 3));
    return cudaGetLastError();
}

cudaError_t launch_rho_mixed(const StepDev& d, const BoxDev& hb, int box, double rho_bg, double* rho,
                             const double h[3], cudaStream_t st)
{
    k_fill<<<512, 256, 0, st>>>(rho, (int64_t)hb.nx * hb.ny * hb.nz, rho_bg);
    k_diag_particles<false><<<hb.nscx * hb.nscy * hb.nscz, 128, 0, st>>>(d, box, rho, nullptr, 1.0 / (h[0] * h[1] * h[2]));
    return cudaGetLastError();
}

}  // namespace pic
