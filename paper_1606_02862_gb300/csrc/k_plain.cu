// k_plain.cu -- the plain FP64 form of the PIC step: absolute FP64 particle
// positions in unsorted SoA arrays, FP64 fields without guards (periodic
// indices wrap), one thread per particle, current deposited straight into
// global memory with FP64 atomics, one box per launch.  It computes the same
// cycle as the mixed form (Sec. 4: gather with the particle shape, Boris,
// Esirkepov, Yee) and serves as the straightforward GPU baseline the mixed,
// supercell-sorted form is measured against.
#include "pic_internal.cuh"
#include "plain.cuh"
#include "quotients.cuh"

#include <cmath>

namespace pic {

__device__ __forceinline__ int wrapi(int i, int n)
{
    i %= n;
    return i < 0 ? i + n : i;
}

__device__ __forceinline__ double S64(int shape, double d)
{
    double a = fabs(d);
    if (shape == 1)
        return a < 1.0 ? 1.0 - a : 0.0;
    if (a <= 0.5)
        return 0.75 - a * a;
    return a < 1.5 ? 0.5 * (1.5 - a) * (1.5 - a) : 0.0;
}

// A particle along one axis: its wrapped nodes and weights for fields sampled
// at the integer nodes (i) and at the half nodes (h), and its offset d0 from
// the node a0 its integer weights are built on (the nearest node for TSC, the
// cell for CIC).  red: one order lower at the half nodes (the
// energy-conserving gather), placed in the same window: CIC inside the TSC
// window, the nearest of the two (a tie goes up) inside the CIC window.
template <int SHAPE>
struct Axis64 {
    static constexpr int NW = SHAPE == 2 ? 3 : 2;
    int ni[NW], nh[NW];
    double wi[NW], wh[NW];
    int a0;
    double d0;

    __device__ __forceinline__ static void weights(double d, double* w)
    {
        if (SHAPE == 2) {
            const double lo = 0.5 - d, hi = 0.5 + d;
            w[0] = 0.5 * lo * lo;
            w[1] = 0.75 - d * d;
            w[2] = 0.5 * hi * hi;
        } else {
            w[0] = 1.0 - d;
            w[1] = d;
        }
    }

    // node v in [-n, 2n) into [0, n)
    __device__ __forceinline__ static int wrap(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

    __device__ __forceinline__ Axis64(double x, int n, bool red)
    {
        const double fl = floor(x);
        const int cell = (int)fl;
        const double o = x - fl;  // exact
        const bool up = o >= 0.5;
        const double dh = o - 0.5;
        int bh;
        if (SHAPE == 2) {
            a0 = cell + (up ? 1 : 0);
            d0 = up ? o - 1.0 : o;
            bh = cell - 1;
            if (red) {
                wh[0] = up ? 0.0 : -dh;
                wh[1] = up ? 1.5 - o : 0.5 + o;
                wh[2] = up ? dh : 0.0;
            } else {
                weights(dh, wh);
            }
        } else {
            a0 = cell;
            d0 = o;
            bh = up ? cell : cell - 1;
            const double f = up ? dh : o + 0.5;
            if (red) {
                wh[0] = f < 0.5 ? 1.0 : 0.0;
                wh[1] = f < 0.5 ? 0.0 : 1.0;
            } else {
                weights(f, wh);
            }
        }
        weights(d0, wi);
        const int bi = SHAPE == 2 ? a0 - 1 : a0;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            ni[k] = wrap(bi + k, n);
            nh[k] = wrap(bh + k, n);
        }
    }
};

// Two components that share their nodes and weights along y and z: the sums
// run along y and z first, so that a product of the two weights serves both
// components and a component's x weights come in once, at the end.
template <int NW>
__device__ __forceinline__ void gather64(const double* __restrict__ F, const int* nf, const double* wf,
                                         const double* __restrict__ H, const int* nhx, const double* wh, int nx, int ny,
                                         const int* nyv, const double* wy, const int* nzv, const double* wz, double* f,
                                         double* h)
{
    double af[NW], ah[NW];
#pragma unroll
    for (int a = 0; a < NW; ++a)
        af[a] = ah[a] = 0.0;
#pragma unroll
    for (int c = 0; c < NW; ++c)
#pragma unroll
        for (int b = 0; b < NW; ++b) {
            const int64_t row = ((int64_t)nzv[c] * ny + nyv[b]) * nx;
            const double w = wy[b] * wz[c];
#pragma unroll
            for (int a = 0; a < NW; ++a) {
                af[a] = fma(__ldg(F + row + nf[a]), w, af[a]);
                if (H)
                    ah[a] = fma(__ldg(H + row + nhx[a]), w, ah[a]);
            }
        }
    *f = 0.0;
#pragma unroll
    for (int a = 0; a < NW; ++a)
        *f = fma(af[a], wf[a], *f);
    if (H) {
        *h = 0.0;
#pragma unroll
        for (int a = 0; a < NW; ++a)
            *h = fma(ah[a], wh[a], *h);
    }
}

// One current component (along axis d) of a move: window nodes (wrapped and
// multiplied by their axis' stride) nd, ne, nf; S0 and DS on the window; the
// last node of an axis is part of the window only where its ext flag is set.
// The transverse factor S0e S0f + (DSe S0f + S0e DSf) / 2 + DSe DSf / 3 is
// taken as A S0f + B DSf with A = S0e + DSe / 2, B = S0e / 2 + DSe / 3.
template <int M>
__device__ __forceinline__ void deposit64(double* J, double cf, const int64_t* nd, const double* DSd, bool extd,
                                          const int64_t* ne, const double* S0e, const double* DSe, bool exte,
                                          const int64_t* nf, const double* S0f, const double* DSf, bool extf)
{
    double P[M - 1];
    P[0] = cf * DSd[0];
#pragma unroll
    for (int k = 1; k < M - 1; ++k)
        P[k] = fma(cf, DSd[k], P[k - 1]);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        if (i == M - 1 && !exte)
            break;
        const double A = fma(0.5, DSe[i], S0e[i]), B = fma(0.5, S0e[i], (1.0 / 3.0) * DSe[i]);
#pragma unroll
        for (int j = 0; j < M; ++j) {
            if (j == M - 1 && !extf)
                break;
            const double T = fma(A, S0f[j], B * DSf[j]);
            double* at = J + ne[i] + nf[j];
#pragma unroll
            for (int k = 0; k < M - 1; ++k)
                if (k < M - 2 || extd)
                    atomicAdd(at + nd[k], P[k] * T);
        }
    }
}

// One particle per thread.  Bound by the FP64 pipe (2 FMA per clock and SM), so
// the work is cut to fewer FP64 operations: each axis' weights once for all six
// components instead of once per component, the sums of the gather factored,
// the transverse factors in the two-term form (deposit64), and the current on 3
// (TSC) or 2 (CIC) nodes per axis, with a fourth (third) only for the axes where
// the move leaves the old support's window.  2.1 million TSC particles in 64^3
// cells: 8.61 -> 2.45 ms per step, 0.86 G particles/s.
template <int SHAPE>
__global__ void __launch_bounds__(128, 3) k_plain_push(const PlainPushArgs a)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= a.n)
        return;
    constexpr int NW = Axis64<SHAPE>::NW, M = NW + 1;
    const int Nd[3] = {a.nx, a.ny, a.nz};
    const int nx = a.nx, ny = a.ny;
    const int64_t nc = (int64_t)nx * ny * a.nz;
    const double p0[3] = {a.x[i], a.y[i], a.z[i]};
    const bool ec = a.ec != 0;
    const Axis64<SHAPE> X(p0[0], Nd[0], ec), Y(p0[1], Nd[1], ec), Z(p0[2], Nd[2], ec);
    double Ex, Ey, Ez, Bx, By, Bz;
    gather64<NW>(a.E, X.nh, X.wh, nullptr, nullptr, nullptr, nx, ny, Y.ni, Y.wi, Z.ni, Z.wi, &Ex, nullptr);
    gather64<NW>(a.E + nc, X.ni, X.wi, a.B + 2 * nc, X.nh, X.wh, nx, ny, Y.nh, Y.wh, Z.ni, Z.wi, &Ey, &Bz);
    gather64<NW>(a.E + 2 * nc, X.ni, X.wi, a.B + nc, X.nh, X.wh, nx, ny, Y.ni, Y.wi, Z.nh, Z.wh, &Ez, &By);
    gather64<NW>(a.B, X.ni, X.wi, nullptr, nullptr, nullptr, nx, ny, Y.nh, Y.wh, Z.nh, Z.wh, &Bx, nullptr);

    // relativistic Boris push
    const double eps = a.eps;
    double ux = a.ux[i], uy = a.uy[i], uz = a.uz[i];
    const double umx = ux + eps * Ex, umy = uy + eps * Ey, umz = uz + eps * Ez;
    const Over64 over_gm(sqrt(1.0 + umx * umx + umy * umy + umz * umz));
    const double tx = over_gm(eps * Bx), ty = over_gm(eps * By), tz = over_gm(eps * Bz);
    const double f = 2.0 / (1.0 + tx * tx + ty * ty + tz * tz);
    const double sx = f * tx, sy = f * ty, sz = f * tz;
    const double upx = umx + (umy * tz - umz * ty);
    const double upy = umy + (umz * tx - umx * tz);
    const double upz = umz + (umx * ty - umy * tx);
    ux = umx + (upy * sz - upz * sy) + eps * Ex;
    uy = umy + (upz * sx - upx * sz) + eps * Ey;
    uz = umz + (upx * sy - upy * sx) + eps * Ez;
    const Over64 over_g(sqrt(1.0 + ux * ux + uy * uy + uz * uz));
    double D[3] = {over_g(a.move[0] * ux), over_g(a.move[1] * uy), over_g(a.move[2] * uz)};
    if (!(fabs(D[0]) < 0.5 && fabs(D[1]) < 0.5 && fabs(D[2]) < 0.5)) {
        atomicOr(a.status, ST_PARTICLE);
        D[0] = D[1] = D[2] = 0.0;
        ux = uy = uz = 0.0;
    }

    // Esirkepov on the union of the old and the new support
    int64_t nd[3][M];
    double S0[3][M], DS[3][M];
    bool ext[3];
    const int64_t stride[3] = {1, nx, (int64_t)nx * ny};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const Axis64<SHAPE>& A = d == 0 ? X : (d == 1 ? Y : Z);
        // new position from the old node: the position as it is stored, so
        // that the current is that of the stored move (exact: |t| < 2)
        const double t = p0[d] + D[d] - (double)A.a0;
        // the node of the new position is a0 + sh, sh = -1, 0, 1
        const int sh = SHAPE == 2 ? (t >= 0.5) - (t < -0.5) : (t >= 1.0) - (t < 0.0);
        double v[NW];
        Axis64<SHAPE>::weights(t - (double)sh, v);
        ext[d] = sh != 0;
#pragma unroll
        for (int k = 0; k < M; ++k) {
            const double lo = k > 0 ? A.wi[k - 1] : 0.0, hi = k < NW ? A.wi[k] : 0.0;
            const double vlo = k > 0 ? v[k - 1] : 0.0, vhi = k < NW ? v[k] : 0.0;
            S0[d][k] = sh < 0 ? lo : hi;
            DS[d][k] = (sh > 0 ? vlo : vhi) - S0[d][k];
            nd[d][k] = Axis64<SHAPE>::wrap(A.a0 - (SHAPE == 2 ? 1 : 0) - (sh < 0 ? 1 : 0) + k, Nd[d]) * stride[d];
        }
    }
    const double w = a.w[i];
    deposit64<M>(a.J, a.jcoef[0] * w, nd[0], DS[0], ext[0], nd[1], S0[1], DS[1], ext[1], nd[2], S0[2], DS[2], ext[2]);
    deposit64<M>(a.J + nc, a.jcoef[1] * w, nd[1], DS[1], ext[1], nd[2], S0[2], DS[2], ext[2], nd[0], S0[0], DS[0],
                 ext[0]);
    deposit64<M>(a.J + 2 * nc, a.jcoef[2] * w, nd[2], DS[2], ext[2], nd[0], S0[0], DS[0], ext[0], nd[1], S0[1], DS[1],
                 ext[1]);
    double out[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        double v = p0[d] + D[d];
        const double N = (double)Nd[d];
        if (v >= N)
            v -= N;
        else if (v < 0.0)
            v += N;
        if (v >= N)
            v = 0.0;
        out[d] = v;
    }
    a.x[i] = out[0];
    a.y[i] = out[1];
    a.z[i] = out[2];
    a.ux[i] = ux;
    a.uy[i] = uy;
    a.uz[i] = uz;
}

cudaError_t launch_plain_push(const PlainPushArgs& a, int shape, cudaStream_t st)
{
    if (a.n == 0)
        return cudaSuccess;
    int blocks = (int)((a.n + 127) / 128);
    if (shape == 2)
        k_plain_push<2><<<blocks, 128, 0, st>>>(a);
    else
        k_plain_push<1><<<blocks, 128, 0, st>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------------ Yee, FP64

__global__ void k_plain_yee_b(PlainYeeArgs a, double tau)
{
    const int64_t nc = (int64_t)a.nx * a.ny * a.nz;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nc;
         t += (int64_t)gridDim.x * blockDim.x) {
        int x = (int)(t % a.nx), y = (int)((t / a.nx) % a.ny), z = (int)(t / ((int64_t)a.nx * a.ny));
        int64_t xp = t - x + wrapi(x + 1, a.nx);
        int64_t yp = t + ((int64_t)wrapi(y + 1, a.ny) - y) * a.nx;
        int64_t zp = t + ((int64_t)wrapi(z + 1, a.nz) - z) * a.nx * a.ny;
        const double *Ex = a.E, *Ey = a.E + nc, *Ez = a.E + 2 * nc;
        double cx = (Ez[yp] - Ez[t]) * a.ih[1] - (Ey[zp] - Ey[t]) * a.ih[2];
        double cy = (Ex[zp] - Ex[t]) * a.ih[2] - (Ez[xp] - Ez[t]) * a.ih[0];
        double cz = (Ey[xp] - Ey[t]) * a.ih[0] - (Ex[yp] - Ex[t]) * a.ih[1];
        a.B[t] -= tau * cx;
        a.B[nc + t] -= tau * cy;
        a.B[2 * nc + t] -= tau * cz;
    }
}

__global__ void k_plain_yee_e(PlainYeeArgs a, double dt)
{
    const int64_t nc = (int64_t)a.nx * a.ny * a.nz;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nc;
         t += (int64_t)gridDim.x * blockDim.x) {
        int x = (int)(t % a.nx), y = (int)((t / a.nx) % a.ny), z = (int)(t / ((int64_t)a.nx * a.ny));
        int64_t xm = t - x + wrapi(x - 1, a.nx);
        int64_t ym = t + ((int64_t)wrapi(y - 1, a.ny) - y) * a.nx;
        int64_t zm = t + ((int64_t)wrapi(z - 1, a.nz) - z) * a.nx * a.ny;
        const double *Bx = a.B, *By = a.B + nc, *Bz = a.B + 2 * nc;
        double cx = (Bz[t] - Bz[ym]) * a.ih[1] - (By[t] - By[zm]) * a.ih[2];
        double cy = (Bx[t] - Bx[zm]) * a.ih[2] - (Bz[t] - Bz[xm]) * a.ih[0];
        double cz = (By[t] - By[xm]) * a.ih[0] - (Bx[t] - Bx[ym]) * a.ih[1];
        a.E[t] += dt * (cx - a.J[t]);
        a.E[nc + t] += dt * (cy - a.J[nc + t]);
        a.E[2 * nc + t] += dt * (cz - a.J[2 * nc + t]);
    }
}

cudaError_t launch_plain_yee(const PlainYeeArgs& a, double dt, cudaStream_t st)
{
    k_plain_yee_b<<<2048, 256, 0, st>>>(a, 0.5 * dt);
    k_plain_yee_e<<<2048, 256, 0, st>>>(a, dt);
    k_plain_yee_b<<<2048, 256, 0, st>>>(a, 0.5 * dt);
    return cudaGetLastError();
}

// ------------------------------------------------------------ load / diagnostics

__global__ void k_plain_load(int64_t n, const double* x, const double* u, const double* w,
                             int nx, int ny, int nz, double* X, double* Y, double* Z, double* UX,
                             double* UY, double* UZ, double* W, int* pid, int id_base,
                             unsigned* status)
{
    const int Nd[3] = {nx, ny, nz};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        double p[3];
        bool bad = false;
        for (int d = 0; d < 3; ++d) {
            double v = x[3 * i + d];
            if (!isfinite(v) || !isfinite(u[3 * i + d]))
                bad = true;
            double N = (double)Nd[d];
            v = v - N * floor(v / N);
            if (!(v < N) || !(v >= 0.0))
                v = 0.0;
            p[d] = v;
        }
        double wv = w ? w[i] : 1.0;
        if (!isfinite(wv))
            bad = true;
        if (bad)
            atomicOr(status, ST_PARTICLE);
        X[i] = p[0];
        Y[i] = p[1];
        Z[i] = p[2];
        UX[i] = u[3 * i];
        UY[i] = u[3 * i + 1];
        UZ[i] = u[3 * i + 2];
        W[i] = wv;
        if (pid)
            pid[i] = id_base + (int)i;
    }
}

cudaError_t launch_plain_load(int64_t n, const double* x, const double* u, const double* w, int nx,
                              int ny, int nz, double* X, double* Y, double* Z, double* UX,
                              double* UY, double* UZ, double* W, int* pid, int id_base,
                              unsigned* status, cudaStream_t st)
{
    if (n == 0)
        return cudaSuccess;
    int blocks = (int)std::min<int64_t>((n + 255) / 256, 8192);
    k_plain_load<<<blocks, 256, 0, st>>>(n, x, u, w, nx, ny, nz, X, Y, Z, UX, UY, UZ, W, pid,
                                         id_base, status);
    return cudaGetLastError();
}

// interleave SoA FP64 particles into n x 3 host layout on the device
__global__ void k_plain_interleave(int64_t n, const double* X, const double* Y, const double* Z,
                                   double* out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        out[3 * i] = X[i];
        out[3 * i + 1] = Y[i];
        out[3 * i + 2] = Z[i];
    }
}

cudaError_t launch_plain_interleave(int64_t n, const double* X, const double* Y, const double* Z,
                                    double* out, cudaStream_t st)
{
    if (n == 0)
        return cudaSuccess;
    int blocks = (int)std::min<int64_t>((n + 255) / 256, 8192);
    k_plain_interleave<<<blocks, 256, 0, st>>>(n, X, Y, Z, out);
    return cudaGetLastError();
}

__device__ __forceinline__ double block_sum64(double v)
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

__global__ void k_plain_diag_fields(int64_t nc, const double* E, const double* B, double* out,
                                    double vol)
{
    double acc = 0.0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 3 * nc;
         t += (int64_t)gridDim.x * blockDim.x)
        acc += E[t] * E[t] + B[t] * B[t];
    double s = block_sum64(acc);
    if (threadIdx.x == 0)
        atomicAdd(out, 0.5 * s * vol);
}

__global__ void k_plain_diag_particles(PlainPushArgs a, int shape, double mass, double q,
                                       double ivol, double* rho, double* out)
{
    double ek = 0.0, qs = 0.0;
    const int Nd[3] = {a.nx, a.ny, a.nz};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.n;
         i += (int64_t)gridDim.x * blockDim.x) {
        double ux = a.ux[i], uy = a.uy[i], uz = a.uz[i], w = a.w[i];
        double u2 = ux * ux + uy * uy + uz * uz;
        ek += w * mass * (u2 / (sqrt(1.0 + u2) + 1.0));
        qs += q * w;
        const double pos[3] = {a.x[i], a.y[i], a.z[i]};
        int base[3];
        double wt[3][4];
        for (int d = 0; d < 3; ++d) {
            base[d] = (int)floor(pos[d]) - 1;
            for (int k = 0; k < 4; ++k)
                wt[d][k] = S64(shape, pos[d] - (double)(base[d] + k));
        }
        for (int kz = 0; kz < 4; ++kz)
            for (int ky = 0; ky < 4; ++ky)
                for (int kx = 0; kx < 4; ++kx) {
                    double v = wt[0][kx] * wt[1][ky] * wt[2][kz];
                    if (v == 0.0)
                        continue;
                    int X = wrapi(base[0] + kx, Nd[0]), Y = wrapi(base[1] + ky, Nd[1]),
                        Z = wrapi(base[2] + kz, Nd[2]);
                    atomicAdd(rho + ((int64_t)Z * a.ny + Y) * a.nx + X, q * w * ivol * v);
                }
    }
    double s1 = block_sum64(ek);
    double s2 = block_sum64(qs);
    if (threadIdx.x == 0) {
        atomicAdd(out + 1, s1);
        atomicAdd(out + 2, s2);
    }
}

__global__ void k_plain_diag_gauss(PlainYeeArgs a, const double* rho, double rho_bg,
                                   unsigned long long* maxbits)
{
    const int64_t nc = (int64_t)a.nx * a.ny * a.nz;
    double m = 0.0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nc;
         t += (int64_t)gridDim.x * blockDim.x) {
        int x = (int)(t % a.nx), y = (int)((t / a.nx) % a.ny), z = (int)(t / ((int64_t)a.nx * a.ny));
        int64_t xm = t - x + wrapi(x - 1, a.nx);
        int64_t ym = t + ((int64_t)wrapi(y - 1, a.ny) - y) * a.nx;
        int64_t zm = t + ((int64_t)wrapi(z - 1, a.nz) - z) * a.nx * a.ny;
        double div = (a.E[t] - a.E[xm]) * a.ih[0] + (a.E[nc + t] - a.E[nc + ym]) * a.ih[1] +
                     (a.E[2 * nc + t] - a.E[2 * nc + zm]) * a.ih[2];
        m = fmax(m, fabs(div - rho[t] - rho_bg));
    }
    for (int o = 16; o > 0; o >>= 1)
        m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(maxbits, (unsigned long long)__double_as_longlong(m));
}

cudaError_t launch_plain_diag_fields(const PlainYeeArgs& a, double* out, double vol, cudaStream_t st)
{
    int64_t nc = (int64_t)a.nx * a.ny * a.nz;
    k_plain_diag_fields<<<512, 256, 0, st>>>(nc, a.E, a.B, out, vol);
    return cudaGetLastError();
}

cudaError_t launch_plain_diag_particles(const PlainPushArgs& a, int shape, double mass, double q,
                                        double ivol, double* rho, double* out, cudaStream_t st)
{
    if (a.n == 0)
        return cudaSuccess;
    k_plain_diag_particles<<<512, 256, 0, st>>>(a, shape, mass, q, ivol, rho, out);
    return cudaGetLastError();
}

cudaError_t launch_plain_diag_gauss(const PlainYeeArgs& a, const double* rho, double rho_bg,
                                    double* out, cudaStream_t st)
{
    k_plain_diag_gauss<<<512, 256, 0, st>>>(a, rho, rho_bg,
                                            reinterpret_cast<unsigned long long*>(out + 3));
    return cudaGetLastError();
}

}  // namespace pic
