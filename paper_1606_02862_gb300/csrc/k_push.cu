// k_push.cu -- the push kernel for any mix of shapes and gathers, and the
// dispatch of the push (the kernels for one shape alone: k_push_cic.cu,
// k_push_tsc.cu, k_push_pcs.cu).
#include "k_push.cuh"

namespace pic {

PIC_PUSH_DEFINE(0, PIC_PUSH_CASES)

// What a configuration needs and whether it is built: by the kernel for any
// mix, which needs the most shared memory and has every configuration.
size_t push_smem_bytes(int LX, int LY, int LZ, int threads, int guard)
{
#define X(a, b, c, t, g)                                                   \
    if (LX == a && LY == b && LZ == c && threads == t && guard == g)       \
        return dyn_smem<Tile<a, b, c, g>, t, 0>();
    PIC_PUSH_CASES(X)
#undef X
    return 0;
}

void push_tile_box(int LX, int LY, int LZ, int guard, int* px, int* ty, int* tz)
{
#define X(a, b, c, t, g)                                                              \
    if (LX == a && LY == b && LZ == c && guard == g) {                                \
        *px = Tile<a, b, c, g>::PX;                                                   \
        *ty = Tile<a, b, c, g>::TY;                                                   \
        *tz = Tile<a, b, c, g>::TZ;                                                   \
        return;                                                                       \
    }
    PIC_PUSH_CASES(X)
#undef X
    *px = *ty = *tz = 0;
}

int push_supported(int LX, int LY, int LZ, int threads, int guard)
{
#define X(a, b, c, t, g) if (LX == a && LY == b && LZ == c && threads == t && guard == g) return 1;
    PIC_PUSH_CASES(X)
#undef X
    return 0;
}

cudaError_t configure_push(int LX, int LY, int LZ, int threads, int guard, int only, int* per_sm)
{
    switch (only) {
    case 1:
        return configure_push_only<1>(LX, LY, LZ, threads, guard, per_sm);
    case 2:
        return configure_push_only<2>(LX, LY, LZ, threads, guard, per_sm);
    case 3:
        return configure_push_only<3>(LX, LY, LZ, threads, guard, per_sm);
    default:
        return configure_push_only<0>(LX, LY, LZ, threads, guard, per_sm);
    }
}

cudaError_t launch_push_deposit(const StepDev& d, int threads, int grid, cudaStream_t st)
{
    switch (d.push_only) {
    case 1:
        return launch_push_only<1>(d, threads, grid, st);
    case 2:
        return launch_push_only<2>(d, threads, grid, st);
    case 3:
        return launch_push_only<3>(d, threads, grid, st);
    default:
        return launch_push_only<0>(d, threads, grid, st);
    }
}

}  // namespace pic
