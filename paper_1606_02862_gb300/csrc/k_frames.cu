// k_frames.cu -- supercell frame maintenance for the mixed particle form
// (Sec. 2.1: particles live in frames of as many slots as a supercell has
// cells; each supercell owns a list of frames).
//
// After the push every list is dense again (the push fills its own holes)
// and holds count[L] particles; narrive[L] particles from neighbouring
// supercells wait in the move buffer, each with its rank among the arrivals
// of its destination list.  One step of maintenance:
//   scan_reduce / scan_top / scan_apply (few lists: scan_small alone): an exclusive prefix sum over the
//     lists of (frames needed, frames to allocate, frames to release) gives
//     every list its place in the next frame table; scan_apply also copies
//     the kept frame indices, pops new frames off the free stack and queues
//     released ones;
//   place: every waiting particle goes to slot abase[L] + rank of its list;
//     the same launch lists the supercells that hold mobile particles for
//     the next push, and the released frames go back on the free stack;
//   finish: the free stack's new height; every sort_every-th step, the TSC
//     and PCS lists are sorted by nearest node / cell for the pushes to come.
// Loading particles from the host uses the same path: a conversion kernel
// fills the move buffer, then the maintenance places them.
#include "pic_internal.cuh"

#include <cmath>
#include <cstddef>

namespace pic {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ int4 operator+(int4 a, int4 b)
{
    return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

__device__ __forceinline__ int4 list_need(const StepDev& d, int L)
{
    int n_new = d.count[L] + d.narrive[L];
    int nf_new = (n_new + d.S - 1) >> d.log2S;
    int nf_old = d.nframes[L];
    return make_int4(nf_new, max(0, nf_new - nf_old), max(0, nf_old - nf_new), 0);
}

template <int NT>
__device__ int4 block_exclusive_scan(int4 v, int4* total)
{
    __shared__ int4 s_warp[NT / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int4 x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int4 y;
        y.x = __shfl_up_sync(0xffffffffu, x.x, o);
        y.y = __shfl_up_sync(0xffffffffu, x.y, o);
        y.z = __shfl_up_sync(0xffffffffu, x.z, o);
        y.w = __shfl_up_sync(0xffffffffu, x.w, o);
        if (lane >= o)
            x = x + y;
    }
    if (lane == 31)
        s_warp[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int4 t = lane < NT / 32 ? s_warp[lane] : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int4 y;
            y.x = __shfl_up_sync(0xffffffffu, t.x, o);
            y.y = __shfl_up_sync(0xffffffffu, t.y, o);
            y.z = __shfl_up_sync(0xffffffffu, t.z, o);
            y.w = __shfl_up_sync(0xffffffffu, t.w, o);
            if (lane >= o)
                t = t + y;
        }
        if (lane < NT / 32)
            s_warp[lane] = t;  // inclusive over warps
    }
    __syncthreads();
    int4 warp_off = wid > 0 ? s_warp[wid - 1] : make_int4(0, 0, 0, 0);
    int4 incl = x + warp_off;
    int4 excl = make_int4(incl.x - v.x, incl.y - v.y, incl.z - v.z, incl.w - v.w);
    if (total)
        *total = s_warp[NT / 32 - 1];
    __syncthreads();
    return excl;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const StepDev d)
{
    const int base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    int4 acc = make_int4(0, 0, 0, 0);
    for (int i = 0; i < kScanItems; ++i) {
        int L = base + i;
        if (L < d.nlists)
            acc = acc + list_need(d, L);
    }
    int4 tot;
    block_exclusive_scan<kScanThreads>(acc, &tot);
    if (threadIdx.x == 0)
        d.blk_sums[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) k_scan_top(const StepDev d, int nblk)
{
    __shared__ int4 s_carry;
    if (threadIdx.x == 0)
        s_carry = make_int4(0, 0, 0, 0);
    __syncthreads();
    for (int b0 = 0; b0 < nblk; b0 += 1024) {
        int b = b0 + threadIdx.x;
        int4 v = b < nblk ? d.blk_sums[b] : make_int4(0, 0, 0, 0);
        int4 tot;
        int4 ex = block_exclusive_scan<1024>(v, &tot);
        int4 carry = s_carry;
        if (b < nblk)
            d.blk_offs[b] = ex + carry;
        __syncthreads();
        if (threadIdx.x == 0)
            s_carry = carry + tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        *d.totals = s_carry;
        if (d.step_ctr) {
            ++*d.step_ctr;
            ++*d.step_no;
        }
    }
}

// Whether the pool holds the frames that the plan `tot` needs; says so in the
// status word if not (the step's arrivals are abandoned).
__device__ __forceinline__ bool pool_holds(const StepDev& d, int4 tot)
{
    if (blockIdx.x == 0 && threadIdx.x == 0)
        *d.nitems = 0;  // k_place counts them anew
    if (tot.y <= *d.free_top)
        return true;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        atomicOr(d.status, ST_FRAME_POOL);
    return false;
}

// This thread's kScanItems lists from `base` on: what each needs, and the sum.
__device__ __forceinline__ int4 lists_need(const StepDev& d, int base, int4 (&need)[kScanItems])
{
    int4 acc = make_int4(0, 0, 0, 0);
    for (int i = 0; i < kScanItems; ++i) {
        const int L = base + i;
        need[i] = L < d.nlists ? list_need(d, L) : make_int4(0, 0, 0, 0);
        acc = acc + need[i];
    }
    return acc;
}

// Writes this thread's lists into the next frame table, `off` being the
// prefix sum over the lists before them.
__device__ __forceinline__ void apply_lists(const StepDev& d, int4 tot, int base, int4 off,
                                            const int4 (&need)[kScanItems])
{
    const int alloc_base = *d.free_top - tot.y;
    for (int i = 0; i < kScanItems; ++i) {
        int L = base + i;
        if (L >= d.nlists)
            break;
        const int nf_new = need[i].x;
        const int nf_old = d.nframes[L];
        const int* src = d.ftab + d.foff[L];
        int* dst = d.ftab_next + off.x;
        const int keep = min(nf_old, nf_new);
        for (int k = 0; k < keep; ++k)
            dst[k] = src[k];
        for (int k = nf_old; k < nf_new; ++k)
            dst[k] = d.free_stack[alloc_base + off.y + (k - nf_old)];
        for (int k = nf_new; k < nf_old; ++k)
            d.released[off.z + (k - nf_new)] = src[k];
        d.foff_next[L] = off.x;
        d.nframes[L] = nf_new;
        const int c = d.count[L], arrivals = d.narrive[L];
        d.abase[L] = c;
        d.count[L] = c + arrivals;
        d.narrive[L] = 0;
        if (arrivals > 0)
            d.joined[L] = 1;
        off = off + need[i];
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const StepDev d)
{
    const int4 tot = *d.totals;
    if (!pool_holds(d, tot))
        return;
    const int base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    int4 need[kScanItems];
    const int4 acc = lists_need(d, base, need);
    apply_lists(d, tot, base, block_exclusive_scan<kScanThreads>(acc, nullptr) + d.blk_offs[blockIdx.x], need);
}

// k_scan_reduce, k_scan_top and k_scan_apply in one block, for at most
// kScanTile lists: a small step is a row of launches of a few microseconds each
// (32^3 CIC, 512 lists: 22.9 us for the five kernels of the maintenance).
__global__ void __launch_bounds__(kScanThreads) k_scan_small(const StepDev d)
{
    const int base = threadIdx.x * kScanItems;
    int4 need[kScanItems], tot;
    const int4 acc = lists_need(d, base, need);
    const int4 off = block_exclusive_scan<kScanThreads>(acc, &tot);
    if (threadIdx.x == 0) {
        *d.totals = tot;
        ++*d.step_ctr;
        ++*d.step_no;
    }
    if (pool_holds(d, tot))
        apply_lists(d, tot, base, off, need);
}

// The work items of the next push: the supercells with a particle of a
// mobile species, 32 at a time (one ballot and one atomic per warp that has
// any; *d.nitems starts at zero).  In a mostly empty box the push otherwise
// spends its time asking for supercells that it then skips: a 256^3 box
// without particles took 0.395 ms per push (131,072 skipped items), of a
// step of 0.83 ms.
__device__ __forceinline__ void list_items(const StepDev& d)
{
    const int lane = threadIdx.x & 31;
    for (int b = (int)(blockIdx.x * blockDim.x + threadIdx.x) - lane; b < d.nsc; b += (int)(gridDim.x * blockDim.x)) {
        const int g = b + lane;
        bool any = false;
        if (g < d.nsc)
            for (int s = 0; s < d.nspecies; ++s)
                any = any || (d.sp[s].mobile && d.count[s * d.nsc + g] > 0);
        const unsigned m = __ballot_sync(0xffffffffu, any);
        if (m == 0)
            continue;
        int base = 0;
        if (lane == 0)
            base = atomicAdd(d.nitems, __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (any)
            d.items[base + __popc(m & ((1u << lane) - 1u))] = g;
    }
}

__global__ void __launch_bounds__(256) k_list_items(const StepDev d) { list_items(d); }

cudaError_t launch_list_items(const StepDev& d, int blocks, cudaStream_t st)
{
    const cudaError_t e = cudaMemsetAsync(d.nitems, 0, sizeof(int), st);
    if (e != cudaSuccess)
        return e;
    k_list_items<<<blocks, 256, 0, st>>>(d);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_place(const StepDev d)
{
    const int4 tot = *d.totals;
    if (tot.y > *d.free_top)
        return;
    list_items(d);
    // the released frames take the places of those that k_scan_apply popped
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < tot.z; i += gridDim.x * blockDim.x)
        d.free_stack[*d.free_top - tot.y + i] = d.released[i];
    const int n = min(*d.mv_count, d.mv_cap);
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < n; m += gridDim.x * blockDim.x) {
        const int L = d.mv_dest[m];
        const int slot = d.abase[L] + d.mv_rank[m];
        const int frame = d.ftab_next[d.foff_next[L] + (slot >> d.log2S)];
        const int64_t idx = (int64_t)frame * d.S + (slot & (d.S - 1));
        d.cell[idx] = d.mv_cell[m];
        d.ox[idx] = d.mv_ox[m];
        d.oy[idx] = d.mv_oy[m];
        d.oz[idx] = d.mv_oz[m];
        d.ux[idx] = d.mv_ux[m];
        d.uy[idx] = d.mv_uy[m];
        d.uz[idx] = d.mv_uz[m];
        d.w[idx] = d.mv_w[m];
        if (d.pid)
            d.pid[idx] = d.mv_pid[m];
    }
}

// ------------------------------------------------------------ list sort
//
// Sorts the frame lists of the mobile TSC and PCS species by nearest node (TSC)
// or cell (PCS) in place, whole lists where they fit a run of kSortRun particles:
// the run comes into shared memory by 16-byte asynchronous copies, a counting
// sort gives every sorted position its source, and the attributes go back as
// contiguous words.  Bound by HBM: 32 B per particle read and 32 B written.
// Against sorting each chunk of 256 by itself inside the push, a warp of the
// push reads fewer different field words (a bank model of the 8x4x4 TSC tile
// at 8 particles per cell: 1.34 against 1.90 wavefronts per load), and the push
// needs neither the sort's shared memory nor its four barriers per chunk.  256^3
// cells, 8 TSC particles each: push 9.73 -> 8.72 ms per step, maintenance 0.19
// -> 0.57 ms (a sort every fourth step takes 1.5 ms, 5.6 TB/s); 128^3 at 16 each
// 2.28 + 0.11 -> 1.99 + 0.20 ms; PCS 96^3 1.26 + 0.07 -> 1.19 + 0.09 ms.
// (CIC lists: see the sort in push_list, k_push.cuh.)
constexpr int kSortThreads = 256;
constexpr int kSortRun = 1536;
constexpr int kSortKeys = 1024;  // >= 729, the nodes of the largest supercell

struct SortSmem {
    int off[kSortKeys];             // histogram, then first sorted position of each key
    unsigned short src[kSortRun];   // sorted position -> run position
    int warp_sum[kSortThreads / 32];
    unsigned st[8][kSortRun];       // cell, offsets, momenta, weight in run order
    unsigned pid[kSortRun];         // ids; allocated only when they are tracked
};

static size_t sort_smem_bytes(bool ids) { return ids ? sizeof(SortSmem) : offsetof(SortSmem, pid); }

__device__ __forceinline__ void sort_copy16(void* smem, const void* gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

// base: a multiple of 4 (16-byte pieces of whole frames, which are allocated
// even past the list's count)
__device__ __forceinline__ void sort_run(const StepDev& d, SortSmem& sm, const int* ft, int base, int cn, int shape)
{
    const int tid = threadIdx.x;
    const int LX = d.LX, LY = d.LY, LZ = d.LZ;  // powers of two
    const int bx = __ffs(LX) - 1, by = __ffs(LY) - 1;
    auto gidx = [&](int slot) -> int64_t { return (int64_t)ft[slot >> d.log2S] * d.S + (slot & (d.S - 1)); };
    unsigned* const attr[8] = {reinterpret_cast<unsigned*>(d.cell), reinterpret_cast<unsigned*>(d.ox),
                               reinterpret_cast<unsigned*>(d.oy),   reinterpret_cast<unsigned*>(d.oz),
                               reinterpret_cast<unsigned*>(d.ux),   reinterpret_cast<unsigned*>(d.uy),
                               reinterpret_cast<unsigned*>(d.uz),   reinterpret_cast<unsigned*>(d.w)};
    for (int k = tid; k < (cn + 3) >> 2; k += kSortThreads) {
        const int64_t idx = gidx(base + 4 * k);
#pragma unroll
        for (int a = 0; a < 8; ++a)
            sort_copy16(sm.st[a] + 4 * k, attr[a] + idx);
        if (d.pid)
            sort_copy16(sm.pid + 4 * k, d.pid + idx);
    }
    const int K = shape == 2 ? (LX + 1) * (LY + 1) * (LZ + 1) : d.S;
    for (int k = tid; k < K; k += kSortThreads)
        sm.off[k] = 0;
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    constexpr int Q = kSortRun / kSortThreads;
    int kr[Q];  // of this thread's particles: key << 16 | rank within the key
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int j = q * kSortThreads + tid;
        if (j >= cn)
            break;
        const int cell = (int)sm.st[0][j];
        int key = cell;
        if (shape == 2) {
            const int lx = (cell & (LX - 1)) + (__uint_as_float(sm.st[1][j]) >= 0.5f);
            const int ly = ((cell >> bx) & (LY - 1)) + (__uint_as_float(sm.st[2][j]) >= 0.5f);
            const int lz = (cell >> (bx + by)) + (__uint_as_float(sm.st[3][j]) >= 0.5f);
            key = lx + (LX + 1) * (ly + (LY + 1) * lz);
        }
        kr[q] = (key << 16) | atomicAdd(&sm.off[key], 1);
    }
    __syncthreads();
    // exclusive prefix of the histogram: every thread takes kSortKeys /
    // kSortThreads keys in a row
    {
        constexpr int P = kSortKeys / kSortThreads;
        const int lane = tid & 31, wid = tid >> 5;
        int v[P], local = 0;
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const int k = P * tid + i;
            v[i] = k < K ? sm.off[k] : 0;
            local += v[i];
        }
        int incl = local;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o)
                incl += y;
        }
        if (lane == 31)
            sm.warp_sum[wid] = incl;
        __syncthreads();
        int run = incl - local;
        for (int w = 0; w < wid; ++w)
            run += sm.warp_sum[w];
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const int k = P * tid + i;
            if (k < K)
                sm.off[k] = run;
            run += v[i];
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int j = q * kSortThreads + tid;
        if (j < cn)
            sm.src[sm.off[kr[q] >> 16] + (kr[q] & 0xffff)] = (unsigned short)j;
    }
    __syncthreads();
    for (int j = tid; j < cn; j += kSortThreads) {
        const int64_t idx = gidx(base + j);
        const int from = sm.src[j];
#pragma unroll
        for (int a = 0; a < 8; ++a)
            attr[a][idx] = sm.st[a][from];
        if (d.pid)
            d.pid[idx] = (int)sm.pid[from];
    }
    __syncthreads();  // the next run fills the stage and clears the histogram
}

// The lists that particles joined since they were last sorted (all: every
// list).  A list's counts are loaded while the block sorts the list before it.
__device__ __forceinline__ void sort_lists(const StepDev& d, SortSmem& sm, const int* foff, const int* ftab, int first,
                                           int stride, bool all)
{
    const int nitems = *d.nitems;
    const int total = nitems * d.nspecies;
    struct List {
        int L, shape, n, off;  // n: 0 for a list that stays as it is
    };
    auto fetch = [&](int t) {
        List l{0, 0, 0, 0};
        if (t < total) {
            const int s = t / nitems;
            l.L = s * d.nsc + d.items[t - s * nitems];
            l.shape = d.sp[s].shape;
            if (d.sp[s].mobile && l.shape != 1) {
                const int n = d.count[l.L];
                l.off = foff[l.L];
                l.n = n > 1 && (all || d.joined[l.L]) ? n : 0;
            }
        }
        return l;
    };
    List next = fetch(first);
    for (int t = first; t < total; t += stride) {
        const List l = next;
        next = fetch(t + stride);
        if (l.n == 0)
            continue;
        const int runs = (l.n + kSortRun - 1) / kSortRun;
        const int per = ((l.n + runs - 1) / runs + 31) & ~31;
        for (int base = 0; base < l.n; base += per)
            sort_run(d, sm, ftab + l.off, base, min(per, l.n - base), l.shape);
        if (threadIdx.x == 0)
            d.joined[l.L] = 0;  // every thread read it before the barriers of sort_run
    }
}

// The lists in the current frame table, before the first push after a load.
__global__ void __launch_bounds__(kSortThreads) k_sort(const StepDev d)
{
    extern __shared__ __align__(16) unsigned char sort_smem[];
    sort_lists(d, *reinterpret_cast<SortSmem*>(sort_smem), d.foff, d.ftab, (int)blockIdx.x, (int)gridDim.x, true);
}

// Last kernel of the maintenance: block 0 settles the free stack and the move
// buffer; on every sort_every-th step the others sort the lists (the frame
// table written in this step is the current one from here on).  A list that no
// particle joined since its last sort is left as it is: what moves within its
// supercell reaches a face about as often as it changes node, so while nothing
// joins, the order is nearly that of the sort, and the slower the particles are
// the more rarely their lists are sorted (cold ions: a thermal list of 1024
// electrons gains about ten a step).  Against sorting every list, maintenance
// per step: half ions, 64x512x64 cells 0.087 -> 0.061 ms, 192x768x192 0.142 ->
// 0.128; 256^3 cells of electrons alone 0.559 -> 0.569 (the marks).
__global__ void __launch_bounds__(kSortThreads) k_finish(const StepDev d)
{
    extern __shared__ __align__(16) unsigned char sort_smem[];
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) {
            const int4 tot = *d.totals;
            const int top = *d.free_top;
            if (tot.y <= top) {
                *d.free_top = top - tot.y + tot.z;
                *d.mv_count = 0;
            }
            *d.work_counter = 0;  // of the next push
        }
        return;
    }
    if (*d.step_ctr % d.sort_every == 0)
        sort_lists(d, *reinterpret_cast<SortSmem*>(sort_smem), d.foff_next, d.ftab_next, (int)blockIdx.x - 1,
                   (int)gridDim.x - 1, false);
}

cudaError_t configure_sort()
{
    cudaError_t e = cudaFuncSetAttribute(k_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem));
    return e;
}

cudaError_t launch_sort(const StepDev& d, int blocks, cudaStream_t st)
{
    k_sort<<<blocks, kSortThreads, sort_smem_bytes(d.pid != nullptr), st>>>(d);
    return cudaGetLastError();
}

// Moving window, part 1: empty the lists of the bottom `rows` supercell
// rows of a box (every species); the next maintenance pass releases their
// frames.
__global__ void k_clear_rows(const StepDev d, const BoxDev b, int rows)
{
    const int per_species = b.nscx * rows * b.nscz;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < d.nspecies * per_species;
         t += gridDim.x * blockDim.x) {
        const int s = t / per_species, r = t % per_species;
        const int scx = r % b.nscx, scy = (r / b.nscx) % rows, scz = r / (b.nscx * rows);
        d.count[s * d.nsc + b.sc_base + (scz * b.nscy + scy) * b.nscx + scx] = 0;
    }
}

// Moving window, part 2: the list of row scy takes over the list (count,
// frames, frame-table offset, mark of its arrivals) of row scy + rows,
// cyclically; the rows that were emptied in part 1 come round to the top.
// old4 = copies of count, nframes, foff and joined (nlists each), taken before
// the kernel.
__global__ void k_rotate_lists(const StepDev d, const BoxDev b, const int* old4, int* foff, int rows)
{
    const int nbox = b.nscx * b.nscy * b.nscz;
    const int* count_old = old4;
    const int* nframes_old = old4 + d.nlists;
    const int* foff_old = old4 + 2 * d.nlists;
    const int* joined_old = old4 + 3 * d.nlists;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < d.nspecies * nbox;
         t += gridDim.x * blockDim.x) {
        const int s = t / nbox, loc = t % nbox;
        const int scx = loc % b.nscx, scy = (loc / b.nscx) % b.nscy, scz = loc / (b.nscx * b.nscy);
        const int sy = (scy + rows) % b.nscy;
        const int L = s * d.nsc + b.sc_base + loc;
        const int Ls = s * d.nsc + b.sc_base + (scz * b.nscy + sy) * b.nscx + scx;
        d.count[L] = count_old[Ls];
        d.nframes[L] = nframes_old[Ls];
        foff[L] = foff_old[Ls];
        d.joined[L] = joined_old[Ls];
    }
}

cudaError_t launch_clear_rows(const StepDev& d, const BoxDev& hb, int rows, cudaStream_t st)
{
    k_clear_rows<<<256, 256, 0, st>>>(d, hb, rows);
    return cudaGetLastError();
}

cudaError_t launch_rotate_lists(const StepDev& d, const BoxDev& hb, const int* old4, int* foff,
                                int rows, cudaStream_t st)
{
    k_rotate_lists<<<256, 256, 0, st>>>(d, hb, old4, foff, rows);
    return cudaGetLastError();
}

int frame_launches(int nlists) { return nlists > kScanTile ? 5 : 3; }

int frame_scan_blocks(int nlists) { return (nlists + kScanTile - 1) / kScanTile; }

cudaError_t launch_frame_plan(const StepDev& d, cudaStream_t st)
{
    const int nblk = frame_scan_blocks(d.nlists);
    k_scan_reduce<<<nblk, kScanThreads, 0, st>>>(d);
    k_scan_top<<<1, 1024, 0, st>>>(d, nblk);
    return cudaGetLastError();
}

static cudaError_t launch_placing(const StepDev& d, int place_blocks, int sort_blocks, cudaStream_t st)
{
    k_place<<<place_blocks, 256, 0, st>>>(d);
    k_finish<<<1 + sort_blocks, kSortThreads, sort_blocks > 0 ? sort_smem_bytes(d.pid != nullptr) : 0, st>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_frame_apply(const StepDev& d, int place_blocks, int sort_blocks, cudaStream_t st)
{
    const int nblk = frame_scan_blocks(d.nlists);
    k_scan_apply<<<nblk, kScanThreads, 0, st>>>(d);
    return launch_placing(d, place_blocks, sort_blocks, st);
}

cudaError_t launch_frames(const StepDev& d, int place_blocks, int sort_blocks, cudaStream_t st)
{
    if (d.nlists > kScanTile) {
        const cudaError_t e = launch_frame_plan(d, st);
        return e != cudaSuccess ? e : launch_frame_apply(d, place_blocks, sort_blocks, st);
    }
    k_scan_small<<<1, kScanThreads, 0, st>>>(d);
    return launch_placing(d, place_blocks, sort_blocks, st);
}

// ------------------------------------------------------------ subdomain migrants

// The migrant message of the neighbouring slab on face `side` of box `box`
// (a one-box subdomain context): every record joins this step's arrivals
// (the move buffer) in supercell (sx, sy, row on that face), where the frame
// plan and k_place then put it like any particle that changed supercell.
__global__ void k_mig_accept(const StepDev d, int box, int side, const char* msg)
{
    const BoxDev b = d.boxes[box];
    const MigHeader h = *reinterpret_cast<const MigHeader*>(msg);
    const int n = min(h.count, h.cap);
    const MigRec* rec = reinterpret_cast<const MigRec*>(msg + sizeof(MigHeader));
    const int sz = side == 0 ? 0 : b.nscz - 1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const MigRec r = rec[i];
        if (r.s < 0 || r.s >= d.nspecies || r.sx < 0 || r.sx >= b.nscx || r.sy < 0 || r.sy >= b.nscy ||
            r.cell < 0 || r.cell >= d.S) {
            atomicOr(d.status, ST_PARTICLE);  // a malformed record is dropped
            continue;
        }
        const int L = r.s * d.nsc + b.sc_base + (sz * b.nscy + r.sy) * b.nscx + r.sx;
        const int m = atomicAdd(d.mv_count, 1);
        if (m >= d.mv_cap) {
            atomicOr(d.status, ST_CAPACITY);
            continue;
        }
        d.mv_rank[m] = atomicAdd(d.narrive + L, 1);
        d.mv_dest[m] = L;
        d.mv_cell[m] = r.cell;
        d.mv_ox[m] = r.ox;
        d.mv_oy[m] = r.oy;
        d.mv_oz[m] = r.oz;
        d.mv_ux[m] = r.ux;
        d.mv_uy[m] = r.uy;
        d.mv_uz[m] = r.uz;
        d.mv_w[m] = r.w;
        if (d.pid)
            d.mv_pid[m] = r.pid;
    }
}

cudaError_t launch_mig_accept(const StepDev& d, int box, int side, const char* msg, cudaStream_t st)
{
    k_mig_accept<<<256, 256, 0, st>>>(d, box, side, msg);
    return cudaGetLastError();
}

// ------------------------------------------------------------ load / read

// Host particles (FP64, n x 3 global cell coordinates) -> move buffer.  A
// block takes 256 particles at a time: their x, u and w runs come into
// shared memory word by word across the threads (each warp load is 256
// contiguous bytes: the source may be page-locked host memory read over the
// host link), then each thread converts one particle.
constexpr int kInsertBlock = 256;

__global__ void __launch_bounds__(kInsertBlock) k_insert_convert(const StepDev d, int box, int species, int n,
                                                                 const double* x, const double* u,
                                                                 const double* w, int id_base,
                                                                 const int64_t* ids)
{
    __shared__ double sx[3 * kInsertBlock], su[3 * kInsertBlock], sw[kInsertBlock];
    const BoxDev b = d.boxes[box];
    const int Nd[3] = {b.nx, b.ny, b.nz};
    const int Ld[3] = {d.LX, d.LY, d.LZ};
    for (int64_t base = (int64_t)blockIdx.x * kInsertBlock; base < n; base += (int64_t)gridDim.x * kInsertBlock) {
        const int m = (int)(n - base < kInsertBlock ? n - base : kInsertBlock);
        __syncthreads();  // the previous group's reads of the stage are done
        for (int j = threadIdx.x; j < 3 * m; j += kInsertBlock) {
            sx[j] = x[3 * base + j];
            su[j] = u[3 * base + j];
        }
        if (threadIdx.x < m)
            sw[threadIdx.x] = w ? w[base + threadIdx.x] : 1.0;
        __syncthreads();
        if (threadIdx.x >= m)
            continue;
        const int t = threadIdx.x;
        const int i = (int)(base + t);
        int scd[3], lc[3];
        float o[3];
        bool bad = false;
        for (int a = 0; a < 3; ++a) {
            double v = sx[3 * t + a];
            if (!isfinite(v) || !isfinite(su[3 * t + a]))
                bad = true;
            double N = (double)Nd[a];
            v = v - N * floor(v / N);
            if (!(v < N))
                v = 0.0;
            if (!(v >= 0.0))
                v = 0.0;
            int ci = (int)floor(v);
            ci = min(max(ci, 0), Nd[a] - 1);
            float of = (float)(v - (double)ci);
            of = fminf(fmaxf(of, 0.0f), 0.99999994f);
            o[a] = of;
            scd[a] = ci / Ld[a];
            lc[a] = ci - scd[a] * Ld[a];
        }
        const double wv = sw[t];
        if (!isfinite(wv))
            bad = true;
        if (bad)
            atomicOr(d.status, ST_PARTICLE);
        else
            atomicMax(d.wmax_bits + species, __float_as_uint(fabsf((float)wv)));
        const int sc = b.sc_base + (scd[2] * b.nscy + scd[1]) * b.nscx + scd[0];
        const int L = species * d.nsc + sc;
        d.mv_dest[i] = L;
        d.mv_rank[i] = bad ? 0 : atomicAdd(d.narrive + L, 1);
        d.mv_cell[i] = lc[0] + d.LX * (lc[1] + d.LY * lc[2]);
        d.mv_ox[i] = o[0];
        d.mv_oy[i] = o[1];
        d.mv_oz[i] = o[2];
        d.mv_ux[i] = (float)su[3 * t + 0];
        d.mv_uy[i] = (float)su[3 * t + 1];
        d.mv_uz[i] = (float)su[3 * t + 2];
        d.mv_w[i] = (float)wv;
        if (d.mv_pid)
            d.mv_pid[i] = ids ? (int)ids[i] : id_base + i;
    }
}

cudaError_t launch_insert_convert(const StepDev& d, int box, int species, int64_t n,
                                  const double* x, const double* u, const double* w, int id_base,
                                  const int64_t* ids, cudaStream_t st)
{
    int blocks = (int)std::min<int64_t>((n + kInsertBlock - 1) / kInsertBlock, 4096);
    if (blocks > 0)
        k_insert_convert<<<blocks, kInsertBlock, 0, st>>>(d, box, species, (int)n, x, u, w, id_base, ids);
    return cudaGetLastError();
}

// One CTA per supercell of the box: copy its particles to FP64 global form
// at list_off[sc] (exclusive prefix of the counts, host-computed).  Thread j
// writes word j of the supercell's run of x (and of u): the destination may be
// page-locked host memory written over the host link, which bounds the kernel.
// Runs start at any word, so the threads are numbered from the 128-byte line
// that the run's first word lies in: a warp store then covers two whole lines.
// 16.8 million particles (x, u, id) to the host 5.84 -> 4.95 ms, 161 -> 190 GB/s
// of the link's 193; four words a thread in flight at once took 6.1 ms.
__global__ void k_read_particles(const StepDev d, int box, int species, const int* list_off,
                                 double* x, double* u, double* w, int64_t* id)
{
    const BoxDev b = d.boxes[box];
    const int loc = blockIdx.x;
    const int g = b.sc_base + loc;
    const int L = species * d.nsc + g;
    const int n = d.count[L];
    const int scx = loc % b.nscx, scy = (loc / b.nscx) % b.nscy, scz = loc / (b.nscx * b.nscy);
    const int* ft = d.ftab + d.foff[L];
    const int64_t o0 = list_off[loc];
    auto words_into_line = [](const void* p) { return (int)((reinterpret_cast<uintptr_t>(p) >> 3) & 15); };
    if (x || u)
        for (int j = (int)threadIdx.x - words_into_line((x ? x : u) + 3 * o0); j < 3 * n; j += blockDim.x) {
            if (j < 0)
                continue;
            const int p = j / 3, a = j - 3 * p;
            const int64_t idx = (int64_t)ft[p >> d.log2S] * d.S + (p & (d.S - 1));
            if (x) {
                const int cell = d.cell[idx];
                const int gc = a == 0 ? scx * d.LX + cell % d.LX
                                      : (a == 1 ? scy * d.LY + (cell / d.LX) % d.LY : scz * d.LZ + cell / (d.LX * d.LY));
                x[3 * o0 + j] = (double)gc + (double)(a == 0 ? d.ox : (a == 1 ? d.oy : d.oz))[idx];
            }
            if (u)
                u[3 * o0 + j] = (double)(a == 0 ? d.ux : (a == 1 ? d.uy : d.uz))[idx];
        }
    if (w || id)
        for (int p = (int)threadIdx.x - (id ? words_into_line(id + o0) : words_into_line(w + o0)); p < n; p += blockDim.x) {
            if (p < 0)
                continue;
            const int64_t idx = (int64_t)ft[p >> d.log2S] * d.S + (p & (d.S - 1));
            if (w)
                w[o0 + p] = (double)d.w[idx];
            if (id)
                id[o0 + p] = d.pid ? (int64_t)d.pid[idx] : -1;
        }
}

cudaError_t launch_read_particles(const StepDev& d, const BoxDev& hb, int box, int species,
                                  const int* list_off, double* x, double* u, double* w,
                                  int64_t* id, cudaStream_t st)
{
    const int nsc_box = hb.nscx * hb.nscy * hb.nscz;
    if (nsc_box == 0)
        return cudaSuccess;
    k_read_particles<<<nsc_box, 128, 0, st>>>(d, box, species, list_off, x, u, w, id);
    return cudaGetLastError();
}

}  // namespace pic
