// LU of the trailing block of the re-factorization (Schedule::tb_p): the
// last m columns, whose part of the factors is nearly dense.
//
// The panels of those columns apply only their dependencies before the block
// and leave the rest in the dense row-major matrix S (zeros where the factor
// has no entry; they stay zeros).  S is then factored right-looking, in
// blocks of 16 columns, without row interchanges, one launch per block b:
//   - S -= L(:, b) U(b, :) on everything behind block b, and
//   - block b+1 itself: its 16 x 16 diagonal block (task D), the rows of L
//     below it (tasks L, 32 rows each) and the columns of U right of it
//     (tasks U, 32 columns each).  Tasks L and U update their tile, then wait
//     for D's flag.
// So the serial part of block b+1 runs beside the update by block b, and the
// chain of the factorization is one launch per 16 columns instead of a
// hand-off between CTAs per panel; the update is spread over the whole
// device.  Every value gets the same multiply-adds in the same (ascending)
// order as in the column kernels: finite factors are the same bits (the
// zeros outside the pattern make NaN of infinite values, which fails the
// column's check; the restart then judges it without them).
// The last launch checks every pivot against its column's largest candidate,
// stores the entries of the columns that pass in the factor's columns and
// publishes them.  The columns before the first failing one were computed
// from passing pivots alone, so first_bad is exact; the failing columns stay
// unpublished, and the restart computes them again.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>

#include "device_util.cuh"
#include "gblu_internal.h"

namespace gblu {

namespace {

using namespace dev;

constexpr int kB = kBlockCols;          // columns of a block
constexpr int kT = 128;                 // threads of a task
constexpr int kTR = 64, kTC = 32;       // tile of the update
constexpr int kEdge = 32;               // rows (columns) of a task L (U)

struct StepShared {
    double a[kB][kTR + 1];              // L(rows, block b), k-major; later the tile's rows
    double u[kB][kTC + 1];              // U(block b, columns)
    double d[kB][kB + 1];               // diagonal block b+1: U and diagonal; unscaled below
    double l[kB][kB + 1];               // its L part, scaled
    double inv[kB];
    unsigned long long mx[kB];
    int ticket, bad;
};

// waits for the diagonal block's flag (thread 0, then the CTA)
__device__ __forceinline__ bool await_diag(const BlockArgs &a, int blk, StepShared &s)
{
    if (threadIdx.x == 0) {
        int bad = 0;
        long long it = 0;
        while (ld_acquire(a.flag + blk) != 1) {
            ++it;
            if ((it & 31) == 0 && ld_volatile(&a.ctl->status)) { bad = 1; break; }
            if (it > a.spin_limit) {
                set_status(a.ctl, GBLU_ERR_DEVICE_TIMEOUT);
                a.ctl->where = 12;
                a.ctl->where_k = a.p + blk * kB;
                bad = 1;
                break;
            }
            if (it > 64) __nanosleep(64);
        }
        s.bad = bad;
    }
    __syncthreads();
    return !s.bad;
}

__device__ __forceinline__ unsigned long long abs_bits(double v)
{
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

// task t of launch `step`
__device__ __forceinline__ void block_task(const BlockArgs &a, int step, int t, StepShared &s)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int kd = step > 0 ? kB : 0;             // depth of the update
    const int kb = (step - 1) * kB;               // first column of block step-1
    const int o = step * kB;                      // first column of block step
    const int nb = min(kB, a.m - o);              // its columns
    const int o2 = o + kB;                        // what lies behind it
    const int rest = max(a.m - o2, 0), ne = (rest + kEdge - 1) / kEdge;
    double *const S = a.S;
    const int64_t ld = a.ld;
    // rows [r0, r0+nr) and columns [c0, c0+nc) of this task
    int r0, c0, nr, nc, kind;
    if (t == 0) { kind = 0; r0 = o; nr = nb; c0 = o; nc = nb; }
    else if (t <= ne) { kind = 1; r0 = o2 + (t - 1) * kEdge; nr = min(kEdge, a.m - r0); c0 = o; nc = kB; }
    else if (t <= 2 * ne) { kind = 2; r0 = o; nr = kB; c0 = o2 + (t - 1 - ne) * kEdge; nc = min(kEdge, a.m - c0); }
    else {
        kind = 3;
        t -= 1 + 2 * ne;
        const int tc = (rest + kTC - 1) / kTC;
        r0 = o2 + (t / tc) * kTR;
        c0 = o2 + (t % tc) * kTC;
        nr = min(kTR, a.m - r0);
        nc = min(kTC, a.m - c0);
        if (kd == 0) return;
    }
    if (kd) {   // the operands: 16 columns of L, 16 rows of U
        for (int i = tid; i < nr * kB; i += kT) s.a[i % kB][i / kB] = __ldcg(S + (int64_t)(r0 + i / kB) * ld + kb + i % kB);
        for (int i = tid; i < nc * kB; i += kT) s.u[i / nc][i % nc] = __ldcg(S + (int64_t)(kb + i / nc) * ld + c0 + i % nc);
    }
    if (kind == 3) {
        // 64 x 32 tile: thread (ty, tx) has rows ty + 16 i, columns tx + 8 j
        const int tx = tid & 7, ty = tid >> 3;
        double c[4][4];
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int r = ty + 16 * i, q = tx + 8 * j;
                c[i][j] = (r < nr && q < nc) ? __ldcg(S + (int64_t)(r0 + r) * ld + c0 + q) : 0.0;
            }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < kB; k++) {
            double x[4], y[4];
#pragma unroll
            for (int i = 0; i < 4; i++) x[i] = s.a[k][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; j++) y[j] = s.u[k][tx + 8 * j];
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) c[i][j] = fma(-y[j], x[i], c[i][j]);
        }
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int r = ty + 16 * i, q = tx + 8 * j;
                if (r < nr && q < nc) S[(int64_t)(r0 + r) * ld + c0 + q] = c[i][j];
            }
        return;
    }
    // an edge task: up to 32 x 16 (or 16 x 32, or 16 x 16) values, four per
    // thread: thread owns row (L) or column (U, D) e = lane and 4 values across
    const bool byrow = kind == 1;
    const int len = byrow ? nr : nc;              // along the lanes
    const int wid = byrow ? nc : nr;              // across: warp * 4 ..
    double v[4];
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const int w = warp * 4 + j;
        const int r = byrow ? lane : w, q = byrow ? w : lane;
        v[j] = (lane < len && w < wid) ? __ldcg(S + (int64_t)(r0 + r) * ld + c0 + q) : 0.0;
    }
    __syncthreads();
    if (kd) {
        for (int k = 0; k < kB; k++) {
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int w = warp * 4 + j;
                const double x = byrow ? s.a[k][lane] : s.a[k][w], y = byrow ? s.u[k][w] : s.u[k][lane];
                v[j] = fma(-y, x, v[j]);
            }
        }
    }
    __syncthreads();   // the operands are no longer needed: s.a becomes the tile, s.a[across][lane]
#pragma unroll
    for (int j = 0; j < 4; j++) s.a[warp * 4 + j][lane] = v[j];
    if (tid < kB) s.mx[tid] = 0;
    __syncthreads();

    if (kind == 0) {
        // diagonal block: thread (q, g) has row q, columns g and g + 8
        const int q = tid & 15, g = tid >> 4;
        double v0 = s.a[q][g], v1 = s.a[q][g + 8];
        s.d[q][g] = v0;
        s.d[q][g + 8] = v1;
        __syncthreads();
        for (int k = 0; k < nb; k++) {
            const double xq = s.d[q][k], u0 = s.d[k][g], u1 = s.d[k][g + 8];
            const double inv = __drcp_rn(s.d[k][k]);   // 1 / x, correctly rounded
            const double l = xq * inv;
            if (tid == 0) s.inv[k] = inv;
            const double n0 = fma(-u0, l, v0), n1 = fma(-u1, l, v1);
            v0 = q > k && g > k ? n0 : v0;
            v1 = q > k && g + 8 > k ? n1 : v1;
            if (q > k && g == 0) s.l[q][k] = l;
            if (q > k && g > k) s.d[q][g] = v0;
            if (q > k && g + 8 > k) s.d[q][g + 8] = v1;
            __syncthreads();
        }
        for (int i = tid; i < nb * nb; i += kT) {
            const int r = i / nb, c = i % nb;
            S[(int64_t)(o + r) * ld + o + c] = r > c ? s.l[r][c] : s.d[r][c];
        }
        if (tid < nb) {
            a.inv[o + tid] = s.inv[tid];
            unsigned long long m = 0;
            for (int r = tid + 1; r < nb; r++) m = max(m, abs_bits(s.d[r][tid]));
            if (m) atomicMax(a.colmax + o + tid, m);
        }
        __syncthreads();
        if (tid == 0) st_release(a.flag + step, 1);
        return;
    }
    if (!await_diag(a, step, s)) return;
    for (int i = tid; i < kB * kB; i += kT) s.d[i / kB][i % kB] = __ldcg(S + (int64_t)(o + i / kB) * ld + o + i % kB);
    if (tid < kB) s.inv[tid] = __ldcg(a.inv + o + tid);
    __syncthreads();
    if (warp == 0) {
        double x[kB];
#pragma unroll
        for (int k = 0; k < kB; k++) x[k] = s.a[k][lane];
        if (kind == 1) {   // L rows: x := x U^-1 (U with the diagonal)
#pragma unroll
            for (int k = 0; k < kB; k++) {
                const unsigned long long key = lane < nr ? abs_bits(x[k]) : 0ull;
                const unsigned hi = __reduce_max_sync(kFull, (unsigned)(key >> 32));
                const unsigned lo = __reduce_max_sync(kFull, (unsigned)(key >> 32) == hi ? (unsigned)key : 0u);
                if (lane == 0) s.mx[k] = ((unsigned long long)hi << 32) | lo;
                x[k] = x[k] * s.inv[k];
#pragma unroll
                for (int c = k + 1; c < kB; c++) x[c] = fma(-s.d[k][c], x[k], x[c]);
            }
        } else {           // U columns: x := L^-1 x (unit diagonal)
#pragma unroll
            for (int k = 0; k < kB; k++)
#pragma unroll
                for (int q = k + 1; q < kB; q++) x[q] = fma(-x[k], s.d[q][k], x[q]);
        }
#pragma unroll
        for (int k = 0; k < kB; k++) s.a[k][lane] = x[k];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const int w = warp * 4 + j;
        if (kind == 2 && lane < nc) S[(int64_t)(r0 + w) * ld + c0 + lane] = s.a[w][lane];
    }
    if (kind == 1) {
        for (int i = tid; i < nr * kB; i += kT) S[(int64_t)(r0 + i / kB) * ld + c0 + i % kB] = s.a[i % kB][i / kB];
        if (tid < kB && s.mx[tid]) atomicMax(a.colmax + o + tid, s.mx[tid]);
    }
}

// launch `step`: update by block step-1 (none for step 0) and factor block
// step; tasks are handed out in order (a diagonal block is never waited for
// before a running CTA has it), one per CTA or, where max_sms leaves fewer
// CTAs than tasks, several
__global__ void __launch_bounds__(kT) block_step_kernel(BlockArgs a, int step, int tasks)
{
    __shared__ StepShared s;
    for (;;) {
        // (a check that failed before the block: nothing to do)
        if (threadIdx.x == 0) s.ticket = ld_volatile(&a.ctl->interrupted) ? tasks : atomicAdd(a.ticket + step, 1);
        __syncthreads();
        const int t = s.ticket;
        if (t >= tasks) return;
        block_task(a, step, t, s);
        if ((int)gridDim.x == tasks) return;
        __syncthreads();
    }
}

// pivot checks, the block's entries into the factor's columns, ready flags:
// column c by one warp
__device__ __forceinline__ void finish_column(const BlockArgs &a, int c, int lane)
{
    // a check that failed before the block (one in the block is not a reason
    // to leave: every column is judged by itself)
    if (ld_volatile(&a.ctl->first_bad) < a.p || ld_volatile(&a.ctl->status)) return;
    const int k = a.p + c;
    const double d = __ldcg(a.S + (int64_t)c * a.ld + c);
    const double m = __longlong_as_double((long long)__ldcg(a.colmax + c));
    if (!(d != 0.0) || !isfinite(d) || !(fabs(d) >= a.eps * m)) {
        if (lane == 0) {
            atomicExch(&a.ctl->interrupted, 1);
            atomicMin(&a.ctl->first_bad, k);
        }
        return;
    }
    const int64_t b = __ldg(a.LUp + k), e = __ldg(a.LUp + k + 1);
    for (int64_t i = b + __ldg(a.nux + c) + lane; i < e; i += 32)
        a.LUx[i] = __ldcg(a.S + (int64_t)(__ldg(a.LUi + i) - a.p) * a.ld + c);
    __syncwarp();
    if (lane == 0) st_release(a.finish + k, a.epoch < 0 ? ld_volatile(&a.ctl->epoch) : a.epoch);
}

__global__ void __launch_bounds__(256) block_finish_kernel(BlockArgs a)
{
    const int step = (int)((gridDim.x * blockDim.x) >> 5);
    for (int c = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); c < a.m; c += step) finish_column(a, c, threadIdx.x & 31);
}

}  // namespace

int block_steps(int m) { return (m + kB - 1) / kB; }

int block_setup(int *ctas_per_sm)
{
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, block_step_kernel, kT, 0);
}

// launches of the block's LU (after the panels' launch on the same stream)
int launch_block_lu(const BlockArgs &a, void *stream, long long *launches)
{
    cudaStream_t st = (cudaStream_t)stream;
    const int steps = block_steps(a.m);
    for (int b = 0; b < steps; b++) {
        const int rest = std::max(a.m - (b + 1) * kB, 0), ne = (rest + kEdge - 1) / kEdge;
        const int tiles = b > 0 ? ((rest + kTR - 1) / kTR) * ((rest + kTC - 1) / kTC) : 0;
        const int tasks = 1 + 2 * ne + tiles;
        block_step_kernel<<<std::min(tasks, a.max_ctas), kT, 0, st>>>(a, b, tasks);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return (int)e;
    }
    block_finish_kernel<<<std::min((a.m + 7) / 8, a.max_ctas), 256, 0, st>>>(a);
    *launches += steps + 1;
    return (int)cudaGetLastError();
}

}  // namespace gblu
