// Panels of the checked re-factorization (Section IV-B, Algorithms 3 and 4):
// up to eight consecutive columns of one supernode of L computed together by
// one CTA.  Included by refactor.cu only.
//
// The work vector is X[slot][LD]: the union of the columns' patterns (slots:
// U rows above the first column, the diagonal block, the L rows of the last
// column), one value per column.  A run of dependencies j .. j+w-1 of one
// supernode of L (PanelRun) updates all columns at once:
//   triangle  - the run's unit lower triangle is solved for every column;
//   rectangle - every row r of R: X[r][c] -= sum_d L(r, j+d) X[j+d][c].
// An entry of L is read, and its row's slot searched, once for all columns.
//
// Warps are specialised.  Producers (warps 4-7) take the stages of the run
// list in turn: they wait for the dependencies' flags, search the rows'
// slots and copy the values of L into a ring of shared-memory stages, up to
// four stages ahead.  Consumers (warps 0-3, one per FP64 pipe) do the
// arithmetic from shared memory, so the latency of L2 and of the flags is
// off their chain.  A stage is up to cap/w rows of a run (its triangle's
// rows first).  Then the diagonal block is factored by one warp, the L rows
// by every thread, the pivots are checked, and the columns are published
// together.
//
// Each value gets the same fused multiply-adds in the same order as when
// its column is computed alone, so finite factors are the same bits.  A column
// without an entry that its neighbours have holds a zero there, and
// subtracts zero times a value: an infinite L (a subnormal pivot, or one that
// passed with a tolerance below the reciprocal of the largest double) makes
// NaN there, also in columns that do not depend on it.
#pragma once

namespace gblu {

namespace {

constexpr int kConsWarps = 4, kProdWarps = kWarps - kConsWarps;
constexpr int kStageRows = 128;                      // most rows of a stage
constexpr int kStagesMax = 4;

template <typename R>
struct PanelShared {
    alignas(16) R mul[kPanelRun * kPanelMax];    // multipliers of the run (work vector in global memory)
    R D[kPanelMax * kPanelMax];                  // diagonal block, unscaled
    R Lb[kPanelMax * kPanelMax];                 // its L part, scaled
    R inv[kPanelMax];
    unsigned long long mx[kWarps][kPanelMax];    // bits of max |x| over the L rows, by warp
    unsigned pass;
    int abort;                                   // a producer gave up: everyone leaves
    int pull_slot;                               // wide columns: the scratch in use
    unsigned long long pull_tag;                 // and its tag
    int step, next;                              // finished columns of the diagonal block; next L row to take
};

// barriers of the stage ring (initialized once per CTA, again per panel)
struct PanelBars {
    unsigned long long full[kStagesMax], empty[kStagesMax];
};

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *b, unsigned count)
{
    asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void init_bars(PanelBars &b)
{
    for (int i = 0; i < kStagesMax; i++) {
        mbar_init(&b.full[i], 1);
        mbar_init(&b.empty[i], kConsWarps);
    }
}
__device__ __forceinline__ void mbar_inval(unsigned long long *b)
{
    asm volatile("mbarrier.inval.shared.b64 [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long *b)
{
    asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.shared.b64 t, [%0];\n\t}" ::"r"(smem_u32(b)) : "memory");
}
// waits for the phase of the given parity; false when the panel is aborted.
// What it waits for is bounded itself (the producers' flag waits by
// spin_limit), so its own limit is only a backstop.
constexpr long long kBarTries = 1ll << 28;
__device__ __forceinline__ bool mbar_wait(unsigned long long *b, unsigned parity, int *abort_flag, DevCtl *ctl)
{
    const volatile int *abort = abort_flag;
    const unsigned addr = smem_u32(b);
    for (long long it = 0;; ++it) {
        unsigned ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(addr), "r"(parity)
                     : "memory");
        if (ok) return true;
        if (*abort) return false;
        if (it > kBarTries) {
            set_status(ctl, GBLU_ERR_DEVICE_TIMEOUT);
            *abort_flag = 1;
            return false;
        }
    }
}

// N values at p, in 16- or 8-byte accesses (p aligned to that)
template <typename R, int N>
__device__ __forceinline__ void ldv(const R *p, R (&v)[N])
{
    if constexpr (N * sizeof(R) % 16 == 0) {
#pragma unroll
        for (int i = 0; i < (int)(N * sizeof(R) / 16); i++) {
            const int4 q = reinterpret_cast<const int4 *>(p)[i];
            memcpy(&v[i * (16 / sizeof(R))], &q, 16);
        }
    } else if constexpr (N * sizeof(R) == 8) {
        const int2 q = *reinterpret_cast<const int2 *>(p);
        memcpy(&v[0], &q, 8);
    } else {
        v[0] = p[0];
    }
}

template <typename R, int N>
__device__ __forceinline__ void stv(R *p, const R (&v)[N])
{
    if constexpr (N * sizeof(R) % 16 == 0) {
#pragma unroll
        for (int i = 0; i < (int)(N * sizeof(R) / 16); i++) {
            int4 q;
            memcpy(&q, &v[i * (16 / sizeof(R))], 16);
            reinterpret_cast<int4 *>(p)[i] = q;
        }
    } else if constexpr (N * sizeof(R) == 8) {
        int2 q;
        memcpy(&q, &v[0], 8);
        *reinterpret_cast<int2 *>(p) = q;
    } else {
        p[0] = v[0];
    }
}

// 1 / x, correctly rounded (as the division is)
__device__ __forceinline__ double recip(double x) { return __drcp_rn(x); }
__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }

__device__ __forceinline__ void st_release_cta(int *p, int v)
{
    asm volatile("st.release.cta.shared.b32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_acquire_cta(const int *p)
{
    int v;
    asm volatile("ld.acquire.cta.shared.b32 %0, [%1];" : "=r"(v) : "r"((unsigned)__cvta_generic_to_shared(p)) : "memory");
    return v;
}

// |x| as an integer of the same order (NaN above infinity), so that maxima
// stay off the FP64 pipe
__device__ __forceinline__ unsigned long long abs_key(double v)
{
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ unsigned long long abs_key(float v)
{
    return (unsigned long long)(__float_as_uint(v) & 0x7fffffffu) << 32;
}
__device__ __forceinline__ double key_abs(unsigned long long k, double) { return __longlong_as_double((long long)k); }
__device__ __forceinline__ float key_abs(unsigned long long k, float) { return __uint_as_float((unsigned)(k >> 32)); }

__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k)
{
    const unsigned hi = (unsigned)(k >> 32);
    const unsigned mh = __reduce_max_sync(kFull, hi);
    const unsigned ml = __reduce_max_sync(kFull, hi == mh ? (unsigned)k : 0u);
    return ((unsigned long long)mh << 32) | ml;
}

// A stage of the ring: header, the rows' slots, and for dependency d < w the
// values of rows i of the stage at val[off[d] + i] (row pitch sp)
struct StageHead {
    int t, w, mask, i0, i1;   // run; rectangle rows [i0, i1) of the stage (those before i0: the triangle's)
    int first, last, pad;     // first stage of its run, last stage of the panel
    int off[kPanelRun];
};
static_assert(sizeof(StageHead) == 96, "StageHead");
constexpr int kHeadBytes = 128;
// value pitch beyond the rows: the copies start and end on 16-byte boundaries
constexpr int kStagePad = 4;
__host__ __device__ constexpr int stage_bytes_of(int cap, int elem) { return kHeadBytes + kStageRows * 4 + cap * elem; }
static_assert(4 * stage_bytes_of(kStageCap, 8) == kPanelRing, "kPanelRing");
static_assert(kStageCap / kPanelRun - kStagePad >= 32, "a stage holds 32 rows of the widest run");
// a panel whose work vector fits beside the ring in doubles fits in floats
constexpr bool fits_in_floats(int smem, int smem32)
{
    const int room = smem - kPanelRing, room32 = smem32 - 4 * stage_bytes_of(kStageCap, 4);
    return room / (4 * 8 + 4) * (4 * 4 + 4) <= room32 && room / (8 * 8 + 4) * (8 * 4 + 4) <= room32 &&
           3 * stage_bytes_of(kStageCapBig, 4) <= smem32 && kRefCapLong * 8 <= smem32;
}
static_assert(fits_in_floats(kRefSmemTwo, kRefSmemTwo32) && fits_in_floats(kRefSmemThree, kRefSmemThree32), "smem32");

// rows of a stage for a run of w dependencies
__device__ __forceinline__ int stage_rows(int cap, int w)
{
    return min(kStageRows, (cap / w - kStagePad) & ~31);
}

// the run descriptors 32 at a time in a warp's lanes, with the stages each
// run takes (st0: the lane's first stage)
struct RunWindow {
    long long lbl;
    int t, wm, nR, j0, rows, st0;
    int base, end;   // first run of the window; first stage after it
    __device__ __forceinline__ void load(const PanelRun *runs, int ri, int n, int cap, int stage0, int lane)
    {
        base = ri;
        const int2 *r = reinterpret_cast<const int2 *>(runs + min(ri + lane, n - 1));   // 24 bytes, 8-byte aligned
        const int2 h0 = __ldg(r), h1 = __ldg(r + 1);
        t = h0.x; wm = h0.y; nR = h1.x; j0 = h1.y;
        lbl = __ldg(reinterpret_cast<const long long *>(r + 2));
        const int w = wm & 0xff;
        rows = stage_rows(cap, w);
        const int cnt = ri + lane < n ? max(1, (w - 1 + nR + rows - 1) / rows) : 0;
        int sum = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, sum, o);
            if (lane >= o) sum += v;
        }
        st0 = stage0 + sum - cnt;
        end = stage0 + __shfl_sync(kFull, sum, 31);
    }
};

// rectangle of one stage: rows [i0, i1) (values val[off[d] + i], slots
// sl[i]), CPT columns per lane, work items of 32 rows x CPT columns (kHalf:
// at most 16 rows, two column groups per warp) dealt to the consumer warps
template <typename R, int LD, int CPT, bool kHalf>
__device__ __forceinline__ void stage_rect(const R *val, const int *off, const int *sl, int i0, int i1, int w,
                                           const R *mul, unsigned mask, R *X, int warp, int lane)
{
    constexpr int G = LD / CPT;
    const int items = kHalf ? G / 2 : ((i1 - i0 + 31) >> 5) * G;
    for (int it = warp; it < items; it += kConsWarps) {
        const int g = kHalf ? it * 2 + (lane >> 4) : it % G;
        const int i = i0 + (kHalf ? (lane & 15) : (it / G) * 32 + lane);
        const unsigned gm = (mask >> (g * CPT)) & ((1u << CPT) - 1u);
        if (i >= i1 || gm == 0) continue;
        R *x = X + (size_t)sl[i] * LD + g * CPT;
        R v[CPT];
        ldv<R, CPT>(x, v);
        const R *l = val + i, *mp = mul + g * CPT;
        if (gm == (1u << CPT) - 1u) {
#pragma unroll 4
            for (int d = 0; d < w; d++) {
                const R lv = l[off[d]];
                R m[CPT];
                ldv<R, CPT>(mp + d * LD, m);
#pragma unroll
                for (int c = 0; c < CPT; c++) v[c] = fma(-m[c], lv, v[c]);
            }
        } else {   // some columns have no entry in this run
            for (int d = 0; d < w; d++) {
                const R lv = l[off[d]];
#pragma unroll
                for (int c = 0; c < CPT; c++)
                    if ((gm >> c) & 1u) v[c] = fma(-mp[d * LD + c], lv, v[c]);
            }
        }
        stv<R, CPT>(x, v);
    }
}

// barrier of the consumer warps; whether any thread's v is set
__device__ __forceinline__ bool cons_sync_or(bool v)
{
    int r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbarrier.red.or.pred q, 1, %2, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
                 : "=r"(r)
                 : "r"((int)v), "n"(kConsWarps * 32)
                 : "memory");
    return r != 0;
}

// the consumers' part of a panel's runs; false = aborted
template <typename R, int LD>
__device__ __forceinline__ bool panel_consume(R *X, bool in_smem, unsigned char *ring, int stage_bytes, int ns,
                                              PanelShared<R> &sh, PanelBars &bars, DevCtl *ctl, int warp, int lane)
{
    int slot = 0;
    unsigned parity = 0;
    bool ok = true;
    const R *mul = sh.mul;
    for (;;) {
        ok = ok && mbar_wait(&bars.full[slot], parity, &sh.abort, ctl);
        unsigned char *st = ring + (size_t)slot * stage_bytes;
        const StageHead &h = *reinterpret_cast<const StageHead *>(st);
        const int *sl = reinterpret_cast<const int *>(st + kHeadBytes);
        const R *val = reinterpret_cast<const R *>(st + kHeadBytes + kStageRows * 4);
        // within a run an aborted warp waits for the others at the next
        // run's barrier (or at the end of the panel): they all leave there
        if (!ok || h.first) {
            // the previous run's rectangle is done everywhere
            if (cons_sync_or(!ok)) return false;
            const int w = h.w;
            if (in_smem) mul = X + (size_t)h.t * LD;
            if (w > 1 || !in_smem) {
                // triangle: lane q holds row q, this warp's columns side by side
                constexpr int C = LD / kConsWarps;
                R *x = X + (size_t)(h.t + lane) * LD + warp;
                R v[C];
#pragma unroll
                for (int c = 0; c < C; c++) v[c] = lane < w ? x[c * kConsWarps] : R(0);
                // (selects, not branches: a divergent step costs several times
                // its arithmetic)
                const R *lp = val + max(lane, 1) - 1;
#pragma unroll 4
                for (int d = 0; d < w - 1; d++) {
                    const R lv = lp[h.off[d]];
#pragma unroll
                    for (int c = 0; c < C; c++) {
                        const R nv = fma(-lv, __shfl_sync(kFull, v[c], d), v[c]);
                        v[c] = lane > d && lane < w ? nv : v[c];
                    }
                }
                if (lane < w) {
#pragma unroll
                    for (int c = 0; c < C; c++) {
                        x[c * kConsWarps] = v[c];
                        if (!in_smem) sh.mul[lane * LD + warp + c * kConsWarps] = v[c];
                    }
                }
                asm volatile("bar.sync 1, %0;" ::"n"(kConsWarps * 32) : "memory");
            }
        }
        const int i0 = h.i0, i1 = h.i1, n = i1 - i0, w = h.w, last = h.last;
        const unsigned mask = (unsigned)h.mask;
        // one item per FP64 pipe where the rows are few, else four columns
        // per lane
        if (n > 0) {
            if (LD == 8 && n <= 16) stage_rect<R, LD, 1, true>(val, h.off, sl, i0, i1, w, mul, mask, X, warp, lane);
            else if (n <= 32) stage_rect<R, LD, LD / 4, false>(val, h.off, sl, i0, i1, w, mul, mask, X, warp, lane);
            else if (LD == 4 && n <= 64) stage_rect<R, LD, 2, false>(val, h.off, sl, i0, i1, w, mul, mask, X, warp, lane);
            else stage_rect<R, LD, 4, false>(val, h.off, sl, i0, i1, w, mul, mask, X, warp, lane);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars.empty[slot]);
        if (last) break;
        if (++slot == ns) { slot = 0; parity ^= 1u; }
    }
    return true;
}

// Waits until the copies that producer warp p has started (fills of them) have
// landed.  Only an aborted panel needs it: otherwise the consumers have waited
// for every stage.  A copy in flight lands without anyone's help, so the limit
// is a backstop.
__device__ __forceinline__ void drain_slot(PanelBars &bars, int p, int fills, DevCtl *ctl)
{
    if (fills == 0) return;
    const unsigned addr = smem_u32(&bars.full[p]), parity = (unsigned)(fills - 1) & 1u;
    unsigned done = 0;
    for (long long it = 0; !done && it < kBarTries; ++it)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(addr), "r"(parity)
                     : "memory");
    if (!done) set_status(ctl, GBLU_ERR_DEVICE_TIMEOUT);
}

// the producers' part: warp p < ns fills slot p of the ring, stages p, p + ns,
// ... (a slot belongs to one warp: a barrier's parity tells two successive
// phases apart, so each phase has to be waited for in turn); false = gave up
// (sh.abort set).  Either way the last fill's copies may still be in flight:
// fills = how many were started (drain_slot).
template <typename R>
__device__ __forceinline__ bool panel_produce(const RefactorArgsT<R> &a, const PanelRun *runs, int nruns,
                                              const int32_t *rows, int nu, int len, int k0, unsigned char *ring,
                                              int cap, int stage_bytes, int ns, PanelShared<R> &sh, PanelBars &bars,
                                              int epoch, bool wait, int p, int lane, int &fills)
{
    fills = 0;
    if (p >= ns) return true;
    const R *const LUx = a.LUx;
    const int32_t *const LUi = a.LUi, *const nUp = a.nU, *const finish = a.finish;
    const int64_t *const LUp = a.LUp;
    volatile int *abort = &sh.abort;
    unsigned char *st = ring + (size_t)p * stage_bytes;
    StageHead &h = *reinterpret_cast<StageHead *>(st);
    int *ssl = reinterpret_cast<int *>(st + kHeadBytes);
    R *val = reinterpret_cast<R *>(st + kHeadBytes + kStageRows * 4);
    // the ring's memory was last written by ordinary stores
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    RunWindow rw;
    rw.load(runs, 0, nruns, cap, 0, lane);
    int ready = 0;   // dependencies [0, ready) are known to be final
    auto give_up = [&]() -> bool {
        if (lane == 0) *abort = 1;
        return false;
    };
    for (int s = p;; s += ns) {
        while (s >= rw.end) {
            if (rw.base + 32 >= nruns) return true;
            rw.load(runs, rw.base + 32, nruns, cap, rw.end, lane);
        }
        // the lane whose run holds stage s (lanes past the list start at rw.end)
        const int q = 31 - __clz(__ballot_sync(kFull, rw.st0 <= s));
        const int t = __shfl_sync(kFull, rw.t, q), wm = __shfl_sync(kFull, rw.wm, q), nR = __shfl_sync(kFull, rw.nR, q);
        const int j0 = __shfl_sync(kFull, rw.j0, q), S = __shfl_sync(kFull, rw.rows, q);
        const int e0 = (s - __shfl_sync(kFull, rw.st0, q)) * S;
        const long long lbl = __shfl_sync(kFull, rw.lbl, q);
        const int w = wm & 0xff, nE = w - 1 + nR, tl = t + w - 1, jl = j0 + w - 1;
        const int n = min(nE - e0, S), i0 = max(w - 1 - e0, 0), nb = (n + 31) >> 5;
        // structure first: lane d < w start of L(:, j0+d); the rows' slots
        const long long lb = lane < w ? __ldg(LUp + j0 + lane) + __ldg(nUp + j0 + lane) : 0;
        int key[4], sl[4];
        bool bad = false;
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const int i = b * 32 + lane;
            key[b] = (i >= i0 && i < n) ? __ldg(LUi + lbl + (e0 + i - (w - 1))) : -1;
        }
        if (nb <= 1) {
            const int r = e0 + lane - (w - 1);
            sl[0] = key[0] >= 0 ? find_slot(rows, tl + 1 + r, tl + (key[0] - jl), len, key[0]) : -1;
            sl[1] = sl[2] = sl[3] = -1;
        } else {
            int lo[4], hi[4];
#pragma unroll
            for (int b = 0; b < 4; b++) {
                lo[b] = tl + 1 + (e0 + b * 32 + lane - (w - 1));
                hi[b] = tl + (key[b] - jl);
            }
            find_slots<4>(rows, lo, hi, len, key, sl);
        }
#pragma unroll
        for (int b = 0; b < 4; b++) bad = bad || (key[b] >= 0 && sl[b] < 0);
        if (__any_sync(kFull, bad)) {   // inconsistent pattern: never index with it
            if (lane == 0) set_status(a.ctl, GBLU_ERR_INTERNAL);
            return give_up();
        }
        if (wait && ready < t + w) {
            long long it = 0;
            for (;;) {
                const int d = ready + lane;
                const bool fin = d >= nu || ld_acquire(finish + rows[d]) == epoch;
                const unsigned m = __ballot_sync(kFull, fin);
                ready += m == kFull ? 32 : __ffs(~m) - 1;
                if (ready >= t + w) break;
                ++it;
                bool stop = *abort != 0;
                if ((it & 31) == 0 && (ld_volatile(&a.ctl->interrupted) || ld_volatile(&a.ctl->status))) stop = true;
                if (it > a.spin_limit) {
                    if (lane == 0) {
                        set_status(a.ctl, GBLU_ERR_DEVICE_TIMEOUT);
                        a.ctl->where = 1;
                        a.ctl->where_k = k0;
                    }
                    stop = true;
                }
                if (__any_sync(kFull, stop)) return give_up();
                if (it > 64) __nanosleep(64);
            }
        }
        // an empty slot (the first fill finds it so)
        if (!mbar_wait(&bars.empty[p], (unsigned)(fills + 1) & 1u, &sh.abort, a.ctl)) return give_up();
#pragma unroll
        for (int b = 0; b < 4; b++)
            if (b < nb) ssl[b * 32 + lane] = sl[b];
        // Values: dependency d's entries of rows i >= d - e0, one bulk copy
        // per dependency (lane d).  Row i's place in the stage is congruent
        // to its address modulo 16 bytes, so the copy takes whole 16-byte
        // units: up to three entries before and after, which stay inside the
        // factor array (a U entry precedes every L part, a column follows
        // it) and inside the pitch.
        constexpr int kE = 16 / (int)sizeof(R);
        const int sp = S + kStagePad;
        const long long src = (long long)(reinterpret_cast<uintptr_t>(LUx) / sizeof(R)) + lb + (e0 - lane);   // element of row 0
        const int sh0 = (int)(src & (kE - 1));
        const int ib = max(lane - e0, 0);
        const int lo = (ib + sh0) & ~(kE - 1), hi = (n + sh0 + kE - 1) & ~(kE - 1);
        const unsigned bytes = (lane < w && n > ib) ? (unsigned)(hi - lo) * (unsigned)sizeof(R) : 0u;
        const unsigned total = __reduce_add_sync(kFull, bytes);
        if (lane < w) h.off[lane] = lane * sp + sh0;
        if (lane == 0) {
            h.t = t;
            h.w = w;
            h.mask = (int)((unsigned)wm >> 8);
            h.i0 = i0;
            h.i1 = n;
            h.first = e0 == 0;
            h.last = rw.base + q == nruns - 1 && e0 + S >= nE;
        }
        __syncwarp();
        if (lane == 0)
            asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.expect_tx.shared.b64 t, [%0], %1;\n\t}" ::"r"(
                             smem_u32(&bars.full[p])),
                         "r"(total)
                         : "memory");
        __syncwarp();
        fills++;
        if (bytes) {
            // the factor values were written by ordinary stores
            asm volatile("fence.proxy.async.global;" ::: "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                             smem_u32(val + lane * sp + lo)),
                         "l"((const void *)((src - sh0 + lo) * (long long)sizeof(R))), "r"(bytes),
                         "r"(smem_u32(&bars.full[p]))
                         : "memory");
        }
    }
}

// the first nu U rows of a panel into the factor's columns (lane c: lup =
// start of column c)
template <typename R, int LD>
__device__ __forceinline__ void store_u_rows(const RefactorArgsT<R> &a, const PanelDesc &p, int nu, const R *X, R *LUx,
                                             int64_t lup, int warp, int lane)
{
    const int nc = p.nc;
    for (int ch0 = warp * 2; ch0 * 32 < nu; ch0 += kWarps * 2) {
        unsigned mk[2];
        int pc[2];
        R x[2][LD];
#pragma unroll
        for (int u = 0; u < 2; u++) {   // two chunks' loads in flight
            const int s = (ch0 + u) * 32 + lane;
            mk[u] = s < nu ? __ldg(a.pmask + p.uoff + s) : 0u;
            pc[u] = (lane < nc && (ch0 + u) * 32 < nu) ? __ldg(a.ppref + p.poff + (int64_t)(ch0 + u) * nc + lane) : 0;
            if (s < nu) ldv<R, LD>(X + (size_t)s * LD, x[u]);
        }
#pragma unroll
        for (int u = 0; u < 2; u++) {
#pragma unroll
            for (int c = 0; c < LD; c++) {
                if (c < nc) {
                    const unsigned b = __ballot_sync(kFull, (mk[u] >> c) & 1u);
                    const int64_t at = __shfl_sync(kFull, lup, c) + __shfl_sync(kFull, pc[u], c) + __popc(b & ((1u << lane) - 1u));
                    if ((mk[u] >> c) & 1u) LUx[at] = x[u][c];
                }
            }
        }
    }
}

// The first p0 slots of a panel of wide columns (pull_rows, for all of the
// panel's columns at once: an entry of L, its row's tag and the wait for a
// value, whose latency bounds the chain, are paid once for four columns; 256
// sets of the bordered 141x141 grid: 334 ms with single columns, 304 ms so.
// A warp per row, with its entries' loads in parallel, took 334 ms, and with
// them pipelined two chunks ahead 345 ms: 256 rows in flight hide more than
// eight).  xd holds
// kPullLd values per row.  A column without an entry that its neighbours
// have holds a zero there.  Returns false if a wait gave up.
template <int LD>
__device__ __noinline__ bool pull_panel(const RefactorArgs *ap, int k0, double *X, const int32_t *rows, int len, int p0,
                                        int epoch, bool wait, PanelShared<double> &sh)
{
    static_assert(LD == kPullLd, "the scratch's pitch");
    const RefactorArgs &a = *ap;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t *const Lrp = a.Lrp;
    const int32_t *const Lcol = a.Lcol, *const Lslot = a.Lslot;
    const double *const LUx = a.LUx;
    bool fail = false;
    auto timeout = [&](int site) {
        set_status(a.ctl, GBLU_ERR_DEVICE_TIMEOUT);
        a.ctl->where = site;
        a.ctl->where_k = k0;
    };
    if (tid == 0) {
        int slot = -1;
        for (long long it = 0; slot < 0; ++it) {
            const int c = (int)((blockIdx.x + it) % a.pull_slots);
            if (atomicCAS(a.pull_lock + c, 0, 1) == 0) slot = c;
            else if (it > a.spin_limit) { timeout(11); break; }
        }
        sh.pull_slot = slot;
        if (slot >= 0) sh.pull_tag = ++a.pull_ctr[slot];
    }
    __syncthreads();
    const int slot = sh.pull_slot;
    if (slot < 0) return false;
    double *const xd = a.pull_x + (size_t)slot * a.n * LD;
    unsigned long long *const xt = a.pull_tag + (size_t)slot * a.n;
    const unsigned long long tag = sh.pull_tag;
    auto release = [&]() {
        __syncthreads();
        if (tid == 0) atomicExch(a.pull_lock + slot, 0);
    };
    auto give_up = [&](long long it, int site) -> bool {
        if ((it & 31) == 0 && (ld_volatile(&a.ctl->interrupted) || ld_volatile(&a.ctl->status))) return true;
        if (it > a.spin_limit) {
            timeout(site);
            return true;
        }
        if (it > 64) __nanosleep(64);
        return false;
    };
    if (wait)   // the prefix's dependencies are final
        for (int s = tid; s < p0 && !fail; s += kThreads) {
            const int j = rows[s];
            for (long long it = 1; ld_acquire(a.finish + j) != epoch; ++it)
                if (give_up(it, 9)) {
                    fail = true;
                    break;
                }
        }
    if (__syncthreads_or(fail)) {
        release();
        return false;
    }
    const double sent = __longlong_as_double((long long)kSentinel);
    for (int s = tid; s < p0; s += kThreads) {
        const int r = rows[s];
#pragma unroll
        for (int c = 0; c < LD; c++) st_relaxed_f64(xd + (size_t)r * LD + c, sent);
        st_relaxed_u64(xt + r, tag);
    }
    __syncthreads();
    for (int s = tid; s < p0 && !fail; s += kThreads) {
        const int r = rows[s];
        double acc[LD];
        ldv<double, LD>(X + (size_t)s * LD, acc);
        const int64_t e1 = __ldg(Lrp + r + 1);
        for (int64_t e = __ldg(Lrp + r); e < e1 && !fail; e++) {
            const int j = __ldg(Lcol + e);
            if (ld_relaxed_u64(xt + j) != tag) continue;
            const double l = __ldcg(LUx + __ldg(Lslot + e));
            const double *v = xd + (size_t)j * LD;
            unsigned long long b[LD];
            for (long long it = 1;; ++it) {
                bool missing = false;
#pragma unroll
                for (int c = 0; c < LD; c++) b[c] = ld_relaxed_u64(v + c);
#pragma unroll
                for (int c = 0; c < LD; c++) missing = missing || b[c] == kSentinel;
                if (!missing) break;
                if (give_up(it, 10)) {
                    fail = true;
                    break;
                }
            }
            if (fail) break;
#pragma unroll
            for (int c = 0; c < LD; c++) acc[c] = fma(-__longlong_as_double((long long)b[c]), l, acc[c]);
        }
        stv<double, LD>(X + (size_t)s * LD, acc);
#pragma unroll
        for (int c = 0; c < LD; c++) st_relaxed_f64(xd + (size_t)r * LD + c, acc[c]);
    }
    if (__syncthreads_or(fail)) {
        release();
        return false;
    }
    const int jlim = rows[p0 - 1];   // the last dependency of the prefix
    for (int s = p0 + warp; s < len; s += kWarps) {
        const int r = rows[s];
        const int64_t e1 = __ldg(Lrp + r + 1);
        double part[LD];
#pragma unroll
        for (int c = 0; c < LD; c++) part[c] = 0.0;
        for (int64_t e0 = __ldg(Lrp + r) + lane; e0 < e1; e0 += 32 * 4) {
            int j[4];
            double l[4];
            unsigned long long tg[4];
#pragma unroll
            for (int u = 0; u < 4; u++) j[u] = e0 + 32 * u < e1 ? __ldg(Lcol + e0 + 32 * u) : INT_MAX;
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const bool in = j[u] <= jlim;   // ascending: the rest is past the prefix
                tg[u] = in ? ld_relaxed_u64(xt + j[u]) : 0ull;
                l[u] = in ? __ldcg(LUx + __ldg(Lslot + e0 + 32 * u)) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (j[u] <= jlim && tg[u] == tag) {
                    const double *v = xd + (size_t)j[u] * LD;
#pragma unroll
                    for (int c = 0; c < LD; c++)
                        part[c] = fma(__longlong_as_double((long long)ld_relaxed_u64(v + c)), l[u], part[c]);
                }
            if (j[3] > jlim) break;
        }
#pragma unroll
        for (int c = 0; c < LD; c++) {
            const double t = warp_sum(part[c]);
            if (lane == 0) X[(size_t)s * LD + c] -= t;
        }
    }
    release();
    __syncthreads();
    return true;
}

// One panel by the whole CTA; true = stop.  Not inlined: its registers are
// allocated apart from the column kernels' (they share a launch bound), and
// the argument block stays where it is (kernel parameter or global memory).
template <typename R, int LD>
__device__ __noinline__ bool col_panel(const RefactorArgsT<R> *ap, int id, unsigned char *smem, int smem_bytes,
                                       PanelShared<R> &sh, PanelBars &bars, int epoch, bool wait)
{
    const RefactorArgsT<R> &a = *ap;
    const PanelDesc p = a.pan[id];
    R *const LUx = a.LUx;
    const int32_t *const LUi = a.LUi, *const nUp = a.nU;
    const int64_t *const LUp = a.LUp;
    int32_t *const finish = a.finish;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nc = p.nc, nu = p.nu, k0 = p.k0;
    if (a.skip_done) {   // every column final already
        bool done = true;
        for (int c = 0; c < nc; c++) done = done && ld_acquire(finish + k0 + c) == epoch;
        if (__syncthreads_and(done)) return false;
    }
    const int64_t lk = __ldg(LUp + k0 + nc - 1) + __ldg(nUp + k0 + nc - 1);   // L part of the last column
    const int nR = (int)(__ldg(LUp + k0 + nc) - lk), len = nu + nc + nR;
    const int32_t *Rk = LUi + lk;
    // the stage ring, then work vector and rows in shared memory; or, with
    // larger stages, the rows alone and the work vector in this CTA's
    // scratch; or both there
    const bool in_smem = (long long)len * (long long)(LD * sizeof(R) + 4) <=
                         smem_bytes - 4 * stage_bytes_of(kStageCap, (int)sizeof(R));
    const int cap = in_smem ? kStageCap : kStageCapBig, ns = in_smem ? 4 : 3;
    const int stage_bytes = stage_bytes_of(cap, (int)sizeof(R));
    unsigned char *area = smem + ns * stage_bytes;
    R *X;
    int32_t *rows;
    if (in_smem) {
        X = reinterpret_cast<R *>(area);
        rows = reinterpret_cast<int32_t *>(area + (size_t)len * LD * sizeof(R));
    } else {
        unsigned char *sc = a.pscratch + (size_t)blockIdx.x * a.pscratch_bytes;
        X = reinterpret_cast<R *>(sc);
        rows = reinterpret_cast<int32_t *>((long long)len * 4 <= smem_bytes - ns * stage_bytes
                                               ? area
                                               : sc + (size_t)len * LD * sizeof(R));
    }
    if (tid == 0) {
        for (int i = 0; i < kStagesMax; i++) {
            mbar_inval(&bars.full[i]);
            mbar_inval(&bars.empty[i]);
            mbar_init(&bars.full[i], 1);
            mbar_init(&bars.empty[i], kConsWarps);
        }
        sh.abort = 0;
        sh.step = 0;
        sh.next = 0;
    }
    for (int i = tid; i < nu + nc; i += kThreads) rows[i] = __ldg(a.prow + p.uoff + i);
    for (int i = tid; i < nR; i += kThreads) rows[nu + nc + i] = __ldg(Rk + i);
    {
        R z[LD];
#pragma unroll
        for (int c = 0; c < LD; c++) z[c] = R(0);
        for (int i = tid; i < len; i += kThreads) stv<R, LD>(X + (size_t)i * LD, z);
    }
    __syncthreads();
    for (int c = warp; c < nc; c += kWarps) {
        const int q = __ldg(a.Q + k0 + c);
        const int ae = __ldg(a.Ap + q + 1);
        for (int e = __ldg(a.Ap + q) + lane; e < ae; e += 32) X[(size_t)__ldg(a.amap + e) * LD + c] = (R)__ldg(a.Ax + e);
    }

    __syncthreads();

    // ---- the runs
    bool go = true;
    // a panel of the trailing block: its dependencies before the block
    const bool blk = k0 >= a.tb_p;
    const int nux = blk ? p.nux : nu;
    int run0 = 0;
    if constexpr (std::is_same<R, double>::value && LD == kPullLd) {
        if (p.pull > 0 && a.pull_start) {   // wide columns: their prefix row by row
            if (!pull_panel<LD>(ap, k0, X, rows, len, p.pull, epoch, wait, sh)) return true;
            run0 = p.runp;
        }
    }
    const int nruns = (blk ? p.nrunsx : p.nruns) - run0;
    int fills = 0;
    if (nruns > 0) {
        const PanelRun *runs = a.prun + p.roff + run0;
        if (warp < kConsWarps)
            go = panel_consume<R, LD>(X, in_smem, smem, stage_bytes, ns, sh, bars, a.ctl, warp, lane);
        else
            go = panel_produce<R>(a, runs, nruns, rows, nux, len, k0, smem, cap, stage_bytes, ns, sh, bars, epoch, wait,
                                  warp - kConsWarps, lane, fills);
    }
    if (__syncthreads_or(!go)) {
        // the one way out of an aborted panel.  Every producer waits for its
        // own copies, also one that had started its last stage when another
        // gave up: the CTA's next panel re-initializes the barriers and fills
        // the ring's memory, and a CTA must not exit before they land.
        if (warp >= kConsWarps) drain_slot(bars, warp - kConsWarps, fills, a.ctl);
        __syncthreads();
        return true;
    }

    const int64_t lup = lane < nc ? __ldg(LUp + k0 + lane) : 0;   // lane c: column c
    if (blk) {   // the block's rows go to the dense matrix
        R *const S = a.tb_S + (k0 - a.tb_p);
        for (int i = nux + tid; i < len; i += kThreads) {
            R *s = S + (int64_t)(rows[i] - a.tb_p) * a.tb_ld;
            for (int c = 0; c < nc; c++) s[c] = X[(size_t)i * LD + c];
        }
        store_u_rows<R, LD>(a, p, nux, X, LUx, lup, warp, lane);
        return false;
    }
    // ---- the diagonal block (warp 0), its columns announced in sh.step as
    // they are done; the other warps follow with the L rows below the block,
    // 32 rows at a time
    const int nuk = lane < nc ? __ldg(nUp + k0 + lane) : 0;
    if (warp == 0) {
        const int q = lane & 7, c0 = lane >> 3, c1 = c0 + 4;   // this lane's entries (q, c0), (q, c1)
        R v0 = (q < nc && c0 < nc) ? X[(size_t)(nu + q) * LD + c0] : R(0);
        R v1 = (LD > 4 && q < nc && c1 < nc) ? X[(size_t)(nu + q) * LD + c1] : R(0);
        for (int s = 0; s < nc; s++) {
            const R src = s < 4 ? v0 : v1;
            const R d = __shfl_sync(kFull, src, s + 8 * (s & 3));
            const R xq = __shfl_sync(kFull, src, q + 8 * (s & 3));
            const R u0 = __shfl_sync(kFull, v0, s + 8 * c0);
            const R u1 = __shfl_sync(kFull, v1, s + 8 * c0);
            if (q == s) {   // row s of U and the diagonal are final
                sh.D[q * kPanelMax + c0] = v0;
                if (LD > 4) sh.D[q * kPanelMax + c1] = v1;
            }
            const R inv = recip(d);
            if (lane == 0) sh.inv[s] = inv;
            __syncwarp();
            if (lane == 0) st_release_cta(&sh.step, s + 1);
            const R l = xq * inv, n0 = fma(-u0, l, v0);
            v0 = q > s && c0 > s ? n0 : v0;
            if (LD > 4) {
                const R n1 = fma(-u1, l, v1);
                v1 = q > s && c1 > s ? n1 : v1;
            }
            if (q > s && c0 == 0) sh.Lb[q * kPanelMax + s] = l;
        }
        // below the diagonal: the unscaled values
        if (q > c0) sh.D[q * kPanelMax + c0] = v0;
        if (LD > 4 && q > c1) sh.D[q * kPanelMax + c1] = v1;
        __syncwarp();
        // the block's U rows, diagonals and L rows
        const unsigned mk = lane < nc ? __ldg(a.pmask + p.uoff + nu + lane) : 0u;
        for (int c = 0; c < nc; c++) {
            const unsigned b = __ballot_sync(kFull, lane <= c && ((mk >> c) & 1u));
            const int64_t col = __shfl_sync(kFull, lup, c) + __shfl_sync(kFull, nuk, c);
            if ((b >> lane) & 1u) LUx[col - __popc(b >> lane)] = sh.D[lane * kPanelMax + c];
            if (lane > c && lane < nc) LUx[col + (lane - c - 1)] = sh.Lb[lane * kPanelMax + c];
        }
    }
    unsigned long long mx[LD];
#pragma unroll
    for (int c = 0; c < LD; c++) mx[c] = 0;
    const int64_t out = lup + nuk + (nc - 1 - lane);   // lane c: column c's first row below the block
    auto take = [&]() -> int {   // this lane's next row
        int r = 0;
        if (lane == 0) r = atomicAdd(&sh.next, 32);
        return __shfl_sync(kFull, r, 0) + lane;
    };
    const R *XL = X + (size_t)(nu + nc) * LD;
    int r = take();
    R x[LD];
    if (r < nR) ldv<R, LD>(XL + (size_t)r * LD, x);
    while (r - lane < nR) {
        // the next rows' values in flight behind these rows' arithmetic
        // (panels of eight columns have few rows)
        const int rn = take();
        R xn[LD];
        if (LD == 4 && rn < nR) ldv<R, LD>(XL + (size_t)rn * LD, xn);
        const bool in = r < nR;
#pragma unroll
        for (int s = 0; s < LD; s++) {
            if (s < nc) {
                for (long long it = 0; ld_acquire_cta(&sh.step) <= s && it < kBarTries; ++it) {}   // warp 0 is on its way
                __syncwarp();
                const int64_t o = __shfl_sync(kFull, out, s);
                if (in) {
                    const unsigned long long key = abs_key(x[s]);
                    mx[s] = key > mx[s] ? key : mx[s];
                    const R l = x[s] * sh.inv[s];
                    LUx[o + r] = l;
#pragma unroll
                    for (int c = s + 1; c < LD; c++)
                        if (c < nc) x[c] = fma(-sh.D[s * kPanelMax + c], l, x[c]);
                }
            }
        }
        r = rn;
        if (LD == 4) {
#pragma unroll
            for (int c = 0; c < LD; c++) x[c] = xn[c];
        } else if (r < nR) {
            ldv<R, LD>(XL + (size_t)r * LD, x);
        }
    }
#pragma unroll
    for (int c = 0; c < LD; c++) {
        if (c < nc) {
            const unsigned long long m = warp_max_key(mx[c]);
            if (lane == 0) sh.mx[warp][c] = m;
        }
    }
    __syncthreads();

    // ---- pivot checks (lane c of warp 0: column c) and publication
    if (warp == 0) {
        bool pass = true;
        // column c = lane & 7: four lanes share its eight warps' maxima and
        // the rows of the diagonal block
        unsigned long long m = 0;
        {
            const int c = lane & 7, h = lane >> 3;
            if (c < nc) {
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    const unsigned long long v = sh.mx[2 * h + i][c];
                    const int r = 2 * h + i;
                    const unsigned long long key = r > c && r < nc ? abs_key(sh.D[r * kPanelMax + c]) : 0ull;
                    m = max(m, max(v, key));
                }
            }
            m = max(m, __shfl_xor_sync(kFull, m, 8));
            m = max(m, __shfl_xor_sync(kFull, m, 16));
        }
        if (lane < nc) {
            pass = check_pivot(a, k0 + lane, sh.D[lane * kPanelMax + lane], key_abs(m, R(0)));
        }
        const unsigned ok = __ballot_sync(kFull, pass);
        if (lane == 0) sh.pass = ok;
        if (ok != kFull) {
            const int f = __ffs(~ok) - 1;   // the first failing column
            if (lane == 0) {
                if (!a.no_stop) atomicExch(&a.ctl->interrupted, 1);
                atomicMin(&a.ctl->first_bad, k0 + f);
            }
            if (!a.no_stop && lane < f) st_release(finish + k0 + lane, epoch);
        } else if (lane < nc) {
            st_release(finish + k0 + lane, epoch);   // the barrier above orders the CTA's stores before it
        }
    }
    store_u_rows<R, LD>(a, p, nu, X, LUx, lup, warp, lane);   // no column of this launch reads them
    __syncthreads();
    if (sh.pass == kFull || !a.no_stop) return false;
    // no-stop mode: a failed column is stored unnormalized (the columns after
    // it are meaningless, whatever they hold)
    for (int r = tid; r < nR; r += kThreads) {
        R x[LD];
        ldv<R, LD>(X + (size_t)(nu + nc + r) * LD, x);
#pragma unroll
        for (int s = 0; s < LD; s++) {
            if (s < nc) {
                if (!((sh.pass >> s) & 1u)) LUx[__ldg(LUp + k0 + s) + __ldg(nUp + k0 + s) + (nc - 1 - s) + r] = x[s];
                const R l = x[s] * sh.inv[s];
#pragma unroll
                for (int c = s + 1; c < LD; c++)
                    if (c < nc) x[c] = fma(-sh.D[s * kPanelMax + c], l, x[c]);
            }
        }
    }
    if (warp == 0)
        for (int c = 0; c < nc; c++) {
            const int64_t col = __shfl_sync(kFull, lup, c) + __shfl_sync(kFull, nuk, c);
            if (!((sh.pass >> c) & 1u) && lane > c && lane < nc) LUx[col + (lane - c - 1)] = sh.D[lane * kPanelMax + c];
        }
    __syncthreads();
    if (tid < nc) st_release(finish + k0 + tid, epoch);
    return false;
}

// panel `id` by the whole CTA; true = stop
template <typename R>
__device__ __forceinline__ bool run_panel(const RefactorArgsT<R> *ap, int id, unsigned char *smem, int smem_bytes,
                                          PanelShared<R> &sh, PanelBars &bars, int epoch, bool wait)
{
    if (__ldg(&ap->pan[id].nc) > 4) return col_panel<R, 8>(ap, id, smem, smem_bytes, sh, bars, epoch, wait);
    return col_panel<R, 4>(ap, id, smem, smem_bytes, sh, bars, epoch, wait);
}

}  // namespace

}  // namespace gblu
