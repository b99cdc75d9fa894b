// Column-distributed leaf of single inversions (L <= 256): the Gauss-Jordan
// of leaf_core.cuh with the block's columns, not its rows, spread over a
// thread-block cluster.
//
// A pivot step is a serial chain (the pivot column's last update, the search
// over its rows, 1/pivot, the next column's update), and on GB300 every FP64
// warp instruction holds its SM sub-partition for 64 cycles, so the chain is
// bound by its own dependent FP64 operations and by whatever lies between
// them.  With rows spread over CTAs (the previous form) that was an exchange
// across the cluster and two block barriers per step: 4080 cycles a step at
// L = 128 on 16 CTAs.  Here every warp owns one column, 32 T rows of it in
// registers, T per lane, and every CTA `w` adjacent columns (a panel):
//  - the pivot search of column k is one warp's own argmax, with no block or
//    cluster barrier;
//  - the step's multipliers (column k before the step), pivot row and
//    1/pivot go into a slot that the warps of the same CTA read from shared
//    memory, and one bulk copy per peer carries to the other CTAs, completing
//    on the slot's mbarrier; every warp updates its column when it sees the
//    slot, so only the first column of the next panel waits for another CTA
//    (once per w steps), and the CTAs to the right follow at their own pace.
//    The owner stores the next panel's copy itself and leaves the others
//    (about 50 cycles each to issue) to one more warp, the sender;
//  - each lane computes the reciprocal of its own best row, on the integer
//    units, while the warp finds the winner among the lanes.
// The arithmetic on every entry, the pivot choice and the order of the
// updates are those of the other forms, so the results are the same bit for
// bit.
//
// Measured (one leaf, back-to-back launches, rows over the cluster before):
// L = 64: 39 us (130 before), L = 128: 104 us (257), L = 256: 357 us (620).
// Inside a panel a step takes 830 / 1010 / 1480 cycles at T = 1 / 2 / 4, of
// which (T = 4) 105 from the publishing warp's arrive to the next warp's
// wake-up, 190 for the scaled pivot entry, 460 for the four dependent-issue
// FMAs (64 cycles each alone, 80 and more with the other sub-partitions at
// work), 170 of bookkeeping and 520 for the search and reciprocal; the first
// column of a panel takes about 600 more.
//
// Slots form a ring of P panels.  The owner of panel q may overwrite panel
// q - P once every warp of the cluster has finished with it: each warp says
// so on the owner's credit barrier (used once per CTA, since a CTA owns one
// panel).  Every wait is bounded.
#pragma once
#include "leaf_core.cuh"
#include "tc_ptx.cuh"

namespace spin {
namespace {

constexpr int kColMaxL = 256;       // 8 rows per lane
constexpr int kColMaxCtas = 16;
constexpr int kColPanelsInRing = 4;  // slots of this many panels (33 KB at L = 128)

// Exchange settings: the wait limit, and (tests only) a CTA that sends
// nothing, so that the others' waits run out.
constexpr uint64_t kLeafWaitLimitNs = 4000000000ull;
struct LeafWait {
    uint64_t limit_ns = kLeafWaitLimitNs;
    int mute_rank = -1;
};

// One lane's wait (the clock is read only after some polls: reading it takes
// longer than a poll).
__device__ __forceinline__ bool slot_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns,
                                          const volatile int* quit = nullptr) {
    for (int i = 0; i < 32; i++)
        if (tc::mbar_try_wait_cluster(bar, parity)) return true;
    const uint64_t t0 = tc::globaltimer_ns();
    for (uint32_t spins = 1;; spins++) {
        if (tc::mbar_try_wait_cluster(bar, parity)) return true;
        if (quit != nullptr && *quit) return false;
        if ((spins & 63u) == 0 && tc::globaltimer_ns() - t0 > limit_ns) return false;
    }
}
// A warp's wait: the same answer in every lane.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns,
                                          const volatile int* quit = nullptr) {
    return __all_sync(FULL, slot_wait(bar, parity, limit_ns, quit));
}

struct ColSmemLayout {
    size_t full_off, credit_off, send_off, go_off, slot_off, pcol_off, stage_off, total;
    int slot_doubles;  // header (1/pivot; pivot row and its position) + the multipliers of 32 T rows
    int stage_ld;      // leading dimension of the staged output columns (odd: no bank conflicts)
};

// Rows per lane for order L.
__host__ __device__ inline int col_rows(int L) { return L <= 32 ? 1 : L <= 64 ? 2 : L <= 128 ? 4 : 8; }

__host__ __device__ inline ColSmemLayout col_layout(int L, int w) {
    ColSmemLayout s;
    auto a16 = [](size_t v) { return (v + 15) & ~(size_t)15; };
    size_t off = 0;
    s.full_off = off; off += (size_t)kColPanelsInRing * w * sizeof(uint64_t);
    s.credit_off = off; off += sizeof(uint64_t);
    s.send_off = off; off += (size_t)w * sizeof(uint64_t);
    s.go_off = off; off += 2 * (size_t)w * w * sizeof(uint64_t);
    s.pcol_off = off; off += 2 * (size_t)L * sizeof(int);  // pivot row of each step, step of each row
    s.slot_off = off = a16(off);
    s.slot_doubles = 2 + 32 * col_rows(L);  // an even count: slots start on 16-byte boundaries
    s.stage_ld = L | 1;
    const size_t ring = (size_t)kColPanelsInRing * w * s.slot_doubles * sizeof(double);
    const size_t stage = (size_t)w * s.stage_ld * sizeof(double);  // reuses the ring at the end
    s.stage_off = s.slot_off;
    off += ring > stage ? ring : stage;
    s.total = a16(off);
    return s;
}

// The words of x, opaque to the compiler: a test of the bits for zero written
// on the 64-bit value is turned into a floating-point compare, which costs an
// FP64-pipe instruction (64 cycles) each.
__device__ __forceinline__ void words_of(double x, unsigned& lo, unsigned& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "d"(x));
}
__device__ __forceinline__ bool is_zero_bits(double x) {
    unsigned lo, hi;
    words_of(x, lo, hi);
    return ((hi << 1) | lo) == 0;
}

// 1/x correctly rounded, on the integer units: a double-precision operation
// takes 64 cycles here and queues behind the other warp's of the
// sub-partition, an integer one about 5.  Newton's iteration y <- y + y e,
// e = 1 - m y, on the significand m in [1, 2) as a 64-bit fraction: a 23-bit
// estimate from the FP32 reciprocal, two iterations (46 and 63 bits).  The
// result is known to a few units of 2^-64, so rounding it to 53 bits is
// right unless it lies that close to a rounding boundary.  Returns false
// then, and for zeros, subnormals, infinities, NaN, powers of two and
// results near the ends of the exponent range: the caller takes __drcp_rn.
__device__ __forceinline__ bool recip_int(double x, double* out) {
    unsigned lo, hi;
    words_of(x, lo, hi);
    const unsigned ex = (hi >> 20) & 0x7FFu;
    const uint64_t M = (1ull << 63) | ((uint64_t)(hi & 0xFFFFFu) << 43) | ((uint64_t)lo << 11);  // m 2^63
    float y0;  // in (1/2, 1]
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(__uint_as_float(0x3F800000u | (unsigned)((M << 1) >> 41))));
    const unsigned Y0 = y0 < 1.0f ? (__float_as_uint(y0) | 0x800000u) << 8 : 0xFFFFFFFFu;  // y 2^32
    // e 2^63, |e| < 2^-21; its top 30 bits suffice here
    const int64_t e0 = (int64_t)((1ull << 63) - __umul64hi(M, (uint64_t)Y0 << 32));
    const uint64_t y1 = ((uint64_t)Y0 << 32) + (uint64_t)(((int64_t)(int)(e0 >> 12) * (int64_t)(uint64_t)Y0) >> 19);
    const int64_t e1 = (int64_t)((1ull << 63) - __umul64hi(M, y1));  // |e| < 2^-40: fits 32 bits
    const uint64_t y2 = y1 + (uint64_t)(((int64_t)(int)e1 * (int64_t)(y1 >> 32)) >> 31);
    const unsigned tail = (unsigned)y2 & 0x7FFu;
    const uint64_t q = (y2 + 0x400u) >> 11;  // in (2^52, 2^53): the significand of 1/m, times 2
    const unsigned eo = 2045u - ex;          // biased exponent of 1/x (m > 1)
    *out = __longlong_as_double((long long)(((uint64_t)(hi & 0x80000000u) << 32) |
                                            (((uint64_t)eo << 52) + (q - (1ull << 52)))));
    return ex - 2u < 2041u && (y2 >> 63) != 0 && (q >> 53) == 0 && tail - 0x3F0u > 0x20u && (M << 1) != 0;
}

// v[t], by a tree of selects (t is the same in every lane; an indexed read
// would put v in local memory).
template <int T>
__device__ __forceinline__ double select_row(const double (&v)[T], int t) {
    double a[T];
#pragma unroll
    for (int i = 0; i < T; i++) a[i] = v[i];
#pragma unroll
    for (int h = 1; h < T; h <<= 1) {
        const bool odd = (t & h) != 0;
#pragma unroll
        for (int i = 0; i + h < T; i += 2 * h) a[i] = odd ? a[i + h] : a[i];
    }
    return a[0];
}

// Columns per CTA (warps) for order L on at most cmax CTAs: few CTAs for
// small blocks, since every panel boundary costs a copy's latency.
constexpr int kColMinPanel = 4;
__host__ __device__ inline int col_panel(int L, int cmax) {
    const int w = (L + cmax - 1) / cmax;
    return w > kColMinPanel ? w : kColMinPanel;
}
template <int T>
constexpr int kColMaxWarps = T == 1 ? 8 : 16;

// One bulk copy of a slot to the same place in CTA `peer`, completing on its
// barrier there.
__device__ __forceinline__ void send_slot(double* slot, uint64_t* bar, uint32_t bytes, int peer) {
    const uint32_t a = tc::smem_u32(slot);
    tc::bulk_copy_to_peer(tc::mapa_u32(a, (uint32_t)peer), a, bytes, tc::mapa_u32(tc::smem_u32(bar), (uint32_t)peer));
}

// T rows per lane: row lane + 32 t.  One warp per column, w warps per CTA,
// and the sender.
template <int T>
__device__ __forceinline__ void leaf_gj_col_body(const double* __restrict__ src, int64_t lds, double* __restrict__ dst,
                                                 int64_t ldd, int L, int w, int32_t* info, int leaf_index,
                                                 const LeafWait& lw) {
    constexpr int P = kColPanelsInRing;
    const int rank = (int)tc::cluster_ctarank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nact = (L + w - 1) / w;  // CTAs that own columns
    const int col = rank * w + warp;
    const bool own = warp < w && col < L;

    __shared__ int quit;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const ColSmemLayout lay = col_layout(L, w);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw + lay.full_off);  // [P][w]
    uint64_t* credit = reinterpret_cast<uint64_t*>(smem_raw + lay.credit_off);
    uint64_t* send = reinterpret_cast<uint64_t*>(smem_raw + lay.send_off);  // [w] slots of this CTA's panel
    uint64_t* go = reinterpret_cast<uint64_t*>(smem_raw + lay.go_off);      // [2][step][warp], see follow
    int* prow_of = reinterpret_cast<int*>(smem_raw + lay.pcol_off);  // [L] pivot row of step k
    int* step_of = prow_of + L;                                      // [L] step that took row i
    double* slots = reinterpret_cast<double*>(smem_raw + lay.slot_off);
    constexpr int SD = 2 + 32 * T;
    const int Lp = (L + 1) & ~1;
    const uint32_t slot_bytes = (uint32_t)(2 + Lp) * sizeof(double);  // what is sent of a slot

    // Slot barriers: one arrival each (this CTA's owner warp, or the arming
    // below, which also expects the copy's bytes).  The credit barrier takes
    // one arrival from every warp that owns a column.
    for (int i = tid; i < P * w; i += blockDim.x) tc::mbar_init(&full[i], 1);
    if (tid == 0) {
        tc::mbar_init(credit, (uint32_t)L);
        quit = 0;
    }
    if (tid < w) tc::mbar_init(&send[tid], 1);
    for (int i = tid; i < 2 * w * w; i += blockDim.x) tc::mbar_init(&go[i], 1);
    tc::fence_mbar_init();
    __syncthreads();
    for (int i = tid; i < P * w; i += blockDim.x)
        if (i / w != rank && i < L) tc::mbar_arrive_expect_tx(&full[i], slot_bytes);

    double v[T];
    int pos[T];  // logical position of each row (the row interchanges are bookkeeping only)
#pragma unroll
    for (int t = 0; t < T; t++) {
        const int i = lane + 32 * t;
        v[t] = (own && i < L) ? src[(size_t)i * lds + col] : 0.0;
        pos[t] = i < L ? i : -1;  // -1: never eligible
    }
    tc::cluster_sync_all();  // every CTA runs, its barriers armed, before the first remote write

    bool timed_out = false;
    int done = 0;
    if (own) {
        const int own0 = rank * w, own1 = min(L, own0 + w);  // this CTA's panel
        int q = 0, s = 0;                                    // step k = q w + s: panel q, slot s of it
        double* slot = slots;
        uint64_t* bar = full;
        uint32_t par = 0;
        int owed = -1;  // a credit put off: the CTA it goes to
        auto give_credit = [&](int to) {
            __syncwarp();
            if (lane == 0) tc::mbar_arrive_cluster(tc::mapa_u32(tc::smem_u32(credit), (uint32_t)to));
        };
        auto advance = [&]() {
            slot += SD;
            bar++;
            if (++s < w) return;
            // the panel is finished here: its slots may be used again by
            // panel q + P, whose owner waits for this from every warp
            const int qn = q + P;
            if (qn < nact) {
                if (warp == 0 && qn != rank && lane < w && qn * w + lane < L)
                    tc::mbar_arrive_expect_tx(&full[(q % P) * w + lane], slot_bytes);
                // (a release at cluster scope takes about 900 cycles: not
                // between the warp that leads the next step and its search)
                if (warp == 0 && q + 1 == rank)
                    owed = qn;
                else
                    give_credit(qn);
            }
            s = 0;
            if (++q % P == 0) {
                slot = slots;
                bar = full;
                par ^= 1u;
            }
        };
        // Steps [k, k1) of other columns; false: stop (a bad pivot or a wait
        // that ran out).  An SM's FP64 units take one warp instruction per
        // 16 to 20 cycles together, each (of warps x, x + 4, ...) one per 64:
        // in the CTA's own panel and the one before it the warps of a
        // sub-partition take a step's update in the order in which their
        // columns come up, each waiting for the one before it, so that the
        // next pivot column is not held up by one that can wait.
        const int ncol = own1 - own0;
        auto follow = [&](int k, int k1) -> bool {
            for (; k < k1; k++) {
                uint64_t* mine = nullptr;  // told when this step's update is done
                uint64_t* wait = bar;
                uint32_t wpar = par;
                if (w > 4 && (q == rank || q + 1 == rank)) {
                    int before = warp - 4;
                    if (q == rank) {
                        if (warp < s)  // a past column: after the last of those to come
                            before = warp + ((ncol - 1 - warp) & ~3);
                        if (before <= s) before = -1;
                    }
                    uint64_t* g = go + (size_t)((q == rank ? 0 : w) + s) * w;
                    mine = g + warp;
                    if (before >= 0) {
                        wait = g + before;
                        wpar = 0;
                    }
                }
                if (!warp_wait(wait, wpar, lw.limit_ns)) {
                    timed_out = true;
                    return false;
                }
                const double2 head = *reinterpret_cast<const double2*>(slot);
                double f[T];
#pragma unroll
                for (int t = 0; t < T; t++) f[t] = slot[2 + lane + 32 * t];
                const int p = __double2loint(head.y), ppos = __double2hiint(head.y);
                if (p < 0) {  // a bad pivot: every warp of the cluster leaves at this step
                    // (a sender whose panel never comes, too; this panel's
                    // own finds the bad slot itself and sends it first)
                    if (tid == 0 && q != rank) *(volatile int*)&quit = 1;
                    if (mine != nullptr && lane == 0) tc::mbar_arrive(mine);
                    return false;
                }
                const double pj = __shfl_sync(FULL, select_row<T>(v, p >> 5), p & 31) * head.x;
                // every FMA before the first use of one: a use in between
                // would hold the next FMA back for the whole latency
                double nv[T];
#pragma unroll
                for (int t = 0; t < T; t++) nv[t] = fma(-f[t], pj, v[t]);
#pragma unroll
                for (int t = 0; t < T; t++) {
                    const int i = lane + 32 * t;
                    if (pos[t] == k) pos[t] = ppos;
                    if (i == p) pos[t] = k;
                    v[t] = i == p ? pj : (is_zero_bits(f[t]) ? v[t] : nv[t]);
                }
                if (mine != nullptr && lane == 0) tc::mbar_arrive(mine);
                if (tid == 0) prow_of[k] = p;
                done = k + 1;
                advance();
            }
            return true;
        };
        // Columns before this one, this one, columns after it.
        bool led = false;
        int k = 0;
        while (follow(k, led ? L : col) && !led) {
            k = col;
            if (s == 0 && q >= P && !warp_wait(credit, 0, lw.limit_ns)) {
                timed_out = true;
                break;
            }
            // the high words of |v| decide unless two rows tie in them
            int h[T], m = -1;
#pragma unroll
            for (int t = 0; t < T; t++) {
                unsigned lo, hi;
                words_of(v[t], lo, hi);
                h[t] = pos[t] >= k ? (int)(hi & 0x7fffffffu) : -1;
                m = max(m, h[t]);
                slot[2 + lane + 32 * t] = v[t];
            }
            const int mh = __reduce_max_sync(FULL, m);
            double val = 1.0;
            int about = 0;  // of this lane's best row: its position, row, whether others tie with it
            int seen = 0;   // (position 0 of row 0 is a word of zeros too)
#pragma unroll
            for (int t = 0; t < T; t++)
                if (h[t] == m) {
                    val = v[t];
                    about = pos[t] | (lane + 32 * t) << 10 | seen;
                    seen = 1 << 30;
                }
            double inv;
            int quick = recip_int(val, &inv);
            asm volatile("" : "+d"(inv), "+r"(quick));  // here, beside the search: not sunk below it
            const unsigned top = __ballot_sync(FULL, m == mh);
            const int from = __ffs(top) - 1;
            inv = __shfl_sync(FULL, inv, from);
            about = __shfl_sync(FULL, quick ? about : about | 1 << 29, from);
            int p = (about >> 10) & 0x3ff, cpos = about & 0x3ff;
            if ((top & (top - 1)) == 0 && !(about >> 30) && mh > 0 && mh < 0x7ff00000) {
                if (about >> 29) inv = __drcp_rn(__shfl_sync(FULL, val, from));  // beyond the quick reciprocal's range
            } else {
                // ties in the high word, zeros, subnormals, infinities, NaN
                uint64_t key = 0;
                val = 0.0;
                int bpos = INT_MAX, bphys = -1;
#pragma unroll
                for (int t = 0; t < T; t++) {
                    if (h[t] < 0) continue;
                    const uint64_t mag = (uint64_t)__double_as_longlong(v[t]) & ~(1ull << 63);
                    const uint64_t kk = mag > kInfBits ? kInfBits : mag;
                    if (kk > key || (kk == key && pos[t] < bpos)) {
                        key = kk;
                        val = v[t];
                        bpos = pos[t];
                        bphys = lane + 32 * t;
                    }
                }
                const Cand c = warp_argmax(key, val, 0.0, bpos, bphys);
                inv = __drcp_rn(c.val);
                cpos = c.pos;
                p = bad_pivot(c) ? -1 : c.phys;
            }
            __syncwarp();  // every lane's part of the column is in the slot
            if (lane == 0) {
                *reinterpret_cast<double2*>(slot) = make_double2(inv, __hiloint2double(cpos, p));
                tc::mbar_arrive(bar);  // this CTA's warps
            }
            if (nact > 1 && rank != lw.mute_rank) {
                // the next panel's CTA waits for this one at the panel's
                // last step: remote stores, which need no proxy fence and
                // arrive sooner than a bulk copy
                const uint32_t peer = (uint32_t)((rank + 1) % nact);
                const uint32_t to = tc::mapa_u32(tc::smem_u32(slot), peer), rbar = tc::mapa_u32(tc::smem_u32(bar), peer);
                if (lane == 0)
                    tc::st_async_v2_b64(to, (uint64_t)__double_as_longlong(inv),
                                        (uint64_t)(uint32_t)cpos << 32 | (uint32_t)p, rbar);
#pragma unroll
                for (int t = 0; t < T; t++)
                    if (lane + 32 * t < Lp)
                        tc::st_async_b64(to + 16 + 8 * (lane + 32 * t), (uint64_t)__double_as_longlong(v[t]), rbar);
            }
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&send[s]);  // the sender: the other CTAs
            if (owed >= 0) give_credit(owed);
            if (p < 0) {
                if (lane == 0) record_failure(info, SPIN_ERR_SINGULAR, leaf_index, k);
                break;
            }
#pragma unroll
            for (int t = 0; t < T; t++) {
                const int i = lane + 32 * t;
                const double f = v[t];
                v[t] = i == p ? inv : (is_zero_bits(f) ? f : fma(-f, inv, 0.0));
                if (pos[t] == k) pos[t] = cpos;
                if (i == p) pos[t] = k;
            }
            if (tid == 0) prow_of[k] = p;
            done = ++k;
            advance();
            led = true;
        }
        if (timed_out && lane == 0) record_failure(info, SPIN_ERR_TIMEOUT, leaf_index, done);
    } else if (warp == w && nact > 2) {
        // the sender: this CTA's slots to every CTA but the next one
        for (int s = 0; s < w && rank * w + s < L; s++) {
            if (!warp_wait(&send[s], 0, lw.limit_ns, &quit)) break;
            double* slot = slots + (size_t)((rank % P) * w + s) * SD;
            if (lane < nact - 2 && rank != lw.mute_rank)
                send_slot(slot, &full[(rank % P) * w + s], slot_bytes, (rank + 2 + lane) % nact);
            if (__double2loint(slot[1]) < 0) break;  // a bad pivot: the last slot
        }
    }
    const int any_late = __syncthreads_or(timed_out);
    // nothing is sent after this: every CTA is through its last step, so the
    // ring may be overwritten and a CTA may leave
    tc::cluster_sync_all();
    if (any_late) {
        // copies to this CTA that nobody waited for (a broken exchange only):
        // let them land before its shared memory goes away
        const uint64_t t0 = tc::globaltimer_ns();
        while (tc::globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    // Step k's row is row k of the inverse, and column k of the eliminated
    // block is the inverse's column p_k (the row interchanges undone as
    // column interchanges): stage the panel, then write runs of a row.
    double* stage = reinterpret_cast<double*>(smem_raw + lay.stage_off);
    const bool complete = done == L;
    int nonfinite = 0;
    if (own && complete) {
#pragma unroll
        for (int t = 0; t < T; t++) {
            const int i = lane + 32 * t;
            if (i < L) {
                stage[(size_t)warp * lay.stage_ld + i] = v[t];
                nonfinite |= !isfinite(v[t]);
                if (warp == 0) step_of[i] = pos[t];
            }
        }
    }
    if (__syncthreads_or(own && !complete)) return;  // failure already recorded; X is undefined
    if (__syncthreads_or(nonfinite) && tid == 0) record_failure(info, SPIN_ERR_SINGULAR, leaf_index, L);
    const int c0 = rank * w, nc = min(w, L - c0);
    if (nc > 0)
        for (int idx = tid; idx < nc * L; idx += blockDim.x) {
            const int r = idx / nc, c = idx % nc;
            dst[(size_t)step_of[r] * ldd + prow_of[c0 + c]] = stage[(size_t)c * lay.stage_ld + r];
        }
}

template <int T>
__global__ void __launch_bounds__(32 * (kColMaxWarps<T> + 1), 1)
leaf_gj_col_kernel(const double* __restrict__ src, int64_t lds, double* __restrict__ dst, int64_t ldd, int L, int w,
                   int32_t* info, int leaf_index, LeafWait lw) {
    leaf_gj_col_body<T>(src, lds, dst, ldd, L, w, info, leaf_index, lw);
}

// Problem blockIdx.y of a batch, on a cluster of its own.
template <int T>
__global__ void __launch_bounds__(32 * (kColMaxWarps<T> + 1), 1)
leaf_gj_col_batched_kernel(BatchView src, BatchView dst, int L, int w, int32_t* info_base, int leaf_index) {
    const int z = blockIdx.y;
    const int64_t lds = src.ld_of(z), ldd = dst.ld_of(z);
    leaf_gj_col_body<T>(src.ptr(z, lds), lds, const_cast<double*>(dst.ptr(z, ldd)), ldd, L, w,
                        info_base + (int64_t)z * INFO_WORDS, leaf_index, LeafWait());
}

}  // namespace
}  // namespace spin
