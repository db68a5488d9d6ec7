// KV compaction: keep the system-prompt, Nexus and current-turn rows of every
// sequence and layer, drop the history bodies.
//
// Retention rule (SONIC Sec. 3.2 "Historical Body Removal" and App. C: the
// effective context is I_sys + Nexus state + current query): a row is kept
// iff its role is not BODY; kept rows keep their order.
//
// Launches, none of which needs a host round trip.  Calls of up to 524,288 rows:
//   keep_plan     the whole scan in one launch (see there);
//   kv_gather     below.
// Larger calls:
//   keep_count    one block per (chunk, sequence), each sequence cut into
//                 kChunks pieces: kept rows of the piece (and a layout check
//                 when segment numbers are given);
//   keep_bases    one block: per-sequence totals and their exclusive scan
//                 (with the reserve rows) -> offsets, ret_len, capacity check;
//   keep_scatter  one block per (chunk, sequence): its output base (the
//                 sequence's offset plus the pieces before it), then a block
//                 prefix scan of the keep flags from warp-shuffle scans,
//                 writing the source row of every output row (-1 in reserve
//                 rows);
//   kv_gather     all layers, K and V: 16-byte vector copy of every kept row
//                 to its output row, grid-stride over rows of each layer.
#include <algorithm>
#include <climits>

#include "sonic_dev.cuh"
#include "sonic_host.h"

namespace sonic {
namespace {

constexpr int kScanThreads = 512;
constexpr int kChunks = 64;  // pieces per sequence in the scans
// the single-launch scan (keep_plan): its largest call (rows; rows x sequences, as every
// block looks at the sequences before its own), and rows per piece
constexpr int kPlanRows = 1 << 19;
constexpr int64_t kPlanWork = 1 << 25;
constexpr int kPlanRowsPerThread = 4;
constexpr int kPlanStep = kScanThreads * kPlanRowsPerThread;  // rows per piece, at least
// rows of a long sequence's pieces; those of the others reach twice as many (where all rows are
// more than half of kPlanRows, both are twice that: a block reads up to all role bytes, at its
// SM's L2 rate, so more blocks do not pay)
__host__ __device__ constexpr int long_piece(int total) {
    return total > kPlanRows / 2 ? 2 * kPlanStep : kPlanStep;
}
constexpr int kSlice = 512;  // rows per slice where sequences share rows (or twice that)

// Rows of sequence (start, len), or 0 when they fall outside [0, total): such a
// sequence is refused, keeps nothing and is never read.
__device__ __forceinline__ int32_t seq_rows(int32_t start, int32_t len, int32_t total) {
    return (start < 0 || len < 0 || (int64_t)start + len > total) ? 0 : len;
}

// Rows [*lo, *hi) of piece c of a sequence of len rows (32-row aligned pieces).
__device__ __forceinline__ void piece(int32_t len, int c, int32_t *lo, int32_t *hi) {
    const long long ch = (((long long)len + kChunks - 1) / kChunks + 31) & ~31LL;
    *lo = (int32_t)min((long long)len, c * ch);
    *hi = (int32_t)min((long long)len, (c + 1) * ch);
}

__global__ void __launch_bounds__(kScanThreads)
keep_count_kernel(const uint8_t *__restrict__ role, const int32_t *__restrict__ seg,
                  const int32_t *__restrict__ k_start, const int32_t *__restrict__ k_len,
                  int32_t total, int32_t *__restrict__ counts, int32_t *status) {
    const int c = blockIdx.x, b = blockIdx.y;
    const int32_t start = k_start[b];
    const int32_t len = seq_rows(start, k_len[b], total);
    if (c == 0 && threadIdx.x == 0 && len != k_len[b]) set_status(status, SONIC_ERR_INVALID_ARGUMENT);
    int32_t lo, hi;
    piece(len, c, &lo, &hi);
    int n = 0;
    bool bad = false;
    for (int32_t t = lo + threadIdx.x; t < hi; t += blockDim.x) {
        uint8_t r = role[start + t];
        n += (r != SONIC_ROLE_BODY);
        bad |= (r > SONIC_ROLE_CURR);
        if (seg != nullptr) {
            int32_t sv = seg[start + t];
            bad |= (r == SONIC_ROLE_BODY && sv <= 0);
            if (t > 0) bad |= (sv < seg[start + t - 1]);
        }
    }
    // block reduction
    __shared__ int red[kScanThreads / 32];
    __shared__ int bad_any;
    if (threadIdx.x == 0) bad_any = 0;
    __syncthreads();
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = n;
    if (bad) bad_any = 1;
    __syncthreads();
    if (threadIdx.x == 0) {
        int sum = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += red[w];
        counts[b * kChunks + c] = sum;
        if (bad_any) set_status(status, SONIC_ERR_LAYOUT);
    }
}

// Inclusive warp scan of v (warp-shuffle).
__device__ __forceinline__ int warp_inclusive_scan(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Exclusive scan over the sequences of (kept rows + reserve): one block.
__global__ void __launch_bounds__(kScanThreads)
keep_bases_kernel(const int32_t *__restrict__ counts, const int32_t *__restrict__ reserve,
                  int32_t B, int32_t capacity, long long *__restrict__ seq_base,
                  int32_t *__restrict__ offsets, int32_t *__restrict__ ret_len,
                  int32_t *status) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = kScanThreads / 32;
    __shared__ long long warp_tot[kWarps];
    long long running = 0;
    for (int32_t b0 = 0; b0 < B; b0 += blockDim.x) {
        const int32_t b = b0 + tid;
        long long v = 0;
        int32_t kept = 0;
        if (b < B) {
            for (int c = 0; c < kChunks; ++c) kept += counts[b * kChunks + c];
            v = (long long)kept + (reserve ? reserve[b] : 0);
        }
        // inclusive warp scan of v
        long long incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) warp_tot[warp] = incl;
        __syncthreads();
        long long wb = 0, tot = 0;
        for (int w = 0; w < kWarps; ++w) {
            if (w < warp) wb += warp_tot[w];
            tot += warp_tot[w];
        }
        if (b < B) {
            const long long base = running + wb + incl - v;
            seq_base[b] = base;
            offsets[b] = (int32_t)base;
            if (ret_len) ret_len[b] = kept;
        }
        running += tot;
        __syncthreads();
    }
    if (tid == 0) {
        offsets[B] = (int32_t)running;
        if (running > capacity || running > 0x7fffffffLL) set_status(status, SONIC_ERR_CAPACITY);
    }
}

__global__ void __launch_bounds__(kScanThreads)
keep_scatter_kernel(const uint8_t *__restrict__ role, const int32_t *__restrict__ seg,
                    const int32_t *__restrict__ k_start, const int32_t *__restrict__ k_len,
                    const int32_t *__restrict__ reserve, const int32_t *__restrict__ counts,
                    const long long *__restrict__ seq_base, int32_t capacity, int32_t total,
                    int32_t *__restrict__ src_idx, uint8_t *__restrict__ out_role,
                    int32_t *__restrict__ out_seg) {
    const int c = blockIdx.x, b = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = kScanThreads / 32;
    __shared__ int warp_tot[kWarps];
    // output base of this piece: the sequence's offset plus the earlier pieces
    long long base = seq_base[b];
    for (int i = 0; i < c; ++i) base += counts[b * kChunks + i];
    const int32_t start = k_start[b], len = seq_rows(start, k_len[b], total);
    int32_t lo, hi;
    piece(len, c, &lo, &hi);
    long long running = base;
    for (int32_t c0 = lo; c0 < hi; c0 += blockDim.x) {
        const int32_t t = c0 + tid;
        const int keep = (t < hi) && (role[start + t] != SONIC_ROLE_BODY);
        int incl = warp_inclusive_scan(keep);
        if (lane == 31) warp_tot[warp] = incl;
        __syncthreads();
        int warp_base = 0, chunk_tot = 0;
        for (int w = 0; w < kWarps; ++w) {
            int v = warp_tot[w];
            if (w < warp) warp_base += v;
            chunk_tot += v;
        }
        const long long o = running + warp_base + incl - keep;
        if (keep && o < capacity) {
            if (src_idx) src_idx[o] = start + t;
            if (out_role) out_role[o] = role[start + t];
            if (out_seg) out_seg[o] = seg ? seg[start + t] : 0;
        }
        running += chunk_tot;
        __syncthreads();
    }
    // Reserve rows (piece 0 writes them): no source.
    if (c == 0 && reserve != nullptr) {
        long long kept = 0;
        for (int i = 0; i < kChunks; ++i) kept += counts[b * kChunks + i];
        const int32_t res = reserve[b];
        for (int32_t r = tid; r < res; r += blockDim.x) {
            const long long o = seq_base[b] + kept + r;
            if (o < capacity) {
                if (src_idx) src_idx[o] = -1;
                if (out_role) out_role[o] = SONIC_ROLE_BODY;
                if (out_seg) out_seg[o] = -1;
            }
        }
    }
}

// Kept rows among n role bytes at p, this thread's share (see count_equal).
__device__ __forceinline__ int count_kept(const uint8_t *p, int n, int lane, int lanes) {
    return (lane == 0 ? n : 0) - count_equal(p, n, SONIC_ROLE_BODY, lane, lanes);
}

// keep_count, keep_bases and keep_scatter in one launch, for calls of at most
// kPlanRows rows: every block counts the kept rows before its own piece itself, from
// the role bytes (16 per load, out of L2; one run where the sequences are packed), so no
// block waits for another and nothing is exchanged between launches.  Bound by its chain
// of dependent loads (lengths, role bytes, then the writes): 5.5 us alone for one
// sequence of 2,688 rows, 8.9 us for 8 ragged ones (~90k rows), 16 us for 64 (~450k
// rows), where every block reads 225 KB on average.  The three launches it replaces
// made the whole call (GPU time, us, three launches / this) 60.2 / 53.9 for one
// sequence of 100k rows, 95.5 / 78.7 for 32 of 3k, 212 / 185 for 64 of 4k and 71.3 / 69.4 for two
// of 250k: the line lies where the gain has run out (the counted bytes grow with the
// square of the rows).
// One long sequence among 63 of 300 rows (three launches / this): 100k rows 37 / 13, 450k
// 43-55 / 29-36.  Sequences that share rows: 16 that share 30k 27 / 23, 64 that share 500k
// 859 / 826, of which the copy most.
// blockIdx = (piece, sequence); gridDim.x pieces per sequence, enough for the mean length (the
// host does not know the others).  One whose pieces would be longer than twice long_piece rows
// is cut into pieces of that many, and helpers (the rows of blocks past the sequences') take
// those past gridDim.x.  The two rare parts are functions of their own: inlined, they cost
// every call 0.3 us or more.

struct PlanShared {
    int total[2][kScanThreads / 32];
    int rows[kScanThreads / 32], from[kScanThreads / 32], to[kScanThreads / 32];
    int slice[kScanThreads + 1];
    int4 mine;  // a helper's sequence (-1: none), piece of it, its first row, its rows
};

// Rows per piece of the long sequences, and a helper's piece (to sh.mine).
__device__ __noinline__ int32_t long_pieces(const int32_t *k_start, const int32_t *k_len, int32_t B,
                                            int32_t total, PlanShared &sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_pieces = gridDim.x, helpers = ((int)gridDim.y - B) * n_pieces;
    const int helper = ((int)blockIdx.y - B) * n_pieces + (int)blockIdx.x;  // (< 0: none)
    if (tid == 0) sh.mine.x = -1;
    for (int32_t rows = long_piece(total);; rows *= 2) {
        int sum = 0;
        for (int i0 = 0, k = 0; i0 < B; i0 += kScanThreads, k ^= 1) {
            const int i = i0 + tid;
            const int32_t s = i < B ? k_start[i] : 0, n = i < B ? seq_rows(s, k_len[i], total) : 0;
            // its pieces that helpers take
            const int v =
                n > 2 * long_piece(total) * n_pieces ? max(0, (n - 1) / rows + 1 - n_pieces) : 0;
            const int incl = warp_inclusive_scan(v);
            if (lane == 31) sh.total[k][warp] = incl;
            __syncthreads();
            int at = sum + incl - v;
            for (int w = 0; w < kScanThreads / 32; ++w) {
                const int t = sh.total[k][w];
                if (w < warp) at += t;
                sum += t;
            }
            if (helper >= at && helper < at + v) sh.mine = make_int4(i, n_pieces + helper - at, s, n);
        }
        __syncthreads();
        if (sum <= helpers) {
            if (helper >= sum && tid == 0) sh.mine.x = -1;
            __syncthreads();
            return rows;
        }
        // (sequences that share rows have more pieces than one array of rows: longer ones)
    }
}

// Rows kept by the first b sequences where these are not packed, this thread's share.
__device__ __noinline__ int count_apart(const uint8_t *role, const int32_t *k_start,
                                        const int32_t *k_len, int b, int32_t total, PlanShared &sh) {
    constexpr int kWarps = kScanThreads / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t listed = 0, from = total, to = 0;  // their rows (at most kPlanWork), in [from, to)
    for (int i = tid; i < b; i += kScanThreads) {
        const int32_t s = k_start[i], n = seq_rows(s, k_len[i], total);
        listed += n;
        from = n > 0 ? min(from, s) : from;
        to = n > 0 ? max(to, s + n) : to;
    }
    listed = __reduce_add_sync(0xffffffffu, listed);
    from = __reduce_min_sync(0xffffffffu, from);
    to = __reduce_max_sync(0xffffffffu, to);
    if (lane == 0) {
        sh.rows[warp] = listed;
        sh.from[warp] = from;
        sh.to[warp] = to;
    }
    __syncthreads();
    listed = 0;
    for (int w = 0; w < kWarps; ++w) {
        listed += sh.rows[w];
        from = min(from, sh.from[w]);
        to = max(to, sh.to[w]);
    }
    int kept = 0;
    if (listed <= 2 * (to - from) + 4 * kSlice * b) {  // (few rows shared, or short sequences)
        int wps = kWarps;  // several warps a sequence while there are few
        while (wps > 1 && wps * b > kWarps) wps >>= 1;
        for (int i = warp / wps; i < b; i += kWarps / wps) {
            const int32_t s = k_start[i], n = seq_rows(s, k_len[i], total);
            kept += count_kept(role + s, n, (warp % wps) * 32 + lane, wps * 32);
        }
        return kept;
    }
    // sequences that share rows: the rows they span are counted once, in slices, and a
    // sequence's are those before its end less those before its start
    const int32_t size = to - from > kScanThreads * kSlice ? 2 * kSlice : kSlice;
    const int32_t used = (to - from + size - 1) / size;  // <= kScanThreads
    for (int k0 = warp; k0 < used; k0 += 4 * kWarps) {
        int n[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int32_t at = from + (k0 + j * kWarps) * size;
            n[j] = at < to ? count_kept(role + at, min(size, to - at), lane, 32) : 0;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            n[j] = __reduce_add_sync(0xffffffffu, n[j]);
            if (lane == 0 && k0 + j * kWarps < used) sh.slice[k0 + j * kWarps] = n[j];
        }
    }
    __syncthreads();
    const int incl = warp_inclusive_scan(tid < used ? sh.slice[tid] : 0);
    if (lane == 31) sh.total[0][warp] = incl;
    __syncthreads();
    int base = 0;
    for (int w = 0; w < warp; ++w) base += sh.total[0][w];
    sh.slice[tid + 1] = base + incl;  // kept rows before slice tid + 1
    if (tid == 0) sh.slice[0] = 0;
    __syncthreads();
    auto upto = [&](int32_t x) {  // kept rows in [from, x), this lane's share
        const int32_t k = (x - from) / size, at = from + k * size;
        return (lane == 0 ? sh.slice[k] : 0) + count_kept(role + at, x - at, lane, 32);
    };
    for (int i = warp; i < b; i += kWarps) {
        const int32_t s = k_start[i], n = seq_rows(s, k_len[i], total);
        if (n > 0) kept += upto(s + n) - upto(s);
    }
    return kept;
}

__global__ void __launch_bounds__(kScanThreads)
keep_plan_kernel(const uint8_t *role, const int32_t *seg,
                 const int32_t *k_start, const int32_t *k_len,
                 const int32_t *reserve, int32_t B, int32_t capacity, int32_t total,
                 int32_t *offsets, int32_t *ret_len,
                 int32_t *src_idx, uint8_t *out_role,
                 int32_t *out_seg, int32_t *status) {
    pdl_wait();
    pdl_trigger();
    const int pieces = gridDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = kScanThreads / 32;
    __shared__ PlanShared sh;
    __shared__ long long seq_part[kWarps];
    __shared__ int own_part[kWarps], warp_tot[kWarps];
    int c = blockIdx.x, b = min((int)blockIdx.y, B - 1);
    int32_t start = k_start[b];
    const int32_t len_in = k_len[b], first = k_start[0];
    int32_t len = seq_rows(start, len_in, total);
    int32_t rows = ((len + pieces - 1) / pieces + 31) & ~31;
    if (blockIdx.y >= B || rows > 2 * long_piece(total)) {
        rows = long_pieces(k_start, k_len, B, total, sh);
        if (blockIdx.y >= B) {
            b = sh.mine.x;
            c = sh.mine.y;
            start = sh.mine.z;
            len = sh.mine.w;
            if (b < 0) return;
        }
    }
    const int32_t lo = min(len, c * rows), hi = min(len, lo + rows);
    if (c > 0 && lo >= len) return;
    // sequences packed one after another (as a batch's mostly are) are counted as one run
    bool packed = true;
    long long before = 0;
    for (int i = tid; i < b; i += kScanThreads) {
        const int32_t s = k_start[i], n = k_len[i];
        packed = packed && s >= 0 && n >= 0 && (int64_t)s + n <= total && s + n == k_start[i + 1];
        if (reserve != nullptr) before += reserve[i];
    }
    if (c == 0 && tid == 0 && len != len_in) set_status(status, SONIC_ERR_INVALID_ARGUMENT);
    // this thread's rows of the piece's first step, loaded ahead of the counts
    int32_t t0 = lo + tid * kPlanRowsPerThread;
    int ro[kPlanRowsPerThread], sg[kPlanRowsPerThread + 1];
    auto load = [&](int32_t t) {
        sg[0] = seg != nullptr && t > 0 && t < hi ? seg[start + t - 1] : INT_MIN;
#pragma unroll
        for (int k = 0; k < kPlanRowsPerThread; ++k) {
            ro[k] = t + k < hi ? role[start + t + k] : -1;
            sg[k + 1] = seg != nullptr && t + k < hi ? seg[start + t + k] : 0;
        }
    };
    load(t0);
    // rows kept (and reserved) by the sequences before this one, and by this sequence's
    // pieces before this one
    if (__syncthreads_and(packed)) {
        if (b > 0) before += count_kept(role + first, start - first, tid, kScanThreads);
    } else {
        before += count_apart(role, k_start, k_len, b, total, sh);
    }
    int own = count_kept(role + start, lo, tid, kScanThreads);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    own = __reduce_add_sync(0xffffffffu, own);
    if (lane == 0) {
        seq_part[warp] = before;
        own_part[warp] = own;
    }
    long long seq_base = 0, running = 0;
    bool bad = false;
    for (int32_t c0 = lo; c0 == lo || c0 < hi; c0 += kPlanStep) {
        int n = 0;  // this thread's kept rows
#pragma unroll
        for (int k = 0; k < kPlanRowsPerThread; ++k) {
            const bool in = ro[k] >= 0, body = ro[k] == SONIC_ROLE_BODY;
            n += in && !body;
            bad |= ro[k] > SONIC_ROLE_CURR;
            if (seg != nullptr && in) bad |= (body && sg[k + 1] <= 0) || sg[k + 1] < sg[k];
        }
        const int incl = warp_inclusive_scan(n);
        if (lane == 31) warp_tot[warp] = incl;
        __syncthreads();
        if (c0 == lo) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                seq_base += seq_part[w];
                running += own_part[w];
            }
            running += seq_base;
        }
        int warp_base = 0, step_tot = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const int v = warp_tot[w];
            if (w < warp) warp_base += v;
            step_tot += v;
        }
        long long o = running + warp_base + incl - n;
#pragma unroll
        for (int k = 0; k < kPlanRowsPerThread; ++k) {
            if (ro[k] < 0 || ro[k] == SONIC_ROLE_BODY) continue;
            if (o < capacity) {
                src_idx[o] = start + t0 + k;
                if (out_role) out_role[o] = (uint8_t)ro[k];
                if (out_seg) out_seg[o] = sg[k + 1];
            }
            ++o;
        }
        running += step_tot;
        t0 += kPlanStep;
        if (c0 + kPlanStep < hi) load(t0);
        __syncthreads();
    }
    if (__syncthreads_or(bad) && tid == 0) set_status(status, SONIC_ERR_LAYOUT);
    if (c == 0 && tid == 0) offsets[b] = (int32_t)seq_base;
    if (hi < len) return;
    // the sequence's last piece: its retained length, its reserve rows (no source), and
    // behind the last sequence the total
    const int32_t res = reserve != nullptr ? reserve[b] : 0;
    for (int32_t r = tid; r < res; r += kScanThreads) {
        const long long o = running + r;
        if (o < capacity) {
            src_idx[o] = -1;
            if (out_role) out_role[o] = SONIC_ROLE_BODY;
            if (out_seg) out_seg[o] = -1;
        }
    }
    if (tid == 0) {
        if (ret_len) ret_len[b] = (int32_t)(running - seq_base);
        if (b == B - 1) {
            offsets[B] = (int32_t)(running + res);
            if (running + res > capacity || running + res > 0x7fffffffLL)
                set_status(status, SONIC_ERR_CAPACITY);
        }
    }
}

// 16-byte vector copy of kept rows.  blockIdx.y = layer * 2 + (0: K, 1: V).
// One warp copies whole rows (lane j takes 16-byte chunks j, j+32, ...); each
// warp works on two rows at a time with all their loads issued before the
// stores, so up to 8 x 16 bytes per thread are in flight.
constexpr int kGatherThreads = 256;


__device__ __forceinline__ int4 ld_stream(const void *p) {
    int4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.s32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// kGatherRows rows a warp moves per pass, kGatherUnroll 16-byte pieces of each
// per lane per step: 2 x 4 for rows under 2 KB, 4 x 2 for larger rows (more
// rows in flight helps the long rows; at 1 KB it measured slower).
template <int kGatherRows, int kGatherUnroll>
__global__ void __launch_bounds__(kGatherThreads)
kv_gather_kernel(const uint8_t *K, const uint8_t *V,
                 uint8_t *out_K, uint8_t *out_V,
                 const int32_t *offsets, const int32_t *src_idx,
                 int32_t B, int32_t capacity, int64_t row_bytes, int64_t in_layer_bytes,
                 int64_t out_layer_bytes) {
    pdl_wait();
    pdl_trigger();
    const int layer = blockIdx.y >> 1;
    const bool is_v = blockIdx.y & 1;
    const uint8_t *src = (is_v ? V : K) + (int64_t)layer * in_layer_bytes;
    uint8_t *dst = (is_v ? out_V : out_K) + (int64_t)layer * out_layer_bytes;
    const int64_t n_rows = min(offsets[B], capacity);
    const int lane = threadIdx.x & 31;
    const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int cpr = (int)(row_bytes >> 4);  // 16-byte chunks per row
    // each warp moves kGatherRows rows per pass (n_warps apart), every lane
    // holding its 16-byte pieces of all of them in flight
    for (int64_t r0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); r0 < capacity;
         r0 += kGatherRows * n_warps) {
        int32_t sr[kGatherRows];
#pragma unroll
        for (int k = 0; k < kGatherRows; ++k) {
            // (read below the capacity, so that it does not wait for the row count:
            // 494 -> 476 us on 3.22 GB of 2 KB rows)
            const int64_t r = r0 + k * n_warps;
            sr[k] = r < capacity ? src_idx[r] : -1;
        }
#pragma unroll
        for (int k = 0; k < kGatherRows; ++k)
            if (r0 + k * n_warps >= n_rows) sr[k] = -1;
        if (r0 >= n_rows) break;
        for (int c0 = lane; c0 < cpr; c0 += 32 * kGatherUnroll) {
            int4 v[kGatherRows][kGatherUnroll];
#pragma unroll
            for (int k = 0; k < kGatherRows; ++k)
#pragma unroll
                for (int u = 0; u < kGatherUnroll; ++u) {
                    const int c = c0 + 32 * u;
                    if (c < cpr && sr[k] >= 0)
                        v[k][u] = ld_stream(src + (int64_t)sr[k] * row_bytes + ((int64_t)c << 4));
                }
#pragma unroll
            for (int k = 0; k < kGatherRows; ++k)
#pragma unroll
                for (int u = 0; u < kGatherUnroll; ++u) {
                    const int c = c0 + 32 * u;
                    if (c < cpr && sr[k] >= 0)
                        *reinterpret_cast<int4 *>(dst + (r0 + k * n_warps) * row_bytes +
                                                  ((int64_t)c << 4)) = v[k][u];
                }
        }
    }
}

}  // namespace
}  // namespace sonic

using namespace sonic;

extern "C" size_t sonic_compact_workspace_size(const sonic_compact_args *a) {
    if (a == nullptr || a->batch < 0) return 0;
    // per-piece counts, then per-sequence 64-bit bases, then (if the caller
    // gives no src_idx) the source row of every output row
    size_t ws = round_up((size_t)a->batch * kChunks * sizeof(int32_t), 256) +
                round_up((size_t)a->batch * sizeof(long long), 256);
    if (a->src_idx == nullptr)
        ws += round_up((size_t)(a->out_capacity_rows > 0 ? a->out_capacity_rows : 0) *
                           sizeof(int32_t),
                       256);
    return ws;
}

extern "C" sonic_status_t sonic_compact_kv(const void *K, const void *V, const int32_t *seg_id,
                                           const uint8_t *role, void *out_K, void *out_V,
                                           int32_t *offsets, const sonic_compact_args *a,
                                           sonic_stream_t stream_) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (a == nullptr || offsets == nullptr) return SONIC_ERR_INVALID_ARGUMENT;
    if (a->batch < 0 || a->n_layers < 1 || a->out_capacity_rows < 0)
        return SONIC_ERR_INVALID_ARGUMENT;
    if (a->batch == 0) {
        if (cudaMemsetAsync(offsets, 0, sizeof(int32_t), stream) != cudaSuccess)
            return SONIC_ERR_CUDA;
        return SONIC_OK;
    }
    if (K == nullptr || V == nullptr || role == nullptr || out_K == nullptr ||
        out_V == nullptr || a->k_start == nullptr || a->k_len == nullptr)
        return SONIC_ERR_INVALID_ARGUMENT;
    if (a->row_bytes <= 0 || (a->row_bytes & 15) || (a->in_layer_bytes & 15) ||
        (a->out_layer_bytes & 15))
        return SONIC_ERR_INVALID_ARGUMENT;
    if (a->n_layers > 1 && (a->in_layer_bytes <= 0 || a->out_layer_bytes <= 0))
        return SONIC_ERR_INVALID_ARGUMENT;
    if (!aligned16(K) || !aligned16(V) || !aligned16(out_K) || !aligned16(out_V))
        return SONIC_ERR_INVALID_ARGUMENT;
    if (a->n_layers > 32767 || a->batch > 65535) return SONIC_ERR_UNSUPPORTED;
    if (a->total_rows <= 0) return SONIC_ERR_INVALID_ARGUMENT;
    const size_t need = sonic_compact_workspace_size(a);
    if (need > 0 && (a->workspace == nullptr || a->workspace_bytes < need))
        return SONIC_ERR_WORKSPACE;

    char *ws = static_cast<char *>(a->workspace);
    int32_t *counts = reinterpret_cast<int32_t *>(ws);
    ws += round_up((size_t)a->batch * kChunks * sizeof(int32_t), 256);
    long long *seq_base = reinterpret_cast<long long *>(ws);
    ws += round_up((size_t)a->batch * sizeof(long long), 256);
    int32_t *src_idx = a->src_idx != nullptr ? a->src_idx : reinterpret_cast<int32_t *>(ws);

    cudaError_t e = cudaSuccess;
    if (a->total_rows <= kPlanRows && (int64_t)a->total_rows * a->batch <= kPlanWork) {
        // pieces per sequence by the mean length, and helpers for longer ones where there can be
        // such: enough for one array of rows, and up to a block per SM where sequences share rows
        // (near 65,535 sequences, the grid's limit, there is no room for them: fewer pieces)
        const int mean = a->total_rows / a->batch;
        const int n = std::min(kChunks, std::max(1, (mean + kPlanStep - 1) / kPlanStep));
        const bool any = a->total_rows > 2 * long_piece(a->total_rows) * n;
        const int64_t packed = any ? a->total_rows / kPlanStep : 0;
        const int64_t helpers =
            std::max(packed, std::min<int64_t>(packed * a->batch, device_sm_count()));
        const int64_t y = std::min<int64_t>(65535, a->batch + (helpers + n - 1) / n);
        e = launch_pdl(keep_plan_kernel, dim3(n, (unsigned)std::max<int64_t>(y, a->batch)),
                       kScanThreads, 0, stream, 1, role, seg_id,
                       a->k_start, a->k_len, a->reserve, a->batch, a->out_capacity_rows,
                       a->total_rows, offsets, a->ret_len, src_idx, a->out_role, a->out_seg,
                       a->status);
    } else {
        const dim3 pieces(kChunks, a->batch);
        keep_count_kernel<<<pieces, kScanThreads, 0, stream>>>(
            role, seg_id, a->k_start, a->k_len, a->total_rows, counts, a->status);
        keep_bases_kernel<<<1, kScanThreads, 0, stream>>>(counts, a->reserve, a->batch,
                                                          a->out_capacity_rows, seq_base, offsets,
                                                          a->ret_len, a->status);
        keep_scatter_kernel<<<pieces, kScanThreads, 0, stream>>>(
            role, seg_id, a->k_start, a->k_len, a->reserve, counts, seq_base, a->out_capacity_rows,
            a->total_rows, src_idx, a->out_role, a->out_seg);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return SONIC_ERR_CUDA;
    const int sms = device_sm_count();
    // ~32 blocks per SM in all (four resident at a time): with many small
    // blocks the SMs run out of work together, where ~8 left a ragged tail
    // (5.9 -> 6.7 TB/s on a 28-layer compaction of 1 KB rows).
    const int per_slice = (sms * 32 + 2 * a->n_layers - 1) / (2 * a->n_layers);
    dim3 grid(per_slice < 1 ? 1 : per_slice, 2 * a->n_layers);
    auto gather = a->row_bytes >= 2048 ? kv_gather_kernel<4, 2> : kv_gather_kernel<2, 4>;
    e = launch_pdl(gather, grid, kGatherThreads, 0, stream, 1, static_cast<const uint8_t *>(K),
                   static_cast<const uint8_t *>(V), static_cast<uint8_t *>(out_K),
                   static_cast<uint8_t *>(out_V), offsets, src_idx, a->batch,
                   a->out_capacity_rows, a->row_bytes, a->in_layer_bytes, a->out_layer_bytes);
    return e == cudaSuccess ? SONIC_OK : SONIC_ERR_CUDA;
}
