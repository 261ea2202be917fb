// Step 1 of the DAF layer (Methods, item 1 "selection" and "gather"; item 2
// "hybrid KV cache") and the stand-alone form of step 4 (item 3 "state fusion").
//
// These steps move bytes and rank 32-bit keys; they are bound by HBM bandwidth
// and launch latency, not by arithmetic, so they are plain coalesced 16-byte
// kernels with no tensor-core work.
#include <cooperative_groups.h>
#include <cuda_fp8.h>

#include <atomic>

#include "daf_common.cuh"

namespace daf {

#ifdef DAF_TRACE
DAF_KT_TABLE;
DAF_KT_READER(daf_dbg_kt_select)
#endif

// ------------------------------------------------------------------ selection
// A cluster of 8 CTAs ranks all L_d aggregated scores.  Each CTA keeps a
// contiguous slice of the keys in its shared memory.  Radix passes over 12, 12
// and 8 bits find the key of the k-th largest score: every CTA counts the digits
// of its slice and adds its counts to the cluster's sums in shared memory, so
// that after one cluster barrier each can pick the same digit.  An ordered
// compaction then emits the selected positions in ascending order.  Ties at the
// threshold are broken by position (lower first), so the result is unique.
//
// Bound by latency: a barrier and a scan per pass.  Twelve bits a pass because
// sign, exponent and three bits of the fraction spread real scores over a hundred
// bins, few of which are not empty, and 24 bits usually leave nothing to tell
// apart.  Where the counts go (times back to back, in us):
//   - straight into the sums while few keys are left, without a histogram of the
//     CTA's own; equal keys of a warp as one count;
//   - into a copy of the sums in every CTA, which then finds them at home, or, as
//     a CTA sends about one word a clock, to one owner per range of bins where
//     many words may have to leave one CTA: from kSelToAll keys left on, and by
//     histogram where a CTA has more than a key per thread.
// Clustered scores at 6k / 16k / 32k / 64k tokens 4.9 / 6.0 / 7.5 / 12.3, with a copy
// everywhere in every pass 4.7 / 5.6 / 7.0 / 11.5 (layers: the same); 2000 equal keys
// around the threshold 6.5 / 7.9 / 9.8 / 14.0, each key counted by itself in every
// CTA 14.2 / 14.0 / 12.1 / 16.9; ascending scores 5.5 / 6.6 / 8.4 / 13.7 and 6.8 / 9.4 /
// 13.3 / 16.2; uniform ones at 64k 11.0 and 14.3.  The loops over passes and CTAs
// stay loops: unrolled they are 0.2 to 0.5 us faster back to back, but in a layer, where
// each kernel's code has to be fetched again, 11k 102.5 -> 105.1 us, 16k 82.3 -> 83.7.

constexpr int kSelCluster = 8;
constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelSmemKeysPerCta = 40960;   // slice kept in shared memory up to this size, in global scratch beyond

// Monotone map fp32 -> uint32: larger score <=> larger key; -0 == +0; NaN -> 0 (ranks lowest).
__device__ __forceinline__ uint32_t score_key(float s) {
    uint32_t b = __float_as_uint(s);
    if ((b & 0x7FFFFFFFu) > 0x7F800000u) return 0u;   // NaN
    if (b == 0x80000000u) b = 0u;                     // -0 -> +0
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// fp32 add, round to nearest, subnormals kept (the library is built with flush-to-zero arithmetic; the
// aggregation of the signal rows must not flush, or tiny sums would all rank as ties at zero).
__device__ __forceinline__ float add_rn_keep_subnormals(float a, float b) {
    float d;
    asm("add.rn.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

// Keys sit in shared memory with one word of padding per 32, so that both access patterns are free of bank
// conflicts: consecutive threads reading consecutive keys, and each thread walking its own run of keys.
__host__ __device__ constexpr int padded(int i) { return i + (i >> 5); }

constexpr int kSelBits = 12;                    // digits of 12, 12 and 8 bits
constexpr int kSelBins = 1 << kSelBits;
constexpr int kSelLastBins = 1 << (32 - 2 * kSelBits);
constexpr int kSelDirect = 2048;                // up to so many keys in a bin are counted straight into the cluster's sums
constexpr int kSelToAll = 256;                  // and up to so many into every CTA's copy

struct SelShared {
    uint32_t hist[kSelBins];                // this CTA's keys
    uint32_t total[2 * kSelBins + kSelLastBins];   // the cluster's, one array per pass: all of them here, or those of the bins this CTA owns
    uint32_t before[2];                     // keys above / equal to the threshold in the CTAs ahead (added by those)
    uint32_t scan_a[kSelWarps];
    uint32_t scan_b[kSelWarps];
    uint32_t pick[3];                       // chosen digit, remaining rank, number of keys in the chosen bin
};

__global__ void __cluster_dims__(kSelCluster, 1, 1) __launch_bounds__(kSelThreads, 1)
select_topk_kernel(const float* __restrict__ scores, int n_sig, int L_d, int k,
                   uint32_t* __restrict__ gkeys, int32_t* __restrict__ idx_out) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    DAF_KT_BEGIN(0);
    extern __shared__ __align__(16) unsigned char sel_smem[];
    SelShared* sh = reinterpret_cast<SelShared*>(sel_smem);
    uint32_t* skeys = reinterpret_cast<uint32_t*>(sel_smem + sizeof(SelShared));

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)cluster.block_rank();
    const int per_cta = (L_d + kSelCluster - 1) / kSelCluster;
    const int lo_cta = min(L_d, rank * per_cta);
    const int n_loc = min(L_d, lo_cta + per_cta) - lo_cta;
    const bool in_smem = per_cta <= kSelSmemKeysPerCta;
    uint32_t* keys = in_smem ? skeys : (gkeys + lo_cta);
    auto at = [&](int i) { return in_smem ? padded(i) : i; };   // padded layout in shared memory only
    for (int i = tid; i < kSelBins; i += kSelThreads) sh->hist[i] = 0u;
    for (int i = tid; i < 2 * kSelBins + kSelLastBins; i += kSelThreads) sh->total[i] = 0u;
    if (tid < 2) sh->before[tid] = 0u;
    cluster.sync();            // every CTA runs, and its sums are zero
    pdl_wait();
    pdl_launch_dependents();   // the gather kernel may start launching; it waits for this grid before reading idx

    // one more key in a bin; a warp whose keys all fall in one bin adds once, otherwise every thread adds for itself
    auto count = [&](bool in, uint32_t bin) {
        const uint32_t active = __ballot_sync(0xFFFFFFFFu, in);
        if (active == 0u) return;
        const uint32_t lead_bin = __shfl_sync(0xFFFFFFFFu, bin, __ffs(active) - 1);
        const uint32_t same = __ballot_sync(0xFFFFFFFFu, in && bin == lead_bin);
        if (same == active) {
            if (lane == __ffs(active) - 1) atomicAdd(&sh->hist[lead_bin], (uint32_t)__popc(active));
        } else if (in) {
            atomicAdd(&sh->hist[bin], 1u);
        }
    };
    // aggregate the signal rows in ascending row order (fp32 adds, no fusing), build keys and count their top digit
    // (four loads in flight per thread: one per trip would serialise on memory latency)
    for (int base = 0; base < n_loc; base += 4 * kSelThreads) {
        float acc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = base + u * kSelThreads + tid;
            acc[u] = i < n_loc ? scores[lo_cta + i] : 0.f;
        }
        for (int l = 1; l < n_sig; ++l) {
            float nxt[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = base + u * kSelThreads + tid;
                nxt[u] = i < n_loc ? scores[(size_t)l * L_d + lo_cta + i] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u] = add_rn_keep_subnormals(acc[u], nxt[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = base + u * kSelThreads + tid;
            if (base + u * kSelThreads >= n_loc) break;       // uniform across the CTA
            const uint32_t key = score_key(acc[u]);
            if (i < n_loc) keys[at(i)] = key;
            count(i < n_loc, key >> (32 - kSelBits));
        }
    }

    // Radix selection from the top digit down.  It stops as soon as every key left in the chosen bin is taken (with distinct
    // scores usually after two passes): the comparisons below then look only at the bits resolved so far.
    uint32_t prefix = 0u, mask = 0u, k_rem = (uint32_t)k, left = 0xFFFFFFFFu;    // left: keys in the chosen bin
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
        const int shift = pass == 0 ? 32 - kSelBits : pass == 1 ? 32 - 2 * kSelBits : 0;
        const int n_bins = pass == 2 ? kSelLastBins : kSelBins;
        uint32_t* const total = sh->total + pass * kSelBins;
        const bool direct = left <= (uint32_t)kSelDirect;
        const bool to_all = pass == 0 || left <= (uint32_t)kSelToAll || (!direct && per_cta <= kSelThreads);    // the same in all CTAs
        const int owner_shift = pass == 2 ? 32 - 2 * kSelBits - 3 : kSelBits - 3;    // CTA r owns the r-th eighth of the bins
        static_assert(kSelCluster == 1 << 3, "");
        auto add = [&](uint32_t bin, uint32_t c) {
            int r = to_all ? 0 : (int)(bin >> owner_shift);
            const int last = to_all ? kSelCluster - 1 : r;
#pragma unroll 1
            for (; r <= last; ++r) atomicAdd(cluster.map_shared_rank(&total[bin], r), c);
        };
        if (pass > 0) {
            for (int base = 0; base < n_loc; base += kSelThreads) {
                const int i = base + tid;
                const uint32_t key = i < n_loc ? keys[at(i)] : 0u;
                const bool in = i < n_loc && (key & mask) == prefix;
                const uint32_t bin = (key >> shift) & (uint32_t)(n_bins - 1);
                if (!direct) {
                    count(in, bin);
                    continue;
                }
                const uint32_t active = __ballot_sync(0xFFFFFFFFu, in);
                if (active == 0u) continue;
                const int lead = __ffs(active) - 1;
                const uint32_t lead_bin = __shfl_sync(0xFFFFFFFFu, bin, lead);
                const bool one_bin = __ballot_sync(0xFFFFFFFFu, in && bin == lead_bin) == active;
                if (one_bin ? lane == lead : in) add(bin, one_bin ? (uint32_t)__popc(active) : 1u);
            }
        }
        if (!direct) {
            __syncthreads();   // this CTA's histogram is complete: its bins go to the cluster's sums (few are not empty)
            for (int bin = tid; bin < n_bins; bin += kSelThreads) {
                const uint32_t c = sh->hist[bin];
                if (c != 0u) {
                    sh->hist[bin] = 0u;
                    add((uint32_t)bin, c);
                }
            }
        }
        cluster.sync();    // the sums of this pass are complete
        // thread t owns the four bins from n_bins - 4 - 4t on: the running count from the top
        const int low = n_bins - 4 - 4 * tid;
        uint4 four = make_uint4(0u, 0u, 0u, 0u);
        if (low >= 0) {
            if (to_all) four = *reinterpret_cast<const uint4*>(&total[low]);
            else four = *reinterpret_cast<const uint4*>(cluster.map_shared_rank(&total[low], low >> owner_shift));
        }
        const uint32_t own = four.x + four.y + four.z + four.w;
        uint32_t incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) sh->scan_a[warp] = incl;
        __syncthreads();
        static_assert(kSelWarps == 32 && kSelBins == 4 * kSelThreads, "one warp's total per lane, four bins per thread");
        const uint32_t w = sh->scan_a[lane];
        const uint32_t ahead = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? w : 0u);
        uint32_t above = ahead + incl - own;
        if (k_rem > above && k_rem <= above + own) {
            uint32_t in_bin = four.w;
            int bin = low + 3;
            if (k_rem > above + in_bin) { above += in_bin; in_bin = four.z; --bin; }
            if (bin == low + 2 && k_rem > above + in_bin) { above += in_bin; in_bin = four.y; --bin; }
            if (bin == low + 1 && k_rem > above + in_bin) { above += in_bin; in_bin = four.x; --bin; }
            sh->pick[0] = (uint32_t)bin;
            sh->pick[1] = k_rem - above;
            sh->pick[2] = in_bin;
        }
        __syncthreads();
        prefix |= sh->pick[0] << shift;
        mask = 0xFFFFFFFFu << shift;
        k_rem = sh->pick[1];
        left = sh->pick[2];
        if (left == k_rem) break;   // every key left in the bin is taken: no need to tell them apart
    }
    const uint32_t thr = prefix;       // the resolved bits of the k-th largest key
    const uint32_t need_eq = k_rem;    // how many keys matching thr are taken (lowest positions first)

    // ordered compaction: thread t owns the contiguous local positions [t*E, (t+1)*E)
    const int E = (per_cta + kSelThreads - 1) / kSelThreads;
    const int lo = min(n_loc, tid * E), hi = min(n_loc, lo + E);
    uint32_t n_gt = 0, n_eq = 0;
    for (int i = lo; i < hi; ++i) {
        const uint32_t key = keys[at(i)] & mask;
        n_gt += key > thr;
        n_eq += key == thr;
    }
    uint32_t in_gt = n_gt, in_eq = n_eq;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t a = __shfl_up_sync(0xFFFFFFFFu, in_gt, o), b = __shfl_up_sync(0xFFFFFFFFu, in_eq, o);
        if (lane >= o) { in_gt += a; in_eq += b; }
    }
    if (lane == 31) { sh->scan_a[warp] = in_gt; sh->scan_b[warp] = in_eq; }
    __syncthreads();
    const uint32_t wa = sh->scan_a[lane], wb = sh->scan_b[lane];
    uint32_t gt_before = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? wa : 0u) + in_gt - n_gt;
    uint32_t eq_before = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? wb : 0u) + in_eq - n_eq;
    if (warp == 0) {       // the CTAs behind this one hear how many keys it has
        const uint32_t all_a = __reduce_add_sync(0xFFFFFFFFu, wa), all_b = __reduce_add_sync(0xFFFFFFFFu, wb);
        if (lane > rank && lane < kSelCluster) {
            atomicAdd(cluster.map_shared_rank(&sh->before[0], lane), all_a);
            atomicAdd(cluster.map_shared_rank(&sh->before[1], lane), all_b);
        }
    }
    cluster.sync();   // (and no CTA's shared memory is touched by another after this)
    gt_before += sh->before[0];
    eq_before += sh->before[1];
    if (k > 0) {
        uint32_t pos = gt_before + min(eq_before, need_eq);
        for (int i = lo; i < hi; ++i) {
            const uint32_t key = keys[at(i)] & mask;
            bool take = key > thr;
            if (key == thr) { take = eq_before < need_eq; ++eq_before; }
            if (take) idx_out[pos++] = lo_cta + i;
        }
    }
    DAF_KT_END(0);
}

// ------------------------------------------------ selection, one CTA (up to 4K tokens)
// Few keys run in one CTA with no cluster traffic.  The keys are first reduced to their offset from the smallest key.  One
// pass over all keys histograms the top 11 of the bits that offset needs (typically 24-27 of 32, fewer
// when the scores are close together) with shared-memory atomics and finds the bin that holds the k-th
// largest key; only the keys of that bin (typically well under one per cent) go on: when they are few,
// each is ranked against the others directly, otherwise passes of 9 bits fix the remaining bits.  Because the offsets of real scores spread over the whole histogram,
// the atomics rarely collide; scores that are all (nearly) equal collide more, and all of them become
// candidates, but the result stays correct.  An ordered compaction then emits the positions.
constexpr int kSel1Threads = 1024;
constexpr int kSel1Warps = kSel1Threads / 32;
constexpr int kSel1MaxKeys = 4096;    // see launch_select
constexpr int kSel1PerThread = kSel1MaxKeys / kSel1Threads;
static_assert(kSel1PerThread * kSel1Threads == kSel1MaxKeys, "every key has a thread that loads it");
constexpr int kSel1TopBits = 11;      // first pass, over all keys
constexpr int kSel1TopBins = 1 << kSel1TopBits;
constexpr int kSel1Bits = 9;          // later passes, over the candidates
constexpr int kSel1Bins = 1 << kSel1Bits;

struct Sel1Shared {
    uint32_t hist[kSel1TopBins];
    uint32_t warp_a[kSel1Warps];
    uint32_t warp_b[kSel1Warps];
    uint32_t pick[2];       // chosen digit, remaining rank
    uint32_t n_cand;
};

// Exclusive prefix sums of (a, b) over the threads of the CTA, in thread order.
__device__ __forceinline__ void block_excl_scan2(uint32_t a, uint32_t b, uint32_t* wa, uint32_t* wb,
                                                 uint32_t& ex_a, uint32_t& ex_b, uint32_t& tot_a, uint32_t& tot_b) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t ia = a, ib = b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, ia, o), y = __shfl_up_sync(0xFFFFFFFFu, ib, o);
        if (lane >= o) { ia += x; ib += y; }
    }
    if (lane == 31) { wa[warp] = ia; wb[warp] = ib; }
    __syncthreads();
    uint32_t va = wa[lane], vb = wb[lane];   // kSel1Warps == 32: one warp total per lane
    uint32_t sa = va, sb = vb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, sa, o), y = __shfl_up_sync(0xFFFFFFFFu, sb, o);
        if (lane >= o) { sa += x; sb += y; }
    }
    tot_a = __shfl_sync(0xFFFFFFFFu, sa, 31);
    tot_b = __shfl_sync(0xFFFFFFFFu, sb, 31);
    ex_a = __shfl_sync(0xFFFFFFFFu, sa - va, warp) + ia - a;
    ex_b = __shfl_sync(0xFFFFFFFFu, sb - vb, warp) + ib - b;
    __syncthreads();   // wa/wb may be reused by the next scan
}

// Finds, from the top, the bin in which the k_rem-th element falls.  Thread t owns `per` consecutive
// bins in descending order; the result goes to pick[0] (bin) and pick[1] (rank inside that bin).
__device__ __forceinline__ void pick_bin(Sel1Shared* sh, int n_bins, int per) {
    const int top = n_bins - 1 - (int)threadIdx.x * per;   // this thread's highest bin
    // the remaining rank is read here, ahead of the scan: the scan's barriers then separate every
    // thread's read from the one thread that writes the reduced rank below
    const uint32_t k_rem = sh->pick[1];
    uint32_t c = 0;
    if (top >= 0)
        for (int b = 0; b < per; ++b) c += sh->hist[top - b];
    uint32_t above, dummy, tot, tot2;
    block_excl_scan2(c, 0u, sh->warp_a, sh->warp_b, above, dummy, tot, tot2);
    if (top >= 0 && k_rem > above && k_rem <= above + c) {
        uint32_t acc = above;
        for (int b = 0; b < per; ++b) {
            const uint32_t cb = sh->hist[top - b];
            if (k_rem <= acc + cb) { sh->pick[0] = (uint32_t)(top - b); sh->pick[1] = k_rem - acc; break; }
            acc += cb;
        }
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kSel1Threads, 1)
select_topk_cta_kernel(const float* __restrict__ scores, int n_sig, int L_d, int k, int32_t* __restrict__ idx_out) {
    extern __shared__ __align__(16) unsigned char sel_smem[];
    Sel1Shared* sh = reinterpret_cast<Sel1Shared*>(sel_smem);
    uint32_t* keys = reinterpret_cast<uint32_t*>(sel_smem + sizeof(Sel1Shared));
    uint32_t* cand = keys + padded(L_d);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    DAF_KT_BEGIN(0);
    pdl_wait();
    pdl_launch_dependents();   // the gather kernel may start launching; it waits for this grid before reading idx

    // aggregate the signal rows in ascending row order (fp32 adds, no fusing), build keys, find their range
    // (a thread's loads of a row in flight together: one after the other would serialise on memory latency)
    uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
    float acc[kSel1PerThread];
#pragma unroll
    for (int u = 0; u < kSel1PerThread; ++u) {
        const int i = tid + u * kSel1Threads;
        acc[u] = i < L_d ? scores[i] : 0.f;
    }
    for (int l = 1; l < n_sig; ++l) {
        float nxt[kSel1PerThread];
#pragma unroll
        for (int u = 0; u < kSel1PerThread; ++u) {
            const int i = tid + u * kSel1Threads;
            nxt[u] = i < L_d ? scores[(size_t)l * L_d + i] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kSel1PerThread; ++u) acc[u] = add_rn_keep_subnormals(acc[u], nxt[u]);
    }
#pragma unroll
    for (int u = 0; u < kSel1PerThread; ++u) {
        const int i = tid + u * kSel1Threads;
        if (i < L_d) {
            const uint32_t key = score_key(acc[u]);
            keys[padded(i)] = key;
            kmin = min(kmin, key);
            kmax = max(kmax, key);
        }
    }
    for (int i = tid; i < kSel1TopBins; i += kSel1Threads) sh->hist[i] = 0u;
    if (tid == 0) { sh->pick[0] = 0u; sh->pick[1] = (uint32_t)k; sh->n_cand = 0u; }
    kmin = __reduce_min_sync(0xFFFFFFFFu, kmin);
    kmax = __reduce_max_sync(0xFFFFFFFFu, kmax);
    if (lane == 0) { sh->warp_a[warp] = kmin; sh->warp_b[warp] = kmax; }
    __syncthreads();
    kmin = __reduce_min_sync(0xFFFFFFFFu, sh->warp_a[lane]);
    kmax = __reduce_max_sync(0xFFFFFFFFu, sh->warp_b[lane]);
    __syncthreads();   // warp_a/warp_b are reused by the scans below
    const uint32_t range = kmax - kmin;
    const int bits = 32 - __clz((int)range);        // bits the offsets need (0 when all keys are equal)
    const int low_bits = max(bits - kSel1TopBits, 0);   // bits left after the first pass

    // first pass, all keys: the top bits of the offset
    for (int i = tid; i < L_d; i += kSel1Threads) atomicAdd(&sh->hist[(keys[padded(i)] - kmin) >> low_bits], 1u);
    __syncthreads();
    pick_bin(sh, kSel1TopBins, kSel1TopBins / kSel1Threads);
    const uint32_t top_digit = sh->pick[0];
    // candidates: the low bits of the keys that fall in the chosen bin
    for (int i = tid; i < L_d; i += kSel1Threads) {
        const uint32_t off = keys[padded(i)] - kmin;
        if ((off >> low_bits) == top_digit) cand[atomicAdd(&sh->n_cand, 1u)] = low_bits > 0 ? off & ((1u << low_bits) - 1u) : 0u;
    }
    if (tid < kSel1Bins) sh->hist[tid] = 0u;
    __syncthreads();
    const int n_cand = (int)sh->n_cand;    // at most L_d, the capacity of the list
    int passes = (low_bits + kSel1Bits - 1) / kSel1Bits;
    uint32_t prefix = 0u;      // the low digits fixed so far
    if (passes > 0 && n_cand <= kSel1Threads) {
        // few candidates (the usual case): each thread ranks one candidate by counting the larger and the
        // equal ones; the candidate whose rank interval holds the remaining rank is the threshold
        const uint32_t k_rem = sh->pick[1];
        __syncthreads();   // every thread has read the rank before one of them replaces it
        if (tid < n_cand) {
            const uint32_t mine = cand[tid];
            uint32_t n_gt = 0, n_eq = 0;
            for (int j = 0; j < n_cand; ++j) {
                const uint32_t other = cand[j];
                n_gt += other > mine;
                n_eq += other == mine;
            }
            if (k_rem > n_gt && k_rem <= n_gt + n_eq) { sh->pick[0] = mine; sh->pick[1] = k_rem - n_gt; }   // equal candidates write the same
        }
        __syncthreads();
        prefix = sh->pick[0];
        passes = 0;
    }
    for (int p = 0; p < passes; ++p) {
        const int shift = (passes - 1 - p) * kSel1Bits;
        for (int i = tid; i < n_cand; i += kSel1Threads) {
            const uint32_t low = cand[i];
            if ((low >> (shift + kSel1Bits)) == prefix) atomicAdd(&sh->hist[(low >> shift) & (kSel1Bins - 1)], 1u);
        }
        __syncthreads();
        pick_bin(sh, kSel1Bins, 1);
        prefix = (prefix << kSel1Bits) | sh->pick[0];
        if (tid < kSel1Bins) sh->hist[tid] = 0u;
        __syncthreads();
    }
    prefix |= top_digit << low_bits;       // the whole offset of the threshold (passes == 0: the top digit alone)
    const uint32_t thr = kmin + prefix;    // key of the k-th largest score (passes == 0: every key equals kmin)
    const uint32_t need_eq = sh->pick[1];  // how many keys equal to thr are taken (lowest positions first)

    // ordered compaction: thread t owns the contiguous positions [t*E, (t+1)*E)
    const int E = (L_d + kSel1Threads - 1) / kSel1Threads;
    const int lo = min(L_d, tid * E), hi = min(L_d, lo + E);
    uint32_t n_gt = 0, n_eq = 0;
    for (int i = lo; i < hi; ++i) {
        const uint32_t key = keys[padded(i)];
        n_gt += key > thr;
        n_eq += key == thr;
    }
    uint32_t gt_before, eq_before, tot_gt, tot_eq;
    block_excl_scan2(n_gt, n_eq, sh->warp_a, sh->warp_b, gt_before, eq_before, tot_gt, tot_eq);
    if (k > 0) {
        uint32_t pos = gt_before + min(eq_before, need_eq);
        for (int i = lo; i < hi; ++i) {
            const uint32_t key = keys[padded(i)];
            bool take = key > thr;
            if (key == thr) { take = eq_before < need_eq; ++eq_before; }
            if (take) idx_out[pos++] = i;
        }
    }
    DAF_KT_END(0);
}

// --------------------------------------------------- gather + hybrid KV update
// One CTA per row.  Rows 0..k-1 are the important tokens: their fresh Q/K/V rows
// go to the packed buffers and (K/V) into the cache rows at their positions.
// Rows k..k+L_q-1 are the question tokens: fresh K/V rows are appended to the cache.
constexpr int kRowThreads = 128;

struct GatherArgs {
    const int4* q_fresh; const int4* k_fresh; const int4* v_fresh;
    int4* kv_k; int4* kv_v;
    int4* q_pack; int4* k_pack; int4* v_pack;
    const int32_t* idx;       // positions to gather (idx_in, or idx_out written by the select kernel)
    int32_t* idx_copy;        // when non-null, also receives idx (the idx_in path)
    int k, L_d, L_q, cq, ckv; // cq/ckv: 16-byte chunks per Q row / per K (or V) row
    int overwrite;
    // rows from host memory only: the caller's cache in host memory (null: not written), and whether the important rows of the device's
    // cache are left to update_cache_kernel because the document rows are still on their way to it
    int4* host_k; int4* host_v;
    int cache_later;
    DeviceStatus* status;
};

// A thread requests kBatch chunks of its row before it stores any (1: the plain loop).  Which form for which row: launch_select.
template <int kBatch, int kThreads>
__global__ void __launch_bounds__(kThreads)
gather_update_kernel(const GatherArgs a) {
    DAF_KT_BEGIN(1);
    pdl_wait();                // idx may come from the selection kernel launched just before; the packed buffers may still be read by the previous layer
    DAF_KT_BEGIN(2);
    pdl_launch_dependents();   // the attention kernel may start launching; it waits for this grid
    const int row = blockIdx.x;
    const int per_row = a.cq + 2 * a.ckv;
    if (row < a.k) {
        const int p = a.idx[row];
        if (a.idx_copy != nullptr && threadIdx.x == 0) a.idx_copy[row] = p;
        if (p < 0 || p >= a.L_d) {
            if (threadIdx.x == 0) report_status(a.status, DAF_ERR_BOUNDS, 1, p);
            return;
        }
        const size_t qsrc = (size_t)p * a.cq, qdst = (size_t)row * a.cq;
        const size_t ksrc = (size_t)p * a.ckv, kdst = (size_t)row * a.ckv;
        // no packed Q wanted: K, V only; no packed K/V wanted and nothing to overwrite in the cache: nothing at all
        const int c_end = (a.k_pack != nullptr || a.overwrite) ? per_row : a.cq;
        const int c0 = (a.q_pack != nullptr ? 0 : a.cq) + threadIdx.x;
        const int k_end = min(a.cq + a.ckv, c_end);      // (a batch may reach past c_end)
        if constexpr (kBatch > 1) {
            for (int base = c0; base < c_end; base += kThreads * kBatch) {
                int4 v[kBatch];
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    const int c = base + u * kThreads;
                    if (c < a.cq) v[u] = __ldg(a.q_fresh + qsrc + c);
                    else if (c < k_end) v[u] = __ldg(a.k_fresh + ksrc + (c - a.cq));
                    else if (c < c_end) v[u] = __ldg(a.v_fresh + ksrc + (c - a.cq - a.ckv));
                }
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    const int c = base + u * kThreads;
                    if (c < a.cq) {
                        a.q_pack[qdst + c] = v[u];
                    } else if (c < k_end) {
                        const int cc = c - a.cq;
                        if (a.k_pack != nullptr) a.k_pack[kdst + cc] = v[u];
                        if (a.overwrite && !a.cache_later) a.kv_k[ksrc + cc] = v[u];
                        if (a.overwrite && a.host_k != nullptr) a.host_k[ksrc + cc] = v[u];
                    } else if (c < c_end) {
                        const int cc = c - a.cq - a.ckv;
                        if (a.v_pack != nullptr) a.v_pack[kdst + cc] = v[u];
                        if (a.overwrite && !a.cache_later) a.kv_v[ksrc + cc] = v[u];
                        if (a.overwrite && a.host_v != nullptr) a.host_v[ksrc + cc] = v[u];
                    }
                }
            }
        } else {
            for (int c = c0; c < c_end; c += kThreads) {
                if (c < a.cq) {
                    a.q_pack[qdst + c] = __ldg(a.q_fresh + qsrc + c);
                } else if (c < a.cq + a.ckv) {
                    const int cc = c - a.cq;
                    const int4 v = __ldg(a.k_fresh + ksrc + cc);
                    if (a.k_pack != nullptr) a.k_pack[kdst + cc] = v;
                    if (a.overwrite) a.kv_k[ksrc + cc] = v;
                } else {
                    const int cc = c - a.cq - a.ckv;
                    const int4 v = __ldg(a.v_fresh + ksrc + cc);
                    if (a.v_pack != nullptr) a.v_pack[kdst + cc] = v;
                    if (a.overwrite) a.kv_v[ksrc + cc] = v;
                }
            }
        }
    } else {
        const size_t off = (size_t)(a.L_d + (row - a.k)) * a.ckv;
        for (int c = threadIdx.x; c < 2 * a.ckv; c += kThreads) {
            const size_t at = off + (c < a.ckv ? c : c - a.ckv);
            const int4 v = __ldg((c < a.ckv ? a.k_fresh : a.v_fresh) + at);
            (c < a.ckv ? a.kv_k : a.kv_v)[at] = v;
            if (kBatch > 1 && a.host_k != nullptr) (c < a.ckv ? a.host_k : a.host_v)[at] = v;
        }
    }
    DAF_KT_END(1);
}

// The important rows of the device's cache from their packed copies (layers from host buffers, where the document rows
// arrive after the rows were gathered).  One warp per row.
__global__ void __launch_bounds__(256)
update_cache_kernel(const int32_t* __restrict__ idx, int k, int L_d, int ckv, const int4* __restrict__ k_pack,
                    const int4* __restrict__ v_pack, int4* __restrict__ kv_k, int4* __restrict__ kv_v) {
    pdl_wait();
    pdl_launch_dependents();
    const int row = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    if (row >= k) return;
    const int p = idx[row];
    if (p < 0 || p >= L_d) return;            // reported by the gather kernel
    for (int c = threadIdx.x & 31; c < ckv; c += 32) {
        kv_k[(size_t)p * ckv + c] = __ldg(k_pack + (size_t)row * ckv + c);
        kv_v[(size_t)p * ckv + c] = __ldg(v_pack + (size_t)row * ckv + c);
    }
}

int launch_update_cache(const ResolvedParams& rp, const int32_t* idx, const void* k_pack, const void* v_pack, void* kv_k,
                        void* kv_v, cudaStream_t stream) {
    if (rp.k <= 0) return DAF_OK;
    const cudaError_t e = launch_kernel(update_cache_kernel, dim3((unsigned)((rp.k + 7) / 8)), dim3(256), 0, stream, idx, rp.k, rp.L_d,
                                        rp.Hkv * 16, reinterpret_cast<const int4*>(k_pack), reinterpret_cast<const int4*>(v_pack),
                                        reinterpret_cast<int4*>(kv_k), reinterpret_cast<int4*>(kv_v));
    count_launch();
    if (e != cudaSuccess) { set_cuda_error(e); return DAF_ERR_CUDA; }
    return check_launch();
}

// ------------------------------------------------------------- state fusion
struct FuseArgs {
    const int4* o_imp; const int4* o_q; int4* hidden;
    const int32_t* idx; int32_t* row_pos;
    int k, L_d, L_q, cq, mode;
};

// Bound by HBM, a few rows by latency: a thread requests its chunks of a row (up to 32 heads) before it stores any.  154 rows of
// 24 / 28 / 40 heads 1.44 / 1.47 / 1.85 us, one chunk after the other 1.64 / 1.74 / 1.84 (192 threads: 1.44 / 1.74 / 1.85); 6554
// rows 8.0 / 10.4 / 20.6 and 9.0 / 12.2 / 21.3 (9.2 / 14.5 / 23.1); five at once are slower from 64 heads on.
constexpr int kFuseChunks = 4;
__global__ void __launch_bounds__(kRowThreads)
fuse_rows_kernel(const FuseArgs a) {
    pdl_wait();
    const int row = blockIdx.x;
    int pos;
    const int4* src;
    if (row < a.k) { pos = a.idx[row]; src = a.o_imp + (size_t)row * a.cq; }
    else { pos = a.L_d + (row - a.k); src = a.o_q + (size_t)(row - a.k) * a.cq; }
    if (a.row_pos != nullptr && threadIdx.x == 0) a.row_pos[row] = pos;
    if (a.hidden == nullptr) return;
    if (pos < 0 || pos >= a.L_d + a.L_q) return;
    int4* dst = a.hidden + (size_t)(a.mode == 0 ? row : pos) * a.cq;
    for (int base = threadIdx.x; base < a.cq; base += kRowThreads * kFuseChunks) {
        int4 v[kFuseChunks];
#pragma unroll
        for (int u = 0; u < kFuseChunks; ++u)
            if (base + u * kRowThreads < a.cq) v[u] = __ldg(src + base + u * kRowThreads);
#pragma unroll
        for (int u = 0; u < kFuseChunks; ++u)
            if (base + u * kRowThreads < a.cq) dst[base + u * kRowThreads] = v[u];
    }
}

// ------------------------------------------------------------ deviation signal
// Per-layer importance signal of a document token: squared deviation of its fresh K and V rows from
// the cached ones, summed over heads and channels (Methods, item 1; the formula is this library's
// reading).  A streaming reduction: one warp per token, 16-byte loads, fp32 accumulation, a fixed
// shuffle tree, so the result does not depend on the launch shape.
__device__ __forceinline__ float sq_dev8(const int4 a, const int4 b) {
    const __nv_bfloat162* x = reinterpret_cast<const __nv_bfloat162*>(&a);
    const __nv_bfloat162* y = reinterpret_cast<const __nv_bfloat162*>(&b);
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 fx = __bfloat1622float2(x[i]), fy = __bfloat1622float2(y[i]);
        const float d0 = fx.x - fy.x, d1 = fx.y - fy.y;
        acc = fmaf(d0, d0, acc);
        acc = fmaf(d1, d1, acc);
    }
    return acc;
}

// 16 bytes that are read once.  An ordinary load that stays behind the wait for the kernel before, which may be the one that
// writes them: not a function of the address alone (volatile, memory), nor of memory that is constant while this kernel is
// there (.nc).
__device__ __forceinline__ int4 ld_once(const int4* p) {
    int4 r;
    asm volatile("ld.global.L1::no_allocate.L2::256B.v4.s32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p) : "memory");
    return r;
}
// A token's value of one layer, this lane's part of it: chunks lane, lane + 32, ... of its rows in that order, the loads of two of
// them written ahead of the arithmetic (at 32 registers the compiler keeps about six of the eight in flight).
__device__ __forceinline__ float sq_dev_rows(const int4* kf, const int4* vf, const int4* kc, const int4* vc, int chunks, int lane) {
    float acc = 0.f;
    int c = lane;
    for (; c + 32 < chunks; c += 64) {
        const int4 kf0 = ld_once(kf + c), kc0 = ld_once(kc + c), vf0 = ld_once(vf + c), vc0 = ld_once(vc + c);
        const int4 kf1 = ld_once(kf + c + 32), kc1 = ld_once(kc + c + 32), vf1 = ld_once(vf + c + 32), vc1 = ld_once(vc + c + 32);
        acc += sq_dev8(kf0, kc0);
        acc += sq_dev8(vf0, vc0);
        acc += sq_dev8(kf1, kc1);
        acc += sq_dev8(vf1, vc1);
    }
    if (c < chunks) {
        const int4 kf0 = ld_once(kf + c), kc0 = ld_once(kc + c), vf0 = ld_once(vf + c), vc0 = ld_once(vc + c);
        acc += sq_dev8(kf0, kc0);
        acc += sq_dev8(vf0, vc0);
    }
    return acc;
}

// One warp per token, as many CTAs as that takes.  Bound by HBM: three layers of 32k tokens of 4 heads, 403 MB, 57 us (7.0 TB/s; it
// only reads).  As a grid of 8 CTAs of 8 warps per SM whose warps walked several tokens, of which 6 were resident and the rest ran
// as a second wave, 67.  The warps of a CTA: signal_warps.
template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps)
deviation_scores_kernel(const int4* __restrict__ k_fresh, const int4* __restrict__ v_fresh,
                        const int4* __restrict__ k_cached, const int4* __restrict__ v_cached,
                        int L_d, int chunks_per_row, float* __restrict__ scores) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int tok = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    if (tok >= L_d) return;
    const size_t base = (size_t)tok * chunks_per_row;
    float acc = sq_dev_rows(k_fresh + base, v_fresh + base, k_cached + base, v_cached + base, chunks_per_row, lane);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
    if (lane == 0) scores[tok] = acc;
}

// The same signal for several layers at once, aggregated on the fly (Methods, item 1: the signals of several
// layers, typically the 2nd to 4th, are aggregated before the tokens are ranked).  One warp per token walks
// the signal layers in ascending order: each layer's value is computed exactly as deviation_scores_kernel
// computes it (same chunk order, same shuffle tree) and added to the running fp32 sum with a plain
// round-to-nearest add, subnormals kept -- the order and arithmetic in which the selection kernels
// aggregate the rows of a score matrix -- so ranking the sums gives the positions that the two-step route
// (one daf_deviation_scores call per layer, then daf_select on the [n_sig, L_d] matrix) would give, without
// that matrix ever being written.
constexpr int kMaxSignalLayers = 8;
struct SignalLayers {
    const int4* k_fresh[kMaxSignalLayers]; const int4* v_fresh[kMaxSignalLayers];
    const int4* k_cached[kMaxSignalLayers]; const int4* v_cached[kMaxSignalLayers];
    int n;
};

template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps)
deviation_sum_kernel(const SignalLayers layers, int L_d, int chunks_per_row, float* __restrict__ sums) {
    pdl_wait();
    pdl_launch_dependents();   // the selection kernel may start launching; it waits for this grid before reading sums
    const int lane = threadIdx.x & 31;
    const int tok = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    if (tok >= L_d) return;
    const size_t base = (size_t)tok * chunks_per_row;
    float total = 0.f;
    for (int l = 0; l < layers.n; ++l) {
        float acc = sq_dev_rows(layers.k_fresh[l] + base, layers.v_fresh[l] + base, layers.k_cached[l] + base,
                                layers.v_cached[l] + base, chunks_per_row, lane);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
        total = l == 0 ? acc : add_rn_keep_subnormals(total, acc);
    }
    if (lane == 0) sums[tok] = total;
}

// ----------------------------------------------------------------- host side
size_t select_scratch_bytes(int L_d) {
    const int per_cta = (L_d + kSelCluster - 1) / kSelCluster;
    return per_cta > kSelSmemKeysPerCta ? ((size_t)per_cta * kSelCluster * sizeof(uint32_t) + 255) / 256 * 256 : 0;
}

static size_t select_smem_bytes(int L_d) {
    const int per_cta = (L_d + kSelCluster - 1) / kSelCluster;
    return sizeof(SelShared) + (per_cta <= kSelSmemKeysPerCta ? (size_t)padded(per_cta) * sizeof(uint32_t) : 0);
}

int launch_select(const ResolvedParams& rp, const float* scores, int n_sig, const int32_t* idx_in,
                  const void* q_fresh, const void* k_fresh, const void* v_fresh, void* kv_k, void* kv_v,
                  int32_t* idx_out, void* q_pack, void* k_pack, void* v_pack,
                  DeviceStatus* status, void* scratch, cudaStream_t stream, const Fp8Cache* fp8, bool select_only, const RowSource* far) {
    const int32_t* idx_src = idx_in;
    if (scores != nullptr && rp.L_d > 0 && rp.k > 0) {
        static std::atomic<bool> attr_done[64];   // per device; a concurrent first call sets the same values
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev >= 0 && dev < 64 && !attr_done[dev].load(std::memory_order_acquire)) {
            const cudaError_t e = cudaFuncSetAttribute(select_topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)(sizeof(SelShared) + (size_t)padded(kSelSmemKeysPerCta) * sizeof(uint32_t)));
            if (e != cudaSuccess) { set_cuda_error(e); return DAF_ERR_CUDA; }
            attr_done[dev].store(true, std::memory_order_release);
        }
        // One CTA and the cluster of eight.  The whole layer, clustered scores: 4000 tokens of 28 / 40 / 4 heads on 4 / 8 / 4 22.6 / 25.0 /
        // 19.0 us and 23.6 / 25.9 / 19.9, 3500 tokens of 28 25.8 and 26.5, 5200 of 28 25.8 and 25.8, 8192 36.9 and 36.6; scores within
        // 2^-17 of each other 22.6 and 25.2 at 4000, 25.6 and 27.4 at 5200; of either sign 24.9 and 23.9, 28.5 and 26.2.  Alone and back
        // to back the cluster is level at 3000 already (4.6 and 4.4): behind other kernels its eight CTAs start later than one.
        if (rp.L_d <= kSel1MaxKeys) {
            static_assert(sizeof(Sel1Shared) + (padded(kSel1MaxKeys) + kSel1MaxKeys) * sizeof(uint32_t) <= 48 * 1024, "within the default limit");
            const size_t smem1 = sizeof(Sel1Shared) + ((size_t)padded(rp.L_d) + rp.L_d) * sizeof(uint32_t);   // keys and candidate list
            const cudaError_t e = launch_kernel(select_topk_cta_kernel, dim3(1), dim3(kSel1Threads), smem1, stream,
                                                scores, n_sig, rp.L_d, rp.k, idx_out);
            if (e != cudaSuccess) { set_cuda_error(e); return DAF_ERR_CUDA; }
        } else {
            const size_t smem = select_smem_bytes(rp.L_d);
            const cudaError_t e = launch_kernel(select_topk_kernel, dim3(kSelCluster), dim3(kSelThreads), smem, stream,
                                                scores, n_sig, rp.L_d, rp.k,
                                                reinterpret_cast<uint32_t*>(scratch), idx_out);
            if (e != cudaSuccess) { set_cuda_error(e); return DAF_ERR_CUDA; }
        }
        count_launch();
        if (int rc = check_launch()) return rc;
        idx_src = idx_out;
    }
    // The expansion of an fp8 cache goes behind the selection kernel, which it does not depend on: it runs beside that one
    // and only waits for it before it retires, so that the gather kernel behind finds both finished.  (The other way round
    // the selection started only with the expansion's last CTAs and was left over at the end.)
    if (fp8 != nullptr)
        if (int rc = launch_expand_fp8(rp, *fp8, kv_k, kv_v, stream, /*beside_selection=*/idx_src == idx_out && idx_src != idx_in)) return rc;
    const int rows = select_only ? 0 : rp.k + rp.L_q;
    if (rows > 0) {
        GatherArgs a;
        a.q_fresh = reinterpret_cast<const int4*>(q_fresh);
        a.k_fresh = reinterpret_cast<const int4*>(k_fresh);
        a.v_fresh = reinterpret_cast<const int4*>(v_fresh);
        a.kv_k = reinterpret_cast<int4*>(kv_k);
        a.kv_v = reinterpret_cast<int4*>(kv_v);
        a.q_pack = reinterpret_cast<int4*>(q_pack);
        a.k_pack = reinterpret_cast<int4*>(k_pack);
        a.v_pack = reinterpret_cast<int4*>(v_pack);
        a.idx = idx_src;
        a.idx_copy = (idx_src == idx_in && idx_out != nullptr && idx_out != idx_in) ? idx_out : nullptr;
        a.k = rp.k; a.L_d = rp.L_d; a.L_q = rp.L_q;
        a.cq = rp.Hq * 16; a.ckv = rp.Hkv * 16;
        a.overwrite = rp.overwrite;
        a.host_k = far != nullptr ? reinterpret_cast<int4*>(far->host_k) : nullptr;
        a.host_v = far != nullptr ? reinterpret_cast<int4*>(far->host_v) : nullptr;
        a.cache_later = far != nullptr && far->cache_later;
        a.status = status;
        // Always a programmatic dependent of whatever kernel precedes it on the stream: the kernel waits for that
        // kernel to complete before it touches anything (so the result is that of a plain launch), but its CTAs are
        // already in place then -- after this library's selection kernel, and equally after the previous layer's
        // merge when layers are issued back to back.
        // Rows from host memory, read over the link, in batches of 12 KB (32 + 2 x 8 heads): one round trip covers a row.  K/V rows
        // alone by the plain loop (6k layer 31.0 us, 31.8 in batches) and 128 threads (with 192 6k layer 31.1 us, 922 rows of 32 KV
        // heads 8.3, 6.6 with 128; from 1480 rows on they no longer all fit on the GPU at once), or 192 where that is one chunk for
        // each (154 rows of 6 KV heads 1.54 us, 1.74 with 128).  With Q rows to pack as well, batches of 12 KB by 192 threads: 154 / 922 / 6554
        // rows of 28 heads on 4, in L2 / from HBM, 1.8 / 1.9, 3.7 / 3.9, 21.3 / 22.6 us; the plain loop with 192 threads 2.1 / 2.0,
        // 3.8 / 4.3, 23.1 / 24.6; batches by 128 threads 1.7 / 1.8, 4.0 / 4.1, 21.3 / 22.6, but 922 rows of 40 heads on 8 6.1 / 6.1,
        // where 192 take 5.6 / 6.1 and the plain loop 5.4 / 6.0.  A row of no more chunks than threads has nothing to batch: 922 rows
        // of 4 heads on 2 (128 chunks) 1.7 us, 2.5 as a batch of which all but one chunk is empty.
        const int chunks = (q_pack != nullptr ? a.cq : 0) + (k_pack != nullptr || a.overwrite ? 2 * a.ckv : 0);   // of an important row
        auto gather = [&](void (*kernel)(GatherArgs), int threads) {
            return launch_kernel(kernel, dim3((unsigned)rows), dim3((unsigned)threads), 0, stream, a);
        };
        const cudaError_t e = far != nullptr                      ? gather(gather_update_kernel<6, 128>, 128)
                              : chunks > 128 && chunks <= 192     ? gather(gather_update_kernel<1, 192>, 192)
                              : chunks > 192 && q_pack != nullptr ? gather(gather_update_kernel<4, 192>, 192)
                                                                  : gather(gather_update_kernel<1, 128>, 128);
        count_launch();
        if (e != cudaSuccess) { set_cuda_error(e); return DAF_ERR_CUDA; }
        if (int rc = check_launch()) return rc;
    }
    return DAF_OK;
}

// Four warps a CTA, which spreads few tokens over more SMs and leaves less of a last wave (three layers of 300 tokens of 4 heads 5.3 us,
// 5.4 with eight; 16k tokens 30.1 and 30.6).  Where four a CTA puts 64 warps on an SM and most of the grid on the GPU at once, eight,
// of which 48 fit, get more out of L2 and HBM: 6840 tokens of 4 heads 13.5 us, 14.4 with four (9 to 12 and 7.7 where L2 holds the
// rows), 11003 of 8 41 and 45.6; one layer of 11003 tokens of 8 heads that L2 holds 8.3, 8 to 13 with four.
static int signal_warps(int L_d) { return L_d > 4096 && L_d <= 12288 ? 8 : 4; }

int launch_deviation_scores(const ResolvedParams& rp, const void* k_fresh, const void* v_fresh, const void* k_cached,
                            const void* v_cached, float* scores, cudaStream_t stream) {
    if (rp.L_d == 0) return DAF_OK;
    const int warps = signal_warps(rp.L_d), blocks = (rp.L_d + warps - 1) / warps;
    const cudaError_t e = launch_kernel(warps == 8 ? deviation_scores_kernel<8> : deviation_scores_kernel<4>, dim3(blocks), dim3(warps * 32), 0, stream,
        reinterpret_cast<const int4*>(k_fresh), reinterpret_cast<const int4*>(v_fresh),
        reinterpret_cast<const int4*>(k_cached), reinterpret_cast<const int4*>(v_cached), rp.L_d, rp.Hkv * 16, scores);
    count_launch();
    if (e != cudaSuccess) { set_cuda_error(e); return DAF_ERR_CUDA; }
    return check_launch();
}

int launch_deviation_sum(const ResolvedParams& rp, int n_sig, const void* const* k_fresh, const void* const* v_fresh,
                         const void* const* k_cached, const void* const* v_cached, float* sums, cudaStream_t stream) {
    if (rp.L_d == 0) return DAF_OK;
    if (n_sig < 1 || n_sig > kMaxSignalLayers) return DAF_ERR_INVALID_ARG;
    SignalLayers layers;
    layers.n = n_sig;
    for (int l = 0; l < kMaxSignalLayers; ++l) {
        const int j = l < n_sig ? l : 0;
        layers.k_fresh[l] = reinterpret_cast<const int4*>(k_fresh[j]);
        layers.v_fresh[l] = reinterpret_cast<const int4*>(v_fresh[j]);
        layers.k_cached[l] = reinterpret_cast<const int4*>(k_cached[j]);
        layers.v_cached[l] = reinterpret_cast<const int4*>(v_cached[j]);
    }
    const int warps = signal_warps(rp.L_d), blocks = (rp.L_d + warps - 1) / warps;
    const cudaError_t e = launch_kernel(warps == 8 ? deviation_sum_kernel<8> : deviation_sum_kernel<4>, dim3(blocks), dim3(warps * 32), 0, stream, layers, rp.L_d,
                                        rp.Hkv * 16, sums);
    count_launch();
    if (e != cudaSuccess) { set_cuda_error(e); return DAF_ERR_CUDA; }
    return check_launch();
}

// ------------------------------------------------ validation of caller-given positions
// The important-token stage treats "causal in packed order" as "causal by position", which holds only if the
// positions are strictly increasing; a caller who passes idx_in can have them checked on the device: each
// position must lie in [0, L_d) and exceed the one before it.  The first offence is recorded in the status
// word (DAF_ERR_BOUNDS; where = 2 out of range, 3 not increasing; detail = the offending index into idx).
__global__ void __launch_bounds__(256)
check_indices_kernel(const int32_t* __restrict__ idx, int k, int L_d, DeviceStatus* status) {
    const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= k) return;
    const int p = idx[i];
    if (p < 0 || p >= L_d) report_status(status, DAF_ERR_BOUNDS, 2, i);
    else if (i > 0 && idx[i - 1] >= p) report_status(status, DAF_ERR_BOUNDS, 3, i);
}

int launch_check_indices(const int32_t* idx, int k, int L_d, DeviceStatus* status, cudaStream_t stream) {
    if (k <= 0) return DAF_OK;
    check_indices_kernel<<<(unsigned)((k + 255) / 256), 256, 0, stream>>>(idx, k, L_d, status);
    count_launch();
    return check_launch();
}

// ------------------------------------------------ offline cache stored in fp8
// Expands the document rows of an offline cache kept as 8-bit floating point (1 sign, 4 exponent, 3 mantissa
// bits, bias 7, no infinities) into the bf16 hybrid-cache buffer: element = bf16(scale[head] * value), the product in
// fp32, both roundings to nearest-even.  A streaming pass (1 byte read, 2 written per element).
__device__ __forceinline__ float mul_rn_keep_subnormals(float a, float b) {
    float d;
    asm("mul.rn.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ uint4 expand8(uint2 bytes, float scale) {
    const __nv_fp8x2_storage_t* pr = reinterpret_cast<const __nv_fp8x2_storage_t*>(&bytes);
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __half2_raw h2 = __nv_cvt_fp8x2_to_halfraw2(pr[i], __NV_E4M3);    // exact: every value is an fp16 value
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h2));
        w[i] = pack_bf16(mul_rn_keep_subnormals(f.x, scale), mul_rn_keep_subnormals(f.y, scale));
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// A streaming pass, read and write.  A CTA takes 256 kPer runs of 8 elements that lie together, a thread kPer of them: each warp
// reads 256 and writes 512 consecutive bytes at a time (16k tokens of 8 heads, 100 MB in all, part of whose writes stay in L2:
// 14.5 us; 18.4 with 16 elements a thread and its two stores 32 bytes apart).  Eight runs a thread keep enough loads under way
// on a full GPU; a cache of which eight would leave SMs without a CTA takes one (322 tokens of 4 heads: 2.4 us, 3.3 with eight).
template <int kPer>
__global__ void __launch_bounds__(256)
expand_fp8_cache_kernel(const uint2* __restrict__ k8, const uint2* __restrict__ v8, const float* __restrict__ k_scale,
                        const float* __restrict__ v_scale, uint4* __restrict__ kv_k, uint4* __restrict__ kv_v,
                        long long n_runs, int Hkv, int beside_selection) {
    if (!beside_selection) pdl_wait();
    pdl_launch_dependents();
    const bool is_v = blockIdx.y != 0;
    const uint2* src = is_v ? v8 : k8;
    const float* sc = is_v ? v_scale : k_scale;
    uint4* dst = is_v ? kv_v : kv_k;
    const long long r0 = (long long)blockIdx.x * (256 * kPer) + threadIdx.x;
    uint2 in[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u)
        if (r0 + u * 256 < n_runs) in[u] = __ldcs(src + r0 + u * 256);
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const long long r = r0 + u * 256;
        if (r < n_runs) dst[r] = expand8(in[u], sc != nullptr ? __ldg(sc + (unsigned)(r >> 4) % (unsigned)Hkv) : 1.0f);   // a head is 16 runs
    }
    if (beside_selection) pdl_wait();      // see launch_select
}

int launch_expand_fp8(const ResolvedParams& rp, const Fp8Cache& c, void* kv_k, void* kv_v, cudaStream_t stream, bool beside_selection) {
    const long long n_runs = (long long)rp.L_d * rp.Hkv * 16;     // per tensor
    if (n_runs == 0) return DAF_OK;
    auto ctas = [&](int per) { return (unsigned)((n_runs + 256 * per - 1) / (256 * per)); };
    const bool small = !beside_selection && 2 * ctas(8) < 148;     // (beside the selection more CTAs would only wait for it)
    const cudaError_t e = launch_kernel(small ? expand_fp8_cache_kernel<1> : expand_fp8_cache_kernel<8>, dim3(ctas(small ? 1 : 8), 2), dim3(256), 0,
                                        stream, reinterpret_cast<const uint2*>(c.k8), reinterpret_cast<const uint2*>(c.v8), c.k_scale, c.v_scale,
                                        reinterpret_cast<uint4*>(kv_k), reinterpret_cast<uint4*>(kv_v), n_runs, rp.Hkv,
                                        beside_selection ? 1 : 0);
    count_launch();
    if (e != cudaSuccess) { set_cuda_error(e); return DAF_ERR_CUDA; }
    return check_launch();
}

int launch_fuse(const ResolvedParams& rp, const int32_t* idx, const void* o_imp, const void* o_q, void* hidden,
                int32_t* row_pos_out, cudaStream_t stream) {
    const int rows = rp.k + rp.L_q;
    if (rows == 0) return DAF_OK;
    FuseArgs a;
    a.o_imp = reinterpret_cast<const int4*>(o_imp);
    a.o_q = reinterpret_cast<const int4*>(o_q);
    a.hidden = reinterpret_cast<int4*>(hidden);
    a.idx = idx; a.row_pos = row_pos_out;
    a.k = rp.k; a.L_d = rp.L_d; a.L_q = rp.L_q; a.cq = rp.Hq * 16; a.mode = rp.fuse_mode;
    const cudaError_t e = launch_kernel(fuse_rows_kernel, dim3(rows), dim3(kRowThreads), 0, stream, a);
    count_launch();
    if (e != cudaSuccess) { set_cuda_error(e); return DAF_ERR_CUDA; }
    return check_launch();
}

}  // namespace daf
