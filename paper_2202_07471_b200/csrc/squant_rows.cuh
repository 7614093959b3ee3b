// 1x1 layers (fully connected and pointwise): a group of 8 to 256 threads takes a whole output channel, up to 32
// weights a thread, or a thread block of 256 or 512 threads a longer one.
//
// Every element is its own kernel, so SQuant-K is a no-op (Sec. 3.4) and the work is absmax, SQuant-E, the channel
// sum and SQuant-C's choice of the k_c largest perturbations of one sign. What bounds such a channel is not bandwidth
// but instructions and the chain of its steps: by way of staged weights, a histogram in shared atomics and a 256-bin
// scan per channel, a ResNet-50 spent 70 thread-instructions per weight, most of them fixed costs of short channels.
// Here
//   - the weights are requested all at once and put into shared memory, each thread's for itself (no barrier); the
//     perturbations take their place, where a thread looks again only if its largest one comes into question;
//   - short channels share a warp (8 or 16 threads each), so the fixed costs are shared too;
//   - SQuant-C needs no histogram.  Each thread knows its largest candidates; a value T0 that at least k_c of those
//     maxima reach is a lower bound of the k_c-th largest candidate whatever the distribution, and few other elements
//     reach it (with k_c of m maxima about m ln(m / (m - k_c)) elements).  T0 is searched among the maxima, the
//     elements from T0 on are listed, and those of the first k_c ranks are flipped.  What that cannot settle (k_c
//     beyond the number of maxima, a full list) goes to an exact search by counting.
// With squant_conv.cuh: ResNet-50 shapes 84.5 -> 65.6 us device time on a B200.  With loops of constant strides over
// a thread's vectors (a warp of a longer row has a contiguous run of them), 22 instead of 30 thread-instructions a
// weight for SQuant-E in rows of 4096, and a list that is made at a guessed bound before any search: 2 x 4096 rows of
// 4096 weights at 8 bit 65.4 -> 55.4 us a call, 16,384 of 512 29.2 -> 23.4, 32,768 of 256 35.9 -> 26.8.
#pragma once

#include <cooperative_groups.h>

#include "squant_device.cuh"

namespace sq {

namespace cg = cooperative_groups;

constexpr int kRowVecs = 8;   // vectors of four weights a thread of a group takes; twice as many where a thread block has a row for itself

// Threads per channel for rows of `vecs` vectors (8, 16, .. 256), 0: too long for a group.
__host__ __device__ inline int row_group(int vecs)
{
    int g = 8;   // (six elements of a row can lie outside its vectors)
    while (g * kRowVecs < vecs) g *= 2;
    return g <= kCtaThreads ? g : 0;
}

// Control words of one group, followed (groups wider than a warp) by what its warps contribute to the channel's
// reductions, then by its list and by the threads' maxima.
struct SelScratch {
    int count;      // listed elements
    int total[3];   // rotating counters of the exact search
    int found[3];   // the same of the search over a cluster
    int pad;
};

// What a warp (of a cluster: a thread block) contributes: absmax (bit pattern of a non-negative float) first, then
// error sum and extremes of the candidates.
constexpr int kMaxWarps = 16;   // of a channel in one thread block
struct WarpPart {
    int lo32, hi32;   // the error sum: modulo 2^32 and, in units of 2^17, its size; or both halves of 64 bits
    int up, down;     // largest candidate of each sign
};

// Who owns a channel: a group inside a thread block, a whole thread block, a cluster of thread blocks
// (each a run of the channel's kernels; they read each other's control words and lists through
// distributed shared memory).
enum Owner { kGroup, kBlock, kCluster };
constexpr int kBlockThreads = 512;   // kBlock, kCluster
// kCluster: room for the lists of all thread blocks together.  Kernels of more than 16 elements are few
// and leave little shared memory: short lists there.
__host__ __device__ constexpr int merged_cap(int K) { return K > 16 ? 128 : 1024; }

// Warps that have a place for their parts.
__host__ __device__ constexpr int sel_warps(int g, Owner own, int K) { return g <= 32 ? 0 : (own == kGroup && K > 1 ? g >> 5 : kMaxWarps); }
// Kernels of more than nine elements: a thread's maximum is put in when the direction of the flips is known, one word
// instead of two and a barrier more, which the few kernels of such a channel hardly notice.
__host__ __device__ constexpr bool late_maxima(int K) { return K > 9; }
// Entries of a list.  Groups of eight threads: 40, with which four thread blocks with 32 rows of 256 weights each
// share a multiprocessor (with 64 three: ResNet-50 shapes 62.3 us on a B200, 57.4 with 40; mixed kernel sizes 47.1,
// 41.9; 65,536 rows of 192 weights alone 38.3, 41.1, a matter of their last wave).  Groups of 64, 128 and 256 threads
// on larger kernels: as many as make the group's selection memory 1,056, 2,144 and 3,104 B, with late maxima 1,056,
// 1,568 and 3,120 B.  The last figure is part of the longest channel of few kernels that a thread block takes; the
// others decide how many channels share one (512 channels of 106 7x7 kernels, four layers: two channels to a thread
// block 49.6 us on a B200, one 70.9).  The weights follow, so a multiple of 32 B: rows of whole 32-byte sectors
// copied to an odd multiple of 16 cost 2000 rows of 21,000 weights 98.0 us instead of 91.8.
__host__ __device__ constexpr int sel_cap(int g, int K = 1)
{
    return K == 1 ? (g == 8 ? 40 : g <= 64 ? 64 : (g > 256 ? 472 : g))   // (472: 4,128 B with the parts)
         : g > 256 ? (K > 16 ? 64 : g)
         : g <= 32 ? 64
         : late_maxima(K) ? (g == 64 ? 91 : (g == 128 ? 118 : 238))
                          : (g == 64 ? 59 : (g == 128 ? 126 : 108));
}
// Maxima that a group leaves in shared memory: one per thread and sign, of 1x1 channels two up to 64 threads.
__host__ __device__ constexpr int sel_maxima(int g, int K) { return K == 1 && g <= 64 ? 4 * g : (late_maxima(K) ? g : 2 * g); }
__host__ __device__ constexpr int sel_list_bytes(int g, Owner own, int K) { return static_cast<int>(sizeof(SelScratch)) + 20 * sel_warps(g, own, K) + 8 * sel_cap(g, K); }
__host__ __device__ constexpr int sel_bytes(int g, Owner own = kGroup, int K = 1)
{
    return sel_list_bytes(g, own, K) +
           (own == kCluster ? 8 * merged_cap(K) : (g > 32 ? 4 * sel_maxima(g, K) : 0));
}
// Shared memory of a 1x1 channel of `vecs` vectors: selection, perturbations, codes.
__host__ __device__ constexpr int row_bytes(int g, int vecs, Owner own = kGroup) { return (own == kBlock ? sel_list_bytes(g, own, 1) : sel_bytes(g, own)) + 20 * vecs; }
// The same in long_row_body (a thread block or a cluster takes the row): weights, and codes if they are to be packed.
__host__ __device__ constexpr int long_row_bytes(int g, int vecs, bool pack, Owner own) { return sel_bytes(g, own) + (pack ? 20 : 16) * vecs; }

// The parts of a group's selection memory.
struct Sel {
    SelScratch *sc;
    WarpPart *part;   // of every warp
    unsigned *amax;   // the same
    unsigned long long *list;
    int *mx;   // the threads' maxima (not kCluster: the lists of all thread blocks are there)
    int cap;
    __device__ __forceinline__ Sel(unsigned char *slice, int g, Owner own, int K)
    {
        const int warps = sel_warps(g, own, K);
        sc = reinterpret_cast<SelScratch *>(slice);
        part = reinterpret_cast<WarpPart *>(sc + 1);
        amax = reinterpret_cast<unsigned *>(part + warps);
        list = reinterpret_cast<unsigned long long *>(amax + warps);
        cap = sel_cap(g, K);
        mx = reinterpret_cast<int *>(list + cap);
    }
};

// How a run of n 4-byte elements that starts anywhere is cut into 16-byte vectors: vector q holds the
// elements 4q - r .. 4q - r + 3; those with q_lo <= q < q_hi are whole, the up to six elements outside
// them go to one thread each (rag, -1: none).
struct Span {
    int r, q_lo, q_hi, rag;
    bool ragged;   // there are such elements (uniform)
    __device__ __forceinline__ Span(const void *p, int n, int t) : Span(static_cast<int>((reinterpret_cast<uintptr_t>(p) >> 2) & 3), n, t) {}
    __device__ __forceinline__ Span(int r_, int n, int t)
    {
        r = r_;
        q_lo = min((r + 3) >> 2, (n + r + 3) >> 2);
        q_hi = max((n + r) >> 2, q_lo);
        const int head = min((4 - r) & 3, n), tail = max(4 * q_hi - r, 0);
        ragged = head > 0 || tail < n;
        rag = t < head ? t : (tail >= head && t - head < n - tail ? tail + t - head : -1);
    }
};

__device__ __forceinline__ void copy_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// max(a, |x|, |y|) in one instruction
__device__ __forceinline__ float absmax3(float a, float x, float y)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(fabsf(x)), "f"(fabsf(y)));
    return d;
}

// The same value, of which the compiler knows nothing: what follows from it is computed anew where it is used instead
// of being kept in registers through the loops before.
__device__ __forceinline__ int again(int v)
{
    asm volatile("" : "+r"(v));
    return v;
}
extern __shared__ __align__(16) unsigned char g_smem[];
__device__ __forceinline__ unsigned char *again(unsigned char *shared)
{
    return g_smem + again(static_cast<int>(smem_addr(shared) - smem_addr(g_smem)));
}

// ---------------------------------------------------------------- reductions inside a warp's group
__device__ __forceinline__ unsigned lanes_max(int g, unsigned v)
{
    if (g >= 32) return __reduce_max_sync(kFull, v);
    for (int o = g >> 1; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

__device__ __forceinline__ int lanes_add(int g, int v)
{
    if (g >= 32) return __reduce_add_sync(kFull, v);
    for (int o = g >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// ---------------------------------------------------------------- reductions over the owner of a channel
// One barrier each: a warp leaves its part in a place of its own, after the barrier every warp reads all of them.  A
// cluster's thread block adds its warps' parts up in one place (S.amax[0], S.part[0]: cleared by clear_parts, a barrier of the block
// later in use), so that a warp reads one part per thread block through distributed shared memory; reading those of all 128
// warps took 200 channels of 12,000 3x3 kernels from 152 to 175 us on a B200.
template <class T>
__device__ __forceinline__ T remote(const T *w, int rank)
{
    return *cg::this_cluster().map_shared_rank(w, rank);
}

template <Owner kOwn>
__device__ __forceinline__ void owner_sync(const Group &G)
{
    if (kOwn == kCluster) cg::this_cluster().sync();
    else if (kOwn == kBlock) __syncthreads();
    else G.sync();
}

template <Owner kOwn>
__device__ __forceinline__ void clear_parts(const Sel &S)
{
    if (kOwn != kCluster) return;
    S.amax[0] = 0u;
    *reinterpret_cast<int4 *>(S.part) = make_int4(0, 0, 0, 0);
    S.sc->found[0] = 0;
}

template <Owner kOwn>
__device__ __forceinline__ float owner_absmax(const Group &G, float amax, const Sel &S)
{
    unsigned u = lanes_max(G.g, __float_as_uint(amax));   // >= 0: uint order = float order
    const int lane = threadIdx.x & 31;
    if (kOwn == kGroup && G.g <= 32) {
        __syncwarp();   // the control words are cleared
        return __uint_as_float(u);
    }
    if (kOwn == kCluster) {
        __syncthreads();   // the words are cleared
        if (lane == 0) atomicMax(S.amax, u);
        owner_sync<kOwn>(G);
        u = lane < static_cast<int>(cg::this_cluster().num_blocks()) ? remote(S.amax, lane) : 0u;
    } else {
        if (lane == 0) S.amax[G.t >> 5] = u;
        owner_sync<kOwn>(G);
        u = S.amax[lane & ((G.g >> 5) - 1)];
    }
    return __uint_as_float(__reduce_max_sync(kFull, u));
}

// Channel-wide error sum and extremes.  k64: the sum of e; else the sum of which lo32 is a thread's value
// modulo 2^32 and apx its size in units of 2^17, off by less than 2^13 units over the channel.  kLargest: up, down
// (both >= 0) become the channel's largest, kTotal: the sums of those of the warps (groups of whole warps).
enum Extra { kNothing, kLargest, kTotal };
template <Owner kOwn, bool k64, Extra kExtra>
__device__ __forceinline__ long long owner_sum(const Group &G, const Sel &S, long long e, unsigned lo32, int apx, int &up, int &down)
{
    const int lane = threadIdx.x & 31;
    if (k64) {
        for (int o = min(G.g, 32) >> 1; o > 0; o >>= 1) e += __shfl_xor_sync(kFull, e, o);
    } else {
        lo32 = static_cast<unsigned>(lanes_add(G.g, static_cast<int>(lo32)));
        apx = lanes_add(G.g, apx);
    }
    if (kExtra == kLargest) {
        up = static_cast<int>(__reduce_max_sync(kFull, static_cast<unsigned>(up)));
        down = static_cast<int>(__reduce_max_sync(kFull, static_cast<unsigned>(down)));
    }
    if (kOwn != kGroup || G.g > 32) {
        int4 q = make_int4(0, 0, 0, 0);
        if (kOwn == kCluster) {
            if (lane == 0) {
                if (k64) {
                    atomicAdd(reinterpret_cast<unsigned long long *>(S.part), static_cast<unsigned long long>(e));   // (lo32, hi32)
                } else {
                    atomicAdd(&S.part->lo32, static_cast<int>(lo32));
                    atomicAdd(&S.part->hi32, apx);
                }
                if (kExtra == kLargest) {
                    atomicMax(&S.part->up, up);
                    atomicMax(&S.part->down, down);
                } else if (kExtra == kTotal) {
                    atomicAdd(&S.part->up, up);
                    atomicAdd(&S.part->down, down);
                }
            }
            owner_sync<kOwn>(G);
            if (lane < static_cast<int>(cg::this_cluster().num_blocks())) q = remote(reinterpret_cast<const int4 *>(S.part), lane);
        } else {
            if (lane == 0)
                *reinterpret_cast<int4 *>(S.part + (G.t >> 5)) = make_int4(k64 ? static_cast<int>(static_cast<unsigned>(e)) : static_cast<int>(lo32),
                                                                           k64 ? static_cast<int>(e >> 32) : apx, up, down);
            owner_sync<kOwn>(G);
            if (lane < (G.g >> 5)) q = reinterpret_cast<const int4 *>(S.part)[lane];
        }
        if (k64) {
            e = (static_cast<long long>(q.y) << 32) | static_cast<unsigned>(q.x);
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(kFull, e, o);
        } else {
            lo32 = static_cast<unsigned>(__reduce_add_sync(kFull, q.x));
            apx = __reduce_add_sync(kFull, q.y);
        }
        if (kExtra == kLargest) {
            up = static_cast<int>(__reduce_max_sync(kFull, static_cast<unsigned>(q.z)));
            down = static_cast<int>(__reduce_max_sync(kFull, static_cast<unsigned>(q.w)));
        } else if (kExtra == kTotal) {
            up = __reduce_add_sync(kFull, q.z);
            down = __reduce_add_sync(kFull, q.w);
        }
    }
    if (k64) return e;
    const unsigned base = static_cast<unsigned>(apx) << 17;
    return static_cast<long long>(apx) * (1ll << 17) + static_cast<int>(lo32 - base);
}

// Sum over the cluster of *w, which every thread block has completed before the barrier in here.
__device__ __forceinline__ int cluster_sum(const int *w)
{
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    const int lane = threadIdx.x & 31;
    return __reduce_add_sync(kFull, lane < static_cast<int>(cl.num_blocks()) ? remote(w, lane) : 0);
}

// absmax / qmax by IEEE division; 1 for a channel below 2^-100.
__device__ __forceinline__ float absmax_scale(float amax, int qmax)
{
    return (amax < 0x1p-100f) ? 1.0f : __fdiv_rn(amax, static_cast<float>(qmax));
}

#ifdef SQUANT_DEBUG_BOUNDS
// The channel's error sum from its final codes and the weights (global memory), compared with ec.  Called by
// every thread of the group after the codes' last barrier; groups that share a warp come together.
__device__ __forceinline__ void debug_check_sum(const Group &G, const float *w, const unsigned char *codes, int n, float s, long long ec, bool valid,
                                                const Sel &S)
{
    unsigned long long *sum64 = reinterpret_cast<unsigned long long *>(S.amax);   // (dead by now)
    long long e = 0;
    for (int j = G.t; j < n; j += G.g) e += debug_error(w[j], s, static_cast<signed char>(codes[j]));
    for (int o = min(G.g, 32) >> 1; o > 0; o >>= 1) e += __shfl_xor_sync(kFull, e, o);
    if (G.g > 32) {
        if (G.t == 0) *sum64 = 0ull;
        G.sync();
        if ((G.t & 31) == 0) atomicAdd(sum64, static_cast<unsigned long long>(e));
        G.sync();
        e = static_cast<long long>(*sum64);
    }
    if (G.t == 0 && valid) {
        SQ_DBG(e == ec, 8);
        atomicAdd(&g_debug_sums, 1u);
    }
}
#endif

// ---------------------------------------------------------------- SQuant-C: the k_c largest candidates
// Entry of a list: larger values first, equal values by lower index; the code byte comes along.
__device__ __forceinline__ unsigned long long list_key(int a, int n, unsigned code)
{
    return (static_cast<unsigned long long>(static_cast<unsigned>(a)) << 32) | (static_cast<unsigned>(~n) << 8) | (code & 255u);
}
// *w += 1, the old value.  (One instruction: the compiler would have the lanes of a warp agree on one of them first.)
__device__ __forceinline__ int shared_count(int *w)
{
    int old;
    asm volatile("atom.shared.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(smem_addr(w)) : "memory");
    return old;
}

// Whether a list from a guessed bound, which holds somewhat more than kc entries, has room for them.  (Of a cluster it is spread over the
// lists of all thread blocks.)
template <Owner kOwn>
__device__ __forceinline__ bool guess_fits(int kc, int cap) { return kOwn == kCluster ? kc < cap : kc + (kc >> 2) + 6 <= cap; }

// a = the value of a candidate in the direction of the flips, n its kernel index in the channel.  listing(t, push) calls
// push(a, n, code) for those of the thread's elements that are at least t units, 1 <= t < top (`top` is one unit above
// the largest possible); code is handed through to flip.  direct: from `start` on somewhat more than kc candidates are expected,
// which are listed without a search.  If there is no such list or it will not do, the bound is searched: the threads know maxima of a
// over parts of their elements, count(t) = how many of the group's nmax maxima are at least t (prepare() once before,
// after a list that will not do: it may write to shared memory.  Without `direct` it is not called, count must do
// without).  For the exact search: settle() once, then tally(v) = how many of the thread's elements have a >= v (any v >= 1, vtop above all),
// each(v, f) calls f(a, n) for those, code_of(n) is the code of one.  spread: the expected distance between the largest candidates in units
// of top / n_all.  flip(a, n, code) is called once for each of the min(kc, candidates) largest (equal values: lower
// index first), by some thread of the group.  want: this group selects at all (kc >= 1).  Returns the number of
// flips.  Every thread of the group calls it, groups that share a warp together; it starts with no barrier and
// ends with none.
template <Owner kOwn, class Prepare, class Count, class Listing, class Settle, class Tally, class Each, class CodeOf, class Flip>
__device__ __forceinline__ int select_top(const Group &G, Prepare prepare, Count count, Listing listing, Settle settle, Tally tally, Each each, CodeOf code_of, Flip flip,
                                          int nmax, bool direct, int start, int top, int vtop, float spread, int kc, int n_all, bool want, const Sel &S, int K)
{
    const int g = G.g, lane = threadIdx.x & 31;
    SelScratch *sc = S.sc;
    unsigned long long *list = S.list;
    const int cap = S.cap;

    // ---- the elements from `lo` on are listed.  Round 0: from `start` on.  Where those are too few or more than the list
    // holds, round 1 lists from a bound that the search has found: at least kc elements.  Where they are still more than the list
    // holds (many to a maximum: k_c is large for the number of maxima), once more from further up, supposing an even
    // spread from there to the top.  Groups that share a warp go to the exact search at once, which takes them 8 to 10 k cycles where
    // the other groups' lists, made again too, bring a second list to 16 to 24 k (ResNet-18 shapes with such a row among the last:
    // 39.0 us on a B200, 36.5).  From a warp a channel on the second list is the shorter way (4096 rows of 2048 weights 24.7 us, 28.0).
    int cnt = 0, all = 0;   // this list, all lists
    int k_eff = want ? kc : 0, lo = max(start, 1);
    const unsigned long long *merged = list;
    bool slow = false, todo = want;
    auto search = [&] {
        // T0: at least kc of the maxima reach it, and not many more.  The first guess supposes an even
        // spread; the distance to the top is doubled until it is enough, then the interval is halved (1x1:
        // 1.1 rounds on normal and heavy-tailed weights of 4 and 8 bit, 3x3: 1.3 to 2.6; the list holds about
        // kc + 3 elements for small, 1.6 kc for large kc).
        int hi = top;
        bool sure = false;   // lo has been counted
        // (Of few maxima nearly all would have to be counted, and with the last ones come far more elements than a list holds.)
        bool done = !todo || kc + (kOwn == kGroup && g < 32 ? kc >> 2 : 0) > nmax;
        const int slack = kc + (kc >> 1) + 6;
        lo = 1;
        int mid = max(top - 1 - __float2int_rz(__fmul_rn(__fmul_rn(static_cast<float>(kc) + 1.0f, spread), __fdividef(static_cast<float>(top), static_cast<float>(n_all)))), 1);
#pragma unroll 1
        for (int it = 0; __any_sync(kFull, !done); ++it) {
            const int c = count(mid, it);
            if (!done) {
                if (c >= kc) { lo = mid; sure = true; done = c <= slack; }
                else hi = mid;
                done = done || hi - lo <= 1;
                mid = sure ? lo + ((hi - lo) >> 1) : max(hi - (top - hi), 1);
            }
        }
        slow = todo && !sure;   // too few maxima
        todo = todo && sure;
    };
#pragma unroll 1
    for (int round = 0;; ++round) {
        if (round > 0 || direct) {
            if (todo && (round > 0 || guess_fits<kOwn>(kc, cap)))
                listing(lo, [&](int a, int n, unsigned code) {
                    const int pos = shared_count(&sc->count);
                    SQ_DBG(a >= 1 && a < vtop && n >= 0 && n < n_all, 12);
                    if (pos < cap) list[pos] = list_key(a, n, code);
                });
            owner_sync<kOwn>(G);
            if (todo) cnt = all = sc->count;
            bool full = false;
            if (kOwn == kCluster) {   // every thread block collects all lists
                unsigned long long *dst = list + cap;
                merged = dst;
                all = 0;
                for (int c = 0; c < static_cast<int>(cg::this_cluster().num_blocks()); ++c) {
                    const int n = remote(&sc->count, c);
                    full = full || n > cap || all + n > merged_cap(K);
                    if (!full)
                        for (int y = G.t; y < n; y += g) dst[all + y] = remote(list + y, c);
                    all += n;
                }
            } else {
                full = cnt > cap;
            }
            full = full && todo;
            bool again = todo && (full || all < kc);
            if (round > 0) {
                if (kOwn == kGroup && g < 32) {
                    slow = slow || full;
                    break;
                }
                if (again && (!full || round > 3)) {   // (fewer than kc: too far up)
                    slow = true;
                    again = false;
                }
            }
            if (kOwn == kCluster) __syncthreads();
            if (!__any_sync(kFull, again)) break;   // (uniform over groups wider than a warp)
            if (round > 0) {
                const int goal = kc + ((min(cap, kOwn == kCluster ? merged_cap(K) : cap) - kc) >> 1);
                const int up = top - __float2int_rz(__fmul_rn(static_cast<float>(top - lo), __fdividef(static_cast<float>(goal), static_cast<float>(all))));
                if (goal <= kc || up <= lo || up >= top) { again = false; slow = true; }
                else lo = up;
            }
            owner_sync<kOwn>(G);   // everybody has read the lists
            if (again && G.t == 0) sc->count = 0;
            if (round == 0 && again) prepare();
            owner_sync<kOwn>(G);
            todo = again;
        }
        if (round == 0) search();
    }
    auto flip_entry = [&](unsigned long long e) {
        const unsigned low = static_cast<unsigned>(e);
        flip(static_cast<int>(e >> 32), static_cast<int>(~low >> 8), low & 255u);
    };
    if (kOwn != kGroup && want && !slow) {   // exact ranks, a warp per entry: keys are distinct
#pragma unroll 1
        for (int x = G.t >> 5; x < cnt; x += g >> 5) {
            const unsigned long long me = list[x];
            int rank = 0;
            for (int y = lane; y < all; y += 32) rank += merged[y] > me ? 1 : 0;
            rank = __reduce_add_sync(kFull, rank);
            if (rank < kc && lane == 0) flip_entry(me);
        }
    }
    if (kOwn == kGroup && want && !slow) {   // exact ranks inside the list: keys are distinct
#pragma unroll 1
        for (int x = G.t; x < cnt; x += g) {
            const unsigned long long me = list[x];
            int rank = 0;
            if (cnt > kc) {
#pragma unroll 4
                for (int y = 0; y < cnt; ++y) rank += list[y] > me ? 1 : 0;
            }
            if (rank < kc) flip_entry(me);
        }
    }

    // ---- exact search: the value v with at most kc - 1 candidates above it and at least kc from it on, by
    // counting (eight rounds interpolate, then the interval is halved); all candidates above v are
    // flipped, and of those that tie at v the ones with the lowest indices.  It starts from the last list's bound where that holds enough.
    // The rows that need it are few, but a launch of one wave waits for them: with counts by tally(), no first list that has no room,
    // no search among too few maxima and this start 4188 rows of 512 weights with scales of half the absmax 22.6 -> 18.5 us on a
    // B200, 4096 of 1024 28.1 -> 25.3, 4096 of 200 16.4 -> 14.7, 32,768 of 512 72.5 -> 68.0, 16,384 of 256 37.0 -> 31.4.
    if (__any_sync(kFull, slow)) {   // group-uniform for groups of whole warps
        if (slow) settle();
        int vlo = 1, vhi = vtop, vm = 1, c_lo = 0, c_hi = 0, tie = 0;   // count(vlo) >= kc > count(vhi)
        int ilo = 0, ihi = n_all, im = 0;                      // ties with index < ihi suffice, with index < ilo do not
        if (kOwn == kGroup && slow && all >= kc) vm = vlo = lo;
        int phase = slow ? 0 : 2;
#pragma unroll 1
        for (int it = 0; __any_sync(kFull, phase < 2); ++it) {
            int c = 0;
            if (phase == 0) c = tally(vm);
            if (phase == 1) each(vlo, [&](int a, int n) { c += (a == vlo && n < im) ? 1 : 0; });
            c = lanes_add(g, c);
            if (g > 32) {
                if (lane == 0) atomicAdd(&sc->total[it % 3], c);
                if (G.t == 0) sc->total[(it + 1) % 3] = 0;
                G.sync();
                c = kOwn == kCluster ? cluster_sum(&sc->total[it % 3]) : sc->total[it % 3];
            }
            if (phase == 0) {
                if (it == 0 && c <= kc) { k_eff = c; vlo = vm; ihi = n_all; phase = 2; }       // all of these are flipped
                else if (c >= kc) { vlo = vm; c_lo = c; if (c == kc) phase = 2; }
                else { vhi = vm; c_hi = c; }
                if (phase == 0) {
                    if (vhi - vlo <= 1) {   // more candidates of value vlo than there is room for
                        tie = kc - c_hi;
                        phase = 1;
                        im = n_all >> 1;
                    } else if (it < 9) {
                        const float f = __fdividef(static_cast<float>(c_lo - kc) + 0.5f, static_cast<float>(c_lo - c_hi) + 0.5f);
                        vm = max(vlo + 1, min(vlo + static_cast<int>(f * static_cast<float>(vhi - vlo)), vhi - 1));
                    } else {
                        vm = vlo + ((vhi - vlo) >> 1);
                    }
                }
            } else if (phase == 1) {
                if (c >= tie) ihi = im;
                else ilo = im;
                if (c == tie || ihi - ilo <= 1) phase = 2;
                im = ilo + ((ihi - ilo) >> 1);
            }
        }
        if (slow) each(vlo, [&](int a, int n) { if (a > vlo || n < ihi) flip(a, n, code_of(n)); });
    }
    return k_eff;
}

// code (low byte of c) * s
__device__ __forceinline__ float row_deq(unsigned c, float s)
{
    return __fmul_rn(__int2float_rn(static_cast<int>(static_cast<signed char>(c & 255u))), s);
}

// two fp32 -> bfloat16, round to nearest, ties to even; a in the low half
__device__ __forceinline__ unsigned bf16_pair(float a, float b)
{
    unsigned d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}

// SQuant-E on four weights by plain IEEE division, codes clamped to [lo, hi]: for scales outside the range of the reciprocal
// sequence.  Out of line: rare, and its code would be in the way.
struct QuadDiv {
    unsigned c4;
    float P[4];
};
__device__ __noinline__ QuadDiv row_div(float4 w, float s, int lo, int hi)
{
    QuadDiv o;
    o.c4 = 0u;
    const float ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float x = __fdiv_rn(ws[c], s);
        const float q = fminf(fmaxf(rintf(x), static_cast<float>(lo)), static_cast<float>(hi));
        o.P[c] = __fmul_rn(__fsub_rn(q, x), 1073741824.0f);
        o.c4 |= (static_cast<unsigned>(__float2int_rn(q)) & 255u) << (8 * c);
    }
    return o;
}

// One element under the clip: its exact perturbation Pf goes into the 64-bit sum and, as a float,
// into o; P (Pf as an integer, saturated) becomes 0 if the element is no candidate in either direction
// because the flipped code (low byte of c) would leave the range - every clipped element among them.
__device__ __forceinline__ void row_clip_one(float Pf, int &P, unsigned c, int qmin, int qmax, long long &sum64, float &o)
{
    const bool large = !(fabsf(Pf) < 0x1p30f);
    sum64 += large ? __float2ll_rn(Pf) : static_cast<long long>(P);
    o = large ? Pf : __int2float_rn(P);
    const int q8 = static_cast<int>(static_cast<signed char>(c & 255u));
    if ((P > 0 && q8 == qmin) || (P < 0 && q8 == qmax)) P = 0;
}

// ---------------------------------------------------------------- one 1x1 channel
// Where a list for SQuant-C starts: from there on kc + kc / 4 + `more` of n_all values that are spread evenly from
// -top / 2 * spread to top / 2 * spread are expected.
__device__ __forceinline__ int list_start(int kc, float spread, int top, int n_all, float more)
{
    const float goal = static_cast<float>(kc) + static_cast<float>(kc >> 2) + more;
    return top - 1 - __float2int_rz(__fmul_rn(__fmul_rn(goal, spread), __fdividef(static_cast<float>(top), static_cast<float>(n_all))));
}

// Weights: SQuant-C of shorter rows (which groups of at most a warp take) searches its bound first, since the guess takes
// in too many of their elements (the guess / the search first, us on a B200: 131,072 rows of 64 49.2 / 45.0, 65,536 of 96
// 31.9 / 30.0, of 128 33.0 / 32.4, of 160 37.1 / 36.9, of 192 39.1 / 41.1, 32,768 of 256 29.7 / 34.4).
constexpr int kRowDirect = 176;
// Where a thread has at most two vectors (launches that do not fill the GPU, whose rows have several times the threads), the
// launch takes the time of its slowest row.  One list in 300 was too short with 6 more than kc * 5 / 4, which cost that
// row a search and a second list; with 10 it is one in 3000.  Groups of up to a warp search first: of so few
// elements to a maximum the search takes hardly too many.  us on a B200, before / with 10 / and that: 300 rows of 700
// 7.5 / 6.2 / 6.2, 1000 of 512 8.2 / 6.7 / 6.7, 2000 of 256 8.2 / 8.2 / 7.2.  With more vectors a thread the longer
// list costs more than it saves (16,384 rows of 512 23.4 / 25.6, ResNet-18 shapes 29.1 / 31.8).
constexpr int kRowFew = 2 * 4;   // elements

// What a thread knows of the perturbations it has made: their sum modulo 2^32 and as floats, the extremes over
// every other vector.
struct RowSums {
    unsigned sum;
    float2 fs;
    int hi[2], lo[2];
};

// SQuant-E on one vector by the reciprocal sequence.  Returns the codes as packed bytes.
__device__ __forceinline__ unsigned row_vector(const float4 w, const E2 &c2, RowSums &R, int which, int4 &p)
{
    float2 ta, tb, Pa, Pb;
    squant_e_fast2<true>(make_float2(w.x, w.y), c2, ta, Pa);
    squant_e_fast2<true>(make_float2(w.z, w.w), c2, tb, Pb);
    p = make_int4(__float2int_rn(Pa.x), __float2int_rn(Pa.y), __float2int_rn(Pb.x), __float2int_rn(Pb.y));
    R.fs = __fadd2_rn(R.fs, Pa);
    R.fs = __fadd2_rn(R.fs, Pb);
    R.sum += static_cast<unsigned>(p.x) + static_cast<unsigned>(p.y);
    R.sum += static_cast<unsigned>(p.z) + static_cast<unsigned>(p.w);
    R.hi[which] = __vimax3_s32(__vimax3_s32(R.hi[which], p.x, p.y), p.z, p.w);
    R.lo[which] = __vimin3_s32(__vimin3_s32(R.lo[which], p.x, p.y), p.z, p.w);
    return __byte_perm(__byte_perm(__float_as_uint(ta.x), __float_as_uint(ta.y), 0x0040),
                       __byte_perm(__float_as_uint(tb.x), __float_as_uint(tb.y), 0x0040), 0x5410);
}
__device__ __forceinline__ float4 row_error_sums(const int4 p)
{
    const float2 k30 = make_float2(0x1p-30f, 0x1p-30f);
    const float2 a = __fmul2_rn(make_float2(__int2float_rn(p.x), __int2float_rn(p.y)), k30);
    const float2 b = __fmul2_rn(make_float2(__int2float_rn(p.z), __int2float_rn(p.w)), k30);
    return make_float4(a.x, a.y, b.x, b.y);
}

// The same where the clip of Sec. 2.2 can fire; `er`: the elements' error sums.  A flip is barred exactly where w/s lies beyond the
// last code: at the last code itself the perturbation is 0 and the element no candidate.  What is left of its perturbation
// only adds to the sum: whole codes and sum64.
struct RowClip {
    float xmin, xmax;
    int whole;   // in codes
    long long sum64;
};
template <bool kErr>
__device__ __forceinline__ unsigned row_vector_clip(const float4 w, const E2 &c2, RowSums &R, RowClip &C, int which, int4 &p, float4 &er)
{
    const float2 wa = make_float2(w.x, w.y), wb = make_float2(w.z, w.w);
    const float2 xa = __fmul2_rn(wa, c2.y), xb = __fmul2_rn(wb, c2.y);
    float2 Xa = __ffma2_rn(__ffma2_rn(xa, c2.ns2, wa), c2.y, xa), Xb = __ffma2_rn(__ffma2_rn(xb, c2.ns2, wb), c2.y, xb);
    float2 ra = make_float2(0.0f, 0.0f), rb = ra;
    const bool beyond = fmaxf(fmaxf(Xa.x, Xa.y), fmaxf(Xb.x, Xb.y)) > C.xmax || fminf(fminf(Xa.x, Xa.y), fminf(Xb.x, Xb.y)) < C.xmin;
    if (beyond) {
        const float2 ya = make_float2(fminf(fmaxf(Xa.x, C.xmin), C.xmax), fminf(fmaxf(Xa.y, C.xmin), C.xmax));
        const float2 yb = make_float2(fminf(fmaxf(Xb.x, C.xmin), C.xmax), fminf(fmaxf(Xb.y, C.xmin), C.xmax));
        ra = __ffma2_rn(Xa, c2.neg1, ya);
        rb = __ffma2_rn(Xb, c2.neg1, yb);
        Xa = ya;
        Xb = yb;
        // whole codes and the rest of each
        const float2 ma = less_magic<true>(__fadd2_rn(ra, c2.magic), c2), mb = less_magic<true>(__fadd2_rn(rb, c2.magic), c2);
        const float2 fa = __ffma2_rn(ma, c2.neg1, ra), fb = __ffma2_rn(mb, c2.neg1, rb);
        const int i0 = __float2int_rn(fa.x), i1 = __float2int_rn(fa.y), i2 = __float2int_rn(fb.x), i3 = __float2int_rn(fb.y);
        C.whole += __float2int_rn(__fmul_rn(__fadd_rn(__fadd_rn(ma.x, ma.y), __fadd_rn(mb.x, mb.y)), 0x1p-30f));
        C.sum64 += static_cast<long long>(i0 + i1) + (i2 + i3);
        if (kErr) {   // (from 2^23 units on an element is whole)
            ra = __fadd2_rn(ma, make_float2(__int2float_rn(i0), __int2float_rn(i1)));
            rb = __fadd2_rn(mb, make_float2(__int2float_rn(i2), __int2float_rn(i3)));
        }
    }
    const float2 ta = __fadd2_rn(Xa, c2.magic), tb = __fadd2_rn(Xb, c2.magic);
    const float2 Pa = __ffma2_rn(Xa, c2.neg1, less_magic<true>(ta, c2)), Pb = __ffma2_rn(Xb, c2.neg1, less_magic<true>(tb, c2));
    p = make_int4(__float2int_rn(Pa.x), __float2int_rn(Pa.y), __float2int_rn(Pb.x), __float2int_rn(Pb.y));
    R.fs = __fadd2_rn(R.fs, Pa);
    R.fs = __fadd2_rn(R.fs, Pb);
    R.sum += static_cast<unsigned>(p.x) + static_cast<unsigned>(p.y);
    R.sum += static_cast<unsigned>(p.z) + static_cast<unsigned>(p.w);
    R.hi[which] = __vimax3_s32(__vimax3_s32(R.hi[which], p.x, p.y), p.z, p.w);
    R.lo[which] = __vimin3_s32(__vimin3_s32(R.lo[which], p.x, p.y), p.z, p.w);
    if (kErr) {   // (one of the two is 0)
        const float2 k30 = make_float2(0x1p-30f, 0x1p-30f);
        const float2 a = __fmul2_rn(__fadd2_rn(make_float2(__int2float_rn(p.x), __int2float_rn(p.y)), ra), k30);
        const float2 b = __fmul2_rn(__fadd2_rn(make_float2(__int2float_rn(p.z), __int2float_rn(p.w)), rb), k30);
        er = make_float4(a.x, a.y, b.x, b.y);
    }
    return __byte_perm(__byte_perm(__float_as_uint(ta.x), __float_as_uint(ta.y), 0x0040),
                       __byte_perm(__float_as_uint(tb.x), __float_as_uint(tb.y), 0x0040), 0x5410);
}

// The loops over a thread's vectors, which lie kStep vectors apart (a constant: the addresses of a step are immediates).
template <int kStep>
__device__ __forceinline__ float row_stage(float4 *w, const float4 *src, int vecs, bool whole)
{
    float amax = 0.0f;
    if (whole) {
#pragma unroll 4
        for (int i = 0; i < vecs; ++i) copy_async16(w + i * kStep, src + i * kStep);
    } else {   // packed codes of a misaligned row
#pragma unroll 1
        for (int i = 0; i < vecs; ++i)
            for (int c = 0; c < 4; ++c) copy_async4(reinterpret_cast<float *>(w + i * kStep) + c, reinterpret_cast<const float *>(src + i * kStep) + c);
    }
    copy_async_wait();
#pragma unroll 4
    for (int i = 0; i < vecs; ++i) {
        const float4 v = w[i * kStep];
        amax = absmax3(absmax3(amax, v.x, v.y), v.z, v.w);
    }
    return amax;
}
template <int kStep, bool kErr, bool kClip>
__device__ __forceinline__ void row_quantize(float4 *w, unsigned *codes, float4 *kerr, int vecs, const E2 &c2, RowSums &R, RowClip &C)
{
    auto vector = [&](int at, int which) {
        int4 p;
        float4 er;
        if (kClip) codes[at] = row_vector_clip<kErr>(w[at], c2, R, C, which, p, er);
        else codes[at] = row_vector(w[at], c2, R, which, p);
        reinterpret_cast<int4 *>(w)[at] = p;
        if (kErr) __stcs(kerr + at, kClip ? er : row_error_sums(p));
    };
#pragma unroll 1
    for (; vecs > 1; vecs -= 2) {
        if (kClip) {
            vector(0, 0);
            vector(kStep, 1);
        } else {
            const float4 w0 = w[0], w1 = w[kStep];
            int4 p0, p1;
            codes[0] = row_vector(w0, c2, R, 0, p0);
            codes[kStep] = row_vector(w1, c2, R, 1, p1);
            reinterpret_cast<int4 *>(w)[0] = p0;
            reinterpret_cast<int4 *>(w)[kStep] = p1;
            if (kErr) {
                __stcs(kerr, row_error_sums(p0));
                __stcs(kerr + kStep, row_error_sums(p1));
            }
        }
        if (kErr) kerr += 2 * kStep;
        w += 2 * kStep;
        codes += 2 * kStep;
    }
    if (vecs > 0) vector(0, 0);
}

// kClip: the clip of Sec. 2.2 can fire (caller-supplied scales): codes are clamped, sums are 64
// bit and an element whose flipped code would leave the range is no candidate.  valid = false: the
// group has no channel (its lanes take part in the warp's steps and write nothing).  kBlock: a row of the row kernel
// (see build_param_plan).  kLanes: lanes of a warp that share the row - 8 or 16: the whole group; 32: a warp or more, each warp has a
// contiguous run of vectors; 0: any of these.
template <bool kClip, Owner kOwn, int kLanes>
__device__ __forceinline__ void row_body(const LayerDesc &L, int m, const Group &group, unsigned char *slice, int qmax, unsigned mode, bool valid)
{
    static_assert(kOwn != kCluster && (kOwn == kGroup || kLanes == 32), "");
    Group G = group;
    if (kLanes != 0 && kLanes < 32) {
        G.g = kLanes;
        G.sh = kLanes == 8 ? 3 : 4;
    }
    const int g = G.g, N = valid ? L.N : 0;
    const Sel S(slice, g, kOwn, 1);
    if (G.t == 0) {
        S.sc->count = 0;
        S.sc->total[0] = 0;
    }
    const size_t first = static_cast<size_t>(m) * L.N;   // of the row in the layer
    const float *wrow = L.w + first;
    // The row is cut into vectors at 16-byte boundaries of the weights (packed codes pair elements from
    // the row's start, so there the vectors start with the row).
    const bool pack = (mode & kModePackInt4) != 0;
    const Span sp(pack ? 0 : static_cast<int>((reinterpret_cast<uintptr_t>(wrow) >> 2) & 3), N, G.t);
    const int r = sp.r, q_hi = sp.q_hi, rag = sp.rag;
    // this thread's vectors: q0, q0 + step, .., `vecs` of them
    const int sh = kLanes == 8 ? 3 : (kLanes == 16 ? 4 : (kLanes == 32 ? 5 : min(G.sh, 5))), step = 1 << sh;
    const int run = kLanes != 0 && kLanes < 32 ? 0 : (G.t >> 5) * (((q_hi - sp.q_lo + g - 1) >> G.sh) << 5);   // of the warps before this one
    const int q0 = sp.q_lo + run + (G.t & (step - 1));
    const int vecs = kLanes != 0 && kLanes < 32 ? (q_hi - q0 + step - 1) >> sh : min((q_hi - q0 + step - 1) >> sh, (q_hi - sp.q_lo + g - 1) >> G.sh);
    SQ_DBG(N >= 0 && N + r <= 4 * L.off_vi && q_hi <= L.off_vi, 14);   // the vectors' places below
    const int sel = kOwn == kBlock ? sel_list_bytes(g, kOwn, 1) : sel_bytes(g);   // (a thread block keeps no maxima in shared memory)
    int4 *Pbuf = reinterpret_cast<int4 *>(slice + sel);              // what SQuant-C may choose from
    unsigned *cbuf = reinterpret_cast<unsigned *>(slice + sel + 16 * L.off_vi);   // codes, by vectors
    int *Pel = reinterpret_cast<int *>(Pbuf) + r;                                   // the same by elements
    unsigned char *cel = reinterpret_cast<unsigned char *>(cbuf) + r;
    float *kerr = L.kerr ? L.kerr + first : nullptr;

    // ---- weights: every thread copies its vectors to shared memory, all requests at once, and takes their
    // absmax.  (Short loops, here and below: unrolled over eight vectors in registers, this body was no
    // faster than the old one, because code that every warp runs through once waits for its instructions.)
    float amax = 0.0f;
    {
        float4 *w = reinterpret_cast<float4 *>(Pbuf) + q0;
        const float4 *src = reinterpret_cast<const float4 *>(wrow - r) + q0;
        if (rag >= 0) copy_async4(Pel + rag, wrow + rag);
        const bool whole = (reinterpret_cast<uintptr_t>(src) & 15) == 0;
        if (kLanes != 0) {
            amax = row_stage<kLanes ? kLanes : 1>(w, src, vecs, whole);
        } else {
#pragma unroll 1
            for (int i = 0; i < vecs; ++i) {
                if (whole) copy_async16(w + i * step, src + i * step);
                else
                    for (int c = 0; c < 4; ++c) copy_async4(reinterpret_cast<float *>(w + i * step) + c, reinterpret_cast<const float *>(src + i * step) + c);
            }
            copy_async_wait();
#pragma unroll 2
            for (int i = 0; i < vecs; ++i) {
                const float4 v = w[i * step];
                amax = absmax3(absmax3(amax, v.x, v.y), v.z, v.w);
            }
        }
    }
    float w_rag = 0.0f;
    if (rag >= 0) w_rag = reinterpret_cast<const float *>(Pel)[rag];
    amax = fmaxf(amax, fabsf(w_rag));

    // ---- scale
    amax = owner_absmax<kOwn>(G, amax, S);
    float s = absmax_scale(amax, qmax);
    if (kClip && valid) {
        s = L.sin[m];
        if (!(s > 0.0f && s < __int_as_float(0x7f800000))) s = 1.0f;
    }

    // ---- SQuant-E: codes and perturbations; the kernels' error sums leave at once (SQuant-C corrects
    // the few it flips)
    const bool fast = s >= 0x1p-60f && s <= 0x1p60f;
    const int qmin = (mode & kModeWideRange) ? -qmax - 1 : -qmax;
    RowSums R;
    R.sum = 0u;
    R.fs = make_float2(0.0f, 0.0f);
    R.hi[0] = R.hi[1] = R.lo[0] = R.lo[1] = 0;   // of the even and the odd ones of the thread's vectors
    RowClip C;
    C.xmin = static_cast<float>(qmin) * 1073741824.0f;
    C.xmax = static_cast<float>(qmax) * 1073741824.0f;
    C.whole = 0;   // kClip: what is not in R.sum
    C.sum64 = 0;
    {
        const float s2 = fast ? __fmul_rn(s, 0x1p-30f) : 0.0f;
        const E2 c2 = make_e2(fast ? __frcp_rn(s2) : 0.0f, s2);
        const bool kvec = ((reinterpret_cast<uintptr_t>(kerr) - 4 * r) & 15) == 0;
        const float tmin = kMagic + C.xmin, tmax = kMagic + C.xmax;
        auto quantize = [&](const float4 w, int4 &p, float2 &oa, float2 &ob, int which) -> unsigned {
            float2 Pa, Pb;
            unsigned c4;
            if (fast) {
                const float2 wa = make_float2(w.x, w.y), wb = make_float2(w.z, w.w);
                float2 ta, tb;
                if (!kClip) {
                    squant_e_fast2<true>(wa, c2, ta, Pa);
                    squant_e_fast2<true>(wb, c2, tb, Pb);
                } else {
                    const float2 xa = __fmul2_rn(wa, c2.y), xb = __fmul2_rn(wb, c2.y);
                    const float2 Xa = __ffma2_rn(__ffma2_rn(xa, c2.ns2, wa), c2.y, xa), Xb = __ffma2_rn(__ffma2_rn(xb, c2.ns2, wb), c2.y, xb);
                    ta = __fadd2_rn(Xa, c2.magic);
                    tb = __fadd2_rn(Xb, c2.magic);
                    ta.x = fminf(fmaxf(ta.x, tmin), tmax);   // the clip of Sec. 2.2
                    ta.y = fminf(fmaxf(ta.y, tmin), tmax);
                    tb.x = fminf(fmaxf(tb.x, tmin), tmax);
                    tb.y = fminf(fmaxf(tb.y, tmin), tmax);
                    Pa = __ffma2_rn(Xa, c2.neg1, less_magic<true>(ta, c2));
                    Pb = __ffma2_rn(Xb, c2.neg1, less_magic<true>(tb, c2));
                }
                c4 = __byte_perm(__byte_perm(__float_as_uint(ta.x), __float_as_uint(ta.y), 0x0040),
                                 __byte_perm(__float_as_uint(tb.x), __float_as_uint(tb.y), 0x0040), 0x5410);
            } else {
                const QuadDiv d = row_div(w, s, kClip ? qmin : -255, kClip ? qmax : 255);
                c4 = d.c4;
                Pa = make_float2(d.P[0], d.P[1]);
                Pb = make_float2(d.P[2], d.P[3]);
            }
            p = make_int4(__float2int_rn(Pa.x), __float2int_rn(Pa.y), __float2int_rn(Pb.x), __float2int_rn(Pb.y));
            if (!kClip) {
                R.fs = __fadd2_rn(R.fs, Pa);
                R.fs = __fadd2_rn(R.fs, Pb);
                R.sum += static_cast<unsigned>(p.x) + static_cast<unsigned>(p.y);
                R.sum += static_cast<unsigned>(p.z) + static_cast<unsigned>(p.w);
                oa = make_float2(__int2float_rn(p.x), __int2float_rn(p.y));
                ob = make_float2(__int2float_rn(p.z), __int2float_rn(p.w));
            } else {
                row_clip_one(Pa.x, p.x, c4, qmin, qmax, C.sum64, oa.x);
                row_clip_one(Pa.y, p.y, c4 >> 8, qmin, qmax, C.sum64, oa.y);
                row_clip_one(Pb.x, p.z, c4 >> 16, qmin, qmax, C.sum64, ob.x);
                row_clip_one(Pb.y, p.w, c4 >> 24, qmin, qmax, C.sum64, ob.y);
            }
            const int h = __vimax3_s32(__vimax3_s32(p.x, p.y, p.z), p.w, 0), l = __vimin3_s32(__vimin3_s32(p.x, p.y, p.z), p.w, 0);
            if (which == 0) { R.hi[0] = max(R.hi[0], h); R.lo[0] = min(R.lo[0], l); }
            else { R.hi[1] = max(R.hi[1], h); R.lo[1] = min(R.lo[1], l); }
            const float2 k30 = make_float2(0x1p-30f, 0x1p-30f);
            oa = __fmul2_rn(oa, k30);
            ob = __fmul2_rn(ob, k30);
            return c4;
        };
        if (kLanes != 0 && __all_sync(kFull, fast && (!kerr || kvec))) {   // (uniform for groups of whole warps)
            constexpr int kStep = kLanes ? kLanes : 1;
            if (kerr) row_quantize<kStep, true, kClip>(reinterpret_cast<float4 *>(Pbuf) + q0, cbuf + q0, reinterpret_cast<float4 *>(kerr - r) + q0, vecs, c2, R, C);
            else row_quantize<kStep, false, kClip>(reinterpret_cast<float4 *>(Pbuf) + q0, cbuf + q0, nullptr, vecs, c2, R, C);
        } else {
#pragma unroll 1
            for (int i = 0; i < vecs; ++i) {
                const int q = q0 + i * step;
                int4 p;
                float2 oa, ob;
                cbuf[q] = quantize(reinterpret_cast<const float4 *>(Pbuf)[q], p, oa, ob, i & 1);
                Pbuf[q] = p;
                if (kerr) {
                    float *ke = kerr + (4 * q - r);
                    if (kvec) __stcs(reinterpret_cast<float4 *>(ke), make_float4(oa.x, oa.y, ob.x, ob.y));
                    else { ke[0] = oa.x; ke[1] = oa.y; ke[2] = ob.x; ke[3] = ob.y; }
                }
            }
        }
        if (sp.ragged) {
            int4 p;
            float2 oa, ob;
            const unsigned c4 = quantize(make_float4(w_rag, 0.0f, 0.0f, 0.0f), p, oa, ob, 0);
            if (rag >= 0) {
                cel[rag] = static_cast<unsigned char>(c4);
                Pel[rag] = p.x;
                if (kerr) kerr[rag] = oa.x;
            }
        }
    }

    // ---- channel sum.  !kClip: its value modulo 2^32 is exact, its size is known from the float sums
    // (2^16 elements of at most one half: the float sums are off by far less than 2^30)
    long long ec = 0;
    if ((mode & 4u) || L.cerr) {
        int up = 0, down = 0;
        const int apx = __float2int_rn(__fmul_rn(__fadd_rn(R.fs.x, R.fs.y), 0x1p-17f));
        if (kClip) C.sum64 += static_cast<long long>(C.whole) * kOne + static_cast<long long>(apx) * (1ll << 17) + static_cast<int>(R.sum - (static_cast<unsigned>(apx) << 17));
        ec = owner_sum<kOwn, kClip, kNothing>(G, S, C.sum64, R.sum, apx, up, down);
    }

    // ---- SQuant-C: Algorithm 2 on the channel, the perturbations are the keys
    if (mode & 4u) {
        const int sgn = ec > 0 ? 1 : -1;
        const long long abs_e = ec > 0 ? ec : -ec;
        const int kc = static_cast<int>(min((abs_e + (kHalf - 1)) >> 30, 1ll << 30));
        const bool want = kc > 0;
        if (g <= 32 ? __any_sync(kFull, want) : want) {
            const int m0 = sgn > 0 ? R.hi[0] : -R.lo[0], m1 = sgn > 0 ? R.hi[1] : -R.lo[1];
            const int sx = sgn > 0 ? 0 : -1;   // p ^ sx = the value in the direction of the flips, less one if that is downward
            // the elements of value t and more, in the vectors of `halves` (bit 0: the even ones, bit 1: the odd ones), of which a word
            // of hits holds at most eight
            SQ_DBG(vecs <= 2 * kRowVecs, 27);
            auto visit = [&](int t, unsigned halves, auto fn) {
                const int tx = t + sx;
#pragma unroll 1
                while (halves != 0u) {
                    const bool both = halves == 3u && vecs <= kRowVecs;   // in one pass
                    const int at = both ? 0 : __ffs(halves) - 1, inc = both ? 1 : 2;
                    halves = both ? 0u : halves & (halves - 1u);
                    unsigned hit = 0u, bit = 1u;   // a bit for each of these (at most 32) elements that counts
#pragma unroll 2
                    for (int i = at; i < vecs; i += inc, bit <<= 4) {
                        const int4 p = Pbuf[q0 + i * step];
                        if ((p.x ^ sx) >= tx) hit |= bit;
                        if ((p.y ^ sx) >= tx) hit |= 2u * bit;
                        if ((p.z ^ sx) >= tx) hit |= 4u * bit;
                        if ((p.w ^ sx) >= tx) hit |= 8u * bit;
                    }
#pragma unroll 1
                    for (; hit != 0u; hit &= hit - 1u) {
                        const int b = __ffs(hit) - 1, n = 4 * (q0 + (at + inc * (b >> 2)) * step) - r + (b & 3);
                        SQ_DBG(n >= 0 && n < N, 15);
                        fn((Pel[n] ^ sx) - sx, n);
                    }
                }
                if (rag >= 0) {
                    const int v = Pel[rag] ^ sx;
                    if (v >= tx) fn(v - sx, rag);
                }
            };
            auto each = [&](int t, auto fn) { visit(t, 3u, fn); };
            auto tally = [&](int t) {
                const int tx = t + sx;
                int c = rag >= 0 && (Pel[rag] ^ sx) >= tx ? 1 : 0;
#pragma unroll 4
                for (int i = 0; i < vecs; ++i) {
                    const int4 p = Pbuf[q0 + i * step];
                    c += ((p.x ^ sx) >= tx ? 1 : 0) + ((p.y ^ sx) >= tx ? 1 : 0) + ((p.z ^ sx) >= tx ? 1 : 0) + ((p.w ^ sx) >= tx ? 1 : 0);
                }
                return c;
            };
            auto listing = [&](int t, auto push) { visit(t, (m0 >= t ? 1u : 0u) | (m1 >= t ? 2u : 0u), [&](int a, int n) { push(a, n, 0u); }); };   // (the codes are here)
            const int lane = threadIdx.x & 31;
            const unsigned gmask = g >= 32 ? kFull : (((1u << g) - 1u) << (lane & ~(g - 1)));
            const int per = g > 64 ? 1 : 2;   // maxima a thread puts in
            auto prepare = [&] {
                if (kOwn == kBlock || g <= 32) return;
                if (per == 2) {
                    S.mx[G.t] = m0;
                    S.mx[G.t + g] = m1;
                } else {
                    S.mx[G.t] = max(m0, m1);
                }
            };
            auto count = [&](int t, int) {
                if (kOwn == kBlock) return __syncthreads_count(max(m0, m1) >= t);
                if (g <= 32) return __popc(__ballot_sync(kFull, m0 >= t) & gmask) + __popc(__ballot_sync(kFull, m1 >= t) & gmask);
                int c = 0;
#pragma unroll 1
                for (int i = lane; i < ((per * g) >> 2); i += 32) {
                    const int4 q = reinterpret_cast<const int4 *>(S.mx)[i];
                    c += (q.x >= t) + (q.y >= t) + (q.z >= t) + (q.w >= t);
                }
                return __reduce_add_sync(kFull, c);
            };
            auto flip = [&](int a, int n, unsigned) {
                SQ_DBG(n >= 0 && n < N, 3);
                unsigned char *cb = cel + n;
                *cb = static_cast<unsigned char>(*cb - sgn);
                if (kerr) kerr[n] = __fmul_rn(__int2float_rn(sgn > 0 ? a - kOne : kOne - a), 0x1p-30f);
            };
            const int vtop = kHalf + (1 << 14) + 1;
            const bool few = L.N <= kRowFew * g;
            // (of a clipped row kc can be huge)
            const bool direct = g > 32 || (!few && L.N >= kRowDirect && __any_sync(kFull, want && guess_fits<kOwn>(kc, S.cap)));
            const int k_eff = select_top<kOwn>(G, prepare, count, listing, [] {}, tally, each, [](int) { return 0u; }, flip, kOwn == kBlock ? g : per * g, direct,
                                               list_start(kc, 2.0f, vtop, max(N, 1), few ? 10.0f : 6.0f), vtop, vtop, 2.0f, kc, N, want, S, 1);
            ec -= static_cast<long long>(sgn) * k_eff * kOne;
        }
    }
    G.sync();   // all codes are final
#ifdef SQUANT_DEBUG_BOUNDS
    if (!kClip && ((mode & 4u) || L.cerr)) debug_check_sum(G, wrow, cel, N, s, ec, valid, S);
#endif
    if (!valid) return;

    // ---- codes, scale, channel error
    const size_t first_code = static_cast<size_t>(again(m)) * L.N;
    if (!pack) {
        unsigned char *crow = reinterpret_cast<unsigned char *>(L.codes) + first_code;
        if (((reinterpret_cast<uintptr_t>(crow) - r) & 3) == 0) {
            unsigned *dst = reinterpret_cast<unsigned *>(crow - r);
            if (((reinterpret_cast<uintptr_t>(crow) | static_cast<unsigned>(N) | (4u * r)) & 15) == 0) {   // the whole row in words of 16 bytes
#pragma unroll 2
                for (int i = G.t; i < (N >> 4); i += g) __stcs(reinterpret_cast<int4 *>(dst) + i, reinterpret_cast<const int4 *>(cbuf)[i]);
            } else {
#pragma unroll 4
                for (int i = 0; i < vecs; ++i) __stcs(dst + q0 + i * step, cbuf[q0 + i * step]);
                if (rag >= 0) crow[rag] = cel[rag];
            }
        } else {
            for (int n = G.t; n < N; n += g) crow[n] = cel[n];
        }
    } else {   // two codes per byte, low nibble = even flat index; r = 0
        unsigned char *crow = reinterpret_cast<unsigned char *>(L.codes) + static_cast<size_t>(m) * ((L.N + 1) >> 1);
        const bool two = (reinterpret_cast<uintptr_t>(crow) & 1) == 0;
#pragma unroll 1
        for (int i = 0; i < vecs; ++i) {
            const int q = q0 + i * step;
            const unsigned b = cbuf[q] & 0x0f0f0f0fu, h = b | (b >> 4);
            if (two) {
                *reinterpret_cast<unsigned short *>(crow + 2 * q) = static_cast<unsigned short>((h & 255u) | ((h >> 8) & 0xff00u));
            } else {
                crow[2 * q] = static_cast<unsigned char>(h);
                crow[2 * q + 1] = static_cast<unsigned char>(h >> 16);
            }
        }
        if (rag >= 0 && (rag & 1) == 0) crow[rag >> 1] = static_cast<unsigned char>((cel[rag] & 15) | (rag + 1 < N ? cel[rag + 1] << 4 : 0));
    }
    if (L.deq) {   // Algorithm 1's own return value: code * s
        float *dg = L.deq + first_code;
        const bool vec = ((reinterpret_cast<uintptr_t>(dg) - 4 * r) & 15) == 0;
#pragma unroll 1
        for (int i = 0; i < vecs; ++i) {
            const int q = q0 + i * step;
            const unsigned c4 = cbuf[q];
            const float4 d = make_float4(row_deq(c4, s), row_deq(c4 >> 8, s), row_deq(c4 >> 16, s), row_deq(c4 >> 24, s));
            float *o = dg + (4 * q - r);
            if (vec) __stcs(reinterpret_cast<float4 *>(o), d);
            else { o[0] = d.x; o[1] = d.y; o[2] = d.z; o[3] = d.w; }
        }
        if (rag >= 0) dg[rag] = row_deq(cel[rag], s);
    }
    if (L.deq16) {   // the same product as bfloat16
        uint16_t *dg = L.deq16 + first_code;
        const bool vec = ((reinterpret_cast<uintptr_t>(dg) - 2 * r) & 7) == 0;
#pragma unroll 1
        for (int i = 0; i < vecs; ++i) {
            const int q = q0 + i * step;
            const unsigned c4 = cbuf[q];
            const unsigned b0 = bf16_bits(row_deq(c4, s)), b1 = bf16_bits(row_deq(c4 >> 8, s));
            const unsigned b2 = bf16_bits(row_deq(c4 >> 16, s)), b3 = bf16_bits(row_deq(c4 >> 24, s));
            uint16_t *o = dg + (4 * q - r);
            if (vec) __stcs(reinterpret_cast<uint2 *>(o), make_uint2(b0 | (b1 << 16), b2 | (b3 << 16)));
            else { o[0] = static_cast<uint16_t>(b0); o[1] = static_cast<uint16_t>(b1); o[2] = static_cast<uint16_t>(b2); o[3] = static_cast<uint16_t>(b3); }
        }
        if (rag >= 0) dg[rag] = static_cast<uint16_t>(bf16_bits(row_deq(cel[rag], s)));
    }
    if (G.t == 0) {
        L.scales[m] = s;
        if (L.cerr) L.cerr[m] = __fmul_rn(__ll2float_rn(ec), 0x1p-30f);
    }
}

}  // namespace sq
