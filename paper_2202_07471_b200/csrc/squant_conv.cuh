// Layers with kernels of more than one element: a group of 32 to 256 threads takes an output channel,
// one thread a whole kernel at a time.
//
// The channel is staged in shared memory by asynchronous copies; a thread reads its kernel's K weights
// from there (for odd K the lanes of a warp fall on different banks), settles SQuant-E, SQuant-K and the
// candidate of Algorithm 3 in registers (3x3) or in place, and leaves candidate, error sum and position
// in the place of the kernel's first three weights.  SQuant-C is select_top over the kernels' candidates.
// What bounds it is the number of instructions: 9 loads, 30 for SQuant-E and about 90 for the selection
// per 3x3 kernel.  A thread with four kernels at once (128-bit loads) needs fewer of them, but leaves half
// of a short channel's threads idle, needs N to be a multiple of four and an aligned row, and its 1500
// instructions of straight code are fetched anew by every warp; this body is a loop of about 170 (ResNet-18 shapes
// 35.9 -> 31.3 us device time on a B200, with supplied scales 81 -> 58, mixed kernel sizes 57 -> 45).
#pragma once

#include "squant_rows.cuh"

namespace sq {

// Shared memory of a group: selection, the staged row (with the misalignment of the row in global
// memory), the codes (likewise).
__host__ __device__ inline int conv_bytes(int g, int nk, int K, Owner own = kGroup)
{
    return sel_bytes(g, own, K) + ((4 * nk + 12 + 15) & ~15) + ((nk + 15 + 15) & ~15);
}

// Exact SQuant-K + Algorithm 3 on a kernel of K elements whose integer perturbations (2^-30 units, sum e)
// are at P and whose SQuant-E code bytes are at cb; both are updated in place.  Out of line.
struct KernelOut64 {
    long long e;
    int v, idx;
};

__device__ __noinline__ KernelOut64 kernel_flip(int *P, unsigned char *cb, int K, bool do_k, long long e)
{
    KernelOut64 o;
    o.v = 0;
    o.idx = 0;
    if (e != 0) {
        const int sgn = e > 0 ? 1 : -1;
        const long long abs_e = e > 0 ? e : -e;
        const int k = do_k ? flip_count(abs_e) : 0;
        int flips = 0, last = -1, cand = -1;
#pragma unroll 1
        for (int r = 0; r <= k; ++r) {
            int best = 0, bi = -1;
#pragma unroll 4
            for (int i = 0; i < K; ++i) {
                const int key = sgn * P[i];
                if (key > best) { best = key; bi = i; }
            }
            if (bi < 0) break;
            if (r < k) {   // a flipped element changes sign and leaves the candidates by itself
                P[bi] -= sgn * kOne;
                cb[bi] = static_cast<unsigned char>(cb[bi] - sgn);
                last = bi;
                ++flips;
            } else {
                cand = bi;
            }
        }
        e -= static_cast<long long>(sgn) * flips * kOne;
        const int pick = (static_cast<long long>(flips) * kOne > abs_e) ? last : cand;   // Over SQuant: flip back
        if (pick >= 0) {
            o.idx = pick;
            o.v = P[pick];
        }
    }
    o.e = e;
    return o;
}

// Straight-line SQuant-K + Algorithm 3 on a kernel of K = 2 .. 7 elements (1x3, 7x1, ..), as kernel9_select:
// P are its integer perturbations, cb its staged code bytes.  With |e| <= K / 2 the flips and the candidate
// are among the (K + 1) / 2 largest keys, which an insertion network finds.  True: not settled (keys below
// 2^27 need not be ordered like the perturbations; the staged codes are then untouched).
template <int K>
__device__ __forceinline__ bool kernel_small_select(const int (&P)[K], unsigned char *cb, int &e_out, int &v_out, int &idx_out)
{
    constexpr int R = (K + 1) / 2;
    long long e = P[0];
#pragma unroll
    for (int i = 1; i < K; ++i) e += P[i];
    const int sgn = e < 0 ? -1 : 1;
    const unsigned eabs = static_cast<unsigned>(e < 0 ? -e : e);   // <= 3.5 * 2^30
    int top[R];
#pragma unroll
    for (int j = 0; j < R; ++j) top[j] = -0x7fffffff;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        int x = ((P[i] * sgn) & ~15) | (15 - i);
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int y = min(top[j], x);
            top[j] = max(top[j], x);
            x = y;
        }
    }
    const unsigned t = (eabs & static_cast<unsigned>(kOne - 1)) != 0u ? 1u : 0u;
    const unsigned jx = (eabs - t) >> 29;   // floor(2 |e|), exact halves falling to the lower value
    const bool zero = eabs == 0u;
    const int c = min(static_cast<int>(jx >> 1), R - 1);   // rank of the candidate, from 0
    int mc = top[0];
#pragma unroll
    for (int j = 1; j < R; ++j) mc = c == j ? top[j] : mc;
    if (!zero && mc < (1 << 27)) return true;
    const int k = zero ? 0 : static_cast<int>((jx + 1u) >> 1);
#pragma unroll
    for (int j = 0; j < R; ++j)
        if (j < k) {
            unsigned char *p = cb + min(~top[j] & 15, K - 1);
            *p = static_cast<unsigned char>(*p - sgn);
        }
    e_out = zero ? 0 : sgn * static_cast<int>(eabs - (static_cast<unsigned>(k) << 30));
    v_out = zero ? 0 : sgn * ((mc & ~15) - static_cast<int>((jx & 1u) << 30));   // Over: value after the flip
    idx_out = min(~mc & 15, K - 1);
    return false;
}

// The same under the clip of Sec. 2.2 and from the weights (kernel_clip), out of line.
__device__ __noinline__ KernelOut64 kernel_clip_out(float *wk, int K, float s, bool do_k, int qmin, int qmax, int8_t *ck)
{
    KernelOut64 o;
    kernel_clip(wk, K, s, do_k, qmin, qmax, ck, o.e, o.v, o.idx);
    return o;
}

// A 3x3 kernel under the clip that the straight-line selection does not settle, from its weights, scale in the range
// of the reciprocal sequence (y, s2: as in squant_e_fast).  Most have elements that lie two codes and more beyond the
// range, and every candidate is flipped.  Out of line.  (Four 512x512x3x3 layers with scales of 0.7 absmax: 59.5 us
// on a B200 with every kernel that has codes on the edge of the range settled by kernel_clip, 41.1 with all but these
// in line.)
__device__ __noinline__ KernelOut64 kernel9_beyond(float *wk, float y, float s2, int qmin, int qmax, unsigned char *ck)
{
    const float xmin = static_cast<float>(qmin) * 1073741824.0f, xmax = static_cast<float>(qmax) * 1073741824.0f;
    unsigned up = 0u, down = 0u;   // candidates
    long long e = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const float X = div_scaled(wk[i], y, s2), Xc = fminf(fmaxf(X, xmin), xmax), t = __fadd_rn(Xc, kMagic);
        const int P = __float2int_rn(__fsub_rn(__fsub_rn(t, kMagic), Xc));
        e += P;
        if (Xc != X) e += __float2ll_rn(__fsub_rn(Xc, X));
        reinterpret_cast<int *>(wk)[i] = P;
        up |= P > 0 ? 1u << i : 0u;
        down |= P < 0 ? 1u << i : 0u;
        ck[i] = static_cast<unsigned char>(__float_as_uint(t));
    }
    const int sgn = e < 0 ? -1 : 1;
    unsigned left = sgn > 0 ? up : down;
    const long long all = static_cast<long long>(__popc(left)) << 30;
    if (e * sgn < all) return kernel_flip(reinterpret_cast<int *>(wk), ck, 9, true, e);
    // at least as many flips are wanted as there are candidates, and none is one too many
#pragma unroll 1
    for (; left != 0u; left &= left - 1u) {
        unsigned char *c = ck + __ffs(left) - 1;
        *c = static_cast<unsigned char>(*c - sgn);
    }
    KernelOut64 o;
    o.e = e - sgn * all;
    o.v = 0;
    o.idx = 0;
    return o;
}

// ---------------------------------------------------------------- codes and their products to global memory
// The n codes at cel (shared memory, visible to the whole group), which are those from element `first` of
// the layer on: int8 or packed int4 (from byte first4 on), and code * s as fp32 and bfloat16.  cel has the
// misalignment of the int8 codes modulo 16.
__device__ __forceinline__ void emit_codes(const LayerDesc &L, size_t first, size_t first4, const Group &G, const unsigned char *cel, int n,
                                           float s, unsigned mode)
{
    if (!(mode & kModePackInt4)) {
        unsigned char *row = reinterpret_cast<unsigned char *>(L.codes) + first;
        const int head = min(static_cast<int>((16 - (reinterpret_cast<uintptr_t>(row) & 15)) & 15), n);
        const int nv = (n - head) >> 4, tail = head + 16 * nv;
#pragma unroll 1
        for (int i = G.t; i < nv; i += G.g)
            __stcs(reinterpret_cast<int4 *>(row + head) + i, reinterpret_cast<const int4 *>(cel + head)[i]);
#pragma unroll 1
        for (int i = G.t; i < head + (n - tail); i += G.g) {
            const int e = i < head ? i : tail + i - head;
            SQ_DBG(tail <= n && e >= 0 && e < n, 17);
            row[e] = cel[e];
        }
    } else {   // two codes per byte, low nibble = even flat index
        unsigned char *row = reinterpret_cast<unsigned char *>(L.codes) + first4;
        // eight codes at a time where the packed row is aligned, the rest byte by byte
        const int head = min(static_cast<int>((4 - (reinterpret_cast<uintptr_t>(row) & 3)) & 3), n >> 1);   // packed bytes
        const int nv = ((n >> 1) - head) >> 2, tail = head + 4 * nv;
#pragma unroll 1
        for (int i = G.t; i < nv; i += G.g) {
            const unsigned char *c = cel + 2 * (head + 4 * i);
            unsigned o = 0u;
#pragma unroll
            for (int k = 0; k < 8; ++k) o |= static_cast<unsigned>(c[k] & 15) << (4 * k);
            __stcs(reinterpret_cast<unsigned *>(row + head) + i, o);
        }
#pragma unroll 1
        for (int i = G.t; i < head + ((n + 1) >> 1) - tail; i += G.g) {
            const int b = i < head ? i : tail + i - head;
            SQ_DBG(2 * tail <= n && b >= 0 && 2 * b < n, 18);
            row[b] = static_cast<unsigned char>((cel[2 * b] & 15) | (2 * b + 1 < n ? cel[2 * b + 1] << 4 : 0));
        }
    }
    if (L.deq) {   // Algorithm 1's own return value: code * s
        float *row = L.deq + first;
        const Span sp(row, n, G.t);
        const bool words = ((reinterpret_cast<uintptr_t>(cel) - sp.r) & 3) == 0;
#pragma unroll 1
        for (int q = sp.q_lo + G.t; q < sp.q_hi; q += G.g) {
            const unsigned char *c = cel + (4 * q - sp.r);
            SQ_DBG(4 * q - sp.r >= 0 && 4 * q - sp.r + 4 <= n, 19);
            const unsigned c4 = words ? *reinterpret_cast<const unsigned *>(c) : c[0] | (c[1] << 8) | (c[2] << 16) | (static_cast<unsigned>(c[3]) << 24);
            __stcs(reinterpret_cast<float4 *>(row + (4 * q - sp.r)), make_float4(row_deq(c4, s), row_deq(c4 >> 8, s), row_deq(c4 >> 16, s), row_deq(c4 >> 24, s)));
        }
        if (sp.rag >= 0) row[sp.rag] = row_deq(cel[sp.rag], s);
    }
    if (L.deq16) {   // the same product as bfloat16
        uint16_t *row = L.deq16 + first;
        const int head = min(static_cast<int>(((8 - (reinterpret_cast<uintptr_t>(row) & 7)) & 7) >> 1), n);
        const int nv = (n - head) >> 2, tail = head + 4 * nv;
        const bool words = (reinterpret_cast<uintptr_t>(cel + head) & 3) == 0;
#pragma unroll 1
        for (int i = G.t; i < nv; i += G.g) {
            const unsigned char *c = cel + head + 4 * i;
            const unsigned c4 = words ? *reinterpret_cast<const unsigned *>(c) : c[0] | (c[1] << 8) | (c[2] << 16) | (static_cast<unsigned>(c[3]) << 24);
            const unsigned b0 = bf16_bits(row_deq(c4, s)), b1 = bf16_bits(row_deq(c4 >> 8, s));
            const unsigned b2 = bf16_bits(row_deq(c4 >> 16, s)), b3 = bf16_bits(row_deq(c4 >> 24, s));
            __stcs(reinterpret_cast<uint2 *>(row + head) + i, make_uint2(b0 | (b1 << 16), b2 | (b3 << 16)));
        }
#pragma unroll 1
        for (int i = G.t; i < head + (n - tail); i += G.g) {
            const int e = i < head ? i : tail + i - head;
            SQ_DBG(tail <= n && e >= 0 && e < n, 20);
            row[e] = static_cast<uint16_t>(bf16_bits(row_deq(cel[e], s)));
        }
    }
}

// ---------------------------------------------------------------- one channel
// KT = 3, 7, 9: kernels of that many elements with SQuant-K in the mode mask; KT = 0: any kernel size and
// mode but E|C.
// kClip: caller-supplied scales, the clip of Sec. 2.2 can fire.
// kCluster: this thread block has the kernels n0 .. n0 + nloc - 1 (n0 even).
template <int KT, bool kClip, Owner kOwn = kGroup>
__device__ __forceinline__ void conv_body(const LayerDesc &L, int m, const Group &G, unsigned char *slice, int qmax, unsigned mode,
                                          int n0 = 0, int nloc = 0)
{
    const int g = G.g, N = kOwn == kCluster ? nloc : L.N, K = KT ? KT : L.K, NK = kOwn == kCluster ? nloc * K : L.NK;   // here
    const size_t first = static_cast<size_t>(m) * L.NK + static_cast<size_t>(n0) * K;   // of these elements in the layer
    const Sel S(slice, g, kOwn, K);
    if (G.t == 0) {
        S.sc->count = 0;
        S.sc->total[0] = 0;
        clear_parts<kOwn>(S);
    }
    // ---- stage the row, take its absmax (each thread over what it has copied itself)
    const float *wrow = L.w + first;
    float *wel;
    float amax = 0.0f;
    {
        const Span sp(wrow, NK, G.t);
        float4 *buf = reinterpret_cast<float4 *>(slice + sel_bytes(g, kOwn, K));
        wel = reinterpret_cast<float *>(buf) + sp.r;
        const float4 *src = reinterpret_cast<const float4 *>(wrow - sp.r);
        const int q0 = sp.q_lo + G.t, vecs = G.rounds(sp.q_lo, sp.q_hi);   // this thread's vectors: q0, q0 + g, ..
#pragma unroll 4
        for (int i = 0; i < vecs; ++i) copy_async16(buf + q0 + i * g, src + q0 + i * g);
        if (sp.rag >= 0) copy_async4(wel + sp.rag, wrow + sp.rag);
        copy_async_wait();
#pragma unroll 4
        for (int i = 0; i < vecs; ++i) {
            const float4 v = buf[q0 + i * g];
            amax = absmax3(absmax3(amax, v.x, v.y), v.z, v.w);
        }
        if (sp.rag >= 0) amax = fmaxf(amax, fabsf(wel[sp.rag]));
    }
    unsigned char *cel;   // codes, with the misalignment of their row in global memory
    {
        unsigned char *c0 = slice + sel_bytes(g, kOwn, K) + ((4 * NK + 12 + 15) & ~15);
        cel = c0 + ((reinterpret_cast<uintptr_t>(L.codes) + first) & 15);
        SQ_DBG(reinterpret_cast<unsigned char *>(wel + NK) <= c0 && cel + NK <= slice + conv_bytes(g, NK, K, kOwn), 16);
    }

    // ---- scale
    amax = owner_absmax<kOwn>(G, amax, S);   // (its barrier: the staged weights are visible)
    float s = absmax_scale(amax, qmax);
    if (kClip && (kOwn != kCluster || L.sin)) {
        s = L.sin[m];
        if (!(s > 0.0f && s < __int_as_float(0x7f800000))) s = 1.0f;
    }

    // ---- SQuant-E, SQuant-K, candidates: one thread per kernel
    const bool do_k = KT != 0 || (mode & 2u) != 0;
    const bool fast = s >= 0x1p-60f && s <= 0x1p60f;
    const int qmin = (mode & kModeWideRange) ? -qmax - 1 : -qmax;
    float *kerr = L.kerr ? L.kerr + static_cast<size_t>(m) * L.N + n0 : nullptr;
    const float s2 = fast ? __fmul_rn(s, 0x1p-30f) : 0.0f;
    const E2 c2 = make_e2(fast ? __frcp_rn(s2) : 0.0f, s2);
    long long esum = 0;
    int hi0 = 0, lo0 = 0;   // extremes of the candidates
    // few kernels of many elements (a 7x7 stem has three per channel): a warp per kernel, lanes over its elements
    const bool by_warp = KT == 0 && !kClip && K >= 16 && 4 * N <= g;
#pragma unroll 1
    for (int n = by_warp ? G.t >> 5 : G.t; n < N; n += by_warp ? g >> 5 : g) {
        float *wk = wel + n * K;
        unsigned char *ck = cel + n * K;
        long long e = 0;
        int v = 0, idx = 0;
        if (by_warp) {
            kernel_warp(wk, K, s, do_k, reinterpret_cast<int8_t *>(ck), G.t & 31, e, v, idx);
            if ((G.t & 31) != 0) continue;
        } else if (KT == 9 && fast) {
            float2 P2[5];
            unsigned beyond = 0u;    // kClip: what clipped elements add to the kernel's sum, modulo 2^32
            float2 rests = make_float2(0.0f, 0.0f);   // the same as floats
            float size = 0.0f;       // and without signs
            {
                float w[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) w[i] = wk[i];
#pragma unroll
                for (int p = 0; p < 5; ++p) {
                    const float2 w2 = make_float2(w[2 * p], p < 4 ? w[2 * p + 1] : 0.0f);
                    float2 t;
                    if (!kClip) {
                        squant_e_fast2<true>(w2, c2, t, P2[p]);
                    } else {
                        // A flip is barred exactly where w/s lies beyond the last code: at the last code itself the perturbation
                        // is 0 and the element no candidate; the rest of its perturbation only adds to the sum.
                        const float2 x0 = __fmul2_rn(w2, c2.y);
                        const float2 X = __ffma2_rn(__ffma2_rn(x0, c2.ns2, w2), c2.y, x0);
                        const float xmax = static_cast<float>(qmax) * 1073741824.0f, xmin = static_cast<float>(qmin) * 1073741824.0f;
                        const float2 Xc = make_float2(fminf(fmaxf(X.x, xmin), xmax), fminf(fmaxf(X.y, xmin), xmax));
                        const float2 rest = __ffma2_rn(X, c2.neg1, Xc);
                        beyond += static_cast<unsigned>(__float2int_rn(rest.x)) + static_cast<unsigned>(__float2int_rn(rest.y));
                        rests = __fadd2_rn(rests, rest);
                        size = __fadd_rn(__fadd_rn(size, fabsf(rest.x)), fabsf(rest.y));
                        t = __fadd2_rn(Xc, c2.magic);
                        P2[p] = __ffma2_rn(Xc, c2.neg1, less_magic<true>(t, c2));
                    }
                    ck[2 * p] = static_cast<unsigned char>(__float_as_uint(t.x));
                    if (p < 4) ck[2 * p + 1] = static_cast<unsigned char>(__float_as_uint(t.y));
                }
            }
            const float2 s01 = __fadd2_rn(__fadd2_rn(P2[0], P2[1]), __fadd2_rn(P2[2], P2[3]));
            float ef = __fadd_rn(__fadd_rn(s01.x, s01.y), P2[4].x);
            if (kClip) ef = size < 0x1p31f ? __fadd_rn(ef, __fadd_rn(rests.x, rests.y)) : 0x1p40f;   // (further beyond: not settled here)
            const float gs = copysignf(1.0f, ef);
            const float2 G2 = make_float2(gs, gs);
            float Pk[9];
#pragma unroll
            for (int p = 0; p < 5; ++p) {
                const float2 q = __fmul2_rn(P2[p], G2);
                Pk[2 * p] = q.x;
                if (p < 4) Pk[2 * p + 1] = q.y;
            }
            int e32;
            unsigned ix;
            if (kernel9_select(Pk, ef, ck, e32, v, ix, beyond)) {   // without the clip about one in 10^5: settled exactly
                if (kClip) {
                    const KernelOut64 o = kernel9_beyond(wk, c2.y.x, s2, qmin, qmax, ck);
                    e = o.e; v = o.v; idx = o.idx;
                } else {
                    int *P = reinterpret_cast<int *>(wk);
                    const int gi = (__float_as_int(ef) >> 31) | 1;
#pragma unroll
                    for (int i = 0; i < 9; ++i) P[i] = gi * __float2int_rn(Pk[i]);
                    long long e64 = 0;
#pragma unroll
                    for (int i = 0; i < 9; ++i) e64 += P[i];
                    const KernelOut64 o = kernel_flip(P, ck, 9, true, e64);
                    e = static_cast<int>(o.e); v = o.v; idx = o.idx;
                }
            } else {
                e = e32;
                idx = static_cast<int>(ix);
            }
        } else if (kClip) {
            const KernelOut64 o = kernel_clip_out(wk, K, s, do_k, qmin, qmax, reinterpret_cast<int8_t *>(ck));
            e = o.e; v = o.v; idx = o.idx;
        } else if (KT > 1 && KT < 9 && fast) {
            int P[KT > 1 ? KT : 2];
#pragma unroll
            for (int i = 0; i < KT; ++i) {
                unsigned tb;
                squant_e_fast(wk[i], c2.y.x, s2, tb, P[i]);
                ck[i] = static_cast<unsigned char>(tb);
            }
            int e32;
            if (kernel_small_select<(KT > 1 && KT < 9 ? KT : 2)>(reinterpret_cast<const int (&)[KT > 1 && KT < 9 ? KT : 2]>(P), ck, e32, v, idx)) {
                int *Ps = reinterpret_cast<int *>(wk);
                e = 0;
#pragma unroll
                for (int i = 0; i < KT; ++i) { Ps[i] = P[i]; e += P[i]; }
                const KernelOut64 o = kernel_flip(Ps, ck, KT, true, e);
                e32 = static_cast<int>(o.e); v = o.v; idx = o.idx;
            }
            e = e32;
        } else {
            int *P = reinterpret_cast<int *>(wk);
#pragma unroll 4
            for (int i = 0; i < K; ++i) {
                int p;
                if (fast) {
                    unsigned tb;
                    squant_e_fast(wk[i], c2.y.x, s2, tb, p);
                    ck[i] = static_cast<unsigned char>(tb);
                } else {
                    int q;
                    squant_e(wk[i], s, q, p);
                    ck[i] = static_cast<unsigned char>(q);
                }
                P[i] = p;
                e += p;
            }
            const KernelOut64 o = kernel_flip(P, ck, K, do_k, e);
            e = o.e; v = o.v; idx = o.idx;
        }
        esum += e;
        if (kerr) kerr[n] = __fmul_rn(KT != 0 && !kClip ? __int2float_rn(static_cast<int>(e)) : __ll2float_rn(e), 0x1p-30f);
        // for SQuant-C, in the place of the kernel's weights (of two elements: the position is the low bit of the sum)
        int *rec = reinterpret_cast<int *>(wk);
        // a kernel that can be flipped has |e| <= 1/2
        const int es = KT != 0 && !kClip ? static_cast<int>(e) : static_cast<int>(max(min(e, 0x3fffffffll), -0x3fffffffll));
        rec[0] = v;
        rec[1] = K > 2 ? es : 2 * es + idx;
        if (K > 2) rec[2] = idx;
        hi0 = max(hi0, v);
        lo0 = min(lo0, v);
    }

    // ---- channel sum
    const bool late = KT == 0 && kOwn != kCluster && g > 32 && late_maxima(K);
    long long ec = 0;
    int up = hi0, down = -lo0;   // the channel's extremes
    if ((mode & 4u) || L.cerr) {
        if (kOwn != kCluster && g > 32 && !late) {   // the maxima that SQuant-C looks for its bound among
            S.mx[G.t] = hi0;
            S.mx[G.t + g] = -lo0;
        }
        ec = owner_sum<kOwn, kClip, kLargest>(G, S, esum, static_cast<unsigned>(esum), static_cast<int>((esum + (1 << 16)) >> 17), up, down);
    }

    // ---- SQuant-C: Algorithm 2 on the channel, keys = the kernels' candidates
    if (mode & 4u) {
        const int sgn = ec > 0 ? 1 : -1;
        const long long abs_e = ec > 0 ? ec : -ec;
        const int kc = static_cast<int>(min((abs_e + (kHalf - 1)) >> 30, 1ll << 30));   // a clipped channel's sum can be huge
        if (kc > 0) {   // uniform in the group
            const int m0 = sgn > 0 ? hi0 : -lo0;
            const Sel S(again(slice), g, kOwn, K);
            const int *mx = sgn > 0 || late ? S.mx : S.mx + g;
            const int lane = threadIdx.x & 31;
            if (late) {
                S.mx[G.t] = m0;
                G.sync();
            }
            auto count = [&](int t, int it) {
                int c;
                if (kOwn == kCluster) {
                    c = __popc(__ballot_sync(kFull, m0 >= t));
                    if (lane == 0) atomicAdd(&S.sc->found[it % 3], c);
                    if (G.t == 0) S.sc->found[(it + 1) % 3] = 0;   // (last read before the previous round's barrier)
                    return cluster_sum(&S.sc->found[it % 3]);
                }
                if (kOwn == kGroup && g <= 32) return __popc(__ballot_sync(kFull, m0 >= t));
                c = 0;
#pragma unroll 1
                for (int i = lane; i < (g >> 2); i += 32) {
                    const int4 q = reinterpret_cast<const int4 *>(mx)[i];
                    c += (q.x >= t) + (q.y >= t) + (q.z >= t) + (q.w >= t);
                }
                return __reduce_add_sync(kFull, c);
            };
            auto each = [&](int t, auto fn) {
                if (m0 < t) return;   // (m0: the thread's largest)
#pragma unroll 1
                for (int n = by_warp ? ((G.t & 31) ? N : G.t >> 5) : G.t; n < N; n += by_warp ? g >> 5 : g) {
                    const int a = reinterpret_cast<const int *>(wel)[n * K] * sgn;
                    if (a >= t) fn(a, n0 + n);
                }
            };
            auto tally = [&](int t) {
                int c = 0;
                each(t, [&](int, int) { ++c; });
                return c;
            };
            auto listing = [&](int t, auto push) { each(t, [&](int a, int n) { push(a, n, 0u); }); };   // (positions are with the kernels)
            auto flip = [&](int, int n_abs, unsigned) {
                const int n = n_abs - n0;
                const int *rec = reinterpret_cast<const int *>(wel + n * K);
                const int idx = K > 2 ? rec[2] : rec[1] & 1;
                SQ_DBG(n >= 0 && n < N && idx >= 0 && idx < K, 2);
                unsigned char *cb = cel + n * K + idx;
                *cb = static_cast<unsigned char>(*cb - sgn);
                if (kerr) kerr[n] = __fmul_rn(__int2float_rn((K > 2 ? rec[1] : rec[1] >> 1) - sgn * kOne), 0x1p-30f);
            };
            // Over-SQuant candidates reach one, but few come near it: the search starts at the largest
            const int top = (sgn > 0 ? up : down) + 1;
            const int nmax = g * (kOwn == kCluster ? static_cast<int>(cg::this_cluster().num_blocks()) : 1);
            const int k_eff = select_top<kOwn>(G, [] {}, count, listing, [] {}, tally, each, [](int) { return 0u; }, flip, nmax, false, 0, top, top, 3.0f, kc, L.N, true, S, K);
            ec -= static_cast<long long>(sgn) * k_eff * kOne;
        }
    }
    G.sync();   // all codes are final
#ifdef SQUANT_DEBUG_BOUNDS
    if (!kClip && kOwn != kCluster && ((mode & 4u) || L.cerr)) debug_check_sum(G, wrow, cel, NK, s, ec, true, S);
#endif

    const size_t ch = static_cast<size_t>(again(m)), k0 = kOwn == kCluster ? static_cast<size_t>(again(n0)) * K : 0;
    emit_codes(L, ch * L.NK + k0, ch * ((L.NK + 1) >> 1) + (k0 >> 1), G, cel, NK, s, mode);
    if (G.t == 0 && n0 == 0) {
        L.scales[m] = s;
        if (L.cerr) L.cerr[m] = __fmul_rn(__ll2float_rn(ec), 0x1p-30f);
    }
}

}  // namespace sq
