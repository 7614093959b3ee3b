// Output channels that are too long for a group of the grouped kernel: 1x1 rows of more than 8 K weights get a thread
// block of 256 or 512 threads each (by row_body, a few sizes by long_row_body here, see build_param_plan), and
// channels that do not fit one thread block's shared memory a cluster of 2, 4 or 8 of them, each with a contiguous
// run of the channel's kernels.  What a channel needs as a whole travels through distributed shared memory (plain
// loads from the other thread blocks' shared memory; no multicast anywhere): absmax, error sum, the counts of
// SQuant-C's search and the short lists of its candidates, which every thread block collects for itself, so that all
// of them take the same decisions without a leader.
//
// Channels this wide can hold 2^16 and more kernels, the size from which the one element that sits on the edge of the
// clip range (|w/s| a shade above qmax) can make it into a top-k: an element whose flipped code would leave the range
// is no candidate.  Rows look for it where it can matter, among candidates of at most 2^16 units of 2^-30, which only
// the exact search takes (rows of the row kernel are shorter); larger kernels run the body that checks every
// candidate.
//
// Two thread blocks per multiprocessor where the channel can be cut that small.
#pragma once

#include "squant_conv.cuh"

namespace sq {

static_assert(kBlockThreads == 1 << 9, "");
constexpr int kWideMaxCluster = 8;
// Longest row of the row kernel (168 KB of shared memory with packed codes or in row_body); up to here it was laid
// out and compared with the staged body of the grouped kernel.  Longer rows that fit one thread block still take that
// body, which is the slower one there: 1024 rows of 32,772 weights 318 us against 99 in this kernel, of 40,000 480
// against 116, 16 rows of 40,000 83 against 22.
constexpr int kRowBlockElems = 32768;
static_assert(kRowBlockElems <= 4 * 2 * kRowVecs * kBlockThreads, "");

// ---------------------------------------------------------------- SQuant-E on four weights of a 1x1 row
struct Quad {
    unsigned c4;       // codes, packed bytes
    int4 p;            // perturbations in units of 2^-30, those that are no candidates by reason of the clip range 0
    float2 Pa, Pb;     // the same as exact floats, nothing left out
    float2 qa, qb;     // codes * 2^30
};

struct RowQuant {
    E2 c2;
    float s;
    int qmin, qmax;
    bool fast;   // the scale is in the range of the reciprocal sequence
};

// An element whose flipped code (low byte of c) would leave the range is no candidate in that direction - every
// clipped element among them (Pf far beyond one half: P has saturated then).
__device__ __forceinline__ int row_barred(int P, unsigned c, int qmin, int qmax)
{
    const int q8 = static_cast<int>(static_cast<signed char>(c & 255u));
    return (P > 0 && q8 == qmin) || (P < 0 && q8 == qmax) ? 0 : P;
}

template <bool kClip>
__device__ __forceinline__ void row_quad_div(const float4 w, const RowQuant &R, Quad &o)
{
    const QuadDiv d = row_div(w, R.s, kClip ? R.qmin : -255, kClip ? R.qmax : 255);
    o.c4 = d.c4;
    o.Pa = make_float2(d.P[0], d.P[1]);
    o.Pb = make_float2(d.P[2], d.P[3]);
    o.qa = o.qb = make_float2(0.0f, 0.0f);   // (no use is made of them)
    o.p = make_int4(__float2int_rn(d.P[0]), __float2int_rn(d.P[1]), __float2int_rn(d.P[2]), __float2int_rn(d.P[3]));
    if (kClip) {
        o.p.x = row_barred(o.p.x, o.c4, R.qmin, R.qmax);
        o.p.y = row_barred(o.p.y, o.c4 >> 8, R.qmin, R.qmax);
        o.p.z = row_barred(o.p.z, o.c4 >> 16, R.qmin, R.qmax);
        o.p.w = row_barred(o.p.w, o.c4 >> 24, R.qmin, R.qmax);
    }
}

template <bool kClip>
__device__ __forceinline__ void row_quad(const float4 w, const RowQuant &R, Quad &o, bool &edge)
{
    const float2 wa = make_float2(w.x, w.y), wb = make_float2(w.z, w.w);
    const float2 xa = __fmul2_rn(wa, R.c2.y), xb = __fmul2_rn(wb, R.c2.y);
    const float2 Xa = __ffma2_rn(__ffma2_rn(xa, R.c2.ns2, wa), R.c2.y, xa), Xb = __ffma2_rn(__ffma2_rn(xb, R.c2.ns2, wb), R.c2.y, xb);
    float2 ta = __fadd2_rn(Xa, R.c2.magic), tb = __fadd2_rn(Xb, R.c2.magic);
    edge = false;
    if (kClip) {   // the clip of Sec. 2.2; a code on the edge of the range can be barred from a flip
        const float tmin = kMagic + static_cast<float>(R.qmin) * 1073741824.0f, tmax = kMagic + static_cast<float>(R.qmax) * 1073741824.0f;
        const float hi = fmaxf(fmaxf(ta.x, ta.y), fmaxf(tb.x, tb.y)), lo = fminf(fminf(ta.x, ta.y), fminf(tb.x, tb.y));
        edge = !(hi < tmax && lo > tmin);
        if (edge) {
            ta.x = fminf(fmaxf(ta.x, tmin), tmax);
            ta.y = fminf(fmaxf(ta.y, tmin), tmax);
            tb.x = fminf(fmaxf(tb.x, tmin), tmax);
            tb.y = fminf(fmaxf(tb.y, tmin), tmax);
        }
    }
    o.qa = less_magic(ta, R.c2);
    o.qb = less_magic(tb, R.c2);
    o.Pa = __ffma2_rn(Xa, R.c2.neg1, o.qa);
    o.Pb = __ffma2_rn(Xb, R.c2.neg1, o.qb);
    o.c4 = __byte_perm(__byte_perm(__float_as_uint(ta.x), __float_as_uint(ta.y), 0x0040),
                       __byte_perm(__float_as_uint(tb.x), __float_as_uint(tb.y), 0x0040), 0x5410);
    o.p = make_int4(__float2int_rn(o.Pa.x), __float2int_rn(o.Pa.y), __float2int_rn(o.Pb.x), __float2int_rn(o.Pb.y));
    if (kClip && edge) {
        o.p.x = row_barred(o.p.x, o.c4, R.qmin, R.qmax);
        o.p.y = row_barred(o.p.y, o.c4 >> 8, R.qmin, R.qmax);
        o.p.z = row_barred(o.p.z, o.c4 >> 16, R.qmin, R.qmax);
        o.p.w = row_barred(o.p.w, o.c4 >> 24, R.qmin, R.qmax);
    }
}

// max(-P, 0) >> 16 (upper half) and max(P, 0) >> 16 (lower half) over the four
__device__ __forceinline__ unsigned row_extremes(const int4 p)
{
    const int mx = __vimax3_s32(__vimax3_s32(p.x, p.y, p.z), p.w, 0), mn = __vimin3_s32(__vimin3_s32(p.x, p.y, p.z), p.w, 0);
    return __byte_perm(static_cast<unsigned>(mx), static_cast<unsigned>(-mn), 0x7632);
}

// ---------------------------------------------------------------- one 1x1 channel
// Rows that a whole thread block (kBlock) or a cluster takes; kCluster: this thread block has the elements n0 .. n0 +
// nloc - 1 (n0 a multiple of four).  kBlock: neither packed codes nor supplied scales.  kClip: the clip of Sec. 2.2
// can fire (caller-supplied scales): codes are clamped, sums are 64 bit and an element whose flipped code would leave
// the range is no candidate.
//
// What bounds it is the number of instructions (and their supply: code outside loops is fetched anew by every warp):
//   - codes, error sums and dequantized weights leave as SQuant-E makes them, and SQuant-C corrects the few elements
//     that it flips in global memory;
//   - the weights stay in shared memory and the perturbations are not kept: a thread remembers the extremes of each
//     quarter of its vectors (both signs, 16 bits each) and makes those of the few quarters that come into question
//     anew, which yields the code of what is flipped too;
//   - only codes that are to be packed wait in shared memory.
// Against the body of the groups, with which wide rows shared their code before: 256 rows of 100,352 weights 156 ->
// 83 us on a B200 (the checked body of supplied scales until then).  Where row_body fits it is the slower one (4096
// rows of 12,000 128 us with 512 threads, in row_body with 256 89.6): the code that runs once counts.
template <bool kClip, Owner kOwn>
__device__ __forceinline__ void long_row_body(const LayerDesc &L, int m, const Group &G, unsigned char *slice, int qmax, unsigned mode,
                                              int n0 = 0, int nloc = 0)
{
    static_assert(kOwn == kCluster || (kOwn == kBlock && !kClip), "");
    const int g = G.g, N = kOwn == kCluster ? nloc : L.N;   // elements here
    constexpr int stride = 32;   // a warp has a contiguous run of vectors
    const Sel S(slice, g, kOwn, 1);
    if (G.t == 0) {
        S.sc->count = 0;
        S.sc->total[0] = 0;
        clear_parts<kOwn>(S);
    }
    const size_t first = static_cast<size_t>(m) * L.N + n0;   // of these elements in the layer
    const float *wrow = L.w + first;
    // The row is cut into vectors at 16-byte boundaries of the weights (packed codes pair elements from
    // the row's start, so there the vectors start with the row).
    const bool pack = kOwn == kCluster && (mode & kModePackInt4) != 0;   // (packed codes of kBlock: row_body)
    int r = 0, q_lo = 0, q_hi = N >> 2, rag = -1;
    bool ragged = false;
    const bool regular = L.off_ev != 0;
    if (!regular) {
        const Span sp(pack ? 0 : static_cast<int>((reinterpret_cast<uintptr_t>(wrow) >> 2) & 3), N, G.t);
        r = sp.r; q_lo = sp.q_lo; q_hi = sp.q_hi; rag = sp.rag; ragged = sp.ragged;
    }
    SQ_DBG(N >= 0 && N + r <= 4 * L.off_vi && q_hi <= L.off_vi, 14);   // the vectors' places below
    // this thread's vectors: q0, q0 + stride, .., `vecs` of them; `rounds` is the most that any thread of the group has
    const int rounds = (q_hi - q_lo + g - 1) >> G.sh;
    const int q0 = q_lo + (G.t >> 5) * (32 * rounds) + (G.t & 31);
    const int vecs = min((q_hi - q0 + 31) >> 5, rounds);
    float4 *const wv = reinterpret_cast<float4 *>(slice + sel_bytes(g, kOwn)) + q0;
    unsigned *cbuf = reinterpret_cast<unsigned *>(slice + sel_bytes(g, kOwn) + 16 * L.off_vi);   // pack: codes, by vectors
    unsigned char *cel = reinterpret_cast<unsigned char *>(cbuf);

    // ---- weights: every thread copies its vectors to shared memory, all requests at once, and takes their absmax
    float amax = 0.0f, w_rag = 0.0f;
    {
        const float4 *src = reinterpret_cast<const float4 *>(wrow - r) + q0;
        if (regular || (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
#pragma unroll 4
            for (int i = 0; i < vecs; ++i) copy_async16(wv + i * stride, src + i * stride);
        } else {   // packed codes of a misaligned row
#pragma unroll 1
            for (int i = 0; i < vecs; ++i)
                for (int c = 0; c < 4; ++c) copy_async4(reinterpret_cast<float *>(wv + i * stride) + c, wrow + 4 * (q0 + i * stride) + c);
        }
        if (rag >= 0) w_rag = __ldcs(wrow + rag);
        copy_async_wait();
#pragma unroll 4
        for (int i = 0; i < vecs; ++i) {
            const float4 v = wv[i * stride];
            amax = absmax3(absmax3(amax, v.x, v.y), v.z, v.w);
        }
        amax = fmaxf(amax, fabsf(w_rag));
    }

    // ---- scale
    amax = owner_absmax<kOwn>(G, amax, S);
    RowQuant R;
    R.s = absmax_scale(amax, qmax);
    if (kClip) {
        R.s = L.sin[m];
        if (!(R.s > 0.0f && R.s < __int_as_float(0x7f800000))) R.s = 1.0f;
    }
    const float s = R.s;
    R.fast = s >= 0x1p-60f && s <= 0x1p60f;
    R.qmax = qmax;
    R.qmin = (mode & kModeWideRange) ? -qmax - 1 : -qmax;
    const float s2 = R.fast ? __fmul_rn(s, 0x1p-30f) : 0.0f;
    R.c2 = make_e2(R.fast ? __frcp_rn(s2) : 0.0f, s2);
    auto quad_of = [&](const float4 w, Quad &o, bool &edge) {
        edge = true;
        if (R.fast) row_quad<kClip>(w, R, o, edge);
        else row_quad_div<kClip>(w, R, o);
    };

    // ---- SQuant-E: codes and perturbations
    unsigned char *crow = reinterpret_cast<unsigned char *>(L.codes) + first;   // not pack
    float *kerr = L.kerr ? L.kerr + first : nullptr;
    float *deq = L.deq ? L.deq + first : nullptr;
    uint16_t *deq16 = L.deq16 ? L.deq16 + first : nullptr;
    unsigned sum = 0u;                      // modulo 2^32
    float2 fs = make_float2(0.0f, 0.0f);    // its size
    long long sum64 = 0;                    // kClip: the sum
    unsigned e0 = 0u, e1 = 0u, e2 = 0u, e3 = 0u;   // extremes of the quarters, the last one in e3
    const int part = (rounds + 3) >> 2;            // vectors of a quarter
    auto account = [&](const Quad &o, bool edge) {
        if (!kClip) {
            fs = __fadd2_rn(fs, __fadd2_rn(o.Pa, o.Pb));
            sum += static_cast<unsigned>(o.p.x) + static_cast<unsigned>(o.p.y);
            sum += static_cast<unsigned>(o.p.z) + static_cast<unsigned>(o.p.w);
        } else if (!edge) {
            sum64 += o.p.x + o.p.y;
            sum64 += o.p.z + o.p.w;
        } else {
            sum64 += __float2ll_rn(o.Pa.x) + __float2ll_rn(o.Pa.y) + __float2ll_rn(o.Pb.x) + __float2ll_rn(o.Pb.y);
        }
        e3 = __vmaxu2(e3, row_extremes(o.p));
    };
    // error sum of an element: its perturbation rounded to units of 2^-30 (beyond 2^23 units the float is whole)
    auto esum_of = [&](float Pf) { return __fmul_rn(fabsf(Pf) < 0x1p30f ? __int2float_rn(__float2int_rn(Pf)) : Pf, 0x1p-30f); };
    const bool plain = R.fast && !pack && !deq && !deq16 &&
                       (regular || (((reinterpret_cast<uintptr_t>(crow) - r) & 3) == 0 && (!kerr || ((reinterpret_cast<uintptr_t>(kerr) - 4 * r) & 15) == 0)));
    {
        unsigned *const cdst = reinterpret_cast<unsigned *>(crow - r) + q0;
        const float2 k30 = make_float2(0x1p-30f, 0x1p-30f);
#pragma unroll 1
        for (int ib = 0; ib < 4 * part; ib += part) {
            const int end = min(ib + part, vecs);
            e0 = e1; e1 = e2; e2 = e3; e3 = 0u;
            if (plain && !kerr) {
#pragma unroll 2
                for (int i = ib; i < end; ++i) {
                    Quad o;
                    bool edge;
                    row_quad<kClip>(wv[i * stride], R, o, edge);
                    __stcs(cdst + i * stride, o.c4);
                    account(o, edge);
                }
            } else if (plain) {
                float4 *const kdst = reinterpret_cast<float4 *>(kerr - r) + q0;
#pragma unroll 2
                for (int i = ib; i < end; ++i) {
                    Quad o;
                    bool edge;
                    row_quad<kClip>(wv[i * stride], R, o, edge);
                    __stcs(cdst + i * stride, o.c4);
                    account(o, edge);
                    float2 a, b;
                    if (!kClip || !edge) {
                        a = __fmul2_rn(make_float2(__int2float_rn(o.p.x), __int2float_rn(o.p.y)), k30);
                        b = __fmul2_rn(make_float2(__int2float_rn(o.p.z), __int2float_rn(o.p.w)), k30);
                    } else {
                        a = make_float2(esum_of(o.Pa.x), esum_of(o.Pa.y));
                        b = make_float2(esum_of(o.Pb.x), esum_of(o.Pb.y));
                    }
                    __stcs(kdst + i * stride, make_float4(a.x, a.y, b.x, b.y));
                }
            } else {   // any outputs, any alignment
#pragma unroll 1
                for (int i = ib; i < end; ++i) {
                    Quad o;
                    bool edge;
                    quad_of(wv[i * stride], o, edge);
                    account(o, edge);
                    const int q = q0 + i * stride, n = 4 * q - r;
                    if (pack) cbuf[q] = o.c4;
                    else if ((reinterpret_cast<uintptr_t>(crow + n) & 3) == 0) __stcs(reinterpret_cast<unsigned *>(crow + n), o.c4);
                    else {
                        for (int c = 0; c < 4; ++c) crow[n + c] = static_cast<unsigned char>(o.c4 >> (8 * c));
                    }
                    if (kerr) {
                        const float4 f = make_float4(esum_of(o.Pa.x), esum_of(o.Pa.y), esum_of(o.Pb.x), esum_of(o.Pb.y));
                        if ((reinterpret_cast<uintptr_t>(kerr + n) & 15) == 0) __stcs(reinterpret_cast<float4 *>(kerr + n), f);
                        else { kerr[n] = f.x; kerr[n + 1] = f.y; kerr[n + 2] = f.z; kerr[n + 3] = f.w; }
                    }
                    if (deq || deq16) {   // Algorithm 1's own return value: code * s; the same product as bfloat16
                        const float4 d = make_float4(row_deq(o.c4, s), row_deq(o.c4 >> 8, s), row_deq(o.c4 >> 16, s), row_deq(o.c4 >> 24, s));
                        if (deq) {
                            if ((reinterpret_cast<uintptr_t>(deq + n) & 15) == 0) __stcs(reinterpret_cast<float4 *>(deq + n), d);
                            else { deq[n] = d.x; deq[n + 1] = d.y; deq[n + 2] = d.z; deq[n + 3] = d.w; }
                        }
                        if (deq16) {
                            const unsigned b0 = bf16_pair(d.x, d.y), b1 = bf16_pair(d.z, d.w);
                            if ((reinterpret_cast<uintptr_t>(deq16 + n) & 7) == 0) __stcs(reinterpret_cast<uint2 *>(deq16 + n), make_uint2(b0, b1));
                            else {
                                deq16[n] = static_cast<uint16_t>(b0); deq16[n + 1] = static_cast<uint16_t>(b0 >> 16);
                                deq16[n + 2] = static_cast<uint16_t>(b1); deq16[n + 3] = static_cast<uint16_t>(b1 >> 16);
                            }
                        }
                    }
                }
            }
        }
    }
    if (ragged) {   // (its extremes go with the last quarter's)
        Quad o;
        bool edge;
        quad_of(make_float4(w_rag, 0.0f, 0.0f, 0.0f), o, edge);
        account(o, edge);
        if (rag >= 0) {
            if (pack) cel[rag] = static_cast<unsigned char>(o.c4);
            else crow[rag] = static_cast<unsigned char>(o.c4);
            if (kerr) kerr[rag] = esum_of(o.Pa.x);
            if (deq) deq[rag] = row_deq(o.c4, s);
            if (deq16) deq16[rag] = static_cast<uint16_t>(bf16_bits(row_deq(o.c4, s)));
        }
    }

    // ---- channel sum.  !kClip: its value modulo 2^32 is exact, its size is known from the float sums
    // (a thread's fewer than 2^7 elements of at most one half give partial sums below 2^36, each addition off by at
    // most 2^11, so its sum by less than 2^18; those of at most 2^12 threads by less than 2^30, and by 2^28 for the
    // rounding to units of 2^17)
    // The list of SQuant-C starts where the number of elements within `near` of one half leads one to expect somewhat
    // more than k_c (near is in units of 2^16; evenly spread values have as many elements there as the channel sum's
    // standard deviation).  The count travels with the channel sum, so that no
    // barrier is spent on a search: 256 rows of 100,352 weights 76.9 -> 71.8 us a call on a B200, 8 of 200,000 19.2
    // -> 17.0, 1000 of 25,001 58.7 -> 56.4.  Too few seen (two bits and outliers) say nothing; a cluster then
    // searches (256 rows of 100,352: 86.6 -> 88.1).
    constexpr int top = (kHalf >> 16) + 1;
    auto near_of = [](int n) { return min(max(__float2int_rn(0.58f * top * rsqrtf(static_cast<float>(n))), 1), top - 1); };
    int above = 0, below = 0;
    long long ec = 0;
    if ((mode & 4u) || L.cerr) {
        if (mode & 4u) {   // quarters whose extremes lie near one half, of either sign
            const unsigned th = static_cast<unsigned>(top - near_of(again(L.N))) << 16;
            for (const unsigned e : {e0, e1, e2, e3}) {
                above += __popc(__ballot_sync(kFull, (e << 16) >= th));
                below += __popc(__ballot_sync(kFull, e >= th));
            }
        }
        ec = owner_sum<kOwn, kClip, kTotal>(G, S, sum64, sum, __float2int_rn(__fmul_rn(__fadd_rn(fs.x, fs.y), 0x1p-17f)), above, below);
    }

    // ---- SQuant-C: Algorithm 2 on the channel, the perturbations are the keys
    if (mode & 4u) {
        const int sgn = ec > 0 ? 1 : -1;
        const long long abs_e = ec > 0 ? ec : -ec;
        const int kc = static_cast<int>(min((abs_e + (kHalf - 1)) >> 30, 1ll << 30));
        const bool want = kc > 0;
        if (want) {
            const int shl = sgn > 0 ? 16 : 0;   // the half of an extremes word that counts, to the top
            const int lane = threadIdx.x & 31;
            // units: 2^16
            auto count = [&](int t, int it) {
                const unsigned th = static_cast<unsigned>(t) << 16;
                int c;
                if (kOwn == kCluster) {
                    c = __popc(__ballot_sync(kFull, (e0 << shl) >= th)) + __popc(__ballot_sync(kFull, (e1 << shl) >= th)) +
                        __popc(__ballot_sync(kFull, (e2 << shl) >= th)) + __popc(__ballot_sync(kFull, (e3 << shl) >= th));
                    if (lane == 0) atomicAdd(&S.sc->found[it % 3], c);
                    if (G.t == 0) S.sc->found[(it + 1) % 3] = 0;   // (last read before the previous round's barrier)
                    return cluster_sum(&S.sc->found[it % 3]);
                }
                c = 0;
#pragma unroll 1
                for (int i = lane; i < (g >> 2); i += 32) {
                    const uint4 q = reinterpret_cast<const uint4 *>(S.mx)[i];
                    c += ((q.x << shl) >= th ? 1 : 0) + ((q.y << shl) >= th ? 1 : 0) + ((q.z << shl) >= th ? 1 : 0) + ((q.w << shl) >= th ? 1 : 0);
                }
                return __reduce_add_sync(kFull, c);
            };
            // of `w`, whose first element has index n, the elements with a >= v
            auto visit = [&](const float4 w, int n, int v, auto fn) {
                Quad o;
                bool edge;
                quad_of(w, o, edge);
                if (max(__vimax3_s32(o.p.x * sgn, o.p.y * sgn, o.p.z * sgn), o.p.w * sgn) < v) return;
                const int a[4] = {o.p.x * sgn, o.p.y * sgn, o.p.z * sgn, o.p.w * sgn};
                unsigned hit = (a[0] >= v ? 1u : 0u) | (a[1] >= v ? 2u : 0u) | (a[2] >= v ? 4u : 0u) | (a[3] >= v ? 8u : 0u);
#pragma unroll 1
                for (; hit != 0u; hit &= hit - 1u) {
                    const int c = __ffs(hit) - 1;
                    SQ_DBG(n + c >= 0 && n + c < N, 15);
                    fn(c & 2 ? (c & 1 ? a[3] : a[2]) : (c & 1 ? a[1] : a[0]), n0 + n + c, (o.c4 >> (8 * c)) & 255u);
                }
            };
            auto visit_rag = [&](int v, auto fn) {
                if (rag >= 0) visit(make_float4(w_rag, 0.0f, 0.0f, 0.0f), rag, v, fn);   // (zeros have no perturbation)
            };
            auto listing = [&](int t, auto push) {
                const unsigned th = static_cast<unsigned>(t) << 16;
                unsigned hit = ((e0 << shl) >= th ? 1u : 0u) | ((e1 << shl) >= th ? 2u : 0u) | ((e2 << shl) >= th ? 4u : 0u) | ((e3 << shl) >= th ? 8u : 0u);
                if (ragged && (hit & 8u)) visit_rag(t << 16, push);
#pragma unroll 1
                for (; hit != 0u; hit &= hit - 1u) {
                    const int ib = (__ffs(hit) - 1) * part, end = min(ib + part, vecs);
#pragma unroll 1
                    for (int i = ib; i < end; ++i) visit(wv[i * stride], 4 * (q0 + i * stride) - r, t << 16, push);
                }
            };
            // the exact search keeps the perturbations in the place of the weights
            int p_rag = 0;
            auto settle = [&] {
                // From 2^16 elements on the one on the edge of the range, a shade beyond it (its perturbation is at most one
                // unit in the last place of qmax), can be among the k_c largest; its flip is barred.
                const bool bar = !kClip && kOwn == kCluster && L.N >= 65536;
                auto of = [&](const float4 w) {
                    Quad o;
                    bool edge;
                    quad_of(w, o, edge);
                    if (bar) {
                        o.p.x = row_barred(o.p.x, o.c4, R.qmin, R.qmax);
                        o.p.y = row_barred(o.p.y, o.c4 >> 8, R.qmin, R.qmax);
                        o.p.z = row_barred(o.p.z, o.c4 >> 16, R.qmin, R.qmax);
                        o.p.w = row_barred(o.p.w, o.c4 >> 24, R.qmin, R.qmax);
                    }
                    return o.p;
                };
#pragma unroll 1
                for (int i = 0; i < vecs; ++i) reinterpret_cast<int4 *>(wv)[i * stride] = of(wv[i * stride]);
                if (rag >= 0) p_rag = of(make_float4(w_rag, 0.0f, 0.0f, 0.0f)).x;
            };
            auto each = [&](int v, auto fn) {
                const int up = sgn > 0 ? v : 0x7fffffff, down = sgn > 0 ? -0x7fffffff - 1 : -v;   // a >= v is p >= up or p <= down
#pragma unroll 1
                for (int i = 0; i < vecs; ++i) {
                    const int4 p = reinterpret_cast<const int4 *>(wv)[i * stride];
                    const int n = n0 + 4 * (q0 + i * stride) - r;
                    if (p.x >= up || p.x <= down) fn(abs(p.x), n);
                    if (p.y >= up || p.y <= down) fn(abs(p.y), n + 1);
                    if (p.z >= up || p.z <= down) fn(abs(p.z), n + 2);
                    if (p.w >= up || p.w <= down) fn(abs(p.w), n + 3);
                }
                if (p_rag >= up || p_rag <= down) fn(abs(p_rag), n0 + rag);
            };
            auto tally = [&](int v) {
                int c = 0;
                each(v, [&](int, int) { ++c; });
                return c;
            };
            auto code_of = [&](int n_abs) { return static_cast<unsigned>(pack ? cel[n_abs - n0] : crow[n_abs - n0]); };
            auto flip = [&](int a, int n_abs, unsigned code) {
                const int n = n_abs - n0;
                SQ_DBG(n >= 0 && n < N, 3);
                const unsigned c = code - static_cast<unsigned>(sgn);
                if (pack) cel[n] = static_cast<unsigned char>(c);
                else crow[n] = static_cast<unsigned char>(c);
                if (kerr) kerr[n] = __fmul_rn(__int2float_rn(sgn > 0 ? a - kOne : kOne - a), 0x1p-30f);
                if (deq) deq[n] = row_deq(c, s);
                if (deq16) deq16[n] = static_cast<uint16_t>(bf16_bits(row_deq(c, s)));
            };
            const int nmax = kOwn == kCluster ? 4 * g * static_cast<int>(cg::this_cluster().num_blocks()) : g;
            auto prepare = [&] {
                if (kOwn != kCluster) S.mx[G.t] = static_cast<int>(__vmaxu2(__vmaxu2(e0, e1), __vmaxu2(e2, e3)));
            };
            const int seen = sgn > 0 ? above : below;
            const float goal = __fadd_rn(__fmul_rn(static_cast<float>(kc), 1.3f), 10.0f);
            const int start = top - 1 - __float2int_rn(__fmul_rn(goal, __fdividef(static_cast<float>(near_of(again(L.N))), static_cast<float>(max(seen, 1)))));
            // (A thread block lists from the guess however few it has seen: a search and its list cost more.  1000 rows of 25,001
            // weights at two bits with outliers 58.4 us on a B200, with the search first 64.6, without outliers 59.2 and 64.2.)
            const bool direct = kOwn != kCluster || seen >= 24;
            const int k_eff = select_top<kOwn>(G, prepare, count, listing, settle, tally, each, code_of, flip, nmax, direct, start, top, kHalf + (1 << 14) + 1, 2.0f, kc, L.N, want, S, 1);
            ec -= static_cast<long long>(sgn) * k_eff * kOne;
        }
    }
#ifdef SQUANT_DEBUG_BOUNDS
    G.sync();   // all codes are final
    if (!kClip && kOwn != kCluster && ((mode & 4u) || L.cerr)) debug_check_sum(G, wrow, pack ? cel : crow, N, s, ec, true, S);
#endif

    // ---- packed codes, scale, channel error
    if (pack) {   // two codes per byte, low nibble = even flat index; r = 0
        G.sync();   // all codes are final
        unsigned char *prow = reinterpret_cast<unsigned char *>(L.codes) + static_cast<size_t>(m) * ((L.N + 1) >> 1) + (n0 >> 1);
        const bool two = (reinterpret_cast<uintptr_t>(prow) & 1) == 0;
#pragma unroll 1
        for (int i = 0; i < vecs; ++i) {
            const int q = q0 + i * stride;
            const unsigned b = cbuf[q] & 0x0f0f0f0fu, h = b | (b >> 4);
            if (two) {
                *reinterpret_cast<unsigned short *>(prow + 2 * q) = static_cast<unsigned short>((h & 255u) | ((h >> 8) & 0xff00u));
            } else {
                prow[2 * q] = static_cast<unsigned char>(h);
                prow[2 * q + 1] = static_cast<unsigned char>(h >> 16);
            }
        }
        if (rag >= 0 && (rag & 1) == 0) prow[rag >> 1] = static_cast<unsigned char>((cel[rag] & 15) | (rag + 1 < N ? cel[rag + 1] << 4 : 0));
    }
    if (G.t == 0 && n0 == 0) {
        L.scales[m] = s;
        if (L.cerr) L.cerr[m] = __fmul_rn(__ll2float_rn(ec), 0x1p-30f);
    }
}

// Rows of more than 8 K weights, one thread block per output channel.  kLong: by long_row_body, else by row_body.
// Which form a row takes: build_param_plan.
template <int kThreads, bool kLong>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads)
squant_row_kernel(const __grid_constant__ LaunchTable tbl, int qmax, unsigned mode)
{
    extern __shared__ __align__(16) unsigned char smem[];
    next_launch_may_start();
    const int item = blockIdx.x;
    int layer = 0;
#pragma unroll 1
    for (int step = tbl.top_step; step > 0; step >>= 1)
        if (layer + step < tbl.n_layers && tbl.first_item[layer + step] <= item) layer += step;
    const LayerDesc &L = tbl.layers[layer];
    Group G;
    G.g = kThreads;
    G.sh = kThreads == 256 ? 8 : 9;
    G.t = threadIdx.x;
    G.bar = 0;
    const int m = item - tbl.first_item[layer];
    if (kLong) {
        SQ_DBG(long_row_bytes(kThreads, L.off_vi, false, kBlock) <= static_cast<int>(dynamic_smem_bytes()) && !L.sin && !(mode & kModePackInt4), 10);
        long_row_body<false, kBlock>(L, m, G, smem, qmax, mode);
    } else {
        SQ_DBG(row_bytes(kThreads, L.off_vi, kBlock) <= static_cast<int>(dynamic_smem_bytes()), 10);
        if (L.sin) row_body<true, kBlock, 32>(L, m, G, smem, qmax, mode, true);
        else row_body<false, kBlock, 32>(L, m, G, smem, qmax, mode, true);
    }
    end_after_launch_before(mode);
}

// Shared memory of one of a cluster's thread blocks that has `kpc` kernels of K weights.
__host__ __device__ inline long long wide_bytes(int kpc, int K, bool pack)
{
    const long long nk = static_cast<long long>(kpc) * K;
    if (nk > (1 << 20)) return 1ll << 30;
    return K == 1 ? long_row_bytes(kBlockThreads, (kpc + 6) >> 2, pack, kCluster) : conv_bytes(kBlockThreads, static_cast<int>(nk), K, kCluster);
}

// One output channel per cluster; grid = channels * cluster size.  L.off_vi = vectors of a run (1x1).
__global__ void __launch_bounds__(kBlockThreads, 2)
squant_wide_kernel(const LayerDesc L, int qmax, unsigned mode, int kpc)
{
    extern __shared__ __align__(16) unsigned char smem[];
    next_launch_may_start();
    cg::cluster_group cluster = cg::this_cluster();
    const int C = static_cast<int>(cluster.num_blocks()), rank = static_cast<int>(cluster.block_rank());
    const int m = static_cast<int>(blockIdx.x) / C;
    const int n0 = min(rank * kpc, L.N), nloc = min(L.N - n0, kpc);   // this thread block's kernels
    Group G;
    G.g = kBlockThreads;
    G.sh = 9;
    G.t = threadIdx.x;
    G.bar = 0;
    SQ_DBG(wide_bytes(kpc, L.K, (mode & kModePackInt4) != 0) <= static_cast<long long>(dynamic_smem_bytes()), 11);
    const bool range = L.sin != nullptr || L.N >= 65536;   // a flip can be barred by the clip range
    if (L.K == 1) {
        if (L.sin) long_row_body<true, kCluster>(L, m, G, smem, qmax, mode, n0, nloc);
        else long_row_body<false, kCluster>(L, m, G, smem, qmax, mode, n0, nloc);
    } else if (L.K == 9 && (mode & 2u)) {
        if (range) conv_body<9, true, kCluster>(L, m, G, smem, qmax, mode, n0, nloc);
        else conv_body<9, false, kCluster>(L, m, G, smem, qmax, mode, n0, nloc);
    } else {
        if (range) conv_body<0, true, kCluster>(L, m, G, smem, qmax, mode, n0, nloc);
        else conv_body<0, false, kCluster>(L, m, G, smem, qmax, mode, n0, nloc);
    }
    cluster.sync();   // no thread block leaves while another may still read its shared memory
    end_after_launch_before(mode);
}

}  // namespace sq
