// The tile passes over window records.
//
// What a lane needs to know of its row of an event's window -- which pixels,
// from which stored column, at which offset u from the chord centre -- depends
// on the event, the grid and the tiling only, not on the image.  k_records
// works it out once per upload (row_span, the same decision as the passes of
// tsp_mlem.cuh take) and stores it: 8 bytes a lane,
//   x = u at the lane's traversal origin (float bits),
//   y = stored index of that pixel in the tile region (16 bits),
//       pairs on the chord of the first / second pixel stream (8 bits each),
// and 64 bytes an event of polynomial coefficients (EvC), so that the passes
// form a row's constants in about twenty multiply-adds.
//
// Why: with the row setup in the pass, 2.5e9 of the 4.3e9 warp instructions of
// a 1e6-event 1 mm pass (58%) were outside the pixel loops' arithmetic and
// memory operations, and issue slots bound the pass.  The records are read once
// per pass at 32 G lanes x 8 bytes an event (1 KB at 1 mm, 512 B at 2 mm, 256 B
// at 4 mm), 10 GB a pass for 1e7 events at 1 mm, copied to shared memory an
// event ahead.  MLEM passes: 1e7 events at 1 mm 42.9 -> 34.4 ms, 1e7 at 4 mm
// 6.22 -> 3.53 ms, 1e6 at 2 mm 2.28 -> 1.66 ms (before the steps below).  Writing
// them costs an upload 1.1 ms per 1e6 events at 1 mm (1.5 with the coefficients
// worked out by one lane a warp), 0.65 at 2 mm.
#pragma once

#include "tsp_mlem.cuh"
#include "tsp_row_bound.h"

namespace tsp {

// Coefficients of an event's row constants as polynomials in y and Dy = y - y~:
//   Q(u) = q0 + y (q1 + q2 y) + g1 y u,    aCb = a1 y u + Dy (b1 y + b2),
//   C0 = log2K - hB Dy^2,   ksu = sqrt(log2(e) iz) of the event,
// stored as float4 (y~, mid, q0, q1), (q2, g1, a1, b1), (b2, hB, log2K, ksu) and
// (max, z~, t, c2i): an upper bound of P over the window (window_bound, row_p_bound), and the
// event's geometry, which the gradient pass needs;
// mid is the middle row of the window (lane rows count outward from it).  P is
// held times 2^-pshift (see Geo).
constexpr int kEvcFloat4 = 4;

__device__ __forceinline__ void make_evc(const Geo& g, const EvSig& es, const float4& ev, int mid,
                                         bool loose, float4* __restrict__ out)
{
    const float yt = ev.x, t = ev.z, c2i = ev.w;
    const float il4 = 4.0f * g.il * c2i, iz2 = 2.0f * es.iz * c2i;
    const float cross = il4 * fmaf(2.0f * t, t, 1.0f);
    float q0 = iz2 * c2i * g.R * g.R;
    float q1 = -cross * yt;
    const float q2 = iz2 * c2i + il4 * t * t + cross;
    float b2 = 0.0f;
    if (g.gR8 != 0.0f) {
        const float sec = sqrtf(c2i), r = g.gR8 * t * c2i * sec;
        q0 = fmaf(r, yt, q0);
        q1 -= 2.0f * r;
        b2 = -g.gR4 * c2i * sec;
    }
    out[0] = make_float4(yt, (float)mid, q0, q1);
    out[1] = make_float4(q2, -2.0f * iz2 * t, -iz2, il4 * t);
    const float log2K = es.log2K - g.pshift;
    out[2] = make_float4(b2, g.half_log2e * il4, log2K, es.ksu);
    const WindowBound b = window_bound(g, es, ev);
    // (row by row from 0 in k_records, if it is loose)
    out[3] = make_float4(loose ? 0.0f
                               : 1.001f * exp2f(fmaf(2.0f * g.half_log2e, b.slack, log2K)) *
                                     rsqrtf(b.q),
                         ev.y, t, c2i);
}

// Lane rows count outward from the middle of the window (see event_rows).
__device__ __forceinline__ int lane_row(int rowi)
{
    return (rowi & 1) ? (rowi >> 1) + 1 : -(rowi >> 1);
}

// Records of the events of the plain items: a block takes an item, or (grid.y > 1,
// short lists) every grid.y-th run of 8 of its events.  A thread an event for the
// coefficients, then a warp per (event, 32-lane block).  (The coefficients by one
// lane of the warp that has an event's first block were 5 to 20% of the kernel's
// instructions, and so was the division of the task index by G.)
template <int LMAX, int NSEG>
__global__ void __launch_bounds__(256)
k_records(Inst p, const int4* __restrict__ items, int n_items, uint2* __restrict__ recs,
          float4* __restrict__ evc)
{
    constexpr int kRun = 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Geo& g = p.g;
    const int G = p.G;
    for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
        const int4 item = items[it];
        const Frame f = tile_frame(g, p.tl, item.x);
        for (int k = threadIdx.x; k < item.z; k += 256) {
            if ((k / kRun) % gridDim.y != blockIdx.y) continue;
            const int e = item.y + k;
            const float4 ev = p.evs.geo[e];
            const int2 rws = p.evs.rows[e];
            make_evc(g, ev_sig(g, ev), ev, rws.x + (((rws.y & kEvRowsMask) - 1) >> 1),
                     (rws.y & kEvLoose) != 0, evc + (size_t)e * kEvcFloat4);
        }
        __syncthreads();        // (the bounds below start at the coefficients' 0)
        for (int j0 = blockIdx.y * kRun; j0 < item.z; j0 += kRun * gridDim.y) {
            const int jn = min(kRun, item.z - j0);
            int j = 0, blk = warp;
            for (;; blk += 8) {
                while (blk >= G) {
                    blk -= G;
                    ++j;
                }
                if (j >= jn) break;
                const int e = item.y + j0 + j;
                const float4 ev = p.evs.geo[e];
                int2 rws = p.evs.rows[e];
                const int evflags = rws.y & ~kEvRowsMask;
                rws.y &= kEvRowsMask;
                const EvSig es = ev_sig(g, ev);
                const int mid = (rws.y - 1) >> 1;
                const int rowi = (NSEG == 1 ? blk : blk >> 1) * 32 + lane;
                const int ri = mid + lane_row(rowi);
                const bool valid = ri >= 0 && ri < rws.y;
                unsigned long long* qc = &p.accum->rec_qclip;
                unsigned long long* lc = &p.accum->rec_lclip;
                RowSpan<true> sp;
                if constexpr (NSEG == 1)
                    sp = row_span<kAlt, LMAX, true, false>(g, es, ev, p.evs.geo64 + e, rws.x + ri, valid,
                                                    evflags, f, qc, lc);
                else if ((blk & 1) == 0)
                    sp = row_span<kPos, LMAX, true, false>(g, es, ev, p.evs.geo64 + e, rws.x + ri, valid,
                                                    evflags, f, qc, lc);
                else
                    sp = row_span<kNeg, LMAX, true, false>(g, es, ev, p.evs.geo64 + e, rws.x + ri, valid,
                                                    evflags, f, qc, lc);
                int la, lb;
                if constexpr (NSEG == 1) {
                    la = sp.lim_odd >> 1;
                    lb = (sp.lim_even + 1) >> 1;
                } else {
                    la = (sp.lim_odd + 1) >> 1;
                    lb = sp.lim_odd >> 1;
                }
                const float u0 = sp.has ? fmaf((float)sp.o, g.dz, g.z0) - sp.c.zc : 0.0f;
                if (evflags & kEvLoose) {
                    float bound = 0.0f;
                    if (sp.has) {
                        float alpha, beta;
                        row_acb(g, es, ev, sp.c, alpha, beta);
                        const float ulo = fmaf((float)sp.c.lo, g.dz, g.z0) - sp.c.zc;
                        bound = row_p_bound(sp.Qc, sp.gam2, alpha, beta, ulo,
                                            fmaf((float)(sp.c.count - 1), g.dz, ulo),
                                            es.log2K - g.pshift - g.half_log2e * sp.c.B0, es.iz,
                                            g.half_log2e);
                    }
                    // (positive floats compare as their bits do)
                    const unsigned most = __reduce_max_sync(0xffffffffu, __float_as_uint(bound));
                    if (lane == 0)
                        atomicMax(reinterpret_cast<unsigned*>(evc + (size_t)e * kEvcFloat4 + 3), most);
                }
                recs[((size_t)e * G + blk) * 32 + lane] =
                    make_uint2(__float_as_uint(u0), (unsigned)sp.sidx | (unsigned)la << 16 |
                                                        (unsigned)lb << 24);
            }
        }
    }
}

// A warp's staging slot in shared memory: its lanes' records, then the event's
// coefficients.  The next event's are copied (cp.async) while this one is
// evaluated, so that their latency stays behind a whole event without holding
// registers (fourteen, which the pixel loops of the 64-register kernels would
// spill).
__device__ __forceinline__ void rec_fetch(unsigned slot, const uint2* rp, const float4* ep, int lane)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(slot + 8u * lane), "l"(rp)
                 : "memory");
    if (lane < kEvcFloat4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(slot + 256u + 16u * lane),
                     "l"(ep + lane)
                     : "memory");
}

__device__ __forceinline__ void rec_wait()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
}

__device__ __forceinline__ float lds32(unsigned a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ float4 lds128(unsigned a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}

// An event's coefficients and a lane's record.
struct RecIn {
    uint2 r;
    float4 a, b, c;
};

__device__ __forceinline__ void rec_take(RecIn& x, unsigned slot, int lane)
{
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];"
                 : "=r"(x.r.x), "=r"(x.r.y) : "r"(slot + 8u * lane) : "memory");
    x.a = lds128(slot + 256u);
    x.b = lds128(slot + 272u);
    x.c = lds128(slot + 288u);
}

// aCb along a row, for the gradient pass: B0 + d dB.
struct GradC {
    float2 B0, dB;
};

// The row's constants, as pairs, from the event's coefficients (rowoff: lane
// row, counted from the window's middle).  GRAD: e0, e1, e2 hold C0, s at the
// origin and its step, so that the exponent is formed as C0 - s^2 (see p1g_pair).
template <int TRAV, bool GRAD>
__device__ __forceinline__ PairC rec_row(const Geo& g, const RecIn& x, float rowoff, float& y,
                                         float& Dy, float& u0, GradC* gc)
{
    u0 = __uint_as_float(x.r.x);
    y = fmaf(x.a.y + rowoff, g.dy, g.y0);
    Dy = y - x.a.x;
    const float Qc = fmaf(y, fmaf(x.b.x, y, x.a.w), x.a.z);
    const float gam = x.b.y * y, al = x.b.z * y, be = Dy * fmaf(x.b.w, y, x.c.x);
    const float Q0 = fmaf(gam, u0, Qc), dQ = gam * g.dz;
    // (the event's coefficients give aCb; the exponent has it times kA)
    float A0 = fmaf(al, u0, be);
    if (GRAD) {
        const float dB = al * g.dz;
        gc->B0 = make_float2(A0, A0);
        gc->dB = make_float2(dB, dB);
    }
    A0 *= g.kA;
    // (not al (kA dz): see rec_grad_row)
    const float dA = al * g.kA * g.dz;
    const float C0 = fmaf(-x.c.y * Dy, Dy, x.c.z);
    const float su0 = x.c.w * u0, dsu = x.c.w * g.dz;
    const float e0 = GRAD ? C0 : fmaf(-su0, su0, C0), e1 = GRAD ? su0 : -2.0f * su0 * dsu,
                e2 = GRAD ? dsu : -(dsu * dsu);
    PairC c;
    c.Q0 = make_float2(Q0, Q0);
    c.dQ = make_float2(dQ, dQ);
    c.A0 = make_float2(A0, A0);
    c.dA = make_float2(dA, dA);
    c.e0 = make_float2(e0, e0);
    c.e1 = make_float2(e1, e1);
    c.e2 = make_float2(e2, e2);
    c.inc = make_float2((float)pair_step0<TRAV>(), (float)pair_step1<TRAV>());
    return c;
}

// Pass 1 of the MLEM and log-likelihood forms: pairs 1 .. kmax, P kept in tensor
// memory (ST), P rho' summed.  GLD: the rho' region is the block's transposed one in
// global memory, a pixel step a column of it.  Chunks of eight and four pairs without any
// test up to kfast, then chunks of four and two that zero P beyond each
// stream's last pair.  Returns the number of pairs stored.
template <int TRAV, int LMAX, bool ST, bool GLD, class Addr>
__device__ __forceinline__ int rec_pass1(Addr base, int la, int lb, const PairC& c, int kfast,
                                         int kmax, float2& D2, unsigned tma)
{
    constexpr int kStep = GLD ? 4 * kScrRows : 4;
    constexpr int s0 = kStep * pair_step0<TRAV>(), s1 = kStep * pair_step1<TRAV>();
    Addr a0 = base + (Addr)(long long)(kStep * pair_d0<TRAV>(1));
    Addr a1 = base + (Addr)(long long)(kStep * pair_d1<TRAV>(1));
    float2 kk = make_float2((float)pair_d0<TRAV>(1), (float)pair_d1<TRAV>(1));
    unsigned col = tma;
    int k = 1;
#define TSP_P1(PRED, J) \
    p1_pair<!GLD, false, PRED, false, (J) * s0, (J) * s1>(a0, a1, k + (J), la, lb, c, kk, D2)
    if constexpr (LMAX >= 24) {
        for (; k + 7 <= kfast; k += 8) {
            float x[16];
            float2 t;
            t = TSP_P1(false, 0), x[0] = t.x, x[1] = t.y;
            t = TSP_P1(false, 1), x[2] = t.x, x[3] = t.y;
            t = TSP_P1(false, 2), x[4] = t.x, x[5] = t.y;
            t = TSP_P1(false, 3), x[6] = t.x, x[7] = t.y;
            t = TSP_P1(false, 4), x[8] = t.x, x[9] = t.y;
            t = TSP_P1(false, 5), x[10] = t.x, x[11] = t.y;
            t = TSP_P1(false, 6), x[12] = t.x, x[13] = t.y;
            t = TSP_P1(false, 7), x[14] = t.x, x[15] = t.y;
            if constexpr (ST) tm_st16(col, x);
            a0 += (Addr)(long long)(8 * s0);
            a1 += (Addr)(long long)(8 * s1);
            col += 16;
        }
    }
    for (; k + 3 <= kfast; k += 4) {
        const float2 pa = TSP_P1(false, 0), pb = TSP_P1(false, 1);
        const float2 pc = TSP_P1(false, 2), pd = TSP_P1(false, 3);
        if constexpr (ST) tm_st8(col, pa.x, pa.y, pb.x, pb.y, pc.x, pc.y, pd.x, pd.y);
        a0 += (Addr)(long long)(4 * s0);
        a1 += (Addr)(long long)(4 * s1);
        col += 8;
    }
    for (; k + 2 <= kmax; k += 4) {
        const float2 pa = TSP_P1(true, 0), pb = TSP_P1(true, 1);
        const float2 pc = TSP_P1(true, 2), pd = TSP_P1(true, 3);
        if constexpr (ST) tm_st8(col, pa.x, pa.y, pb.x, pb.y, pc.x, pc.y, pd.x, pd.y);
        a0 += (Addr)(long long)(4 * s0);
        a1 += (Addr)(long long)(4 * s1);
        col += 8;
    }
    for (; k <= kmax; k += 2) {
        const float2 pa = TSP_P1(true, 0), pb = TSP_P1(true, 1);
        if constexpr (ST) tm_st4(col, pa.x, pa.y, pb.x, pb.y);
        a0 += (Addr)(long long)(2 * s0);
        a1 += (Addr)(long long)(2 * s1);
        col += 4;
    }
#undef TSP_P1
    return k - 1;
}

// Two pairs' terms (four pixels; pa = pair k, pb = pair k + 1) added to the words at
// a0, a1, a0 + S0, a1 + S1.  s2 = 2^-149 / (D quantum): the product, rounded to
// nearest, is a subnormal number (or in the first binade above, of the same
// spacing), whose bits are the count of quanta, up to 2^24.
template <int S0, int S1>
__device__ __forceinline__ void add4(unsigned a0, unsigned a1, float2 pa, float2 pb, float2 s2)
{
    const float2 va = __fmul2_rn(pa, s2), vb = __fmul2_rn(pb, s2);
#ifdef TSP_DEBUG_CHECKS
    if (!(tsp_sh_ok(a0, 4, 2) && tsp_sh_ok(a1, 4, 2) && tsp_sh_ok(a0 + (unsigned)S0, 4, 2) &&
          tsp_sh_ok(a1 + (unsigned)S1, 4, 2)))
        return;
#endif
    asm volatile(
        "red.shared.add.u32 [%0], %4;\n\tred.shared.add.u32 [%1], %5;\n\t"
        "red.shared.add.u32 [%0+%2], %6;\n\tred.shared.add.u32 [%1+%3], %7;"
        ::"r"(a0), "r"(a1), "n"(S0), "n"(S1),
        "r"(__float_as_uint(va.x)), "r"(__float_as_uint(va.y)), "r"(__float_as_uint(vb.x)),
        "r"(__float_as_uint(vb.y))
        : "memory");
}

// Pass 2: the values of pairs 1 .. n (n a multiple of two), 0 beyond each stream's
// last pair, added to the item's accumulator at base.
template <int TRAV>
__device__ __forceinline__ void rec_pass2(unsigned base, int n, unsigned tma, float2 s2)
{
    constexpr int s0 = 4 * pair_step0<TRAV>(), s1 = 4 * pair_step1<TRAV>();
    unsigned a0 = base + (unsigned)(4 * pair_d0<TRAV>(1));
    unsigned a1 = base + (unsigned)(4 * pair_d1<TRAV>(1));
    unsigned col = tma;
    int k = n;
    for (; k >= 8; k -= 8) {
        float x[16];
        tm_ld16(col, x);
        tm_wait_ld();
        add4<s0, s1>(a0, a1, make_float2(x[0], x[1]), make_float2(x[2], x[3]), s2);
        add4<s0, s1>(a0 + (unsigned)(2 * s0), a1 + (unsigned)(2 * s1), make_float2(x[4], x[5]),
                     make_float2(x[6], x[7]), s2);
        add4<s0, s1>(a0 + (unsigned)(4 * s0), a1 + (unsigned)(4 * s1), make_float2(x[8], x[9]),
                     make_float2(x[10], x[11]), s2);
        add4<s0, s1>(a0 + (unsigned)(6 * s0), a1 + (unsigned)(6 * s1), make_float2(x[12], x[13]),
                     make_float2(x[14], x[15]), s2);
        a0 += (unsigned)(8 * s0);
        a1 += (unsigned)(8 * s1);
        col += 16;
    }
    if (k >= 4) {
        float x[8];
        tm_ld8(col, x);
        tm_wait_ld();
        add4<s0, s1>(a0, a1, make_float2(x[0], x[1]), make_float2(x[2], x[3]), s2);
        add4<s0, s1>(a0 + (unsigned)(2 * s0), a1 + (unsigned)(2 * s1), make_float2(x[4], x[5]),
                     make_float2(x[6], x[7]), s2);
        a0 += (unsigned)(4 * s0);
        a1 += (unsigned)(4 * s1);
        col += 8;
        k -= 4;
    }
    if (k >= 2) {
        float x0, x1, x2, x3;
        tm_ld4(col, x0, x1, x2, x3);
        tm_wait_ld();
        add4<s0, s1>(a0, a1, make_float2(x0, x1), make_float2(x2, x3), s2);
    }
}

// Sum over the group's warps of each warp's value (lane 0's), the same in every
// lane: kMinWarps slots of which those beyond the group's warps stay zero, summed by
// a butterfly without a loop's control.
__device__ __forceinline__ float group_sum(float v, int G, int wig, int lane, int bar_id, float* slot)
{
    static_assert(kMinWarps == 16, "four steps");
    if (lane == 0) slot[wig] = v;
    named_barrier(bar_id, G * 32);
    v = slot[lane & (kMinWarps - 1)];
#pragma unroll
    for (int o = kMinWarps / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// 1/D to float precision (one Newton step); not finite or 0 where D is far out of
// range, which the callers' test of the largest term excludes.
__device__ __forceinline__ float recip(float D)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(D));
    return fmaf(r, fmaf(-D, r, 1.0f), r);
}

// Gradient pass, one pair: the kernel value's pair (0 beyond the streams' last
// pairs), and the sums that D and the sigma gradients are made of.  With
// X = aCb / Q and S = X^2 + 1/Q, every term of the derivatives is a polynomial in
// the offset d times 1, X or S (see rec_grad_row), so the moments
//   sum v, sum v d, sum v d^2, sum v X, sum v X d, sum v S, sum v S d   (v = P rho')
// are all that the loop has to sum: eleven packed operations a pair beside the
// kernel's own, against fifteen when the derivatives are formed per pixel.  The
// exponent is formed as C0 - s^2 with s linear in d, not as a quadratic in d, and
// X from aCb itself, not from the scaled one of the exponent: with windows wide
// enough that the truncated tails are negligible the derivatives nearly cancel
// over a window, and the rounding of a coefficient that is the same for every
// event would show in their sum.
struct GradSums {
    float2 m0, m1, m2, x0, x1, s0, s1;
};

template <bool GLD, bool PRED, int OFF0, int OFF1, class Addr>
__device__ __forceinline__ float2 p1g_pair(Addr a0, Addr a1, int k, int la, int lb,
                                           const PairC& c, const GradC& g, float2& kk,
                                           GradSums& m)
{
    const float2 q = __ffma2_rn(kk, c.dQ, c.Q0);
    float2 rq;
    rq.x = rsqrt_approx(q.x);
    rq.y = rsqrt_approx(q.y);
    if constexpr (PRED) {
        // (with 1/sqrt(Q) set to 0 P is 0 and everything else finite)
        rq.x = k <= la ? rq.x : 0.0f;
        rq.y = k <= lb ? rq.y : 0.0f;
    }
    const float2 a = __ffma2_rn(kk, c.dA, c.A0);
    const float2 su = __ffma2_rn(kk, c.e2, c.e1);
    const float2 e = __ffma2_rn(su, __fmul2_rn(su, make_float2(-1.0f, -1.0f)), c.e0);
    const float2 w = __fmul2_rn(a, rq);
    const float2 ar = __ffma2_rn(w, w, e);
    float2 x;
    x.x = ex2_approx(ar.x);
    x.y = ex2_approx(ar.y);
    const float2 p = __fmul2_rn(rq, x);
    float2 v;
    v.x = ld_rhop<!GLD, false, GLD && PRED, OFF0>(a0, k, la);
    v.y = ld_rhop<!GLD, false, GLD && PRED, OFF1>(a1, k, lb);
    const float2 pv = __fmul2_rn(p, v), pvd = __fmul2_rn(pv, kk);
    const float2 iq = __fmul2_rn(rq, rq);
    const float2 X = __fmul2_rn(__ffma2_rn(kk, g.dB, g.B0), iq), S = __ffma2_rn(X, X, iq);
    m.m0 = __fadd2_rn(m.m0, pv);
    m.m1 = __fadd2_rn(m.m1, pvd);
    m.m2 = __ffma2_rn(pvd, kk, m.m2);
    m.x0 = __ffma2_rn(pv, X, m.x0);
    m.x1 = __ffma2_rn(pvd, X, m.x1);
    m.s0 = __ffma2_rn(pv, S, m.s0);
    m.s1 = __ffma2_rn(pvd, S, m.s1);
    kk = __fadd2_rn(kk, c.inc);
    return p;
}

// Gradient pass over pairs 1 .. kmax, P kept in tensor memory, two pairs a step
// (the sums and constants leave no registers for more).  Returns the number of
// pairs stored.
template <int TRAV, bool GLD, class Addr>
__device__ __forceinline__ int rec_pass1_grad(Addr base, int la, int lb, const PairC& c,
                                              const GradC& g, int kfast, int kmax, GradSums& m,
                                              unsigned tma)
{
    constexpr int kStep = GLD ? 4 * kScrRows : 4;
    constexpr int s0 = kStep * pair_step0<TRAV>(), s1 = kStep * pair_step1<TRAV>();
    Addr a0 = base + (Addr)(long long)(kStep * pair_d0<TRAV>(1));
    Addr a1 = base + (Addr)(long long)(kStep * pair_d1<TRAV>(1));
    float2 kk = make_float2((float)pair_d0<TRAV>(1), (float)pair_d1<TRAV>(1));
    unsigned col = tma;
    int k = 1;
    for (; k + 1 <= kfast; k += 2) {
        const float2 pa = p1g_pair<GLD, false, 0, 0>(a0, a1, k, la, lb, c, g, kk, m);
        const float2 pb = p1g_pair<GLD, false, s0, s1>(a0, a1, k + 1, la, lb, c, g, kk, m);
        tm_st4(col, pa.x, pa.y, pb.x, pb.y);
        a0 += (Addr)(long long)(2 * s0);
        a1 += (Addr)(long long)(2 * s1);
        col += 4;
    }
    for (; k <= kmax; k += 2) {
        const float2 pa = p1g_pair<GLD, true, 0, 0>(a0, a1, k, la, lb, c, g, kk, m);
        const float2 pb = p1g_pair<GLD, true, s0, s1>(a0, a1, k + 1, la, lb, c, g, kk, m);
        tm_st4(col, pa.x, pa.y, pb.x, pb.y);
        a0 += (Addr)(long long)(2 * s0);
        a1 += (Addr)(long long)(2 * s1);
        col += 4;
    }
    return k - 1;
}

// (Ez, El) of a lane from its moments: the sums of v dlogP/d(iz) and
// v dlogP/d(il),
//   d log P / d iz = 1/iz - u^2 + X Cz - (Qz/2) S
//   d log P / d il = 1/(2 il) - Bl/2 + X Cl - (Ql/2) S
// with u, Cz and Qz linear in d (formulas in make_row), the z terms with
// respect to the base iz (times inv_f2).
__device__ __forceinline__ float2 rec_grad_row(const Geo& g, const float4& ev, float y, float Dy,
                                               float u0, const GradSums& m)
{
    const EvSig es = ev_sig(g, ev);
    const float t = ev.z, c2i = ev.w, y2 = y * y, dz = g.dz;
    const float m0 = m.m0.x + m.m0.y, m1 = m.m1.x + m.m1.y, m2 = m.m2.x + m.m2.y;
    const float x0 = m.x0.x + m.x0.y, x1 = m.x1.x + m.x1.y;
    const float s0 = m.s0.x + m.s0.y, s1 = m.s1.x + m.s1.y;
    const float qzs = -2.0f * y * t * c2i, qz0 = fmaf(qzs, u0, (g.R * g.R + y2) * c2i * c2i);
    const float czs = -2.0f * y * c2i;
    // sum v u^2 = u0^2 m0 + 2 u0 dz m1 + dz^2 m2 (dz dz, rounded the same for every
    // event, would move the sum of these nearly cancelling terms by up to 1e-6)
    const float vu2 = fmaf(u0, fmaf(u0, m0, 2.0f * dz * m1), dz * (dz * m2));
    const float Ez = fmaf(es.ldz, m0, -vu2) + czs * fmaf(u0, x0, dz * x1) - fmaf(qz0, s0, qzs * dz * s1);
    const float Bl = 4.0f * Dy * Dy * c2i;
    const float cl = 4.0f * y * t * Dy * c2i;
    const float qlh = 2.0f * y2 * t * t * c2i + 2.0f * y * fmaf(2.0f * t, t, 1.0f) * Dy * c2i;
    const float El = fmaf(es.ldl - 0.5f * Bl, m0, fmaf(cl, x0, -qlh * s0));
    return make_float2(Ez * es.inv_f2, El);
}

// Room of the fixed-point accumulator (see k_tiles_rec), in quanta.
constexpr float kTopTerm = 0.99f * 0x1p24f;   // one event's largest term, of add4
constexpr float kRoom = 0.99f * 0x1p32f;      // all the events of an item

// The fixed point of the item at hand, a copy for each warp in shared memory (the pixel
// loops have no registers for it).
struct RecScale {
    float inv_q;        // 1 over the quantum of the terms P / D
    float plain;        // the same for the plain scatter; infinite in a peaked item, which
                        // it then takes no event of
    float share;        // of the word's room, a group's
    float cap;          // the most of it that one event may take
};

// How the terms of an event that the plain scatter does not take are added: not at all, by
// float adds to the global A, or in quanta, by a conversion (up to 2^32 of them; add4's
// arithmetic ends at 2^24).
enum How : int { kNone, kFloat, kFixed };

// An offset in [-1/2, 1/2) from the bits of an event's D: with it, a term is rounded to
// the nearest quantum up or down in proportion, and terms that many events have alike
// (1 / rho' at a pixel that is most of their D) keep their mean.
__device__ __forceinline__ float dither(float D)
{
    return (float)((__float_as_uint(D) * 2654435761u) >> 8) * 0x1p-24f - 0.5f;
}

__device__ __forceinline__ void add_fixed(unsigned a, float p, float s, float u)
{
    const unsigned v = p > 0.0f ? __float2uint_rn(__fmaf_rn(p, s, u)) : 0u;
#ifdef TSP_DEBUG_CHECKS
    if (!tsp_sh_ok(a, 4, 2)) return;
#endif
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// Image pixel of a stored index (see Frame).
__device__ __forceinline__ int frame_pixel(const Frame& f, int nz, int i)
{
    const int rr = i / f.stride, iy = f.oy + rr;
    return iy * nz + f.zbase + (int)rintf(__fmul_rn(f.shear, (float)(iy - f.Y0))) + i - rr * f.stride;
}

// The scatter of an event that the plain one does not take (see How): into the accumulator
// (base: as rec_pass2), s = 1 / (D quantum), or to the global A, s = 1/D, each
// pixel (idx: stored index of the row's origin) under its predicate; with MASK only where
// rho' > 0 (as the flush does).  (Called from one place: a second caller costs the pixel
// loops beside the call 6%.)
template <int TRAV, bool MASK>
__device__ __noinline__ void rec_scatter_slow(unsigned base, const Inst* I, const Frame* fp,
                                              int idx, int la, int lb, int n, unsigned tma,
                                              float s, float u, int how)
{
    const int pix = how == kFloat ? frame_pixel(*fp, I->g.nz, idx) : 0;
    float* const A = I->A;
    const float* const rhop = I->rhop;
    auto add = [&](int q, float p) {
        if (p != 0.0f && (!MASK || rhop[q] > 0.0f)) atomicAdd(A + q, p * s);
    };
    for (int k = 1; k <= n; k += 2) {
        float x0, x1, x2, x3;
        tm_ld4(tma, x0, x1, x2, x3);
        tm_wait_ld();
        const int d0 = pair_d0<TRAV>(k), d1 = pair_d1<TRAV>(k);
        const int d2 = pair_d0<TRAV>(k + 1), d3 = pair_d1<TRAV>(k + 1);
        if (how == kFixed) {
            add_fixed(base + (unsigned)(4 * d0), x0, s, u);
            add_fixed(base + (unsigned)(4 * d1), x1, s, u);
            add_fixed(base + (unsigned)(4 * d2), x2, s, u);
            add_fixed(base + (unsigned)(4 * d3), x3, s, u);
        } else {
            if (k <= la) add(pix + d0, x0);
            if (k <= lb) add(pix + d1, x1);
            if (k < la) add(pix + d2, x2);
            if (k < lb) add(pix + d3, x3);
        }
        __syncwarp();
        tma += 4;
    }
}

// The events first + grp, first + grp + ngroups, ... of an item, by one group
// of G warps.
template <int TRAV, int LMAX, int MODE, int NSEG, bool GLD>
__device__ __forceinline__ void rec_events(const Inst& I, const Frame* fp, const RecScale* sc,
                                           int first, int count, int grp, int ngroups, int wig,
                                           int lane, unsigned rp_addr, unsigned acc_off,
                                           unsigned slot, float* part, BlockSums* bs, unsigned tma,
                                           const float* scr)
{
    constexpr bool GRAD = MODE == kGrad;
    const Geo& g = I.g;
    const int G = I.G;
    int left = (count - grp + ngroups - 1) / ngroups;
    if (left <= 0) return;
    first += grp;
    // the row block of a warp is rotated by its group (see process_event)
    int blk;
    if constexpr (NSEG == 1) {
        blk = wig + grp % G;
        blk -= blk >= G ? G : 0;
    } else {
        const int nb = G >> 1;
        blk = (wig >> 1) + grp % nb;
        blk -= blk >= nb ? nb : 0;
    }
    const float rowoff = (float)lane_row(blk * 32 + lane);
    const int rslot = NSEG == 1 ? blk * 32 + lane : (blk * 2 + (wig & 1)) * 32 + lane;
    // (GRAD: an index, not two pointers that step, which spills less)
    const uint2* rp = I.evs.recs + (size_t)first * (32 * G) + rslot;
    const float4* ep = I.evs.evc + (size_t)first * kEvcFloat4;
    rec_fetch(slot, rp, ep, lane);
    const float inv_q = MODE == kLoglik ? 0.0f : sc->plain;
    float room = MODE == kLoglik ? 0.0f : sc->share;
    unsigned used = 0;
    double logD = 0.0, giz = 0.0, gil = 0.0;
    int parity = 0;
    for (;;) {
        RecIn x;
        rec_wait();
        rec_take(x, slot, lane);
        float y, Dy, u0;
        GradC gc;
        const PairC c = rec_row<TRAV, GRAD>(g, x, rowoff, y, Dy, u0, &gc);
        const unsigned idx = x.r.y & 0xffffu, base = rp_addr + 4u * idx;
        const int la = (x.r.y >> 16) & 0xff, lb = x.r.y >> 24;
        const int kmax = __reduce_max_sync(0xffffffffu, max(la, lb));
        const int kfast = __reduce_min_sync(0xffffffffu, min(la, lb));
        float4 ev = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if constexpr (GRAD) ev = lds128(slot + 304u);
        else if (MODE != kLoglik) ev.x = lds32(slot + 304u);
        __syncwarp();   // every lane has its values: the slot may be refilled
        if (--left > 0) {
            if (GRAD) {
                first += ngroups;
                rec_fetch(slot, I.evs.recs + (size_t)first * (32 * G) + rslot,
                          I.evs.evc + (size_t)first * kEvcFloat4, lane);
            } else {
                rp += (size_t)ngroups * (32 * G);
                ep += ngroups * kEvcFloat4;
                rec_fetch(slot, rp, ep, lane);
            }
        }
        int n;
        float D;
        using Addr = typename std::conditional<GLD, unsigned long long, unsigned>::type;
        Addr rbase;
        if constexpr (GLD) {
            const int rr = (int)(x.a.y + rowoff) - fp->oy;
            const int off = min(max(rr, 0), I.tl.RH - 1) * (1 - kScrRows * I.tl.RS) + (int)idx * kScrRows;
            rbase = (unsigned long long)(scr + off);
        } else {
            rbase = base;
        }
        float2 E = make_float2(0.0f, 0.0f);
        if constexpr (GRAD) {
            GradSums m;
            m.m0 = m.m1 = m.m2 = m.x0 = m.x1 = m.s0 = m.s1 = make_float2(0.0f, 0.0f);
            n = rec_pass1_grad<TRAV, GLD>(rbase, la, lb, c, gc, kfast, kmax, m, tma);
            E = rec_grad_row(g, ev, y, Dy, u0, m);
            D = warp_sum(m.m0.x + m.m0.y);
        } else {
            float2 D2 = make_float2(0.0f, 0.0f);
            n = rec_pass1<TRAV, LMAX, MODE != kLoglik, GLD>(rbase, la, lb, c, kfast, kmax, D2, tma);
            D = warp_sum(D2.x + D2.y);
        }
        if (MODE != kLoglik) tm_wait_st();
        if (G > 1) {
            D = group_sum(D, G, wig, lane, 1 + grp, part + parity);
            parity ^= kMinWarps;
        }
        if (D > 0.0f) {
            if (MODE != kLoglik) {
                const float r = recip(D), s = r * inv_q, top = s * ev.x;
                // (false for a NaN, and for a D that recip has no value of)
                float w = r;
                if ((top > 0.0f) & (top <= room) & (top <= kTopTerm)) {
                    // (some more than the bound: the rounding of the terms)
                    room = fmaf(top, -1.0001f, room - 1.0f);
                    const float q = s * 0x1p-149f;
                    rec_pass2<TRAV>(base + acc_off, n, tma, make_float2(q, q));
                } else {
                    const float s1 = r * sc->inv_q, top1 = s1 * ev.x;
                    const bool fit = top1 > 0.0f && top1 <= fminf(room, sc->cap);
                    if (fit) room = fmaf(top1, -1.0001f, room - 1.0f);
                    else w = 1.0f / D;
                    rec_scatter_slow<TRAV, MODE == kMlem && !GLD>(
                        base + acc_off, &I, fp, (int)idx, la, lb, n, tma, fit ? s1 : w, dither(D),
                        fit ? kFixed : kFloat);
                }
                if (GRAD) {
                    // per-lane sums: the rows' terms of an event cancel to a small
                    // part of themselves, so they are added in double precision
                    giz += (double)(E.x * w);
                    gil += (double)(E.y * w);
                }
            }
            ++used;
            if (MODE != kMlem && wig == 0 && lane == 0) logD += (double)logf(D);
        }
        if (left == 0) break;
    }
    if (wig == 0 && lane == 0) {
        if (used) atomicAdd(&bs->used, (unsigned long long)used);
        if (MODE != kMlem) atomicAdd(&bs->logD, logD + used * (g.pshift * 0.69314718055994530942));
    }
    if (GRAD) {
        for (int o = 16; o > 0; o >>= 1) {
            giz += __shfl_xor_sync(0xffffffffu, giz, o);
            gil += __shfl_xor_sync(0xffffffffu, gil, o);
        }
        if (lane == 0) {
            atomicAdd(&bs->giz, giz);
            atomicAdd(&bs->gil, gil);
        }
    }
}

// ---- Two rows a lane -----------------------------------------------------------
//
// The MLEM and log-likelihood passes of chords up to 32 pixels: a lane takes two rows, the
// neighbours of the lane-row order (mid - p and mid + p + 1, of about the same
// length), as the two components of the packed operations.  An event of up to 32
// rows (4 mm grids) then takes half a warp, one of 64 (2 mm) one warp and no
// barrier, where a row a lane took twice as much; its pairs take the same time, but
// what is done once a warp and event (record, constants, reductions, 1/D, loop
// control: some 250 instructions of the 370 that an event of a 4 mm grid took) is
// halved.  Longer chords have no room: a lane has 64 tensor-memory columns.
//   1e7 events at 4 mm 3.38 -> 2.96 ms, three updates of 3e5 at 2 mm (chords of 25
//   pixels) 1.36 -> 1.15 ms, 1e6 from host buffers at 2 mm (three updates and the
//   log-likelihood) 6.53 -> 5.68 ms, mixed batch 18.15 -> 17.99 ms.
// The gradient pass keeps a row a lane: with two, and its sums, 64 registers a thread
// spill (1e6 events at 2 mm 3.30 -> 4.37 ms).
// A window of an odd number of 32-row blocks above one keeps a row a lane: with two it
// would leave a quarter of the lanes idle and every step predicated (12 mixed
// reconstructions, one in three of them of such windows: 18.7 ms with two rows a lane
// for all that their chords allow, 18.0 ms with this rule).
// Step k of a row is the pixels at k and 1 - k from its origin, as with kAlt.

__device__ __forceinline__ bool two_rows_fit(int G) { return G == 1 || (G & 1) == 0; }

__host__ __device__ constexpr bool two_rows(int lmax, int mode, int nseg, bool gld)
{
    return lmax <= 32 && mode != kGrad && nseg == 1 && !gld;
}

// The two rows' constants (.x, .y): see rec_row.
struct Row2 {
    float2 Q0, dQ, A0, dA, e0, e1, e2;
};

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }

__device__ __forceinline__ Row2 rec_row2(const Geo& g, const RecIn& x, float2 rowoff, float2 u0)
{
    const float2 y = __ffma2_rn(__fadd2_rn(dup(x.a.y), rowoff), dup(g.dy), dup(g.y0));
    const float2 Dy = __fadd2_rn(y, dup(-x.a.x));
    const float2 Qc = __ffma2_rn(y, __ffma2_rn(dup(x.b.x), y, dup(x.a.w)), dup(x.a.z));
    const float2 gam = __fmul2_rn(dup(x.b.y), y), al = __fmul2_rn(dup(x.b.z), y);
    const float2 be = __fmul2_rn(Dy, __ffma2_rn(dup(x.b.w), y, dup(x.c.x)));
    Row2 c;
    c.Q0 = __ffma2_rn(gam, u0, Qc);
    c.dQ = __fmul2_rn(gam, dup(g.dz));
    c.A0 = __fmul2_rn(__ffma2_rn(al, u0, be), dup(g.kA));
    c.dA = __fmul2_rn(al, dup(g.dz * g.kA));
    const float2 C0 = __ffma2_rn(__fmul2_rn(dup(-x.c.y), Dy), Dy, dup(x.c.z));
    const float2 su0 = __fmul2_rn(dup(x.c.w), u0);
    const float dsu = x.c.w * g.dz;
    c.e0 = __ffma2_rn(make_float2(-su0.x, -su0.y), su0, C0);
    c.e1 = __fmul2_rn(su0, dup(-2.0f * dsu));
    c.e2 = dup(-(dsu * dsu));
    return c;
}

// One pixel of each row, at kk from the origins: P, 0 beyond the rows' ends (in0, in1).
template <int OFF>
__device__ __forceinline__ float2 p2_eval(unsigned a0, unsigned a1, bool in0, bool in1, float2 kk,
                                          const Row2& c, float2& D2)
{
    const float2 q = __ffma2_rn(kk, c.dQ, c.Q0);
    // (with 1/sqrt(Q) set to 0 everything after it is finite)
    const float r0 = rsqrt_approx(q.x), r1 = rsqrt_approx(q.y);
    const float2 rq = make_float2(in0 ? r0 : 0.0f, in1 ? r1 : 0.0f);
    const float2 a = __ffma2_rn(kk, c.dA, c.A0);
    const float2 e = __ffma2_rn(kk, __ffma2_rn(kk, c.e2, c.e1), c.e0);
    const float2 w = __fmul2_rn(a, rq);
    const float2 h = __ffma2_rn(w, w, e);
    const float2 p = __fmul2_rn(rq, make_float2(ex2_approx(h.x), ex2_approx(h.y)));
    float2 v;
    v.x = ld_rhop<true, false, false, OFF>(a0, 0, 0);
    v.y = ld_rhop<true, false, false, OFF>(a1, 0, 0);
    D2 = __ffma2_rn(p, v, D2);
    return p;
}

// Pass 1, steps 1 .. kmax.  a0, a1: addresses of the rows' origins.
template <int MODE>
__device__ __forceinline__ void rec2_pass1(unsigned a0, unsigned a1, int la0, int lb0, int la1,
                                           int lb1, const Row2& c, int kmax, float2& D2,
                                           unsigned tma)
{
    const float2 one = dup(1.0f), mone = dup(-1.0f);
    float2 kp = one, km = dup(0.0f);
    unsigned u0 = a0 + 4u, u1 = a1 + 4u, d0 = a0, d1 = a1, col = tma;
    auto step = [&](auto J, int k, float2& pu, float2& pd) {
        constexpr int j = decltype(J)::value;
        const bool i0 = k + j <= la0, i1 = k + j <= la1, j0 = k + j <= lb0, j1 = k + j <= lb1;
        pu = p2_eval<4 * j>(u0, u1, i0, i1, kp, c, D2);
        pd = p2_eval<-4 * j>(d0, d1, j0, j1, km, c, D2);
        kp = __fadd2_rn(kp, one);
        km = __fadd2_rn(km, mone);
    };
    int k = 1;
    for (; k + 1 <= kmax; k += 2) {
        float2 p, q, r, s;
        step(std::integral_constant<int, 0>{}, k, p, q);
        step(std::integral_constant<int, 1>{}, k, r, s);
        if (MODE != kLoglik) tm_st8(col, p.x, p.y, q.x, q.y, r.x, r.y, s.x, s.y);
        u0 += 8u;
        u1 += 8u;
        d0 -= 8u;
        d1 -= 8u;
        col += 8;
    }
    if (k <= kmax) {
        float2 p, q;
        step(std::integral_constant<int, 0>{}, k, p, q);
        if (MODE != kLoglik) tm_st4(col, p.x, p.y, q.x, q.y);
    }
}

// The terms of one step (p at k, q at 1 - k): counts of quanta (see add4).
template <int OFF>
__device__ __forceinline__ void add2x2(unsigned u0, unsigned u1, unsigned d0, unsigned d1, float2 p,
                                       float2 q, float2 s2)
{
    const float2 vp = __fmul2_rn(p, s2), vq = __fmul2_rn(q, s2);
#ifdef TSP_DEBUG_CHECKS
    if (!(tsp_sh_ok(u0 + (unsigned)OFF, 4, 2) && tsp_sh_ok(u1 + (unsigned)OFF, 4, 2) &&
          tsp_sh_ok(d0 - (unsigned)OFF, 4, 2) && tsp_sh_ok(d1 - (unsigned)OFF, 4, 2)))
        return;
#endif
    asm volatile(
        "red.shared.add.u32 [%0+%4], %6;\n\tred.shared.add.u32 [%1+%4], %7;\n\t"
        "red.shared.add.u32 [%2+%5], %8;\n\tred.shared.add.u32 [%3+%5], %9;"
        ::"r"(u0), "r"(u1), "r"(d0), "r"(d1), "n"(OFF), "n"(-OFF),
        "r"(__float_as_uint(vp.x)), "r"(__float_as_uint(vp.y)), "r"(__float_as_uint(vq.x)),
        "r"(__float_as_uint(vq.y))
        : "memory");
}

// Pass 2, steps 1 .. n, into the item's accumulator.
__device__ __forceinline__ void rec2_pass2(unsigned a0, unsigned a1, int n, unsigned tma, float2 s2)
{
    unsigned u0 = a0 + 4u, u1 = a1 + 4u, d0 = a0, d1 = a1, col = tma;
    for (; n >= 4; n -= 4) {
        float x[16];
        tm_ld16(col, x);
        tm_wait_ld();
        add2x2<0>(u0, u1, d0, d1, make_float2(x[0], x[1]), make_float2(x[2], x[3]), s2);
        add2x2<4>(u0, u1, d0, d1, make_float2(x[4], x[5]), make_float2(x[6], x[7]), s2);
        add2x2<8>(u0, u1, d0, d1, make_float2(x[8], x[9]), make_float2(x[10], x[11]), s2);
        add2x2<12>(u0, u1, d0, d1, make_float2(x[12], x[13]), make_float2(x[14], x[15]), s2);
        u0 += 16u;
        u1 += 16u;
        d0 -= 16u;
        d1 -= 16u;
        col += 16;
    }
    if (n >= 2) {
        float x[8];
        tm_ld8(col, x);
        tm_wait_ld();
        add2x2<0>(u0, u1, d0, d1, make_float2(x[0], x[1]), make_float2(x[2], x[3]), s2);
        add2x2<4>(u0, u1, d0, d1, make_float2(x[4], x[5]), make_float2(x[6], x[7]), s2);
        u0 += 8u;
        u1 += 8u;
        d0 -= 8u;
        d1 -= 8u;
        col += 8;
        n -= 2;
    }
    if (n >= 1) {
        float x0, x1, x2, x3;
        tm_ld4(col, x0, x1, x2, x3);
        tm_wait_ld();
        add2x2<0>(u0, u1, d0, d1, make_float2(x0, x1), make_float2(x2, x3), s2);
    }
}

// The scatter of rows whose event rec2_pass2 does not take (see rec_scatter_slow; a0, a1:
// addresses of the lane's rows' origins, i0, i1: their stored indexes).
template <bool MASK>
__device__ __noinline__ void rec2_scatter_slow(unsigned a0, unsigned a1, const Inst* I,
                                               const Frame* fp, unsigned i0, unsigned i1,
                                               unsigned n0, unsigned n1, int n, unsigned tma,
                                               float s, float u, int how)
{
    const int p0 = how == kFloat ? frame_pixel(*fp, I->g.nz, (int)i0) : 0;
    const int p1 = how == kFloat ? frame_pixel(*fp, I->g.nz, (int)i1) : 0;
    float* const A = I->A;
    const float* const rhop = I->rhop;
    auto add = [&](int q, float p) {
        if (p != 0.0f && (!MASK || rhop[q] > 0.0f)) atomicAdd(A + q, p * s);
    };
    for (int k = 1; k <= n; ++k) {
        float x0, x1, x2, x3;
        tm_ld4(tma, x0, x1, x2, x3);
        tm_wait_ld();
        if (how == kFloat) {
            if (k <= (int)(n0 & 0xff)) add(p0 + k, x0);
            if (k <= (int)(n1 & 0xff)) add(p1 + k, x1);
            if (k <= (int)(n0 >> 8)) add(p0 + 1 - k, x2);
            if (k <= (int)(n1 >> 8)) add(p1 + 1 - k, x3);
        } else if (how == kFixed) {
            add_fixed(a0 + 4u * k, x0, s, u);
            add_fixed(a1 + 4u * k, x1, s, u);
            add_fixed(a0 - 4u * (k - 1), x2, s, u);
            add_fixed(a1 - 4u * (k - 1), x3, s, u);
        }
        __syncwarp();
        tma += 4;
    }
}

// The groups of the two-row form: with G = 1 (up to 32 rows) a half warp an event, else
// (G + 1) / 2 warps.  The first group of this warp, and their number.
__device__ __forceinline__ int2 rec2_groups(int G, int warp)
{
    if (G == 1) return make_int2(2 * warp, 2 * kMaxWarps);
    const int G2 = (G + 1) >> 1;
    return make_int2(warp / G2, group_count(kMaxWarps, G2));
}

// The events of an item for this warp's groups.
template <int MODE>
__device__ __forceinline__ void rec2_events(const Inst& I, const Frame* fp, const RecScale* sc,
                                            int first, int count, int warp, int lane,
                                            unsigned rp_addr, unsigned acc_off, unsigned slot,
                                            float* s_part, BlockSums* bs, unsigned tma)
{
    const Geo& g = I.g;
    const int G = I.G;
    const bool halves = G == 1;
    const int G2 = (G + 1) >> 1;
    const int wgrp = warp / G2, wig = warp - wgrp * G2;
    const int2 gr = rec2_groups(G, warp);
    const int ngroups = gr.y;
    // (the row block of a warp is rotated by its group)
    int blk = wig + wgrp % G2;
    blk -= blk >= G2 ? G2 : 0;
    int p = halves ? lane & 15 : blk * 32 + lane;
    const bool has_rows = p < 16 * G;
    const float2 rowoff = make_float2((float)-p, (float)(p + 1));
    p = min(p, 16 * G - 1);
    // events left of the warp's first group (the second half's may end one sooner)
    int left = gr.x < ngroups ? (count - gr.x + ngroups - 1) / ngroups : 0;
    if (left <= 0) return;
    int e = gr.x + (halves ? lane >> 4 : 0);
    const uint4* const recs = reinterpret_cast<const uint4*>(I.evs.recs) + p;
    const float4* const evc = I.evs.evc;
    const int cl = halves ? lane & 15 : lane;
    const unsigned cslot = slot + 512u + (halves ? (lane >> 4) * 64u : 0u);
    auto fetch = [&](int ev) {
        const long long j = first + min(ev, count - 1);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(slot + 16u * lane),
                     "l"(recs + j * (16 * G))
                     : "memory");
        if (cl < kEvcFloat4)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(cslot + 16u * cl),
                         "l"(evc + j * kEvcFloat4 + cl)
                         : "memory");
    };
    fetch(e);
    float* const part = s_part + wgrp * 2 * kMinWarps;
    int parity = 0;
    const float inv_q = MODE == kLoglik ? 0.0f : sc->plain;
    float room = MODE == kLoglik ? 0.0f : sc->share;
    unsigned used = 0;
    double logD = 0.0;
    for (;;) {
        RecIn x;
        unsigned w[4];
        rec_wait();
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(slot + 16u * lane)
                     : "memory");
        x.a = lds128(cslot);
        x.b = lds128(cslot + 16u);
        x.c = lds128(cslot + 32u);
        const float pmax = lds32(cslot + 48u);
        const bool live = e < count && has_rows;
        __syncwarp();   // every lane has its values: the slot may be refilled
        e += ngroups;
        if (--left > 0) fetch(e);
        const float2 u0 = make_float2(__uint_as_float(w[0]), __uint_as_float(w[2]));
        const unsigned i0 = w[1] & 0xffffu, i1 = w[3] & 0xffffu;
        const unsigned n0 = live ? w[1] >> 16 : 0u, n1 = live ? w[3] >> 16 : 0u;
        const int la0 = n0 & 0xff, lb0 = n0 >> 8, la1 = n1 & 0xff, lb1 = n1 >> 8;
        const int kmax = __reduce_max_sync(0xffffffffu, max(max(la0, lb0), max(la1, lb1)));
        const unsigned a0 = rp_addr + 4u * i0, a1 = rp_addr + 4u * i1;
        float2 D2 = make_float2(0.0f, 0.0f);
        rec2_pass1<MODE>(a0, a1, la0, lb0, la1, lb1, rec_row2(g, x, rowoff, u0), kmax, D2, tma);
        float D = D2.x + D2.y;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) D += __shfl_xor_sync(0xffffffffu, D, o);
        if (!halves) D += __shfl_xor_sync(0xffffffffu, D, 16);
        if (MODE != kLoglik) tm_wait_st();
        if (G2 > 1) {
            D = group_sum(D, G2, wig, lane, 1 + wgrp, part + parity);
            parity ^= kMinWarps;
        }
        // (a second half beyond the list has no pixels: D = 0)
        const bool on = D > 0.0f;
        if (MODE != kLoglik) {
            const float r = recip(D), s = r * inv_q, top = s * pmax;
            // (false for a NaN, and for a D that recip has no value of)
            const bool fast = on & (top > 0.0f) & (top <= room) & (top <= kTopTerm);
            if (!__any_sync(0xffffffffu, on & !fast)) {
                // (some more than the bound: the rounding of the terms)
                if (on) room = fmaf(top, -1.0001f, room - 1.0f);
                rec2_pass2(a0 + acc_off, a1 + acc_off, kmax, tma, dup(on ? s * 0x1p-149f : 0.0f));
            } else {
                const float s1 = r * sc->inv_q, top1 = s1 * pmax;
                const bool fit = on && top1 > 0.0f && top1 <= fminf(room, sc->cap);
                if (fit) room = fmaf(top1, -1.0001f, room - 1.0f);
                rec2_scatter_slow<MODE == kMlem>(a0 + acc_off, a1 + acc_off, &I, fp, i0, i1, n0, n1,
                                                 kmax, tma, fit ? s1 : 1.0f / D, dither(D),
                                                 !on ? kNone : fit ? kFixed : kFloat);
            }
        }
        if (on) {
            ++used;
            if (MODE != kMlem && (halves ? (lane & 15) == 0 : wig == 0 && lane == 0))
                logD += (double)logf(D);
        }
        if (left == 0) break;
    }
    if (used && (halves ? (lane & 15) == 0 : wig == 0 && lane == 0)) {
        atomicAdd(&bs->used, (unsigned long long)used);
        if (MODE != kMlem) atomicAdd(&bs->logD, logD + used * (g.pshift * 0.69314718055994530942));
    }
}

// An item's scale: a lane has the sum and the largest of rho' over its
// band of rows (Inst::fx_*).  r, what an event of the item sees, is the mean of rho' over
// a box of a window's size about the bands that hold window centres, averaged with itself
// for weight, as events are distributed.  (With the largest mean in its place the items
// at the body's edge had no room for their events from the third update on, and some
// thousands of float adds in a few items held the whole pass up: 5e6 events at 1 mm
// 15.1 -> 20 to 24 ms.)
// (Not the mean over the region: after a few updates most of it, outside
// the body, is near 0, and the largest terms would lose four to five bits.)
__device__ __forceinline__ void item_scale(const Inst& I, float2 band, int n, int ngroups, int lane,
                                           RecScale* sc)
{
    const float peak =
        __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(band.y))) * I.fx_peak;
    float S = band.x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float v = __shfl_up_sync(0xffffffffu, S, o);
        if (lane >= o) S += v;
    }
    const float hi = __shfl_sync(0xffffffffu, S, min(lane + I.fx_half, 31));
    const float lo = __shfl_sync(0xffffffffu, S, max(lane - I.fx_half - 1, 0));
    float b = lane > I.fx_half ? hi - lo : hi;
    b = b > 0.0f && lane >= I.fx_first && lane <= I.fx_last ? b : 0.0f;
    const float m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(b)));
    const float x = m > 0.0f ? __fdividef(b, m) : 0.0f;
    float r = m > 0.0f ? __fdividef(m * warp_sum(x * x), warp_sum(x)) * I.fx_box : 0.0f;
    const bool peaked = peak > 0.5f * r;
    if (peaked) r = fmaxf(r, peak);
    const float share = __fdividef(kRoom, (float)ngroups);
    // an eighth of the share, or what each of a group's events can have, if that is more
    const float cap = share * fminf(fmaxf(__fdividef((float)ngroups, (float)n), 0.125f), 1.0f);
    // (peaked: the bits that leave events with a 2^-7.5th of the pixel's largest P, those at
    // the edge of a window of 3 sigma, within the cap)
    const int t = peaked ? min(18, (int)(__float_as_uint(cap) >> 23) - 127 - 8)
                         : min(I.fx_bits, 29 - (32 - __clz(n - 1)));
    const float v = __fdividef(r, I.fx_peak) * (float)(1 << t);
    // a power of two, so that neither scaling by it nor the flush rounds (peaked: not above v,
    // for the cap's sake); infinite for an image of no usable scale, whose events all
    // take the float scatter
    const unsigned up = peaked ? 0u : 0x7fffffu;
    const float inv_q = v >= 1e-30f && v <= 1e30f
                            ? __uint_as_float((__float_as_uint(v) + up) & 0x7f800000u)
                            : INFINITY;
    if (lane == 0) {
        sc->inv_q = inv_q;
        sc->plain = peaked ? INFINITY : inv_q;
        sc->share = share;
        sc->cap = cap;
    }
    __syncwarp();
}

// Persistent tile kernel over window records.  Work items and batches are those of
// k_tiles; the first item of a block is its index, later ones come from the queue, asked
// for while an item is worked on.
//
// The scatter sums P / D in fixed point, one word a pixel, with native integer adds
// (a float add to shared memory is a compare-and-swap loop).  The quantum is the item's:
// the largest term of an event that sees a mean rho' of r, as the item's events do on the
// average (item_scale), is fx_peak / r, and takes t = fx_bits (17 to 20) bits, or fewer to
// leave the word room for eight times the item's events (17 at 4000).  What an event
// really adds at most, its bound of P over D, is known before it is added, so that no sum
// can overflow: one above 2^24 quanta takes a slower loop (up to 2.4% of the events in
// 50 updates of phantoms), and one that the group's share of the word has no room left for,
// or an eighth of it, float adds to global memory (up to 0.8%).
//   A term is rounded to 2^-(t + 1) of the event's largest one, and over the cov events
// of a pixel the rounding of A is 0.3 x 2^(2.2 - t) / sqrt(cov) of it (fx_bits), within
// the 2^-22 of a term that its exponential and square root carry.  Two words of the
// responsibilities P rho' / D, as in k_tiles, need no estimate, but twice the
// adds and five more packed operations a pair: 1e7 events at 1 mm 34.3 -> 30.4 ms,
// five updates of 2e5 at 1 mm 5.07 -> 4.29 ms, three of 3e5 at 2 mm 1.57 -> 1.36 ms.
//
// Where one pixel can hold much of an event's D (peaked: the region's largest rho' alone
// would give half of r), the events' terms there are equal multiples 1 / rho' of the
// quantum, and rounded to the nearest one they would all err alike (a point source from a
// spike image: 4e-5 of the counts lost).  The events of such an item all take the
// slower loop, whose rounding is up or down in proportion (dither), with 15 to 18 bits for
// that pixel's terms: 0.4 x 2^-t / sqrt(events) = 2e-7 of their sum for 4000 events, 2e-8
// for 6e5.  (Float adds would not do: they round the many equal terms alike as well.)
//
// GLD: the windows are too large to stage rho' beside the accumulator.  The block
// writes the item's rho' region to its own part of global memory, transposed
// (column-major, kScrRows rows): the lanes of a warp, neighbouring rows at the
// same sheared column, then read neighbouring words, which a row-major image gives
// one cache line each.  It stays in the L1 and L2 caches.  2e6 events at
// 0.5 mm: 64.2 ms with the row-major image, float adds and rows set up in the pass,
// 28.1 ms now.
template <int LMAX, int MODE, int NSEG, bool BATCH, bool GLD>
__global__ void __launch_bounds__(pass_threads(LMAX, MODE, NSEG, BATCH), 1)
k_tiles_rec(const __grid_constant__ Inst p, const Inst* __restrict__ table, const int4* __restrict__ items, int n_items,
            int* queue)
{
    constexpr int kThreads = pass_threads(LMAX, MODE, NSEG, BATCH);
    constexpr int kWarps = kThreads / 32;
    constexpr bool kTwo = two_rows(LMAX, MODE, NSEG, GLD);
    constexpr int kSlot = rec_slot_floats(kTwo);
    constexpr int kTm = kTwo ? 2 * LMAX : LMAX;    // tensor-memory columns of a lane
    extern __shared__ float4 smem_f4[];
    float* const smem = reinterpret_cast<float*>(smem_f4);
    float* const s_part = smem;
    float* const s_rp = smem + kPartFloats + kMaxWarps * kSlot + kPadFloats;
    __shared__ int s_item[2];
    __shared__ BlockSums s_sums;
    __shared__ Inst s_inst;
    __shared__ unsigned s_tmem;
    __shared__ Frame s_frame;
    __shared__ RecScale s_scale[kWarps];
    __shared__ float2 s_band[kWarps];      // rho' of a 32nd of the region's rows: sum, largest
    const Inst& I = BATCH ? s_inst : p;

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    constexpr int kCols = tm_block_cols(kTm, kWarps);
    if (warp == 0) tm_alloc<kCols>(&s_tmem);
    init_block_sums(&s_sums);
#ifdef TSP_DEBUG_CHECKS
    if (tid == 0) tsp_dbg_word = 0ull;
#endif
    // slots of warps that a group does not have stay zero (group_sum)
    for (int k = tid; k < kPartFloats; k += kThreads) s_part[k] = 0.0f;
    if (tid < kWarps) s_band[tid] = make_float2(0.0f, 0.0f);
    int cur = -1, it = blockIdx.x, par = 0;
    bool fresh = true;
    tm_sync_threads();
    const unsigned tma = tm_thread_addr<kTm>(s_tmem, warp);

    while (it < n_items) {
        int next = 0;
        if (tid == 0) next = (int)gridDim.x + atomicAdd(queue, 1);
        const int4 item = items[it];
        if (BATCH && item.w != cur) {
            if (cur >= 0 && tid == 0) {
                flush_block_sums(&s_sums, s_inst.accum, MODE);
                init_block_sums(&s_sums);
#ifdef TSP_DEBUG_CHECKS
                if (tsp_dbg_word) atomicCAS(&s_inst.accum->dbg, 0ull, tsp_dbg_word);
                tsp_dbg_word = 0ull;
#endif
            }
            __syncthreads();
            const unsigned long long* src = reinterpret_cast<const unsigned long long*>(table + item.w);
            unsigned long long* dst = reinterpret_cast<unsigned long long*>(&s_inst);
            for (int k = tid; k < (int)(sizeof(Inst) / 8); k += kThreads) dst[k] = src[k];
            cur = item.w;
            fresh = true;
            __syncthreads();
        }
        const Geo& g = I.g;
        const Tiling& tl = I.tl;
        const int region = tl.RH * tl.RS;
        float* const s_acc = GLD ? s_rp : s_rp + region + 2 * kPadFloats;
        unsigned* const s_cnt = reinterpret_cast<unsigned*>(s_acc);
        float* const scr = GLD ? I.scratch + (size_t)blockIdx.x * tl.RS * kScrRows : nullptr;
        if (fresh) {
            // the slack around the regions is read (times P = 0) and added
            // zeros to by the unpredicated accesses: finite values
            for (int k = tid; k < kPadFloats; k += kThreads) {
                s_rp[-kPadFloats + k] = 0.0f;
                s_rp[region + k] = 0.0f;
                s_acc[-kPadFloats + k] = 0.0f;
                s_acc[region + k] = 0.0f;
            }
            for (int rr = tid; rr < tl.RH; rr += kThreads)
                for (int cc = tl.RW; cc < tl.RS; ++cc) {
                    if (!GLD) s_rp[rr * tl.RS + cc] = 0.0f;
                    s_cnt[rr * tl.RS + cc] = 0u;
                }
            fresh = false;
            // the groups' slots change their layout with G
            if (BATCH)
                for (int k = tid; k < kPartFloats; k += kThreads) s_part[k] = 0.0f;
        }
        const Frame f = tile_frame(g, tl, item.x);
        float sum = 0.0f, most = 0.0f;     // rho' over the warp's band of rows
        const int rpw = I.fx_rows;
        if constexpr (GLD) {
            if (MODE != kLoglik)
                for (int k = tid; k < region; k += kThreads) s_cnt[k] = 0u;
            // 32 rows of a run of columns a warp: the image's rows come through L1
            const int nr = (tl.RH + 31) >> 5;
            for (int k = warp; k < 4 * nr; k += kWarps) {
                const int rr = (k >> 2) * 32 + lane, iy = f.oy + rr;
                if (rr >= tl.RH) continue;
                const bool row_in = iy >= 0 && iy < g.ny;
                const int z0row = f.zbase + (int)rintf(__fmul_rn(f.shear, (float)(iy - f.Y0)));
                const int w = (tl.RW + 3) >> 2, c1 = min(tl.RW, ((k & 3) + 1) * w);
                float row = 0.0f;
#pragma unroll 4
                for (int cc = (k & 3) * w; cc < c1; ++cc) {
                    const int iz = z0row + cc;
                    float v = 0.0f;
                    if (row_in && iz >= 0 && iz < g.nz) v = __ldg(I.rhop + (size_t)iy * g.nz + iz);
                    scr[cc * kScrRows + rr] = v;
                    row += v;
                    most = fmaxf(most, v);
                }
                if (MODE != kLoglik) atomicAdd(&s_band[rr / rpw].x, row);
            }
        } else {
            for (int rr = warp * rpw; rr < min(tl.RH, (warp + 1) * rpw); ++rr) {
                const int iy = f.oy + rr;
                const bool row_in = iy >= 0 && iy < g.ny;
                const int z0row = f.zbase + (int)rintf(__fmul_rn(f.shear, (float)(iy - f.Y0)));
#pragma unroll 4
                for (int cc = lane; cc < tl.RW; cc += 32) {
                    const int iz = z0row + cc;
                    float v = 0.0f;
                    // (the read-only path: loads may pass the stores of earlier columns)
                    if (row_in && iz >= 0 && iz < g.nz) v = __ldg(I.rhop + (size_t)iy * g.nz + iz);
                    s_rp[rr * tl.RS + cc] = v;
                    if (MODE != kLoglik) s_cnt[rr * tl.RS + cc] = 0u;
                    sum += v;
                    most = fmaxf(most, v);
                }
            }
        }
        if (MODE != kLoglik) {
            most = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(most)));
            if constexpr (!GLD) sum = warp_sum(sum);
            if (lane == 0) {
                if constexpr (!GLD) s_band[warp].x = sum;
                s_band[warp].y = most;
            }
        }
        if (tid == 0) {
            s_item[par] = next;
            s_frame = f;
            // pixels that the records left out, counted once a pass
            if (item.y == 0) {
                s_sums.qclip += I.accum->rec_qclip;
                s_sums.lclip += I.accum->rec_lclip;
            }
        }
        __syncthreads();
        const int G = I.G;
        const int ngroups = group_count(kWarps, G);
        const int grp = warp / G, wig = warp - grp * G;
        RecScale* const sc = s_scale + warp;
        if (MODE != kLoglik) {
            static_assert(kWarps == 32, "a lane a band");
            const int groups = kTwo && two_rows_fit(G) ? rec2_groups(G, warp).y : ngroups;
            item_scale(I, s_band[lane], item.z, groups, lane, sc);
        }
        const unsigned rp_addr = (unsigned)__cvta_generic_to_shared(s_rp);
        const unsigned acc_off = GLD ? 0u : 4u * (unsigned)(region + 2 * kPadFloats);
        const unsigned slot = (unsigned)__cvta_generic_to_shared(smem + kPartFloats + warp * kSlot);
        float* part = s_part + grp * 2 * kMinWarps;
#define TSP_REC_EVENTS(TRAV) \
    rec_events<TRAV, LMAX, MODE, NSEG, GLD>(I, &s_frame, sc, item.y, item.z, grp, ngroups, wig, lane, \
                                            rp_addr, acc_off, slot, part, &s_sums, tma, scr)
        if (kTwo && two_rows_fit(G)) {
            if constexpr (kTwo)
                rec2_events<MODE>(I, &s_frame, sc, item.y, item.z, warp, lane, rp_addr, acc_off, slot,
                                  s_part, &s_sums, tma);
        } else if (grp < ngroups) {
            if (NSEG == 1)
                TSP_REC_EVENTS(kAlt);
            else if ((wig & 1) == 0)
                TSP_REC_EVENTS(kPos);
            else
                TSP_REC_EVENTS(kNeg);
        }
#undef TSP_REC_EVENTS
        __syncthreads();
        if (MODE != kLoglik) {
            if (GLD && tid < kWarps) s_band[tid].x = 0.0f;
            const float quantum = 1.0f / sc->inv_q;
            const Frame fl = s_frame;
            for (int rr = warp; rr < tl.RH; rr += kWarps) {
                const int iy = fl.oy + rr;
                if (iy < 0 || iy >= g.ny) continue;
                const int z0row = fl.zbase + (int)rintf(__fmul_rn(fl.shear, (float)(iy - fl.Y0)));
                for (int cc = lane; cc < tl.RW; cc += 32) {
                    const int iz = z0row + cc;
                    const int k = rr * tl.RS + cc;
                    float v = (float)s_cnt[k] * quantum;
                    // (the update is 0 where rho' = 0, whatever A holds)
                    if (MODE == kMlem && !GLD && !(s_rp[k] > 0.0f)) v = 0.0f;
                    if (iz >= 0 && iz < g.nz && v != 0.0f)
                        atomicAdd(I.A + (size_t)iy * g.nz + iz, v);
                }
            }
            __syncthreads();
        }
        it = s_item[par];
        par ^= 1;
    }
    tm_sync_threads();
    if (!BATCH || cur >= 0) flush_block_sums(&s_sums, I.accum, MODE);
#ifdef TSP_DEBUG_CHECKS
    if (tid == 0 && tsp_dbg_word && (!BATCH || cur >= 0))
        atomicCAS(&I.accum->dbg, 0ull, tsp_dbg_word);
#endif
    if (warp == 0) tm_dealloc<kCols>(s_tmem);
}

}  // namespace tsp
