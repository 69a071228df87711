// sic_item.cuh -- the device code that the step kernels share: a work item's
// push and deposit (do_item), the block's copy of the mesh, exact sums, the
// staging of items through shared memory and the field solve's arithmetic.
// Included by sic_kernels.cu (k_step) and sic_run.cu (k_run).
//
// Positions are 32-bit: P = x / L 2^30 modulo 2^32 (2 bits of winding).  The
// cell coordinate of a position, 32.32 fixed point with the cell in [0, nx),
// is one multiply (P 2^2) nx; a segment is the 32-bit difference of its ends'
// P times nx 2^2, so both ends are known in the frame of the lower one.
//
// Deposit arithmetic: a segment [a, b] of q units in 32.32 fixed-point cell
// coordinates gives its first cell F = round(q (e_1 - a) / (b - a)) (FP32,
// with an approximate reciprocal, clamped to [0, q]), every whole cell inside
// P = floor(q 2^32 / (b - a)) (exact integer), and the
// last cell the rest, q - F - (cells inside) P.  The pieces always sum to q
// exactly and never go negative; the integer mesh does not depend on the
// order of the atomic adds, so results are bit-identical however the work is
// split.  Whole cells inside a long segment are added through a difference
// array, so a segment costs O(1) shared-memory atomics at any length.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "sic_internal.h"

namespace sic {

namespace {

constexpr int B = SIC_K1_BLOCK;
constexpr int R = SIC_K1_R;
constexpr int NW = SIC_K1_WARPS;
constexpr int WT = SIC_K1_WARP_TRACERS;

__device__ __forceinline__ int cell_of(long long u) { return (int)(u >> 32); }
__device__ __forceinline__ unsigned frac_of(long long u) { return (unsigned)(unsigned long long)u; }

// 32.32 fixed-point cell coordinate of a position P (x / L 2^30 modulo 2^32):
// the cell in [0, nx) in the high word, the fraction of the cell in the low
// word, exactly (one 32 x 32 -> 64 multiply of the box fraction P 2^2 by nx)
__device__ __forceinline__ long long cell_coord(unsigned p, int nx)
{
    return (long long)((unsigned long long)(p << SIC_POS_WIND_BITS) * (unsigned)nx);
}

// The segment from position pa to pb in 32.32 cell units: the 32-bit
// difference of the positions (exact for segments shorter than 2 box lengths)
// times nx 2^2
__device__ __forceinline__ long long seg_span(unsigned pa, unsigned pb, int nx4)
{
    return (long long)(int)(pb - pa) * (long long)nx4;
}

// fraction of a cell in [0, 1) from the low word (its top 23 bits)
__device__ __forceinline__ float frac_float(unsigned lo)
{
    return __fsub_rn(__uint_as_float(0x3f800000u | (lo >> 9)), 1.0f);
}

// gather (linear weighting between nodes j and j+1), kick, drift; j is the
// cell of the new position on return.  ek[j] = (Ek_j, Ek_{j+1} - Ek_j).  The
// drift adds the velocity rounded to whole position units (exact integer
// arithmetic, wrapping modulo 4 box lengths); vmax keeps the largest |v|, and
// a step of half a box (2^29 units) or more is an error.
__device__ __forceinline__ void push_one(unsigned &p, float &v, int &j, const float2 *ek, int nx, float ks,
                                         int drift, float &vmax)
{
    const long long c = cell_coord(p, nx);
    j = cell_of(c);
    const float2 e = ek[j];
    const float a = __fmaf_rn(frac_float(frac_of(c)), e.y, e.x);
    const float vn = __fmaf_rn(ks, a, v);
    v = vn;
    if (drift) {
        vmax = fmaxf(vmax, fabsf(vn));
        p += (unsigned)__float2int_rn(vn);
        j = cell_of(cell_coord(p, nx));
    }
}

// The block's copy of the charge mesh: cell j holds hi[j] * 2^32 + lo[j].
// Adds use 32-bit shared-memory atomics (a carry out of the low word goes to
// the high word), which the hardware executes natively.
struct Hist {
    unsigned *lo;
    unsigned *hi;
    __device__ __forceinline__ void add(int j, long long v) const
    {
        const unsigned l = (unsigned)(unsigned long long)v;
        const unsigned h = (unsigned)((unsigned long long)v >> 32);
        const unsigned old = atomicAdd(lo + j, l);
        const unsigned c = h + ((old + l < old) ? 1u : 0u);
        if (c)
            atomicAdd(hi + j, c);
    }
    __device__ __forceinline__ void add32(int j, unsigned v) const
    {
        const unsigned old = atomicAdd(lo + j, v);
        if (old + v < old)
            atomicAdd(hi + j, 1u);
    }
    __device__ __forceinline__ void sub32(int j, unsigned v) const  // v > 0
    {
        if (atomicAdd(lo + j, 0u - v) < v)
            atomicAdd(hi + j, 0xffffffffu);
    }
    __device__ __forceinline__ unsigned long long get(int j) const
    {
        return ((unsigned long long)hi[j] << 32) | lo[j];
    }
    __device__ __forceinline__ void set(int j, unsigned long long v) const
    {
        lo[j] = (unsigned)v;
        hi[j] = (unsigned)(v >> 32);
    }
};

// Per-thread run of consecutive contributions to one cell; a cell change
// commits the run to the block's mesh.
struct RunAcc {
    Hist h;
    int cell;
    long long sum;
    __device__ __forceinline__ explicit RunAcc(const Hist &hist) : h(hist), cell(-1), sum(0) {}
    __device__ __forceinline__ void add(int j, long long v)
    {
        if (j == cell) {
            sum += v;
            return;
        }
        if (sum)
            h.add(cell, sum);
        cell = j;
        sum = v;
    }
    __device__ __forceinline__ void flush()
    {
        if (sum)
            h.add(cell, sum);
        sum = 0;
        cell = -1;
    }
};

// A 64-bit integer rounded to nearest in FP32 (as __ll2float_rn and
// __float2ll_rn round, which run on the FP64 pipe, 64 cycles a warp
// instruction): the top 32 bits with the bits below them as a sticky bit
// round as the whole does.
__device__ __forceinline__ float u64_to_float(unsigned long long v)
{
    const unsigned hi = (unsigned)(v >> 32);
    if (hi == 0)
        return __uint2float_rn((unsigned)v);
    const int s = 32 - __clz((int)hi);  // 1..32
    const unsigned w = (unsigned)(v >> s) | ((v << (64 - s)) ? 1u : 0u);
    return __fmul_rn(__uint2float_rn(w), __uint_as_float((unsigned)(127 + s) << 23));
}

__device__ __forceinline__ float i64_to_float(long long v)
{
    const float f = u64_to_float((unsigned long long)(v < 0 ? -v : v));
    return v < 0 ? -f : f;
}

__device__ __forceinline__ long long float_to_i64(float x)
{
    if (fabsf(x) < 2147483648.0f)
        return __float2int_rn(x);
    return __float2ll_rn(x);
}

__device__ __forceinline__ float span_to_float(long long span)
{
    if ((unsigned long long)span < (1ull << 32))
        return __uint2float_rn((unsigned)span);
    return __fmaf_rn(__int2float_rn((int)(span >> 32)), 4294967296.0f, __uint2float_rn(frac_of(span)));
}

// floor(q 2^32 / span) for 0 <= q <= 2^28 and 2^32 <= span < 2^46 (a particle
// that covers whole cells): the whole-cell charge of a box particle, at most
// q.  qf and inv are q and an approximate 1 / span in FP32.  The estimate's
// relative error is below 2^-21, so it is within 130 of the quotient; the
// exact remainder then gives the rest of it to the nearest integer (error
// below 0.5 + 2^-14), and its sign the floor.  Only 32-bit conversions: the
// 64-bit ones run on the FP64 pipe, 64 cycles a warp instruction.
__device__ __forceinline__ unsigned whole_cell_charge(unsigned q, float qf, unsigned long long span, float inv)
{
    const unsigned P0 = __float2uint_rz(__fmul_rn(__fmul_rn(qf, 4294967296.0f), inv));
    long long r = (long long)(((unsigned long long)q << 32) - (unsigned long long)P0 * span);
    const float rf = __fmaf_rn(__int2float_rn((int)(r >> 32)), 4294967296.0f, __uint2float_rn((unsigned)r));
    const int k = __float2int_rn(__fmul_rn(rf, inv));
    r -= (long long)k * (long long)span;
    return P0 + (unsigned)k - (r < 0 ? 1u : 0u);
}

// n whole cells starting at cell js (mod nx) each receive p units: +p at js
// and -p after the range in the block's difference array (two's complement
// in the same 32-bit lo/hi form as the mesh, so the adds are native shared
// atomics), summed into the mesh when the block leaves the simulation
__device__ __noinline__ void range_add(int js, long long n, long long p, int nx, const Hist &dh, int *diff_used)
{
    const long long full = n < nx ? 0 : n / nx;  // 0 or 1 for a particle shorter than 1.5 box lengths
    const int rem = (int)(n - full * nx);
    if (full)
        dh.add(0, full * p);
    if (rem) {
        const int e = js + rem;
        dh.add(js, p);
        if (e <= nx) {
            dh.add(e, -p);
        } else {
            dh.add(0, p);
            dh.add(e - nx, -p);
        }
    }
    *diff_used = 1;
}

// Deposit one segment that crosses at least one cell edge, between
// fixed-point positions ua (cell ja mod nx) and ub (cell jb mod nx), carrying
// q units.  maxseg tracks the longest such segment, in 2^-16 cells
// (saturating).
// Adds each piece straight into the block's mesh.
struct DirectAdd {
    Hist h;
    __device__ __forceinline__ void add(int j, long long v) const
    {
        if (v)
            h.add(j, v);
    }
};

template <class ACC>
__device__ __forceinline__ void emit_cross(long long ua, int ja, long long ub, int jb, int q, int nx, ACC &acc,
                                           const Hist &diff, int *diff_used, unsigned &maxseg)
{
    if (ub < ua) {
        const long long t = ua;
        ua = ub;
        ub = t;
        const int tj = ja;
        ja = jb;
        jb = tj;
    }
    const long long span = ub - ua;
    maxseg = max(maxseg, (unsigned)min((unsigned long long)span >> 16, 0xffffffffull));
    const unsigned la = frac_of(ua);
    const float df = la ? __uint2float_rn(0u - la) : 4294967296.0f;  // a to the first edge
    // an approximate reciprocal is enough: F is clamped to [0, q] and the
    // other end takes q - F, so the charge stays exact
    float inv;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(span_to_float(span)));
    int F = __float2int_rn(__fmul_rn(__fmul_rn(df, inv), __int2float_rn(q)));
    F = min(max(F, 0), q);
    const long long ncut = (long long)cell_of(ub) - (long long)cell_of(ua);
    if (ncut == 1) {
        acc.add(ja, F);
        acc.add(jb, q - F);
        return;
    }
    const long long nint = ncut - 1;
    const long long P = whole_cell_charge((unsigned)q, __int2float_rn(q), (unsigned long long)span, inv);
    const long long inner = nint * P;
    if ((long long)F > (long long)q - inner)
        F = (int)((long long)q - inner);
    acc.add(ja, F);
    int j = (ja + 1 == nx) ? 0 : ja + 1;
    if (nint <= 2) {
        acc.add(j, P);
        if (nint == 2) {
            j = (j + 1 == nx) ? 0 : j + 1;
            acc.add(j, P);
        }
    } else {
        range_add(j, nint, P, nx, diff, diff_used);
    }
    acc.add(jb, (long long)q - F - inner);
}

// First-order weighting of a box particle (Sec. 2.4), between 32.32 cell
// coordinates ua and ub (any order, the lower end's cell possibly outside
// [0, nx)), q units.  Its zero-order piece in each cell (the pieces of
// emit_cross: first, whole cells inside, the rest) is shared between the
// cell's two nodes by the piece's centroid: the upper node gets round(piece
// (s0 + s1) / 2) of a piece over [s0, s1] of the cell, the lower one the
// rest.  That is the hat weighting of a uniform density exactly, up to the
// rounding of each share, and the node charges sum to q.
__device__ __forceinline__ int wrap_near(int c, int nx)
{
    while (c < 0)
        c += nx;
    while (c >= nx)
        c -= nx;
    return c;
}

template <class ACC>
__device__ __forceinline__ void emit_first(long long ua, long long ub, int q, int nx, ACC &acc,
                                           const Hist &diff, int *diff_used, unsigned &maxseg)
{
    if (ub < ua) {
        const long long t = ua;
        ua = ub;
        ub = t;
    }
    const int ja = wrap_near(cell_of(ua), nx);
    const int ja1 = (ja + 1 == nx) ? 0 : ja + 1;
    const unsigned la = frac_of(ua), lb = frac_of(ub);
    const long long ncut = (long long)cell_of(ub) - (long long)cell_of(ua);
    const long long span = ub - ua;
    maxseg = max(maxseg, (unsigned)min((unsigned long long)span >> 16, 0xffffffffull));
    if (ncut == 0) {  // inside one cell (or a point): centroid (la + lb) / 2
        const long long Y =
            (long long)(((unsigned long long)q * ((unsigned long long)la + lb) + (1ull << 32)) >> 33);
        acc.add(ja, (long long)q - Y);
        acc.add(ja1, Y);
        return;
    }
    const float df = la ? __uint2float_rn(0u - la) : 4294967296.0f;  // a to the first edge
    float inv;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(span_to_float(span)));
    long long F = __float2int_rn(__fmul_rn(__fmul_rn(df, inv), __int2float_rn(q)));
    F = min(max(F, 0ll), (long long)q);
    const long long nint = ncut - 1;
    const long long P = nint > 0 ? whole_cell_charge((unsigned)q, __int2float_rn(q), (unsigned long long)span, inv) : 0;
    const long long inner = nint * P;
    if (F > (long long)q - inner)
        F = (long long)q - inner;
    const long long Lr = (long long)q - F - inner;  // the last cell's piece
    // shares of the upper nodes: first piece over [la, 1], whole cells 1/2,
    // last piece over [0, lb]
    const long long YF = (long long)(((unsigned long long)F * ((1ull << 32) + la) + (1ull << 32)) >> 33);
    const long long YP = (P + 1) >> 1;
    const long long YL = (long long)(((unsigned long long)Lr * lb + (1ull << 32)) >> 33);
    const int jb = wrap_near(cell_of(ub), nx);
    const int jb1 = (jb + 1 == nx) ? 0 : jb + 1;
    acc.add(ja, F - YF);
    if (nint == 0) {  // first and last cells adjacent: node ja + 1 is jb
        acc.add(jb, YF + Lr - YL);
    } else {
        acc.add(ja1, YF + P - YP);
        // nodes ja + 2 .. ja + nint get P each (the upper share of the cell
        // below and the lower share of their own)
        if (nint > 1) {
            const int js = (ja1 + 1 == nx) ? 0 : ja1 + 1;
            if (nint - 1 <= 2) {
                acc.add(js, P);
                if (nint - 1 == 2)
                    acc.add((js + 1 == nx) ? 0 : js + 1, P);
            } else {
                range_add(js, nint - 1, P, nx, diff, diff_used);
            }
        }
        acc.add(jb, YP + Lr - YL);
    }
    acc.add(jb1, YL);
}

// Piecewise-linear particles (Sec. 2.5).  The particle from ua to ub (tracers
// i, i+1) has neighbours from up (tracer i-1) and to un (tracer i+2) along
// the sheet, all in 32.32 cell coordinates, with charges qp, qs, qn.  Its
// density rho0 + g (x - c) gives, from its lower end, the cumulative charge
// qs (t + kappa t (t - 1)) at the fraction t of its length, with
// kappa = g l / (2 rho0) and g the central difference of Eq.
// gradient_rho_estimate.  The centroids are in order along the sheet exactly
// when up < ub and ua < un (or both reversed); otherwise (a fold corner), or
// when a length or the charge is zero, kappa = 0: the box particle.
__device__ __forceinline__ float pl_kappa(long long up, long long ua, long long ub, long long un, int qp, int qs,
                                          int qn)
{
    const bool inc = up < ub && ua < un, dec = up > ub && ua > un;
    const long long lp = ua > up ? ua - up : up - ua;
    const long long ls = ub > ua ? ub - ua : ua - ub;
    const long long ln = un > ub ? un - ub : ub - un;
    if (!(inc || dec) || lp == 0 || ls == 0 || ln == 0 || qs == 0)
        return 0.f;
    const float fp = i64_to_float(lp), fs = i64_to_float(ls), fn = i64_to_float(ln);
    const float rp = __fdiv_rn(__int2float_rn(qp), fp);
    const float rs = __fdiv_rn(__int2float_rn(qs), fs);
    const float rn = __fdiv_rn(__int2float_rn(qn), fn);
    // twice the centroid distance c_{s+1} - c_{s-1}, signed
    const float dc2 = i64_to_float((ub - up) + (un - ua));
    const float k = __fdiv_rn(__fmul_rn(__fsub_rn(rn, rp), fs), __fmul_rn(rs, dc2));
    return fabsf(k) < 1e30f ? k : 0.f;
}

// Piecewise-linear particles of a warp, one per lane (n cells of it, 0: none),
// shorter than the box each.  From the lower end's cell jl, at the fraction la
// of it, the cell between the cuts k and k+1 gets round(q phi(t_{k+1})) -
// round(q phi(t_k)), phi(t) = t + kappa t (t - 1), t_k the fraction of the
// length at the k-th edge (phi(0) = 0, phi(1) = 1), so the pieces sum to q
// exactly.  A piece may be negative when |kappa| > 1 (the linear density
// changes sign inside the particle).
//
// The cells of all 32 particles are laid out one after another and dealt to
// the lanes 32 at a time, each lane finding its particle in the running count
// and taking its parameters from the owner: on folded sheets particles range
// from two cells to half the box, and a loop per lane (or a warp per long
// particle) left most lanes idle for a chain of divisions and conversions.
// A step of 256 x 2048 folded tracers on 256 cells takes 71 us, 122 us with those
// loops (42 us of many steps a launch).
__device__ __forceinline__ void emit_linear(int jl, unsigned la, float inv, int q, float kappa, int n, int nx,
                                            const Hist &hist)
{
    const int lane = threadIdx.x & 31;
    // round(q phi) at the edge above cell jl + k
    auto cum = [](int k, unsigned la_, float inv_, float kap_, int q_) -> long long {
        const float t = __fmul_rn(u64_to_float(((unsigned long long)(unsigned)(k + 1) << 32) - la_), inv_);
        const float phi = __fmaf_rn(__fmul_rn(kap_, t), __fsub_rn(t, 1.0f), t);
        return float_to_i64(__fmul_rn(__int2float_rn(q_), phi));
    };
    if (!__any_sync(0xffffffffu, n > 2)) {
        // Particles of two cells only, as on quiet sheets: one edge each and
        // nothing to deal.  Single steps, us with the dealing and this: 256
        // sheets of 600 on 512 cells 37.1 and 28.4, 512 of 4096 on 1024 41.3 and
        // 35.7 (many steps a launch 18.3 and 14.0, 35.6 and 30.3); folded 256 x
        // 2048 on 256 take 1 % longer.
        if (n == 2) {
            const long long first = cum(0, la, inv, kappa, q);
            if (first)
                hist.add(jl, first);
            if (q - first)
                hist.add(jl + 1 == nx ? 0 : jl + 1, q - first);
        }
        return;
    }
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += t;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    long long last = 0;  // round(q phi) at the upper cut of the cell before this pass's first
    for (int p0 = 0; p0 < total; p0 += 32) {
        const int p = p0 + lane;
        int own = 0;  // particles that end at or before p
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, incl, own + o - 1) <= p)
                own += o;
        own = min(own, 31);  // past the end: any
        const int n_o = __shfl_sync(0xffffffffu, n, own);
        const int k = p - (__shfl_sync(0xffffffffu, incl, own) - n_o);  // cell jl + k
        const int jl_o = __shfl_sync(0xffffffffu, jl, own);
        const unsigned la_o = __shfl_sync(0xffffffffu, la, own);
        const float inv_o = __shfl_sync(0xffffffffu, inv, own);
        const float kap_o = __shfl_sync(0xffffffffu, kappa, own);
        const int q_o = __shfl_sync(0xffffffffu, q, own);
        long long up = q_o;  // round(q phi) at the cell's upper cut
        if (k + 1 < n_o)
            up = cum(k, la_o, inv_o, kap_o, q_o);
        long long lo = __shfl_up_sync(0xffffffffu, up, 1);
        if (lane == 0)
            lo = last;
        last = __shfl_sync(0xffffffffu, up, 31);
        if (p < total) {
            const long long piece = up - (k == 0 ? 0 : lo);
            int j = jl_o + k;  // k <= nx
            if (j >= nx)
                j -= nx;
            if (piece)
                hist.add(j, piece);
        }
    }
}

// A 128-bit integer as two words (the warp's and block's fixed-point sums).
struct Acc128 {
    unsigned long long lo;
    long long hi;
};

__device__ __forceinline__ void acc_add(Acc128 &a, const Acc128 &b)
{
    const unsigned long long nlo = a.lo + b.lo;
    a.hi = a.hi + b.hi + (nlo < b.lo ? 1 : 0);
    a.lo = nlo;
}

// The sum of the warp's 64-bit values, in every lane: four sums of 16-bit
// pieces (the top one signed), 21 bits each, by the warp's own reduction
__device__ __forceinline__ Acc128 i64_warp_sum(long long v)
{
    const unsigned long long u = (unsigned long long)v;
    const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)u & 0xffffu);
    const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 16) & 0xffffu);
    const unsigned s2 = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 32) & 0xffffu);
    const int s3 = __reduce_add_sync(0xffffffffu, (int)(v >> 48));
    Acc128 t{(unsigned long long)s0 + ((unsigned long long)s1 << 16) + ((unsigned long long)s2 << 32), 0ll};
    acc_add(t, Acc128{(unsigned long long)(long long)s3 << 48, (long long)s3 >> 16});
    return t;
}

// 128-bit add into a (lo, hi) pair of 64-bit words with two atomics
__device__ __forceinline__ void atomic_add_i128(unsigned long long *lohi, __int128 v)
{
    if (v == 0)
        return;
    const unsigned long long lo = (unsigned long long)v;
    const unsigned long long hi = (unsigned long long)(v >> 64);
    const unsigned long long old = atomicAdd(lohi, lo);
    const unsigned long long carry = (old + lo < old) ? 1ull : 0ull;
    if (hi + carry)
        atomicAdd(lohi + 1, hi + carry);
}

struct Spill {
    long long a;
    unsigned err;
};

// The rare path of sum_add, for the whole warp: the sums of the lanes that ask
// for it go into the block's 128-bit sum (shared memory), and so do their terms
// y unless they fit a fresh 64-bit sum.  y is integer-valued when it is 2^63 or
// more (below 2^124; inf, NaN or larger set bit 31 of the error word instead).
// The lanes are summed first: plasmas that start at rest have units so fine
// that every lane comes here, and 256 64-bit adds to one word, loops of
// compare-and-swap, were most of their step (a cold oscillation of 4096 tracers
// on 64 cells, us a step: 26.3 lane by lane, 6.3).
__device__ __noinline__ Spill acc_spill(long long a, float y, unsigned long long *blk, bool mine)
{
    Spill r{a, 0u};
    Acc128 t{0ull, 0ll};
    if (mine) {
        r.a = 0;
        __int128 v = a;
        if (fabsf(y) < 9223372036854775808.0f) {
            r.a = __float2ll_rz(y);
        } else {
            const unsigned b = __float_as_uint(y);
            const int sh = (int)((b >> 23) & 0xffu) - 150;  // y = m 2^sh, sh >= 40 here
            if (sh > 100) {
                r.err = 0x80000000u;
            } else {
                const __int128 m = (__int128)((b & 0x7fffffu) | 0x800000u) << sh;
                v += (b >> 31) ? -m : m;
            }
        }
        t = Acc128{(unsigned long long)v, (long long)(v >> 64)};
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Acc128 b;
        b.lo = __shfl_down_sync(0xffffffffu, t.lo, o);
        b.hi = __shfl_down_sync(0xffffffffu, t.hi, o);
        acc_add(t, b);
    }
    if ((threadIdx.x & 31) == 0)
        atomic_add_i128(blk, (__int128)(((unsigned __int128)(unsigned long long)t.hi << 64) | t.lo));
    return r;
}

// Add y (a term already in the sum's fixed-point unit), truncated to an
// integer, to a lane's 64-bit sum.  Below 2^53 the integer is the exact sum
// of two 32-bit conversions, y's multiple of 2^22 and the rest (both exact in
// FP32: y has 24 bits); one 64-bit conversion would take the FP64 pipe 64
// cycles a warp.  A term of 2^53 or more, or one that would overflow the sum,
// takes the rare path, which moves the lane's sum into the block's 128-bit
// sum: the total stays exact, so it does not depend on the order of the
// additions.
__device__ __forceinline__ void sum_add(long long &a, float y, unsigned long long *blk, unsigned &err)
{
    const int h = __float2int_rz(__fmul_rn(y, 0x1p-22f));
    const int l = __float2int_rz(__fmaf_rn(__int2float_rn(h), -0x1p22f, y));
    const long long v = (long long)h * (1ll << 22) + l;
    const long long s = (long long)((unsigned long long)a + (unsigned long long)v);
    const bool over = !(fabsf(y) < 9007199254740992.0f) || ((a ^ s) & (v ^ s)) < 0;
    if (__builtin_expect(__any_sync(0xffffffffu, over), 0)) {
        const Spill r = acc_spill(a, y, blk, over);
        a = over ? r.a : s;
        err |= r.err;
    } else {
        a = s;
    }
}

__device__ __forceinline__ double i128_words_to_double(unsigned long long lo, unsigned long long hi)
{
    return __fma_rn((double)(long long)hi, 18446744073709551616.0, __ull2double_rn(lo));
}

// ---- programmatic dependent launch: a step launched with it may start while
// the step before it in the stream finishes; it waits for that step's end
// (and its memory) before it reads anything that step writes, and lets the
// next one start once it has no more items to begin.  Without the launch
// attribute both are no-ops.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- bulk-copy staging (cp.async.bulk into shared memory, mbarrier completion)

__device__ __forceinline__ unsigned smem_u32(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity)
{
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(smem_u32(bar)), "r"(parity)
                 : "memory");
    return ok != 0;
}

// The tracer state is read once per step and is larger than L2: its copies
// are marked first to be evicted, so the kernel's code, the simulation
// tables and the meshes stay in L2 from step to step.
__device__ __forceinline__ unsigned long long l2_evict_first()
{
    unsigned long long pol;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, unsigned long long *bar,
                                         unsigned long long pol)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}

// A bounded wait on a stage barrier: true once the phase of this parity has
// completed; false after about a second of polling (the caller raises an
// error instead of hanging).
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long *bar, unsigned parity)
{
    for (int i = 0; i < (1 << 24); ++i)
        if (mbar_try_wait(bar, parity))
            return true;
    return false;
}

// A warp that gave up on its copies waits for them once more (as long at most)
// before it goes on to leave the kernel: they must not land in the shared memory
// of a block that has exited.
__device__ __noinline__ void mbar_drain(unsigned long long *bar, unsigned parity)
{
    (void)mbar_wait_bounded(bar, parity);
}

constexpr int kStageBytesU = SIC_STAGE_U_BYTES;
constexpr int kStageBytesV = SIC_STAGE_V_BYTES;
constexpr int kStageBytesQ = SIC_STAGE_Q_BYTES;
// the box deposit's table of a warp's positions (and as much again of running
// charges), entry r of lane l at 32 r + l, r = 0..R
constexpr int kTabWords = 32 * (SIC_K1_R + 1);
constexpr int kTabBytes = 4 * kTabWords;

// Per-warp buffer: two stages when staging (U | V | Q each), otherwise one
// scratch of new positions (U | Q) for the cross-cell pass.
template <bool PER_Q, bool STAGED>
struct WarpBuf {
    static constexpr int q_offset = STAGED ? kStageBytesU + kStageBytesV : kStageBytesU;
    // (without staging the box deposit's table is the larger use)
    static constexpr int stage = STAGED ? q_offset + (PER_Q ? kStageBytesQ : 0) : (PER_Q ? 2 : 1) * kTabBytes;
    static_assert(stage >= (PER_Q ? 2 : 1) * kTabBytes && stage >= q_offset + (PER_Q ? kStageBytesQ : 0),
                  "a stage holds the item and the table");
    static constexpr int bytes = (STAGED ? 2 : 1) * stage;
};

// Lane 0 of a warp: copy a work item's descriptor into shared memory
// without waiting for it (five 8-byte asynchronous copies, one group)
__device__ __forceinline__ void desc_fetch(WorkItem *dst, const WorkItem *src)
{
    const unsigned d = smem_u32(dst);
    unsigned long long g;
    asm("cvta.to.global.u64 %0, %1;" : "=l"(g) : "l"(src));
#pragma unroll
    for (int k = 0; k < 5; ++k)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d + 8 * k), "l"(g + 8 * k) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void desc_wait()
{
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Lane 0 of a warp: start the bulk copies of item W (and its halo when the
// halo is the next tracer in memory) into one stage.
template <bool PER_Q>
__device__ __forceinline__ void stage_issue(const WorkItem &W, const unsigned *Uin, const float *Vin,
                                            const int32_t *Qh, char *st, unsigned long long *bar)
{
    const bool contiguous_halo = (W.halo == W.t0 + W.count);
    const int n = W.count + (contiguous_halo ? 1 : 0);
    const unsigned b = (unsigned)(n * 4 + 15) & ~15u;  // the same for positions, velocities, charges
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_expect_tx(bar, (PER_Q ? 3u : 2u) * b);
    const unsigned long long pol = l2_evict_first();
    bulk_g2s(st, Uin + W.t0, b, bar, pol);
    bulk_g2s(st + kStageBytesU, Vin + W.t0, b, bar, pol);
    if (PER_Q)
        bulk_g2s(st + kStageBytesU + kStageBytesV, Qh + W.t0, b, bar, pol);
}

// What a warp that keeps its item in shared memory from step to step (k_run)
// holds besides: the tracers outside the item that it pushes for itself, the
// one after the item and, for piecewise-linear particles, the one before it
// and the one after the next
struct Beside {
    unsigned hu, pu, nu;
    float hv, pv, nv;
    int hq, pq, nq;
};

struct Shared {
    SimDev sim;              // the current simulation's descriptor
    unsigned long long mbar[NW][2];
    struct alignas(16) Slot {
        WorkItem w;
    } desc[NW][2];  // staging: each warp's descriptors of the items in its two stages
    int diff_used;
    int last;
    unsigned pl_prev[NW];    // piecewise-linear particles: each warp's tracer before its item
    int pl_prevq[NW];
    int taken;               // items of the current simulation the block's warps took
    int pick_n[NW], pick_s[NW];  // per warp: most unclaimed items, in which slot
    unsigned long long ke[2], p[2];          // 128-bit sums of the rare path (sum_add)
    long long wke[NW][2], wp[NW][2];         // each warp's KE and P sums (lo, hi)
    unsigned wmseg[NW];                      // each warp's longest segment
    unsigned hold, buf;                      // the simulation's scalars at entry
    long long w64[NW];
    long long hi[NW], lo[NW];
    double da[NW];
    // the epilogue's inputs, read in one round trip with the mesh: the sums'
    // limbs (ke 0-3, p 4-7), the longest segment (8), and the scalars
    unsigned long long pre[9];
    long long pre_step;
    double pre_we, pre_wk;
    unsigned pre_err, pre_hold;
    float mre[NW], mim[NW];  // each warp's part of the Fourier mode sum
    // k_run: the step's longest segment and error bits, the block's sums, and
    // whether the wait for the other blocks gave up
    unsigned long long step_mseg;
    unsigned step_err, gave_up, last_out;
    unsigned long long tot[2][2];  // KE, P: lo, hi
    WorkItem own[NW];              // each warp's first item of a step
    Beside beside[NW];
};

constexpr size_t kSharedHead = (sizeof(Shared) + 15) / 16 * 16;

// shared head, mesh lo/hi [nx], diff [nx + 2], kick pairs [nx] (float2);
// staging starts on a 128-byte boundary (bulk copies need 16)
__host__ __device__ __forceinline__ size_t stage_offset(int nx_max)
{
    const size_t end = kSharedHead + (size_t)8 * nx_max + (size_t)8 * (nx_max + 2) + (size_t)8 * nx_max;
    return (end + 127) / 128 * 128;
}

// ------------------------------------------------------------ epilogue ----

__device__ __forceinline__ double i128_to_double(__int128 v)
{
    const long long hi = (long long)(v >> 64);
    const unsigned long long lo = (unsigned long long)v;
    return __fma_rn((double)hi, 18446744073709551616.0, __ull2double_rn(lo));
}

__device__ __forceinline__ __int128 shfl_down_i128(__int128 v, int o)
{
    long long lo = (long long)(unsigned long long)v;
    long long hi = (long long)(v >> 64);
    lo = __shfl_down_sync(0xffffffffu, lo, o);
    hi = __shfl_down_sync(0xffffffffu, hi, o);
    return (__int128)(((unsigned __int128)(unsigned long long)hi << 64) | (unsigned long long)lo);
}

__device__ __forceinline__ __int128 make_i128(long long hi, long long lo)
{
    return (__int128)(((unsigned __int128)(unsigned long long)hi << 64) | (unsigned long long)lo);
}

// v * 2^e2 as a float, without FP64: normalise |v|, keep its top 32 bits,
// round them to 24 (relative error < 2^-24 + 2^-31), then scale by 2^(...)
__device__ __forceinline__ float pow2f(int e)
{
    e = max(-126, min(127, e));
    return __uint_as_float((unsigned)(e + 127) << 23);
}

// |v| normalised to its top 32 bits t (|v| = t 2^(e - 96) up to the bits
// below them), once for several scalings
struct Norm128 {
    unsigned t;
    int e;  // 96 - leading zeros
    bool neg, zero;
};

__device__ __forceinline__ Norm128 norm128(__int128 v)
{
    Norm128 r;
    r.zero = v == 0;
    r.neg = v < 0;
    const unsigned __int128 m = r.neg ? (unsigned __int128)(-v) : (unsigned __int128)v;
    const unsigned long long hi = (unsigned long long)(m >> 64), lo = (unsigned long long)m;
    // the top two nonzero 32-bit words and a funnel shift, instead of a
    // 128-bit one
    const unsigned long long top = hi ? hi : lo;
    const unsigned th = (unsigned)(top >> 32), tl = (unsigned)top;
    const unsigned a = th ? th : tl;
    const unsigned b = th ? tl : (hi ? (unsigned)(lo >> 32) : 0u);
    const int lz = __clz((int)a);
    r.t = __funnelshift_l(b, a, lz);
    r.e = (hi ? 64 : 0) + (th ? 32 : 0) - lz;
    return r;
}

// v 2^e2 as a float from its normalised form
__device__ __forceinline__ float norm_to_float(const Norm128 &n, int e2)
{
    if (n.zero)
        return 0.f;
    const int e = n.e + e2;  // |v| 2^e2 = t 2^e
    float f = __uint2float_rn(n.t);
    if (e >= -126 && e <= 95) {  // one exact scaling
        f = __fmul_rn(f, __uint_as_float((unsigned)(e + 127) << 23));
    } else {
        const int e_a = e / 2, e_b = e - e / 2;
        f = __fmul_rn(__fmul_rn(f, pow2f(e_a)), pow2f(e_b));
    }
    return n.neg ? -f : f;
}

__device__ __forceinline__ float i128_to_float(__int128 v, int e2) { return norm_to_float(norm128(v), e2); }

// x 2^k exactly (x 2^k a normal double or zero)
__device__ __forceinline__ double times_pow2(double x, int k)
{
    return x * __hiloint2double((1023 + k) << 20, 0);
}

// One term of the Fourier sum sum_j y_j exp(-2 pi i j k / nx) (Sec. 3.2: the
// energy in the excited mode), the phase reduced exactly to j k mod nx.
__device__ __noinline__ void mode_add(float y, int j, int k, int nx, float &re, float &im)
{
    const int idx = (int)(((long long)j * k) % nx);
    float sn, cs;
    sincospif(__fdiv_rn(__int2float_rn(2 * idx), __int2float_rn(nx)), &sn, &cs);
    re = __fmaf_rn(y, cs, re);
    im = __fmaf_rn(-y, sn, im);
}

// inclusive prefix sum of diff[0..nx) added into hist (block-wide)
__device__ void add_diff_prefix(const Hist &hist, const Hist &diff, int nx, Shared &sh)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (nx + B - 1) / B;
    const int j0 = min(tid * per, nx), j1 = min(j0 + per, nx);
    long long lsum = 0;
    for (int j = j0; j < j1; ++j)
        lsum += (long long)diff.get(j);
    long long incl = lsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += t;
    }
    if (lane == 31)
        sh.w64[warp] = incl;
    __syncthreads();
    long long run = incl - lsum;
    for (int w = 0; w < warp; ++w)
        run += sh.w64[w];
    for (int j = j0; j < j1; ++j) {
        run += (long long)diff.get(j);
        hist.set(j, hist.get(j) + (unsigned long long)run);
    }
    __syncthreads();
}

// ---------------------------------------------------------------- kernel ----

// The box deposit of one warp's tracers, R consecutive ones per lane at u with
// cells jn (nu, nj, nq: the tracer after the lane's last one; nseg: segments
// starting at the lane's tracers, nseg_item: at the item's).
//
// Along a lane, charge is carried in `pend` until the sheet leaves the cell it
// is in: a segment inside a cell adds its charge to it, one that crosses edges
// commits it together with its share of the cell it leaves and carries on with
// its share of the cell it arrives in.  So a lane makes one commit per crossing
// segment and one at its end, and the crossing segments of the lanes are dealt
// with side by side: the loop runs as often as the lane with the most of them
// asks (once on quiet sheets).  With one charge per sheet, lanes without a
// crossing make no commit: the lane with a crossing before them takes their
// segments into its last one (they lie in one cell), which also spares
// the adds of many lanes into one word.  No list of the crossing ones is made
// and no lane works for another, but in short items (below).  Against per-cell
// counts and a warp-wide task list for the crossing ones (us per step, before and
// after): 4.2 M folded
// tracers 72 and 51, 2.3 M folded 50 and 34, 8.4 M quiet 43 and 41; a batch of
// 66 M quiet 278 and 246.  (With the whole cells through the general
// range_add, a call of 64-bit adds: 60, 42.)
//
// A crossing segment of q units in 32.32 cell coordinates: its lower end's
// cell gets F = round(q (e_1 - a) / (b - a)) (FP32, approximate reciprocal,
// clamped), every whole cell inside P = floor(q 2^32 / (b - a)), the upper
// end's the rest: all below 2^28, so the arithmetic is 32 bits wide.
// tab: the lane's positions (and running charges) by index, entry r of lane l
// at 32 r + l, so that a lane's own choice of r never conflicts.
template <bool PER_Q, bool FULL>
__device__ __forceinline__ void deposit_boxes(const unsigned (&u)[R], const int (&jn)[R], const int (&q)[R], unsigned nu,
                                              int nj, int nq, int nseg, int rn, int nseg_item, int qs_sheet, int segq,
                                              int nx, const Hist &hist, const Hist &diff, int *diff_used, unsigned *tab,
                                              unsigned &mlen)
{
    const int lane = threadIdx.x & 31;
    const unsigned nx4 = (unsigned)nx << SIC_POS_WIND_BITS;
    unsigned cross = 0;
    unsigned qsum = 0;  // per-tracer charges: of the segments before r
    __syncwarp();       // every lane has read its tracers: the table takes their place
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const bool end = FULL ? r + 1 == R : r + 1 >= rn;  // the next tracer is the one after the lane's
        const unsigned ub = end ? nu : u[r + 1 < R ? r + 1 : r];
        const int jb = end ? nj : jn[r + 1 < R ? r + 1 : r];
        // inside one cell: both ends in it and shorter than half a box (a
        // longer one could end in the same cell one box on)
        const bool in = jb == jn[r] && (ub - u[r] + (1u << 29)) < (1u << 30);
        const bool seg = (FULL && r + 1 < R) || r < nseg;
        if (seg && !in)
            cross |= 1u << r;
        if (PER_Q) {
            const int qb = end ? nq : q[r + 1 < R ? r + 1 : r];
            tab[kTabWords + 32 * r + lane] = qsum;
            qsum += seg ? (unsigned)(segq ? q[r] : q[r] + qb) : 0u;
        }
    }
    const unsigned who = __ballot_sync(0xffffffffu, cross != 0);
    unsigned pend = 0;  // charge waiting for cell c (below 2^32: at most 9 shares of 2^28)
    int c = jn[0];
    int done = 0;       // segments of the lane dealt with
    bool spread = false;  // the item's particles are dealt over the lanes
    if (who) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            tab[32 * r + lane] = u[r];
        if (FULL || rn == R) {
            tab[32 * R + lane] = nu;
        } else if (rn > 0) {
#pragma unroll
            for (int r = 1; r < R; ++r)
                if (r == rn)
                    tab[32 * r + lane] = nu;
        }
        if (PER_Q)
            tab[kTabWords + 32 * R + lane] = qsum;
        // A short item (a short sheet, or what is left of one) leaves most lanes
        // without a tracer and the others a long loop each: where half of its
        // particles or more cross, they are dealt over all lanes instead, those
        // inside a cell too, each adding its own shares.  Single steps of one
        // launch, us with the loops and this: 172 sheets of up to 60 tracers on
        // 114 cells 20.7 and 15.1, 2000 of up to 100 on 500 28.3 and 20.8 (one
        // launch for many 14.2 and 11.5), 2048 of 64 on 1024 25.5 and 19.8.  At 120
        // tracers on 64 cells, 40 % of them crossing, 15.8 with the loops: the
        // lanes inside a cell would all add into the same few words.  Up to 128
        // particles, four a lane: up to 64 only, 500 sheets of up to 100 on 2048
        // cells took 31.6 and not 25.5.
        if (!FULL) {
            spread = nseg_item <= 4 * 32 && 2 * (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(cross)) >= nseg_item;
            if (spread) {
                const int left = nseg_item - lane;
                cross = left > 0 ? (2u << ((left - 1) >> 5)) - 1u : 0u;
                __syncwarp();
            }
        }
        while (cross) {
            const int k = __ffs(cross) - 1;
            cross &= cross - 1u;
            int at = 32 * k + lane;
            if (!FULL && spread)
                at = 32 * (lane & (R - 1)) + (at >> 3);
            const unsigned pa = tab[at], pb = tab[at + 32];
            unsigned qs, before;
            if (PER_Q) {
                const unsigned q0 = tab[kTabWords + at], q1 = tab[kTabWords + at + 32];
                qs = q1 - q0;
                before = q0 - tab[kTabWords + 32 * done + lane];
            } else {
                qs = (unsigned)qs_sheet;
                before = (unsigned)(k - done) * qs;
            }
            done = k + 1;
            const int cb = cell_of(cell_coord(pb, nx));
            const int d = (int)(pb - pa);
            const bool back = d < 0;
            const unsigned len = (unsigned)abs(d);
            if (!FULL && spread) {
                before = 0u;
                c = cell_of(cell_coord(pa, nx));
                if (c == cb && (pb - pa + (1u << 29)) < (1u << 30)) {  // inside its cell
                    hist.add32(c, qs);
                    continue;
                }
            }
            mlen = max(mlen, len);
            const unsigned la = (back ? pb : pa) * nx4;  // the lower end's fraction of its cell
            const unsigned long long span = (unsigned long long)len * nx4;
            const float df = la ? __uint2float_rn(0u - la) : 4294967296.0f;  // to the first edge
            const float sf = __fmaf_rn(__int2float_rn((int)(span >> 32)), 4294967296.0f, __uint2float_rn((unsigned)span));
            // an approximate reciprocal is enough: F is clamped to [0, q] and
            // the other end takes the rest, so the charge stays exact
            float inv;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(sf));
            const float qf = __int2float_rn((int)qs);
            unsigned F = (unsigned)min(max(__float2int_rn(__fmul_rn(__fmul_rn(df, inv), qf)), 0), (int)qs);
            const int nint = (int)((span + la) >> 32) - 1;  // whole cells inside
            unsigned inner = 0;
            if (nint > 0) {
                const unsigned P = whole_cell_charge(qs, qf, span, inv);
                inner = (unsigned)nint * P;  // at most qs
                F = min(F, qs - inner);
                int js = (back ? cb : c) + 1;
                js = js == nx ? 0 : js;
                if (nint >= nx) {
                    range_add(js, nint, (long long)P, nx, diff, diff_used);
                } else if (P) {
                    // One or two cells: into the mesh; more: +P at the first and
                    // -P after the last in the difference array.  For two cells
                    // that would be as many adds, and then the array's sum over
                    // the mesh for a step that may need it for nothing else: 8
                    // sheets of 2.5 cells a particle, us a step with two cells
                    // through the array and this, 8192 cells 80 and 48, 4096 30
                    // and 22, 1024 12 and 11.  Both ways take the same atomics, so
                    // that the lanes do not part (with a branch for each, folded
                    // sheets took 5 % longer; so, 0.4 to 0.9 %).
                    const bool far = nint > 2;
                    const Hist to{far ? diff.lo : hist.lo, far ? diff.hi : hist.hi};
                    to.add32(js, P);
                    if (nint > 1) {
                        int je = js + (far ? nint : 1);
                        if (je > (far ? nx : nx - 1)) {
                            je -= nx;
                            if (far)
                                diff.add32(0, P);
                        }
                        const unsigned val = far ? 0u - P : P;
                        const unsigned before_it = atomicAdd(to.lo + je, val);
                        if ((before_it + val < before_it) != far)  // a carry, or a borrow
                            atomicAdd(to.hi + je, far ? 0xffffffffu : 1u);
                        if (far)
                            *diff_used = 1;
                    }
                }
            }
            const unsigned rest = qs - F - inner;
            hist.add32(c, pend + before + (back ? rest : F));
            pend = back ? F : rest;
            c = cb;
            if (!FULL && spread) {
                hist.add32(c, pend);
                pend = 0u;
            }
        }
    }
    if (!FULL && spread)
        return;
    // what is left of the lane, in the cell its sheet is in now
    if (PER_Q) {
        const unsigned left = pend + (qsum - (done ? tab[kTabWords + 32 * done + lane] : 0u));
        if (left)
            hist.add32(c, left);
    } else {
        const unsigned owners = who | 1u;
        if ((owners >> lane) & 1u) {
            const unsigned above = owners & (0xfffffffeu << lane);           // the lanes with a crossing after this one
            const int upto = above ? R * (__ffs(above) - 1) : nseg_item;     // (the first of them; the item's end)
            const int mine = min(upto, nseg_item) - (lane * R + done);
            const unsigned long long left = pend + (unsigned long long)(unsigned)max(mine, 0) * (unsigned)qs_sheet;
            if (left)
                hist.add(c, (long long)left);
        }
    }
}

// One work item (up to 32 R tracers, R per lane) of the current simulation.
// FULL: the item has all 32 R tracers, so no lane needs a bounds test.  KEPT:
// the item stays in its stage st from step to step (k_run): it is written back
// there, and the tracers beside it are kept in sh.beside; tab is then a table
// of its own.
template <bool PUSH, bool DEPOSIT, bool PER_Q, bool FULL, bool STAGED, bool GEN, bool KEPT, class MID>
__device__ __forceinline__ void do_item(const WorkItem &W, const unsigned *__restrict__ Uin,
                                        const float *__restrict__ Vin, unsigned *__restrict__ Uout,
                                        float *__restrict__ Vout, const int32_t *__restrict__ Qh,
                                        const float2 *ek, const Hist &hist, const Hist &diff,
                                        Shared &sh, int nx, float ks, int drift, unsigned &rerr,
                                        char *st, char *tab, unsigned short *tasks, long long &ake, long long &ap, unsigned &mseg, unsigned &mlen,
                                        const WorkItemPL *pw, int dep, int segq, bool track_all, const MID &mid)
{
    const unsigned *stU = reinterpret_cast<const unsigned *>(st);
    const float *stV = reinterpret_cast<const float *>(st + kStageBytesU);
    const int *stQ = reinterpret_cast<const int *>(st + kStageBytesU + kStageBytesV);
    const int lane = threadIdx.x & 31;
    const int nx4 = nx << SIC_POS_WIND_BITS;
    const int m = FULL ? WT : W.count;
    const long long base = W.t0;
    const int l0 = lane * R;
    const int rn = FULL ? R : max(0, min(R, m - l0));
    const int lane_last = FULL ? 31 : (m - 1) / R;

    unsigned u[R];
    float v[R];
    int q[R];
    int jn[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        u[r] = 0u;
        v[r] = 0.f;
        q[r] = W.qh;
        jn[r] = 0;
    }
    // the tracer after the item's last one (next item, or the sheet's first)
    unsigned hu = 0u;
    float hv = 0.f;
    int hq = W.qh, hj = 0;
    bool has_halo = false;
    Beside &beside = sh.beside[threadIdx.x >> 5];
    if (DEPOSIT && lane == lane_last && W.halo >= 0) {
        has_halo = true;
        if (KEPT) {
            hu = beside.hu;
            hv = beside.hv;
            if (PER_Q)
                hq = beside.hq;
        } else if (STAGED && W.halo == base + m) {
            hu = stU[m];
            if (PUSH)
                hv = stV[m];
            if (PER_Q)
                hq = stQ[m];
        } else {
            // (from L2: inside k_run another SM may have written it a step ago)
            hu = __ldcg(Uin + W.halo);
            if (PUSH)
                hv = __ldcg(Vin + W.halo);
            if (PER_Q)
                hq = Qh[W.halo];
        }
    }
    static_assert(R % 4 == 0, "a lane's tracers load as 16-byte vectors");
    if (STAGED || FULL || rn == R) {
        // the stage holds the whole item (and garbage past its end)
        const unsigned *pu = STAGED ? stU + l0 : Uin + base + l0;
        const float *pvv = STAGED ? stV + l0 : Vin + base + l0;
        const int *pqq = STAGED ? stQ + l0 : Qh + base + l0;
#pragma unroll
        for (int k = 0; k < R / 4; ++k) {
            // from global memory (unstaged): streaming loads, first out of L2
            const uint4 t = STAGED ? reinterpret_cast<const uint4 *>(pu)[k] : __ldcs(reinterpret_cast<const uint4 *>(pu) + k);
            u[4 * k] = t.x;
            u[4 * k + 1] = t.y;
            u[4 * k + 2] = t.z;
            u[4 * k + 3] = t.w;
            if (PUSH) {
                const float4 f =
                    STAGED ? reinterpret_cast<const float4 *>(pvv)[k] : __ldcs(reinterpret_cast<const float4 *>(pvv) + k);
                v[4 * k] = f.x;
                v[4 * k + 1] = f.y;
                v[4 * k + 2] = f.z;
                v[4 * k + 3] = f.w;
            }
            if (PER_Q) {
                const int4 c = STAGED ? reinterpret_cast<const int4 *>(pqq)[k] : __ldcs(reinterpret_cast<const int4 *>(pqq) + k);
                q[4 * k] = c.x;
                q[4 * k + 1] = c.y;
                q[4 * k + 2] = c.z;
                q[4 * k + 3] = c.w;
            }
        }
    } else {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r < rn) {
                u[r] = Uin[base + l0 + r];
                if (PUSH)
                    v[r] = Vin[base + l0 + r];
                if (PER_Q)
                    q[r] = Qh[base + l0 + r];
            }
        }
    }

    float acc_a = 0.f, acc_b = 0.f;
    if (PUSH) {
        float vmax = 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (FULL || r < rn) {
                const float vo = v[r];
                push_one(u[r], v[r], jn[r], ek, nx, ks, drift, vmax);
                const float vn = v[r];
                if (PER_Q) {
                    const float qq = __int2float_rn(q[r]);
                    acc_a = __fmaf_rn(qq, __fmaf_rn(vo, vo, __fmul_rn(vn, vn)), acc_a);
                    acc_b = __fmaf_rn(qq, __fadd_rn(vo, vn), acc_b);
                } else {
                    acc_a = __fmaf_rn(vo, vo, __fmaf_rn(vn, vn, acc_a));
                    acc_b = __fadd_rn(acc_b, __fadd_rn(vo, vn));
                }
            }
        }
        if (!(vmax < 536870912.0f))  // a step of half a box or more
            rerr |= 1u << 30;
        if (has_halo) {
            float ignore = 0.f;
            push_one(hu, hv, hj, ek, nx, ks, drift, ignore);
            if (KEPT) {
                beside.hu = hu;
                beside.hv = hv;
            }
        }
        if (KEPT) {
            // back to the stage (past the item's end: what was there)
            unsigned *bu = reinterpret_cast<unsigned *>(st) + l0;
            float *bv = reinterpret_cast<float *>(st + kStageBytesU) + l0;
#pragma unroll
            for (int k = 0; k < R / 4; ++k) {
                reinterpret_cast<uint4 *>(bu)[k] = make_uint4(u[4 * k], u[4 * k + 1], u[4 * k + 2], u[4 * k + 3]);
                reinterpret_cast<float4 *>(bv)[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
            }
        } else if (FULL || rn == R) {
#pragma unroll
            for (int k = 0; k < R / 4; ++k) {
                __stcs(reinterpret_cast<uint4 *>(Uout + base + l0) + k,
                       make_uint4(u[4 * k], u[4 * k + 1], u[4 * k + 2], u[4 * k + 3]));
                __stcs(reinterpret_cast<float4 *>(Vout + base + l0) + k,
                       make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]));
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (r < rn) {
                    Uout[base + l0 + r] = u[r];
                    Vout[base + l0 + r] = v[r];
                }
            }
        }
    } else {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (FULL || r < rn)
                jn[r] = cell_of(cell_coord(u[r], nx));
        if (has_halo)
            hj = cell_of(cell_coord(hu, nx));
    }
    mid();  // staging: the next item's copies start here

    // piecewise-linear particles (pw set): the tracer before the item and the
    // one after its halo too, for the gradients of the item's first and last
    // particles (Sec. 2.5)
    unsigned pu = 0u, nu2 = 0u;
    int pq = W.qh, nq2 = W.qh;
    bool has_prev = false, has_next2 = false;
    if (GEN && DEPOSIT && pw != nullptr) {
        const long long ip = pw->prev, in2 = pw->next2;
        has_prev = ip >= 0;
        has_next2 = in2 >= 0;
        if (lane == 0 && has_prev) {
            pu = KEPT ? beside.pu : __ldcg(Uin + ip);
            if (PER_Q)
                pq = KEPT ? beside.pq : Qh[ip];
            if (PUSH) {
                float pv = KEPT ? beside.pv : __ldcg(Vin + ip);
                int pj;
                float ignore = 0.f;
                push_one(pu, pv, pj, ek, nx, ks, drift, ignore);
                if (KEPT) {
                    beside.pu = pu;
                    beside.pv = pv;
                }
            }
            pu -= pw->prev_shift;
        }
        if (lane == lane_last && has_next2) {
            nu2 = KEPT ? beside.nu : __ldcg(Uin + in2);
            if (PER_Q)
                nq2 = KEPT ? beside.nq : Qh[in2];
            if (PUSH) {
                float nv = KEPT ? beside.nv : __ldcg(Vin + in2);
                int nj;
                float ignore = 0.f;
                push_one(nu2, nv, nj, ek, nx, ks, drift, ignore);
                if (KEPT) {
                    beside.nu = nu2;
                    beside.nv = nv;
                }
            }
            nu2 += pw->next2_shift;
        }
    }

    if (GEN && DEPOSIT && (dep == SIC_DEPOSIT_PIC_NGP || dep == SIC_DEPOSIT_PIC_CIC)) {
        // PIC comparison deposits (Sec. 2.4): every tracer a point charge of
        // 2 Qh units, in its cell (nearest grid point) or shared between the
        // two cells whose centres bracket it (cloud in cell: the second gets
        // round(Q f), f the distance past the first centre in cells)
        DirectAdd acc{hist};
        RunAcc run(hist);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (FULL || r < rn) {
                const long long Qt = 2ll * (long long)q[r];
                if (dep == SIC_DEPOSIT_PIC_NGP) {
                    run.add(jn[r], Qt);
                } else {
                    const long long pc = cell_coord(u[r], nx) - (1ll << 31);  // centres on integers
                    int j0 = cell_of(pc);                                      // -1 before the first centre
                    j0 += (j0 < 0) ? nx : 0;
                    const int j1 = (j0 + 1 == nx) ? 0 : j0 + 1;
                    const long long p1 =
                        (long long)(((unsigned long long)Qt * (unsigned long long)frac_of(pc) + (1ull << 31)) >> 32);
                    acc.add(j0, Qt - p1);
                    acc.add(j1, p1);
                }
            }
        }
        run.flush();
    } else if (DEPOSIT && !(GEN && (pw != nullptr || dep == SIC_DEPOSIT_FIRST))) {
        hu += W.halo_shift;  // closing segment: the sheet's first tracer one winding on
        // the tracer after each lane's last one: the next lane's first, or the halo
        unsigned nu = __shfl_down_sync(0xffffffffu, u[0], 1);
        int nj = __shfl_down_sync(0xffffffffu, jn[0], 1);
        int nq = __shfl_down_sync(0xffffffffu, q[0], 1);
        int nseg = rn;  // segments that start at this lane's tracers
        if (lane >= lane_last) {
            nu = hu;
            nj = hj;
            nq = hq;
            if (lane == lane_last && !has_halo)
                --nseg;
        }
        deposit_boxes<PER_Q, FULL>(u, jn, q, nu, nj, nq, nseg, rn, m - (W.halo >= 0 ? 0 : 1), 2 * W.qh, segq, nx,
                                   hist, diff, &sh.diff_used, reinterpret_cast<unsigned *>(tab), mlen);
        if (track_all) {
            // a refinement length shorter than a cell: particles inside one
            // cell count towards the longest one too
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (r < nseg) {
                    const unsigned ub = (r + 1 < R && r + 1 < rn) ? u[r + 1 < R ? r + 1 : r] : nu;
                    mlen = max(mlen, (unsigned)abs((int)(ub - u[r])));
                }
        }
    } else if (DEPOSIT) {
        hu += W.halo_shift;  // closing segment: the sheet's first tracer one winding on
        // publish the new positions (and charges) of the item in shared
        // memory, so the cross-cell segments can be shared out over the warp
        unsigned *pts = reinterpret_cast<unsigned *>(st);
        int *qpts = reinterpret_cast<int *>(st + WarpBuf<PER_Q, STAGED>::q_offset);
        // (every lane has written its tracers back there, the lane after the
        // last one too, whose first words may be the halo's)
        if (KEPT)
            __syncwarp();
        if (FULL || rn == R) {
#pragma unroll
            for (int k = 0; k < R / 4; ++k) {
                reinterpret_cast<uint4 *>(pts + l0)[k] = make_uint4(u[4 * k], u[4 * k + 1], u[4 * k + 2], u[4 * k + 3]);
                if (PER_Q)
                    reinterpret_cast<int4 *>(qpts + l0)[k] = make_int4(q[4 * k], q[4 * k + 1], q[4 * k + 2], q[4 * k + 3]);
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (r < rn) {
                    pts[l0 + r] = u[r];
                    if (PER_Q)
                        qpts[l0 + r] = q[r];
                }
        }
        if (lane == lane_last && has_halo) {
            pts[m] = hu;
            if (PER_Q)
                qpts[m] = hq;
        }
        if (GEN && lane == lane_last && has_next2) {
            pts[m + 1] = nu2;
            if (PER_Q)
                qpts[m + 1] = nq2;
        }
        if (GEN && lane == 0 && has_prev) {
            sh.pl_prev[threadIdx.x >> 5] = pu;
            sh.pl_prevq[threadIdx.x >> 5] = pq;
        }
        // the next tracer of each lane's last one comes from the lane above
        const unsigned nu = __shfl_down_sync(0xffffffffu, u[0], 1);
        const int nj = __shfl_down_sync(0xffffffffu, jn[0], 1);
        const int nq = __shfl_down_sync(0xffffffffu, q[0], 1);
        const int qs_sheet = 2 * W.qh;
        __syncwarp();

        if (GEN && dep == SIC_DEPOSIT_FIRST) {
            // first-order weighting (Sec. 2.4): every particle shared out to
            // nodes by emit_first, straight into the block's mesh
            DirectAdd acc{hist};
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (FULL || r < rn) {
                    unsigned ub;
                    int qb;
                    bool seg = true;
                    if (r + 1 < R && (FULL || r + 1 < rn)) {
                        ub = u[r + 1 < R ? r + 1 : r];
                        qb = q[r + 1 < R ? r + 1 : r];
                    } else if (lane < lane_last) {
                        ub = nu;
                        qb = nq;
                    } else {
                        ub = hu;
                        qb = hq;
                        seg = has_halo;
                    }
                    if (seg) {
                        const long long ua64 = cell_coord(u[r], nx);
                        emit_first(ua64, ua64 + seg_span(u[r], ub, nx4),
                                   PER_Q ? (segq ? q[r] : q[r] + qb) : qs_sheet, nx, acc, diff, &sh.diff_used,
                                   mseg);
                    }
                }
            }
        } else {
        // segments inside one cell: whole charges summed per lane into three
        // buckets for the cells c0, c0 + 1, c0 + 2 of its first tracer (a lane
        // that reaches other cells falls back to run merging); the segments
        // that cross a cell edge are marked for the second pass.  A segment
        // lies inside one cell when its two ends share a cell and it is
        // shorter than half a box (a longer one could end in the same cell
        // one box on).
        unsigned cross = 0;
        {
            const int c0 = jn[0];
            unsigned b0 = 0, b1 = 0, b2 = 0;  // charges per tracer: charge per bucket
            unsigned cnt = 0;                 // one charge per sheet: byte k counts the segments in cell c0 + k
            int nsame = 0;
            bool wide = false;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (FULL || r < rn) {
                    unsigned ub;
                    int jb, qb;
                    bool seg = true;
                    if (r + 1 < R && (FULL || r + 1 < rn)) {
                        ub = u[r + 1 < R ? r + 1 : r];
                        jb = jn[r + 1 < R ? r + 1 : r];
                        qb = q[r + 1 < R ? r + 1 : r];
                    } else if (lane < lane_last) {
                        ub = nu;
                        jb = nj;
                        qb = nq;
                    } else {
                        ub = hu;
                        jb = hj;
                        qb = hq;
                        seg = has_halo;
                    }
                    const bool shrt = (ub - u[r] + (1u << 29)) < (1u << 30);
                    const bool same = seg && shrt && jn[r] == jb;
                    const int d = jn[r] - c0;
                    if (PER_Q) {
                        const unsigned qv = (unsigned)(segq ? q[r] : q[r] + qb);
                        b0 += (same && d == 0) ? qv : 0u;
                        b1 += (same && d == 1) ? qv : 0u;
                        b2 += (same && d == 2) ? qv : 0u;
                        wide = wide || (same && (unsigned)d > 2u);
                    } else {
                        // 2^(8 d), or 0 for d outside [0, 3] (the funnel shift
                        // clamps its count at 32; a negative d is a huge count)
                        cnt += same ? __funnelshift_lc(0u, 1u, (unsigned)d << 3) : 0u;
                        nsame += same ? 1 : 0;
                    }
                    cross |= (seg && !same) ? (1u << r) : 0u;
                }
            }
            // every inside segment of the lane in one of the four bytes (the
            // bytes cannot carry: each counts at most R)
            if (!PER_Q)
                wide = ((cnt * 0x01010101u) >> 24) != (unsigned)nsame;
            if (__builtin_expect(!wide, 1)) {
                // the cells c0 + k (k <= 3) of non-empty buckets are below nx
                if (PER_Q) {
                    if (b0)
                        hist.add(c0, b0);
                    if (b1)
                        hist.add(c0 + 1, b1);
                    if (b2)
                        hist.add(c0 + 2, b2);
                } else {
                    const long long qs = qs_sheet;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const unsigned c = (cnt >> (8 * k)) & 0xffu;
                        if (c)
                            hist.add(c0 + k, (long long)c * qs);
                    }
                }
            } else {
                RunAcc acc(hist);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if ((FULL || r < rn) && !((cross >> r) & 1u)) {
                        int qb;
                        bool seg = true;
                        if (r + 1 < R && (FULL || r + 1 < rn)) {
                            qb = q[r + 1 < R ? r + 1 : r];
                        } else if (lane < lane_last) {
                            qb = nq;
                        } else {
                            qb = hq;
                            seg = has_halo;
                        }
                        if (seg)
                            acc.add(jn[r], PER_Q ? (segq ? q[r] : q[r] + qb) : qs_sheet);
                    }
                }
                acc.flush();
            }
        }

        // a refinement length shorter than a cell: particles inside one cell
        // count towards the longest one too (the cross-cell ones are measured
        // where they are deposited)
        if (track_all) {
            unsigned longest = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (FULL || r < rn) {
                    unsigned ub;
                    bool seg = true;
                    if (r + 1 < R && (FULL || r + 1 < rn))
                        ub = u[r + 1 < R ? r + 1 : r];
                    else if (lane < lane_last)
                        ub = nu;
                    else {
                        ub = hu;
                        seg = has_halo;
                    }
                    if (seg)
                        longest = max(longest, (unsigned)abs((int)(ub - u[r])));
                }
            }
            mseg = max(mseg, (unsigned)min(((unsigned long long)longest * (unsigned)nx4) >> 16, 0xffffffffull));
        }

        // cross-cell segments: compact them into a task list and let every lane take
        // one in turn; a lane's slot is the count before it, summed from one
        // ballot per bit of the per-lane counts (0..R) when there are any
        unsigned lt;
        asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
        const int total = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(cross));  // tasks of the warp
        int excl = 0;
        if (total) {
#pragma unroll
            for (int bit = 0; (1 << bit) <= R; ++bit) {
                const unsigned bb = __ballot_sync(0xffffffffu, (__popc(cross) >> bit) & 1);
                excl += __popc(bb & lt) << bit;
            }
        }
        if (total) {
            int pos = excl;
#pragma unroll
            for (int r = 0; r < R; ++r) {  // predicated stores, no loop to diverge on
                if ((cross >> r) & 1u)
                    tasks[pos++] = (unsigned short)(l0 + r);
            }
            cross = 0;
            __syncwarp();
            DirectAdd acc{hist};
            // piecewise-linear particles: kappa of the particle at idx, from
            // its neighbours' positions in the frame of its own lower end ua;
            // 0 keeps it a box (no neighbour on one side, or a box length or
            // longer)
            auto kappa_of = [&](int idx, long long ua, long long ub, int qs) -> float {
                const bool hp = idx > 0 || has_prev;
                const bool hn = idx + 2 < m || (idx + 2 == m && W.halo >= 0) || (idx + 2 == m + 1 && has_next2);
                const long long len = ub > ua ? ub - ua : ua - ub;
                if (!(hp && hn && len < ((long long)nx << 32)))
                    return 0.f;
                const int w8 = threadIdx.x >> 5;
                const unsigned pp = idx > 0 ? pts[idx - 1] : sh.pl_prev[w8];
                const long long up = ua - seg_span(pp, pts[idx], nx4);
                const long long un = ub + seg_span(pts[idx + 1], pts[idx + 2], nx4);
                const int qp = PER_Q ? (idx > 0 ? qpts[idx - 1] : sh.pl_prevq[w8]) + (segq ? 0 : qpts[idx]) : qs_sheet;
                const int qn = PER_Q ? qpts[idx + 1] + (segq ? 0 : qpts[idx + 2]) : qs_sheet;
                return pl_kappa(up, ua, ub, un, qp, qs, qn);
            };
            for (int k0 = 0; k0 < total; k0 += 32) {
                const int k = k0 + lane;
                int jl = 0, qs = 0, n = 0;
                unsigned la = 0u;
                float inv = 0.f, kappa = 0.f;
                if (k < total) {
                    const int idx = tasks[k];
                    const unsigned pa = pts[idx], pb = pts[idx + 1];
                    const long long ua = cell_coord(pa, nx);
                    const long long ub = ua + seg_span(pa, pb, nx4);
                    qs = PER_Q ? qpts[idx] + (segq ? 0 : qpts[idx + 1]) : qs_sheet;
                    kappa = kappa_of(idx, ua, ub, qs);
                    const int ja = cell_of(ua), jb = cell_of(cell_coord(pb, nx));
                    if (kappa == 0.f) {
                        emit_cross(ua, ja, ub, jb, qs, nx, acc, diff, &sh.diff_used, mseg);
                    } else {
                        const long long lo = min(ua, ub), span = max(ua, ub) - lo;
                        mseg = max(mseg, (unsigned)min((unsigned long long)span >> 16, 0xffffffffull));
                        jl = ub < ua ? jb : ja;
                        la = frac_of(lo);
                        inv = __frcp_rn(u64_to_float((unsigned long long)span));
                        n = cell_of(max(ua, ub)) - cell_of(lo) + 1;
                    }
                }
                __syncwarp();
                emit_linear(jl, la, inv, qs, kappa, n, nx, hist);
            }
        }
        }  // not first-order
        __syncwarp();  // pts and tasks are rewritten by the next item
    }

    // this lane's kinetic-energy and momentum terms (times the sheet's half
    // charge, unless the tracers carry their own, and in the sums' fixed-point
    // units), added exactly to its running sums (summed over the warp when it
    // leaves the simulation)
    if (PUSH) {
        sum_add(ake, __fmul_rn(acc_a, W.ke_mult), sh.ke, rerr);
        sum_add(ap, __fmul_rn(acc_b, W.p_mult), sh.p, rerr);
    }
}

}  // namespace
}  // namespace sic
