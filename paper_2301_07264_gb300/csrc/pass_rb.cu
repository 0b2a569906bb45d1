// Register-blocked fused tile pass (complex64, tiles of 2^t >= 2^10 amplitudes).
//
// A CTA of 2^(t-5) threads owns one tile of one trajectory; every thread
// keeps 32 amplitudes in registers. The tile-local index of register ri of
// thread tid is deposit(ri, R) | deposit(tid, complement of R), where R, the 5
// "register bits", changes only between phases (a swizzled shared-memory
// transpose). Register bit 0 is always tile bit 0, so registers 2k and 2k+1
// hold the neighbours j and j|1; they are kept split as two FP32x2 pairs,
// re[k] = (Re a_j, Re a_j|1) and im[k] = (Im a_j, Im a_j|1), and one packed
// instruction (FFMA2 / FMUL2 / FADD2) updates both. Within a phase:
//  * dense one-qubit gates, H and CX targets act on register bits, entirely
//    in registers;
//  * diagonal gates (T, S, Z, RZ, P, CZ, CP) act on any bit in place;
//  * X gates and Pauli errors never touch the data: the tile keeps masks m and z with
//    state[j] = (-1)^(z . (j ^ m)) stored[j ^ m] (Eq. (2): X swaps the pair (a0, a1), i.e.
//    flips bit q of the index; Z is a sign on it), later gates act on the stored
//    data conjugated by the masks, and the final store writes the signed stored[k] to
//    index k ^ m; Y = i X Z adds a factor i tracked as a power gp and applied at the store.
// Global loads and stores are 16-byte vector accesses in the mapping
// R = {0, t-4, t-3, t-2, t-1}, whose thread bits 1..t-5 are contiguous.
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>

#include "prof.h"
#include "sim_common.cuh"
#include "umma.cuh"

namespace arso {

// slot of pair J: eight 16-byte slots make a bank row, so the higher bits fold into three
__device__ __forceinline__ uint32_t swz(uint32_t j) { return j ^ (((j >> 3) ^ (j >> 6) ^ (j >> 9) ^ (j >> 12)) & 7u); }

// register bit b of a packed register set (the five bits are stored in ascending order)
__device__ __forceinline__ uint32_t rbit(uint32_t packed, int b) { return (packed >> (5 * b)) & 31u; }

// tid's bits deposited into the tile bits that are not register bits, ascending:
// a zero bit inserted at each register bit position, lowest first
__device__ __forceinline__ uint32_t thread_part(uint32_t tid, uint32_t packed) {
    uint32_t x = tid;
#pragma unroll
    for (int b = 0; b < REG_BITS; ++b) {
        const uint32_t r = rbit(packed, b);
        x = ((x >> r) << (r + 1)) | (x & ((1u << r) - 1u));
    }
    return x;
}


// register part of the local index of register ri (ri is a constant after unrolling)
__device__ __forceinline__ uint32_t reg_part(int ri, uint32_t packed) {
    uint32_t o = 0;
#pragma unroll
    for (int b = 0; b < REG_BITS; ++b)
        if ((ri >> b) & 1) o |= 1u << rbit(packed, b);
    return o;
}

// ----------------------------------------------------------- amplitudes ---
struct Amps {
    float2 re[16], im[16];  // re[k] = (Re of register 2k, Re of register 2k+1)
};

__device__ __forceinline__ float2 amp_get(const Amps &a, int ri) {
    const float2 r = a.re[ri >> 1], i = a.im[ri >> 1];
    return (ri & 1) ? make_float2(r.y, i.y) : make_float2(r.x, i.x);
}
__device__ __forceinline__ void amp_set(Amps &a, int ri, float2 v) {
    if (ri & 1) {
        a.re[ri >> 1].y = v.x;
        a.im[ri >> 1].y = v.y;
    } else {
        a.re[ri >> 1].x = v.x;
        a.im[ri >> 1].x = v.y;
    }
}

__device__ __forceinline__ float2 bc2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 swp2(float2 a) { return make_float2(a.y, a.x); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// ------------------------------------------------------- register gates ---
// Code size matters: warps stall for instructions more than for anything else
// when the phase loop outgrows the instruction cache (with 46 CZ variants by
// positions and mask bits 2.9 of 9.2 warps per issue waited for them, with a
// position-free form 1.4 of 8.4), so only dense one-qubit gates, odd phases and CZ
// are specialised per register position; everything else is position-free. CZ has
// 16 variants of 8 negations since the z mask took the mask bits out of its signs:
// 24-qubit brickwork, 177 trajectories, passes 336 -> 305 ms against the position-free
// form (about 165 instructions per warp for a layer of them).

// U on register bit P >= 1: packed registers k and k | 2^(P-1) hold the pairs
template <int P>
__device__ __forceinline__ void rg_dense1(Amps &a, float2 u00, float2 u01, float2 u10, float2 u11) {
    const float2 u00r = bc2(u00.x), u00i = bc2(u00.y), n00i = bc2(-u00.y);
    const float2 u01r = bc2(u01.x), u01i = bc2(u01.y), n01i = bc2(-u01.y);
    const float2 u10r = bc2(u10.x), u10i = bc2(u10.y), n10i = bc2(-u10.y);
    const float2 u11r = bc2(u11.x), u11i = bc2(u11.y), n11i = bc2(-u11.y);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        if (k & (1 << (P - 1))) continue;
        const int k1 = k | (1 << (P - 1));
        const float2 r0 = a.re[k], i0 = a.im[k], r1 = a.re[k1], i1 = a.im[k1];
        a.re[k] = fma2(n01i, i1, fma2(u01r, r1, fma2(n00i, i0, mul2(u00r, r0))));
        a.im[k] = fma2(u01i, r1, fma2(u01r, i1, fma2(u00i, r0, mul2(u00r, i0))));
        a.re[k1] = fma2(n11i, i1, fma2(u11r, r1, fma2(n10i, i0, mul2(u10r, r0))));
        a.im[k1] = fma2(u11i, r1, fma2(u11r, i1, fma2(u10i, r0, mul2(u10r, i0))));
    }
}

// G(x) = [[1, x], [-conj x, 1]] on register bit P >= 1 (the frame form of a one-qubit
// unitary, RegOpCode in internal.h): half the instructions of the full matrix and four
// broadcast constants instead of seven.
template <int P> __device__ __forceinline__ void rg_giv(Amps &a, float2 xr, float2 xi) {
    const float2 nxr = make_float2(-xr.x, -xr.y), nxi = make_float2(-xi.x, -xi.y);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        if (k & (1 << (P - 1))) continue;
        const int k1 = k | (1 << (P - 1));
        const float2 r0 = a.re[k], i0 = a.im[k], r1 = a.re[k1], i1 = a.im[k1];
        a.re[k] = fma2(nxi, i1, fma2(xr, r1, r0));
        a.im[k] = fma2(xi, r1, fma2(xr, i1, i0));
        a.re[k1] = fma2(nxi, i0, fma2(nxr, r0, r1));
        a.im[k1] = fma2(xi, r0, fma2(nxr, i0, i1));
    }
}
// the same for a real x
template <int P> __device__ __forceinline__ void rg_givr(Amps &a, float2 xr) {
    const float2 nxr = make_float2(-xr.x, -xr.y);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        if (k & (1 << (P - 1))) continue;
        const int k1 = k | (1 << (P - 1));
        const float2 r0 = a.re[k], i0 = a.im[k], r1 = a.re[k1], i1 = a.im[k1];
        a.re[k] = fma2(xr, r1, r0);
        a.im[k] = fma2(xr, i1, i0);
        a.re[k1] = fma2(nxr, r0, r1);
        a.im[k1] = fma2(nxr, i0, i1);
    }
}
// on register bit 0 (the two lanes of each packed register): xr = (Re x, -Re x)
__device__ __forceinline__ void rg_giv_lanes(Amps &a, float2 xr, float2 xi) {
    const float2 nxi = make_float2(-xi.x, -xi.y);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float2 r = a.re[k], i = a.im[k], rs = swp2(r), is = swp2(i);
        a.re[k] = fma2(nxi, is, fma2(xr, rs, r));
        a.im[k] = fma2(xi, rs, fma2(xr, is, i));
    }
}
__device__ __forceinline__ void rg_givr_lanes(Amps &a, float2 xr) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float2 r = a.re[k], i = a.im[k];
        a.re[k] = fma2(xr, swp2(r), r);
        a.im[k] = fma2(xr, swp2(i), i);
    }
}

// Special unitary U = [[a, b], [-conj b, conj a]] on register bit P >= 1:
// seven broadcast constants instead of twelve keep the phase loop spill-free.
template <int P> __device__ __forceinline__ void rg_su2(Amps &a, float2 ua, float2 ub) {
    const float2 ar = bc2(ua.x), ai = bc2(ua.y), nai = bc2(-ua.y);
    const float2 br = bc2(ub.x), bi = bc2(ub.y), nbi = bc2(-ub.y), nbr = bc2(-ub.x);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        if (k & (1 << (P - 1))) continue;
        const int k1 = k | (1 << (P - 1));
        const float2 r0 = a.re[k], i0 = a.im[k], r1 = a.re[k1], i1 = a.im[k1];
        a.re[k] = fma2(nbi, i1, fma2(br, r1, fma2(nai, i0, mul2(ar, r0))));
        a.im[k] = fma2(bi, r1, fma2(br, i1, fma2(ai, r0, mul2(ar, i0))));
        a.re[k1] = fma2(ai, i1, fma2(ar, r1, fma2(nbi, i0, mul2(nbr, r0))));
        a.im[k1] = fma2(nai, r1, fma2(ar, i1, fma2(bi, r0, mul2(nbr, i0))));
    }
}

// U on register bit 0: the pair sits in the two lanes of one packed register;
// lane 0 takes (u00, u01) against (a0, a1), lane 1 takes (u11, u10) against (a1, a0).
__device__ __forceinline__ void rg_dense1_lanes(Amps &a, float2 u00, float2 u01, float2 u10, float2 u11) {
    const float2 dr = make_float2(u00.x, u11.x), di = make_float2(u00.y, u11.y), ndi = make_float2(-u00.y, -u11.y);
    const float2 xr = make_float2(u01.x, u10.x), xi = make_float2(u01.y, u10.y), nxi = make_float2(-u01.y, -u10.y);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float2 r = a.re[k], i = a.im[k], rs = swp2(r), is = swp2(i);
        a.re[k] = fma2(nxi, is, fma2(xr, rs, fma2(ndi, i, mul2(dr, r))));
        a.im[k] = fma2(xi, rs, fma2(xr, is, fma2(di, r, mul2(dr, i))));
    }
}

// H on register bit P: (a0, a1) -> (a0 + a1, a0 - a1) / sqrt2 with 1/sqrt2
// applied as the compensated pair hi + lo. FLIP gives (a0 + a1, a1 - a0) /
// sqrt2, i.e. Z H, which is H on a qubit whose mask bit is set (H X = Z H:
// the caller then clears the mask bit).
template <int P, bool FLIP> __device__ __forceinline__ void rg_h(Amps &a) {
    const float2 hi = bc2(RSQRT2_HI), lo = bc2(RSQRT2_LO), m1 = bc2(-1.f);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        if (k & (1 << (P - 1))) continue;
        const int k1 = k | (1 << (P - 1));
        const float2 r0 = a.re[k], i0 = a.im[k], r1 = a.re[k1], i1 = a.im[k1];
        const float2 sr = add2(r0, r1), si = add2(i0, i1);
        const float2 dr = FLIP ? fma2(m1, r0, r1) : fma2(m1, r1, r0);
        const float2 di = FLIP ? fma2(m1, i0, i1) : fma2(m1, i1, i0);
        a.re[k] = fma2(hi, sr, mul2(lo, sr));
        a.im[k] = fma2(hi, si, mul2(lo, si));
        a.re[k1] = fma2(hi, dr, mul2(lo, dr));
        a.im[k1] = fma2(hi, di, mul2(lo, di));
    }
}
template <int P> __device__ __forceinline__ void rg_h(Amps &a, uint32_t flip) {
    if (flip) rg_h<P, true>(a);
    else rg_h<P, false>(a);
}
__device__ __forceinline__ void rg_h_lanes(Amps &a, float sg) {
    const float2 pm = make_float2(1.f, -1.f);
    const float2 h = make_float2(RSQRT2_HI, sg * RSQRT2_HI), l = make_float2(RSQRT2_LO, sg * RSQRT2_LO);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float2 tr = fma2(pm, a.re[k], swp2(a.re[k]));  // (a0 + a1, a0 - a1)
        const float2 ti = fma2(pm, a.im[k], swp2(a.im[k]));
        a.re[k] = fma2(h, tr, mul2(l, tr));
        a.im[k] = fma2(h, ti, mul2(l, ti));
    }
}

// Exchange the members of the pairs along register bit P where the mask (over registers;
// both members of a pair have the same bit) is set.
template <int P> __device__ __forceinline__ void rg_flip_if(Amps &a, uint32_t mask) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        constexpr int bit = P > 0 ? 1 << (P > 0 ? P - 1 : 0) : 0;
        if (k & bit) continue;
        const bool x = (mask >> (2 * k)) & 1u, y = P > 0 ? ((mask >> (2 * k + 1)) & 1u) : x;
        if (P == 0) {
            const float2 r = a.re[k], i = a.im[k];
            a.re[k] = make_float2(x ? r.y : r.x, x ? r.x : r.y);
            a.im[k] = make_float2(x ? i.y : i.x, x ? i.x : i.y);
        } else {
            const int k1 = k | bit;
            const float2 r0 = a.re[k], i0 = a.im[k], r1 = a.re[k1], i1 = a.im[k1];
            a.re[k] = make_float2(x ? r1.x : r0.x, y ? r1.y : r0.y);
            a.re[k1] = make_float2(x ? r0.x : r1.x, y ? r0.y : r1.y);
            a.im[k] = make_float2(x ? i1.x : i0.x, y ? i1.y : i0.y);
            a.im[k1] = make_float2(x ? i0.x : i1.x, y ? i0.y : i1.y);
        }
    }
}

// CX on stored data, target register bit P; control is register bit cpos
// (0..4) or, when cpos == 15, the thread-level bit value cth.
template <int P> __device__ __forceinline__ void rg_cx(Amps &a, uint32_t cpos, uint32_t cth) {
#pragma unroll
    for (int ri = 0; ri < 32; ++ri) {
        if (ri & (1 << P)) continue;
        const uint32_t ctl = cpos < REG_BITS ? (((uint32_t)ri >> cpos) & 1u) : cth;
        const float2 a0 = amp_get(a, ri), a1 = amp_get(a, ri | (1 << P));
        amp_set(a, ri, ctl ? a1 : a0);
        amp_set(a, ri | (1 << P), ctl ? a0 : a1);
    }
}

// Value of tile bit q of the true index (stored index ^ m) for register ri:
// register bit pos < 5 -> (ri >> pos) ^ mq; else the thread-level value th.
__device__ __forceinline__ uint32_t bit_of(int ri, uint32_t pos, uint32_t mq, uint32_t th) {
    return pos < REG_BITS ? ((((uint32_t)ri >> pos) & 1u) ^ mq) : th;
}

struct TileCtx {
    uint32_t R;          // register bits of the current phase, 5 bits each (bit 0 of the tile first)
    uint32_t tpart;      // thread part of the local index
    uint32_t m;          // X mask (stored[j] = state[j ^ m])
    uint32_t z;          // Z mask on stored indices (register programs)
    uint32_t gp;         // global phase i^gp
    uint32_t tid, nthr;  // thread index within the tile's thread group, group size
};

__device__ __forceinline__ uint32_t reg_pos(const TileCtx &c, uint32_t q) {
    uint32_t p = 15;
#pragma unroll
    for (int b = 0; b < REG_BITS; ++b)
        if (rbit(c.R, b) == q) p = (uint32_t)b;
    return p;
}
// true value of tile bit q held at thread level
__device__ __forceinline__ uint32_t thread_bit(const TileCtx &c, uint32_t q) { return ((c.tpart ^ c.m) >> q) & 1u; }

// diag(d0, d1) on tile bit q (true index) at register position pos (15: thread bit)
__device__ __forceinline__ void rg_diag1(Amps &a, const TileCtx &c, uint32_t q, uint32_t pos, float2 d0, float2 d1) {
    const uint32_t mq = (c.m >> q) & 1u, th = thread_bit(c, q);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t bx = bit_of(2 * k, pos, mq, th), by = bit_of(2 * k + 1, pos, mq, th);
        const float2 fr = make_float2(bx ? d1.x : d0.x, by ? d1.x : d0.x);
        const float2 fi = make_float2(bx ? d1.y : d0.y, by ? d1.y : d0.y);
        const float2 nfi = make_float2(-fi.x, -fi.y);
        const float2 r = a.re[k], i = a.im[k];
        a.re[k] = fma2(nfi, i, mul2(fr, r));
        a.im[k] = fma2(fi, r, mul2(fr, i));
    }
}

// diag(1, e^{i k pi/4}) on tile bit q, written per lane as kappa (A + i B)
// with A, B in {0, +-1} and kappa = 1/sqrt2 (odd k, compensated hi + lo) or 1.
// (R, I) -> kappa (A R - B I, B R + A I): the products by 0 and +-1 are exact,
// so lanes with (A, B, hi, lo) = (1, 0, 1, 0) pass through unchanged.
struct PhaseOp {
    float2 A, B, nB, H, L;
};
__device__ __forceinline__ void phase_pk(float2 &r, float2 &i, const PhaseOp &o) {
    float2 t1 = fma2(o.nB, i, mul2(o.A, r));
    float2 t2 = fma2(o.B, r, mul2(o.A, i));
    r = fma2(o.H, t1, mul2(o.L, t1));
    i = fma2(o.H, t2, mul2(o.L, t2));
}
__device__ __forceinline__ void omega_ab(uint32_t k, float &A, float &B, float &H, float &L) {
    const uint32_t q = (k >> 1) & 3u;
    const float cq = q == 0 ? 1.f : (q == 2 ? -1.f : 0.f), sq = q == 1 ? 1.f : (q == 3 ? -1.f : 0.f);
    if (k & 1u) {  // i^q (1 + i) / sqrt2
        A = cq - sq;
        B = cq + sq;
        H = RSQRT2_HI;
        L = RSQRT2_LO;
    } else {
        A = cq;
        B = sq;
        H = 1.f;
        L = 0.f;
    }
}
template <int P> __device__ __forceinline__ void rg_omega_half(Amps &a, const PhaseOp &op, uint32_t want) {
    if (want) {
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (k & (1 << (P - 1))) phase_pk(a.re[k], a.im[k], op);
    } else {
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (!(k & (1 << (P - 1)))) phase_pk(a.re[k], a.im[k], op);
    }
}
__device__ __forceinline__ void rg_omega(Amps &a, const TileCtx &c, uint32_t q, uint32_t pos, uint32_t k) {
    float A, B, H, L;
    omega_ab(k, A, B, H, L);
    if (pos >= REG_BITS) {
        if (thread_bit(c, q)) {
            const PhaseOp op{bc2(A), bc2(B), bc2(-B), bc2(H), bc2(L)};
#pragma unroll
            for (int kk = 0; kk < 16; ++kk) phase_pk(a.re[kk], a.im[kk], op);
        }
        return;
    }
    const uint32_t want = ((c.m >> q) & 1u) ^ 1u;  // stored bit value whose true bit is 1
    if (pos == 0) {
        // lane `want` of every packed register
        const PhaseOp op = want ? PhaseOp{make_float2(1.f, A), make_float2(0.f, B), make_float2(0.f, -B),
                                          make_float2(1.f, H), make_float2(0.f, L)}
                                : PhaseOp{make_float2(A, 1.f), make_float2(B, 0.f), make_float2(-B, 0.f),
                                          make_float2(H, 1.f), make_float2(L, 0.f)};
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) phase_pk(a.re[kk], a.im[kk], op);
        return;
    }
    const PhaseOp op{bc2(A), bc2(B), bc2(-B), bc2(H), bc2(L)};
    switch (pos) {
        case 1: rg_omega_half<1>(a, op, want); break;
        case 2: rg_omega_half<2>(a, op, want); break;
        case 3: rg_omega_half<3>(a, op, want); break;
        default: rg_omega_half<4>(a, op, want); break;
    }
}

// Registers whose tile bit q (of the true index) is 1, as a 32-bit mask.
__device__ __forceinline__ uint32_t reg_pattern(uint32_t pos) {
    return pos == 0 ? 0xAAAAAAAAu : pos == 1 ? 0xCCCCCCCCu : pos == 2 ? 0xF0F0F0F0u : pos == 3 ? 0xFF00FF00u : 0xFFFF0000u;
}
__device__ __forceinline__ uint32_t bit_mask(const TileCtx &c, uint32_t q) {
    const uint32_t pos = reg_pos(c, q);
    if (pos < REG_BITS) return ((c.m >> q) & 1u) ? ~reg_pattern(pos) : reg_pattern(pos);
    return thread_bit(c, q) ? 0xFFFFFFFFu : 0u;
}
__device__ __forceinline__ uint32_t sign_bit(uint32_t mask, int ri) { return (mask << (31 - ri)) & 0x80000000u; }
// negate the registers selected by mask: flip the sign bits
__device__ __forceinline__ void negate_masked(Amps &a, uint32_t mask) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t sx = sign_bit(mask, 2 * k), sy = sign_bit(mask, 2 * k + 1);
        a.re[k].x = __uint_as_float(__float_as_uint(a.re[k].x) ^ sx);
        a.im[k].x = __uint_as_float(__float_as_uint(a.im[k].x) ^ sx);
        a.re[k].y = __uint_as_float(__float_as_uint(a.re[k].y) ^ sy);
        a.im[k].y = __uint_as_float(__float_as_uint(a.im[k].y) ^ sy);
    }
}

// CZ: negate the registers whose stored bits at positions PA and PB equal
// (WA, WB). Both bits in registers: 8 of the 32 amplitudes, fixed at compile
// time (40 variants); packed registers are negated with one FMUL2 by (-1, -1)
// or (-1, 1) per plane.
template <int PA, int PB, int WA, int WB> __device__ __forceinline__ void neg_quarter(Amps &a) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const bool nx = ((((2 * k) >> PA) & 1) == WA) && ((((2 * k) >> PB) & 1) == WB);
        const bool ny = ((((2 * k + 1) >> PA) & 1) == WA) && ((((2 * k + 1) >> PB) & 1) == WB);
        if (!nx && !ny) continue;
        const float2 s = make_float2(nx ? -1.f : 1.f, ny ? -1.f : 1.f);
        a.re[k] = mul2(s, a.re[k]);
        a.im[k] = mul2(s, a.im[k]);
    }
}
template <int P, int W> __device__ __forceinline__ void neg_half(Amps &a) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const bool nx = (((2 * k) >> P) & 1) == W, ny = (((2 * k + 1) >> P) & 1) == W;
        if (!nx && !ny) continue;
        const float2 s = make_float2(nx ? -1.f : 1.f, ny ? -1.f : 1.f);
        a.re[k] = mul2(s, a.re[k]);
        a.im[k] = mul2(s, a.im[k]);
    }
}
__device__ __forceinline__ void negate_all(Amps &a) {
    const float2 m1 = bc2(-1.f);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        a.re[k] = mul2(m1, a.re[k]);
        a.im[k] = mul2(m1, a.im[k]);
    }
}
__host__ __device__ constexpr int cz_pa(int pp) { return pp < 4 ? 0 : pp < 7 ? 1 : pp < 9 ? 2 : 3; }
__host__ __device__ constexpr int cz_pb(int pp) {
    return pp < 4 ? pp + 1 : pp < 7 ? pp - 2 : pp < 9 ? pp - 4 : 4;
}
template <int IDX> __device__ __forceinline__ void cz_case(Amps &a) {
    neg_quarter<cz_pa(IDX >> 2), cz_pb(IDX >> 2), (IDX >> 1) & 1, IDX & 1>(a);
}

// multiply the registers selected by mask by f
__device__ __forceinline__ void phase_masked(Amps &a, uint32_t mask, float2 f) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const bool x = (mask >> (2 * k)) & 1u, y = (mask >> (2 * k + 1)) & 1u;
        const float2 fr = make_float2(x ? f.x : 1.f, y ? f.x : 1.f), fi = make_float2(x ? f.y : 0.f, y ? f.y : 0.f);
        const float2 nfi = make_float2(-fi.x, -fi.y);
        const float2 r = a.re[k], i = a.im[k];
        a.re[k] = fma2(nfi, i, mul2(fr, r));
        a.im[k] = fma2(fi, r, mul2(fr, i));
    }
}
// multiply the registers selected by mask by f, the others by its conjugate
__device__ __forceinline__ void phase_pair(Amps &a, uint32_t mask, float2 f) {
    const float2 fr = bc2(f.x);
    const uint32_t b = __float_as_uint(f.y) ^ 0x80000000u;  // -f.y, the sign flipped by the mask
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float2 fi = make_float2(__uint_as_float(b ^ sign_bit(mask, 2 * k)), __uint_as_float(b ^ sign_bit(mask, 2 * k + 1)));
        const float2 nfi = make_float2(-fi.x, -fi.y);
        const float2 r = a.re[k], i = a.im[k];
        a.re[k] = fma2(nfi, i, mul2(fr, r));
        a.im[k] = fma2(fi, r, mul2(fr, i));
    }
}
// the same with d added to the real part of f (EvSlot), for constants that a trajectory's errors
// bring in. d is less than a rounding of the product, so it goes in before the last two: a
// factor 1 + d on the result would round back. Norm of 64 trajectories, largest error: 16-qubit
// Clifford+T circuit of 3,000 gates, some 70 errors each, 9.9e-7 without d, 2.8e-7 with such a
// factor, 8.4e-8 so.
__device__ __forceinline__ void phase_pair_exact(Amps &a, uint32_t mask, float2 f, float d) {
    const float2 fr = bc2(f.x), dd = bc2(d);
    const uint32_t b = __float_as_uint(f.y) ^ 0x80000000u;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float2 fi = make_float2(__uint_as_float(b ^ sign_bit(mask, 2 * k)), __uint_as_float(b ^ sign_bit(mask, 2 * k + 1)));
        const float2 nfi = make_float2(-fi.x, -fi.y);
        const float2 r = a.re[k], i = a.im[k];
        a.re[k] = fma2(fr, r, fma2(nfi, i, mul2(dd, r)));
        a.im[k] = fma2(fr, i, fma2(fi, r, mul2(dd, i)));
    }
}
// diag(1, 1, 1, f) on tile bits qa, qb
__device__ __forceinline__ void rg_cp(Amps &a, const TileCtx &c, uint32_t qa, uint32_t qb, float2 f) {
    const uint32_t mask = bit_mask(c, qa) & bit_mask(c, qb);
    if (mask) phase_masked(a, mask, f);
}

// Pauli error on tile bit q of the true state (Eq. (2)): Z -> phase -1 on
// bit q; X -> index mask; Y = i X Z.
__device__ __forceinline__ void rg_pauli(Amps &a, TileCtx &c, uint32_t q, uint32_t code) {
    if (code & 2u) {  // Z part (Z or Y): negate where bit q of the true index is 1
        const uint32_t mask = bit_mask(c, q);
        if (mask) negate_masked(a, mask);
    }
    if (code & 1u) c.m ^= 1u << q;          // X part (X or Y)
    if (code == 3u) c.gp = (c.gp + 1u) & 3u;  // Y = i X Z
}

// multiply every amplitude by i^gp (exact) and reset gp
__device__ __forceinline__ void apply_global_phase(Amps &a, TileCtx &c) {
    if (!c.gp) return;
    const float2 A = bc2(c.gp == 2 ? -1.f : (c.gp == 0 ? 1.f : 0.f)), B = bc2(c.gp == 1 ? 1.f : (c.gp == 3 ? -1.f : 0.f));
    const float2 nB = make_float2(-B.x, -B.y);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float2 r = a.re[k], i = a.im[k];
        a.re[k] = fma2(nB, i, mul2(A, r));
        a.im[k] = fma2(B, r, mul2(A, i));
    }
    c.gp = 0;
}

// stored index -> tile-local index bits for the load/store mapping
__device__ __forceinline__ void set_phase(TileCtx &c, uint32_t packed, int t) {
    c.R = packed;
    c.tpart = thread_part(c.tid, packed);
}

// Shared memory holds a tile as packed neighbour pairs, 16 bytes each: slot swz(J) = (Re a_2J,
// Re a_2J+1, Im a_2J, Im a_2J+1), so a register set changes with 16 writes and 16 reads a
// thread instead of 32 and 32 of 8 bytes (the same bytes: half the issue slots). Eight slots
// are one turn of the banks: the swizzle folds the higher bits into three. It is linear over XOR, so the slot of packed
// register k is swz(tpart >> 1) ^ (XOR of swz(2^(r[b]-1)) over the set bits
// b-1 of k); walking the registers in Gray-code order costs one XOR each.
__host__ __device__ constexpr int ctz4(int x) { return x & 1 ? 0 : x & 2 ? 1 : x & 4 ? 2 : 3; }

__device__ __forceinline__ void smem_basis(const TileCtx &c, uint32_t &base, uint32_t (&sw)[REG_BITS - 1]) {
    base = swz(c.tpart >> 1);
#pragma unroll
    for (int b = 1; b < REG_BITS; ++b) sw[b - 1] = swz(1u << (rbit(c.R, b) - 1));
}
__device__ __forceinline__ void to_smem(const Amps &a, float2 *sm, const TileCtx &c, int t) {
    uint32_t idx, sw[REG_BITS - 1];
    smem_basis(c, idx, sw);
    float4 *p = reinterpret_cast<float4 *>(sm);
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
        const int k = kk ^ (kk >> 1);
        p[idx] = make_float4(a.re[k].x, a.re[k].y, a.im[k].x, a.im[k].y);
        if (kk < 15) idx ^= sw[ctz4(kk + 1)];
    }
}
__device__ __forceinline__ void from_smem(Amps &a, const float2 *sm, const TileCtx &c, int t) {
    uint32_t idx, sw[REG_BITS - 1];
    smem_basis(c, idx, sw);
    const float4 *p = reinterpret_cast<const float4 *>(sm);
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
        const int k = kk ^ (kk >> 1);
        const float4 w = p[idx];
        a.re[k] = make_float2(w.x, w.y);
        a.im[k] = make_float2(w.z, w.w);
        if (kk < 15) idx ^= sw[ctz4(kk + 1)];
    }
}

// SYNCED: the caller has just synced the CTA after the last shared-memory
// read (a phase start), so the first barrier is not needed.
template <bool SYNCED = false>
__device__ __forceinline__ void remap(Amps &a, float2 *sm, TileCtx &c, uint32_t packed, int t) {
    if (!SYNCED) __syncthreads();
    to_smem(a, sm, c, t);
    set_phase(c, packed, t);
    __syncthreads();
    from_smem(a, sm, c, t);
}

// Dense two-qubit gates and SWAP are rare: they run through shared memory on
// the stored data (U already conjugated by the mask) with runtime indices.
__device__ __forceinline__ void smem_dense2(float2 *sm, int t, uint32_t q0, uint32_t q1, const float2 *__restrict__ U,
                                            uint32_t tid, uint32_t nthr) {
    float *pre = reinterpret_cast<float *>(sm), *pim = pre + 2;
    const uint32_t lo = q0 < q1 ? q0 : q1, hi = q0 < q1 ? q1 : q0;
    const uint32_t m0 = 1u << q0, m1 = 1u << q1;
    if (lo > 0) {
        // neither qubit is tile bit 0: both amplitudes of a slot at once, one 16-byte read and write
        // per slot and packed arithmetic. Bound by shared-memory reads and the 64 FMA of a group (12-qubit
        // quantum volume, 4,000 trajectories: 1.08 ms with the scalar loop below for all pairs, 0.86 so)
        float4 *s4 = reinterpret_cast<float4 *>(sm);
        for (uint32_t p = tid; p < (1u << (t - 3)); p += nthr) {
            const uint32_t i = insert_zero2(p, lo - 1, hi - 1);
            const uint32_t ix[4] = {swz(i), swz(i | m0 >> 1), swz(i | m1 >> 1), swz(i | m0 >> 1 | m1 >> 1)};
            float2 xr[4], xi[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 w = s4[ix[k]];
                xr[k] = make_float2(w.x, w.y);
                xi[k] = make_float2(w.z, w.w);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float2 r, c;
#pragma unroll
                for (int l = 0; l < 4; ++l) {
                    const float2 u = U[4 * k + l];
                    const float2 ur = bc2(u.x), ui = bc2(u.y), nui = bc2(-u.y);
                    r = l ? fma2(nui, xi[l], fma2(ur, xr[l], r)) : fma2(nui, xi[l], mul2(ur, xr[l]));
                    c = l ? fma2(ui, xr[l], fma2(ur, xi[l], c)) : fma2(ui, xr[l], mul2(ur, xi[l]));
                }
                s4[ix[k]] = make_float4(r.x, r.y, c.x, c.y);
            }
        }
        return;
    }
    float2 M[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) M[k] = U[k];
    for (uint32_t p = tid; p < (1u << (t - 2)); p += nthr) {
        const uint32_t i = insert_zero2(p, lo, hi);
        const uint32_t jx[4] = {i, i | m0, i | m1, i | m0 | m1};
        uint32_t ix[4];
        float2 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            ix[k] = 4u * swz(jx[k] >> 1) + (jx[k] & 1u);
            v[k] = make_float2(pre[ix[k]], pim[ix[k]]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float2 acc = cmac2(M[4 * k], v[0], M[4 * k + 1], v[1]);
            const float2 acc2 = cmac2(M[4 * k + 2], v[2], M[4 * k + 3], v[3]);
            pre[ix[k]] = acc.x + acc2.x;
            pim[ix[k]] = acc.y + acc2.y;
        }
    }
}

// CZ from the host-resolved code: pair of register positions, or one
// register position and a thread bit; the mask bits of the qubits select the
// sign pattern (want = 1 ^ mask bit).
#define ARSO_CZ_CASE(i) case OP_CZ_RR + (i): cz_case<(i)>(a); break;
#define ARSO_CZ_CASE4(i) ARSO_CZ_CASE(4 * (i)) ARSO_CZ_CASE(4 * (i) + 1) ARSO_CZ_CASE(4 * (i) + 2) ARSO_CZ_CASE(4 * (i) + 3)
__device__ __forceinline__ void rg_cz_code(Amps &a, const TileCtx &c, uint32_t x, uint32_t q0, uint32_t q1,
                                           uint32_t p0) {
    const uint32_t ba = ((c.m >> q0) ^ (x >> 12)) & 1u, bb = ((c.m >> q1) ^ (x >> 13)) & 1u;
    const uint32_t code = (x & 255u) + ba * ((x >> 8) & 3u) + bb * ((x >> 10) & 3u);
    if (code >= (uint32_t)OP_CZ_RT) {
        if (code == (uint32_t)OP_CZ_TT) {
            if (thread_bit(c, q0) && thread_bit(c, q1)) negate_all(a);
            return;
        }
        if (!thread_bit(c, p0 < REG_BITS ? q1 : q0)) return;
        switch (code - OP_CZ_RT) {
            case 0: neg_half<0, 0>(a); break;
            case 1: neg_half<0, 1>(a); break;
            case 2: neg_half<1, 0>(a); break;
            case 3: neg_half<1, 1>(a); break;
            case 4: neg_half<2, 0>(a); break;
            case 5: neg_half<2, 1>(a); break;
            case 6: neg_half<3, 0>(a); break;
            case 7: neg_half<3, 1>(a); break;
            case 8: neg_half<4, 0>(a); break;
            default: neg_half<4, 1>(a); break;
        }
        return;
    }
    switch (code) {
        ARSO_CZ_CASE4(0) ARSO_CZ_CASE4(1) ARSO_CZ_CASE4(2) ARSO_CZ_CASE4(3) ARSO_CZ_CASE4(4)
        ARSO_CZ_CASE4(5) ARSO_CZ_CASE4(6) ARSO_CZ_CASE4(7) ARSO_CZ_CASE4(8) ARSO_CZ_CASE4(9)
        default: break;
    }
}
#undef ARSO_CZ_CASE
#undef ARSO_CZ_CASE4

// Dense two-qubit gate M (or SWAP) on tile bits q0, q1, through shared memory
__device__ __forceinline__ void tile_two(Amps &a, TileCtx &c, bool swap, uint32_t q0, uint32_t q1,
                                         const float2 *__restrict__ M, float2 *sm, float2 *ubuf, int t) {
    const uint32_t mab = ((c.m >> q0) & 1u) | (((c.m >> q1) & 1u) << 1);
    const uint32_t zab = ((c.z >> q0) & 1u) | (((c.z >> q1) & 1u) << 1);
    if (c.tid < 16) {
        const uint32_t k = c.tid >> 2, l = c.tid & 3u;
        float2 u;
        if (swap) {
            const uint32_t perm[4] = {0, 2, 1, 3};
            u = make_float2(perm[k] == l ? 1.f : 0.f, 0.f);
        } else {
            u = M[4 * (k ^ mab) + (l ^ mab)];
            if (__popc(zab & (k ^ l)) & 1) u = make_float2(-u.x, -u.y);
        }
        ubuf[c.tid] = u;
    }
    __syncthreads();
    to_smem(a, sm, c, t);
    __syncthreads();
    smem_dense2(sm, t, q0, q1, ubuf, c.tid, c.nthr);
    __syncthreads();
    from_smem(a, sm, c, t);
    __syncthreads();
    // SWAP X^m = X^{m with bits q0, q1 exchanged} SWAP
    if (swap && (((c.m >> q0) ^ (c.m >> q1)) & 1u)) c.m ^= (1u << q0) | (1u << q1);
    if (swap && (((c.z >> q0) ^ (c.z >> q1)) & 1u)) c.z ^= (1u << q0) | (1u << q1);
}

#define ARSO_CZ_ALL \
    case OP_CZ_RR + 0: case OP_CZ_RR + 4: case OP_CZ_RR + 8: case OP_CZ_RR + 12: case OP_CZ_RR + 16: \
    case OP_CZ_RR + 20: case OP_CZ_RR + 24: case OP_CZ_RR + 28: case OP_CZ_RR + 32: case OP_CZ_RR + 36: \
    case OP_CZ_RT + 0: case OP_CZ_RT + 2: case OP_CZ_RT + 4: case OP_CZ_RT + 6: case OP_CZ_RT + 8: \
    case OP_CZ_TT

// One dispatch per gate on the host-resolved base op code (class and
// register positions); mask-dependent details (H on a flipped qubit, the CZ
// sign pattern) are resolved inside the case, so cheap gates pay no extra
// decoding.
#define ARSO_P4(BASE, CALL) \
    case BASE + 1: CALL(1); break; \
    case BASE + 2: CALL(2); break; \
    case BASE + 3: CALL(3); break; \
    case BASE + 4: CALL(4); break;
__device__ __forceinline__ void apply_op(Amps &a, TileCtx &c, const RegOp &op, const float2 *__restrict__ mats,
                                         float2 *sm, float2 *ubuf, int t) {
    const uint32_t p0 = (op.w0 >> 8) & 15u;
    const uint32_t q0 = (op.w0 >> 16) & 255u, q1 = op.w0 >> 24;
    const float2 *M = mats + op.aux;
    // X U X for the qubit's mask bit: for SU(2) [[conj a, -conj b], [b, a]], the same form;
    // for a general U [[u11, u10], [u01, u00]]
#define ARSO_FLIP ((c.m >> q0) & 1u)
#define ARSO_UA (ARSO_FLIP ? make_float2(op.c0.x, -op.c0.y) : op.c0)
#define ARSO_UB (ARSO_FLIP ? make_float2(-op.c1.x, op.c1.y) : op.c1)
#define ARSO_SU2(P) rg_su2<P>(a, ARSO_UA, ARSO_UB)
#define ARSO_D1(P) \
    rg_dense1<P>(a, M[ARSO_FLIP ? 3 : 0], M[ARSO_FLIP ? 2 : 1], M[ARSO_FLIP ? 1 : 2], M[ARSO_FLIP ? 0 : 3])
    // H on a flipped qubit: H X = Z H, so apply Z H and clear the mask bit
#define ARSO_HADAMARD(P) rg_h<P>(a, ARSO_FLIP); c.m &= ~(1u << q0)
    // CX X^m = X^{m'} CX with m' = m ^ (target bit if the control bit is in m)
#define ARSO_CX(P) rg_cx<P>(a, p0, (c.tpart >> q0) & 1u); if (ARSO_FLIP) c.m ^= 1u << q1
    switch (op.pad[0] & 255u) {
        case OP_SU2: {
            const float2 ua = ARSO_UA, ub = ARSO_UB;
            rg_dense1_lanes(a, ua, ub, make_float2(-ub.x, ub.y), make_float2(ua.x, -ua.y));
            break;
        }
        ARSO_P4(OP_SU2, ARSO_SU2)
        case OP_DENSE1: {
            const uint32_t f = ARSO_FLIP;
            rg_dense1_lanes(a, M[f ? 3 : 0], M[f ? 2 : 1], M[f ? 1 : 2], M[f ? 0 : 3]);
            break;
        }
        ARSO_P4(OP_DENSE1, ARSO_D1)
        case OP_H: rg_h_lanes(a, ARSO_FLIP ? -1.f : 1.f); c.m &= ~(1u << q0); break;
        case OP_H + 2: ARSO_HADAMARD(1); break;
        case OP_H + 4: ARSO_HADAMARD(2); break;
        case OP_H + 6: ARSO_HADAMARD(3); break;
        case OP_H + 8: ARSO_HADAMARD(4); break;
        ARSO_CZ_ALL: rg_cz_code(a, c, op.pad[0], q0, q1, p0); break;
        case OP_X: c.m ^= 1u << q0; break;
        case OP_OMEGA: rg_omega(a, c, q0, p0, op.aux); break;
        case OP_DIAG1: rg_diag1(a, c, q0, p0, op.c0, op.c1); break;
        case OP_CP: rg_cp(a, c, q0, q1, op.c0); break;
        case OP_CX: ARSO_CX(0); break;
        ARSO_P4(OP_CX, ARSO_CX)
        case OP_DENSE2:
        case OP_SWAP: tile_two(a, c, (op.pad[0] & 255u) == OP_SWAP, q0, q1, M, sm, ubuf, t); break;
        default: break;
    }
#undef ARSO_UA
#undef ARSO_UB
#undef ARSO_SU2
#undef ARSO_HADAMARD
}

// Raw sums (kernels.h) of the pairs along register bit P of this thread's registers.
// flip: the qubit's bit of m (s0 and s1 change places); g: the sign of its bit of z.
template <int P> __device__ __forceinline__ void rg_probe(const Amps &a, uint32_t flip, float g, float *w) {
    float2 z = make_float2(0.f, 0.f), cr = z, ci = z;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        if (k & (1 << (P - 1))) continue;
        const int k1 = k | (1 << (P - 1));
        const float2 r0 = a.re[k], i0 = a.im[k], r1 = a.re[k1], i1 = a.im[k1];
        const float2 nr1 = make_float2(-r1.x, -r1.y), ni1 = make_float2(-i1.x, -i1.y), ni0 = make_float2(-i0.x, -i0.y);
        z = fma2(ni1, i1, fma2(nr1, r1, fma2(i0, i0, fma2(r0, r0, z))));
        cr = fma2(i0, i1, fma2(r0, r1, cr));
        ci = fma2(ni0, r1, fma2(r0, i1, ci));
    }
    const float zs = z.x + z.y, cs = ci.x + ci.y;
    w[0] = flip ? -zs : zs;
    w[1] = g * (cr.x + cr.y);
    w[2] = flip ? -g * cs : g * cs;
}
__device__ __forceinline__ void rg_probe_lanes(const Amps &a, uint32_t flip, float g, float *w) {
    float z = 0.f, cr = 0.f, ci = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float2 r = a.re[k], i = a.im[k];
        z = fmaf(-i.y, i.y, fmaf(-r.y, r.y, fmaf(i.x, i.x, fmaf(r.x, r.x, z))));
        cr = fmaf(i.x, i.y, fmaf(r.x, r.y, cr));
        ci = fmaf(-i.x, r.y, fmaf(r.x, i.y, ci));
    }
    w[0] = flip ? -z : z;
    w[1] = g * cr;
    w[2] = flip ? -g * ci : g * ci;
}
// psi in lane 0, phi in lane 1 of every packed register
template <int P> __device__ __forceinline__ void rg_probe_dual(const Amps &a, uint32_t flip, float g, float *w) {
    float x[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        if (k & (1 << (P - 1))) continue;
        const int k1 = k | (1 << (P - 1));
        const float ar0 = a.re[k].x, ai0 = a.im[k].x, ar1 = a.re[k1].x, ai1 = a.im[k1].x;
        const float br0 = a.re[k].y, bi0 = a.im[k].y, br1 = a.re[k1].y, bi1 = a.im[k1].y;
        x[0] = fmaf(bi0, ai1, fmaf(br0, ar1, x[0]));
        x[1] = fmaf(-bi0, ar1, fmaf(br0, ai1, x[1]));
        x[2] = fmaf(bi1, ai0, fmaf(br1, ar0, x[2]));
        x[3] = fmaf(-bi1, ar0, fmaf(br1, ai0, x[3]));
        x[4] = fmaf(-bi1, ai1, fmaf(-br1, ar1, fmaf(bi0, ai0, fmaf(br0, ar0, x[4]))));
        x[5] = fmaf(bi1, ar1, fmaf(-br1, ai1, fmaf(-bi0, ar0, fmaf(br0, ai0, x[5]))));
    }
    w[0] = g * (flip ? x[2] : x[0]);
    w[1] = g * (flip ? x[3] : x[1]);
    w[2] = g * (flip ? x[0] : x[2]);
    w[3] = g * (flip ? x[1] : x[3]);
    w[4] = flip ? -x[4] : x[4];
    w[5] = flip ? -x[5] : x[5];
}
// The measurements of one OP_PROBE: the values of all positions summed over the warp by
// halving exchanges (one shuffle per value instead of five), then added to the warp's row,
// one value per lane (pair of lanes).
template <bool DUAL> __device__ __forceinline__ void run_probe(const Amps &a, const TileCtx &c, const uint4 h, uint32_t slot0,
                                                            double *row) {
    constexpr int SUMS = DUAL ? 6 : 3, N = DUAL ? 32 : 16, P0 = DUAL ? 1 : 0;
    float w[N];
#pragma unroll
    for (int i = 0; i < N; ++i) w[i] = 0.f;
    const uint32_t act = (h.x >> (8 + P0)) & 31u;
#define ARSO_PROBE_P(P)                                                          \
    if (h.x & (0x100u << P)) {                                                   \
        const uint32_t f = (c.m >> rbit(c.R, P)) & 1u;                           \
        const float g = (c.z >> rbit(c.R, P)) & 1u ? -1.f : 1.f;                 \
        if constexpr (DUAL) rg_probe_dual<P>(a, f, g, w + SUMS * (P - P0));      \
        else rg_probe<P>(a, f, g, w + SUMS * (P - P0));                          \
    }
    if constexpr (!DUAL) {
        if (h.x & 0x100u) rg_probe_lanes(a, c.m & 1u, c.z & 1u ? -1.f : 1.f, w);
    }
    ARSO_PROBE_P(1) ARSO_PROBE_P(2) ARSO_PROBE_P(3) ARSO_PROBE_P(4)
#undef ARSO_PROBE_P
    const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
    for (int o = 16, n = N / 2; n >= 1; o >>= 1, n >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            if (i >= n) break;
            const float send = up ? w[i] : w[i + n], keep = up ? w[i + n] : w[i];
            w[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    if constexpr (!DUAL) w[0] += __shfl_xor_sync(0xffffffffu, w[0], 1);
    const uint32_t v = DUAL ? lane : lane >> 1, p = v / SUMS;
    if (((DUAL || !(lane & 1u))) && ((act >> p) & 1u)) {
        const uint32_t slot = h.z - slot0 + __popc(act & ((1u << p) - 1u));
        atomicAdd(row + slot * SUMS + v - p * SUMS, (double)w[0]);  // its own row: no result is waited for
    }
}

// One macro-op of a register program (internal.h): h its header, u its further units.
__device__ __forceinline__ void apply_macro(Amps &a, TileCtx &c, const uint4 h, const uint4 *u,
                                            const float2 *__restrict__ mats, float2 *sm, float2 *ubuf, int t) {
    const uint32_t code = h.x & 255u;
    if (code == OP_LAYER) {
        c.m ^= h.w;
        // X G(x) X = G(-conj x), Z G(x) Z = G(-x): the qubit's bit of z flips the sign of x,
        // that of m the sign of Re x
        const uint32_t mz = c.m ^ c.z;
#define ARSO_LAYER_X                                                           \
    const uint4 w = *u++;                                                      \
    const uint32_t f = (mz >> rbit(c.R, P)) << 31, g = (c.z >> rbit(c.R, P)) << 31; \
    const float2 xr = make_float2(__uint_as_float(w.x ^ f), __uint_as_float(w.y ^ f)); \
    const float2 xi = make_float2(__uint_as_float(w.z ^ g), __uint_as_float(w.w ^ g));
        if (h.x & 0x100u) {
            constexpr int P = 0;
            ARSO_LAYER_X
            if (h.x & 0x2000u) rg_givr_lanes(a, xr);
            else rg_giv_lanes(a, xr, xi);
        }
#define ARSO_LAYER_P(PP)                                        \
        if (h.x & (0x100u << PP)) {                             \
            constexpr int P = PP;                               \
            ARSO_LAYER_X                                        \
            if (h.x & (0x2000u << PP)) rg_givr<P>(a, xr);       \
            else rg_giv<P>(a, xr, xi);                          \
        }
        ARSO_LAYER_P(1)
        ARSO_LAYER_P(2)
        ARSO_LAYER_P(3)
        ARSO_LAYER_P(4)
#undef ARSO_LAYER_X
#undef ARSO_LAYER_P
        return;
    }
    const uint32_t q0 = h.z & 255u, q1 = (h.z >> 8) & 255u, p0 = (h.z >> 16) & 15u;
    // Z M Z: the off-diagonal entries change sign
    const float zs = (c.z >> q0) & 1u ? -1.f : 1.f;
#define ARSO_ZS(v) make_float2(zs * (v).x, zs * (v).y)
#define ARSO_D1Z(P)                                                                                     \
    {                                                                                                   \
        const float2 *M = mats + u->x;                                                                  \
        const uint32_t f = ARSO_FLIP;                                                                   \
        rg_dense1<P>(a, M[f ? 3 : 0], ARSO_ZS(M[f ? 2 : 1]), ARSO_ZS(M[f ? 1 : 2]), M[f ? 0 : 3]);        \
    }
    switch (code) {
        // CZ X^m = X^m CZ with Z on a qubit whose partner is flipped: the signs do not depend on m
#define ARSO_CZ_MASKS                                                          \
    {                                                                          \
        const uint32_t b0 = (c.m >> q0) & 1u, b1 = (c.m >> q1) & 1u;           \
        c.z ^= (b0 << q1) ^ (b1 << q0);                                        \
        c.gp ^= (b0 & b1) << 1;                                                \
    }
        case OP_CZ_RR + 0: neg_quarter<0, 1, 1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RR + 1: neg_quarter<0, 2, 1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RR + 2: neg_quarter<0, 3, 1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RR + 3: neg_quarter<0, 4, 1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RR + 4: neg_quarter<1, 2, 1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RR + 5: neg_quarter<1, 3, 1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RR + 6: neg_quarter<1, 4, 1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RR + 7: neg_quarter<2, 3, 1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RR + 8: neg_quarter<2, 4, 1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RR + 9: neg_quarter<3, 4, 1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RT + 0: if ((c.tpart >> q1) & 1u) neg_half<0, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RT + 1: if ((c.tpart >> q1) & 1u) neg_half<1, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RT + 2: if ((c.tpart >> q1) & 1u) neg_half<2, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RT + 3: if ((c.tpart >> q1) & 1u) neg_half<3, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_RT + 4: if ((c.tpart >> q1) & 1u) neg_half<4, 1>(a); ARSO_CZ_MASKS break;
        case OP_CZ_TT:
            if ((c.tpart >> q0) & (c.tpart >> q1) & 1u) negate_all(a);
            ARSO_CZ_MASKS break;
#undef ARSO_CZ_MASKS
        case OP_OMEGA: rg_omega(a, c, q0, p0, (h.x >> 20) & 7u); break;
        case OP_PHASE: phase_pair(a, bit_mask(c, q0), make_float2(__uint_as_float(u->x), __uint_as_float(u->y))); break;
        case OP_CP: rg_cp(a, c, q0, q1, make_float2(__uint_as_float(u->x), __uint_as_float(u->y))); break;
        case OP_SIGN:
        case OP_CX: case OP_CX + 1: case OP_CX + 2: case OP_CX + 3: case OP_CX + 4: {
            const uint4 w = *u;
            const uint32_t tm = c.tpart ^ c.m;
            const uint32_t A = w.x ^ (uint32_t)((int)(tm << (w.z & 31u)) >> 31);
            const uint32_t B = w.y ^ (uint32_t)((int)(tm << ((w.z >> 8) & 31u)) >> 31);
            const uint32_t mask = (w.w & 1u ? A : 0u) ^ (w.w & 2u ? B : 0u) ^ (w.w & 4u ? A & B : 0u);
            if (mask) {
                switch (code) {
                    case OP_CX: rg_flip_if<0>(a, mask); break;
                    case OP_CX + 1: rg_flip_if<1>(a, mask); break;
                    case OP_CX + 2: rg_flip_if<2>(a, mask); break;
                    case OP_CX + 3: rg_flip_if<3>(a, mask); break;
                    case OP_CX + 4: rg_flip_if<4>(a, mask); break;
                    default: break;
                }
            }
            uint32_t sg = 0;
            if ((w.w & 7u) && ((c.z >> (31u - ((w.z >> 16) & 31u))) & 1u)) {
                // Z on the target: a sign where it flips; for CX, Z on the control
                if ((w.w & 7u) == 1u) {
                    const uint32_t qa = 31u - (w.z & 31u);
                    c.z ^= 1u << qa;
                    c.gp ^= ((c.m >> qa) & 1u) << 1;
                } else {
                    sg = mask;
                }
            }
            c.m ^= h.w;
            if (w.w & 0x78u) {
                const uint32_t pc = w.z >> 24;
                const uint32_t C = (pc < REG_BITS ? reg_pattern(pc) : 0u) ^
                                   (uint32_t)((int)((c.tpart ^ c.m) << ((w.z >> 16) & 31u)) >> 31);
                sg ^= (w.w & 8u ? A & B : 0u) ^ (w.w & 16u ? A & C : 0u) ^ (w.w & 32u ? B & C : 0u) ^
                      (w.w & 64u ? A & B & C : 0u);
            }
            if (sg) negate_masked(a, sg);
            break;
        }
        case OP_PARITY:
            phase_pair(a, bit_mask(c, q0) ^ bit_mask(c, q1), make_float2(__uint_as_float(u->x), __uint_as_float(u->y)));
            break;
        case OP_SCALE:
            phase_pair_exact(a, ~0u, make_float2(__uint_as_float(u->x), __uint_as_float(u->y)), __uint_as_float(u->z));
            break;
        case OP_DENSE1: {
            const float2 *M = mats + u->x;
            const uint32_t f = ARSO_FLIP;
            rg_dense1_lanes(a, M[f ? 3 : 0], ARSO_ZS(M[f ? 2 : 1]), ARSO_ZS(M[f ? 1 : 2]), M[f ? 0 : 3]);
            break;
        }
        case OP_DENSE1 + 1: ARSO_D1Z(1); break;
        case OP_DENSE1 + 2: ARSO_D1Z(2); break;
        case OP_DENSE1 + 3: ARSO_D1Z(3); break;
        case OP_DENSE1 + 4: ARSO_D1Z(4); break;
        case OP_DENSE2: tile_two(a, c, false, q0, q1, mats + u->x, sm, ubuf, t); break;
        case OP_SWAP: tile_two(a, c, true, q0, q1, nullptr, sm, ubuf, t); break;
        default: break;
    }
}
#undef ARSO_FLIP
#undef ARSO_D1
#undef ARSO_D1Z
#undef ARSO_ZS
#undef ARSO_CX
#undef ARSO_CZ_ALL
#undef ARSO_P4

// Gates [g, ge) of one phase of a tensor circuit with the Pauli events that fall inside
// them; ops[0] is the record of gate g0 (the phase's first gate). The inner loop
// runs up to and including the next event's gate without touching the event
// state, which stays out of the hot registers. Records whose tensor role has
// its bit set in `skip` are passed over (tensor phases, which hold no event).
__device__ __forceinline__ void run_gates(Amps &v, TileCtx &c, uint32_t g, uint32_t ge, const RegOp *ops, uint32_t g0,
                                          const float2 *__restrict__ mats, float2 *sm, float2 *ubuf, int t,
                                          const uint32_t *&ev, const uint32_t *ev_end, uint32_t &next, uint32_t skip) {
    while (g < ge) {
        const uint32_t np = next == NO_EVENT ? ge : ev_pos(next);
        const uint32_t stop = np < ge ? np + 1 : ge;
        for (; g < stop; ++g) {
            const RegOp &op = ops[g - g0];
            if ((skip >> op.pad[1]) & 1u) continue;
            apply_op(v, c, op, mats, sm, ubuf, t);
        }
        if (np >= ge) break;
        const uint32_t w0 = ops[np - g0].w0;
        while (next != NO_EVENT && ev_pos(next) == np) {
            rg_pauli(v, c, ev_slot(next) ? (w0 >> 24) : ((w0 >> 16) & 255u), ev_code(next));
            ++ev;
            next = ev < ev_end ? *ev : NO_EVENT;
        }
    }
}

// The macro-ops [u, ue) of one phase with the Pauli events that fall inside them. An X
// or Y error would turn the frame's diag(1, phi) on its qubit into diag(phi, 1);
// diag(phi, conj phi) on the flipped state keeps the frame the same for every trajectory.
// (The float cosine of a phase below 2.4e-4 is 1: both parts of phi tell whether it is.)
__device__ __forceinline__ void run_prog(Amps &v, TileCtx &c, const uint4 *u, const uint4 *ue,
                                         const float2 *__restrict__ mats, float2 *sm, float2 *ubuf, int t,
                                         const uint32_t *&ev, const uint32_t *ev_end, uint32_t &next,
                                         const EvSlot *__restrict__ evs) {
    uint32_t skip = 0;  // units after the next macro-op
    while (u < ue) {
        const uint4 h = *u;
        if ((h.x & 255u) == OP_BLOCK) {  // fused, unless an event falls inside
            if (ev_pos(next) < h.y) u += 1 + (u[1].x >> 24);
            else ++u, skip = h.z;
            continue;
        }
        apply_macro(v, c, h, u + 1, mats, sm, ubuf, t);
        u += (h.x >> 24) + skip;
        skip = 0;
        while (ev_pos(next) < h.y) {
            const float4 e = __ldg(reinterpret_cast<const float4 *>(evs + 2 * ev_pos(next) + ev_slot(next)));
            const uint32_t q = __float_as_uint(e.z), pc = ev_code(next);
            if (pc & 2u) {  // Z part (Eq. (2)): on the true bit, so a sign of all where the bit is flipped
                c.z ^= 1u << q;
                c.gp ^= ((c.m >> q) & 1u) << 1;
            }
            if (pc & 1u) c.m ^= 1u << q;
            if (pc == 3u) c.gp = (c.gp + 1u) & 3u;  // Y = i X Z
            if ((pc & 1u) && (e.x != 1.f || e.y != 0.f)) phase_pair_exact(v, ~bit_mask(c, q), make_float2(e.x, e.y), e.w);
            ++ev;
            next = ev < ev_end ? *ev : NO_EVENT;
        }
    }
}

// A phase's program is staged in shared memory: stage_units starts cp.async copies of
// the next phase's 16-byte units while the current phase runs (a tensor circuit's gate
// records are two units each); stage_wait waits for this thread's copies and syncs the
// CTA, after which the staged units are visible to all threads and the other buffer is
// free again.
__device__ __forceinline__ void stage_units(uint4 *dst, const void *src, uint32_t n, uint32_t tid, uint32_t nthr) {
    n = n < (uint32_t)MAX_PHASE_UNITS ? n : (uint32_t)MAX_PHASE_UNITS;
    const char *s = static_cast<const char *>(src);
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    for (uint32_t i = tid; i < n; i += nthr)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 16 * i), "l"(s + 16 * i) : "memory");
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void stage_wait() {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
}

// ------------------------------------------------------- tensor phases ---
// A phase with a fused unitary U (see the tensor-phase notes of internal.h) as
// one contraction on the tensor cores. The tile is a matrix of 2^(t-5) rows
// (row = thread) by 64 reals (the thread's 32 amplitudes in packed-register
// order: for packed register p, Re a_2p, Re a_2p+1, Im a_2p, Im a_2p+1), and
// D = A B^T with B the real 64 x 64 form of U in the same order on both sides.
// FP32 accuracy from FP16 operands, with no bias from the tensor core's
// accumulation (which is not rounded to nearest): each row is scaled by a power
// of two so that its entries stay below 2^9 and split into the integer
// hi = rint(x) and lo = fp16(x - hi) (|lo| <= 1/2); B comes from the host scaled
// by 2^8 and split the same way (|hi| <= 256). The hi x hi products are integers
// below 2^17 and their sums below 2^23, so their accumulator D0 is exact; the
// other three products (hi lo, lo hi, lo lo) go to a second accumulator D1 about
// 2^-9 of D0's size, whose rounding is negligible; D0 + D1 is formed in
// registers. A (both terms) fills the tile's shared-memory buffer exactly; rows
// are grouped in blocks of 128 (MMAs of M = 128, N = 64), each block with its
// two accumulators in 128 tensor-memory columns.
constexpr uint32_t TP_ROWS = 128;
constexpr uint32_t TP_TERM_BYTES = TP_ROWS * 64 * 2;          // one term of one row block: 16 KiB
constexpr uint32_t TP_IMAGE_BYTES = TENSOR_IMAGE_HALVES * 2;  // B hi and lo: 16 KiB
constexpr uint32_t TP_IDESC = idesc_f16_f32(128, 64);

__device__ __forceinline__ uint32_t h2_bits(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);  // a in the low half (the lower K index)
    return *reinterpret_cast<const uint32_t *>(&h);
}
__device__ __forceinline__ float2 h2_value(uint32_t u) {
    const __half2 h = *reinterpret_cast<const __half2 *>(&u);
    return __half22float2(h);
}

// cp.async copies of one phase's B images (16 KiB) into shared memory, in the
// caller's commit group
__device__ __forceinline__ void stage_image(unsigned char *dst, const unsigned char *src, uint32_t tid, uint32_t nthr) {
    const uint32_t d = smem_u32(dst);
    for (uint32_t i = tid; i < TP_IMAGE_BYTES / 16; i += nthr)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 16 * i), "l"(src + 16 * i) : "memory");
}

// v <- U v for every row of the tile. Each block of 128 rows (four warps) is an
// independent group: it writes its rows of A, syncs on its own named barrier,
// and its first thread issues the block's MMAs and commits them to the block's
// mbarrier, which the group waits on before reading D back. The caller has
// synced the CTA after its last read of the tile buffer `abuf`; `img` holds
// this phase's staged B images (their cp.async copies waited for and synced).
// Returns false when the wait for the tensor cores gave up (v then holds no
// valid state).
__device__ __forceinline__ bool tensor_apply(Amps &v, unsigned char *abuf, const unsigned char *img, uint32_t nblk,
                                             uint32_t tmem, uint64_t *bars, uint32_t &parity) {
    const uint32_t tid = threadIdx.x, blk = tid >> 7, r = tid & (TP_ROWS - 1u);
    // row scale 2^k: sum of squares in [2^E, 2^(E+1)) bounds every entry below 2^ceil((E+1)/2)
    float2 s2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int p = 0; p < 16; ++p) {
        s2 = fma2(v.re[p], v.re[p], s2);
        s2 = fma2(v.im[p], v.im[p], s2);
    }
    const int E = (int)((__float_as_uint(s2.x + s2.y) >> 23) & 255u) - 127;
    const int k = min(max(9 - ((E + 2) >> 1), -100), 100);
    const float2 sc = bc2(__uint_as_float((uint32_t)(127 + k) << 23));
    const float2 inv = bc2(__uint_as_float((uint32_t)(127 - k - 8) << 23));  // undoes the row and B scales
    {
        unsigned char *row_hi = abuf + blk * TP_TERM_BYTES + (r >> 3) * 1024u + (r & 7u) * 16u;
        unsigned char *row_lo = row_hi + nblk * TP_TERM_BYTES;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int p = 2 * u + (h >> 1);
                const float2 x = mul2(h & 1 ? v.im[p] : v.re[p], sc);
                const float2 rx = make_float2(rintf(x.x), rintf(x.y));
                hi[h] = h2_bits(rx.x, rx.y);
                lo[h] = h2_bits(x.x - rx.x, x.y - rx.y);
            }
            *reinterpret_cast<uint4 *>(row_hi + u * 128) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4 *>(row_lo + u * 128) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
    }
    fence_proxy_async_smem();  // A (and the staged B) visible to the tensor core
    tc_fence_before();         // the previous phase's tensor-memory loads precede the next MMA
    asm volatile("bar.sync %0, %1;\n" ::"r"(1u + blk), "r"(TP_ROWS) : "memory");
    if (r == 0) {
        tc_fence_after();
        // descriptors of K step 0; a K step of 16 advances every operand by 256 bytes (16 in
        // the descriptor's address field, which has room: shared addresses stay below 256 KiB)
        const uint32_t ah = smem_u32(abuf) + blk * TP_TERM_BYTES, b0 = smem_u32(img);
        const uint64_t dah = smem_desc_kmajor(ah, 128, 1024), dal = smem_desc_kmajor(ah + nblk * TP_TERM_BYTES, 128, 1024);
        const uint64_t dbh = smem_desc_kmajor(b0, 128, 1024), dbl = smem_desc_kmajor(b0 + TP_IMAGE_BYTES / 2, 128, 1024);
        const uint32_t d0 = tmem + blk * 128, d1 = d0 + 64;
#pragma unroll
        for (uint32_t s = 0; s < 4; ++s) {
            const uint64_t o = 16u * s;
            umma_bf16(d0, dah + o, dbh + o, TP_IDESC, s);
            umma_bf16(d1, dah + o, dbl + o, TP_IDESC, s);
            umma_bf16(d1, dal + o, dbh + o, TP_IDESC, 1);
            umma_bf16(d1, dal + o, dbl + o, TP_IDESC, 1);
        }
        umma_commit(bars + blk);
    }
    bool ok = mbar_wait_bounded(bars + blk, parity);
    if (!ok) (void)mbar_wait_bounded(bars + blk, parity);  // give a slow contraction one more bounded wait
    parity ^= 1u;
    tc_fence_after();
    // this thread's row: tensor-memory lane 32 (warp mod 4) + lane = tid mod 128, block tid / 128
    const uint32_t taddr = tmem + ((((tid >> 5) & 3u) * 32u) << 16) + blk * 128u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t e[32], f[32];
        tmem_ld32_nowait(taddr + 32 * h, e);
        tmem_ld32_nowait(taddr + 64 + 32 * h, f);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 er = make_float2(__uint_as_float(e[4 * i]), __uint_as_float(e[4 * i + 1]));
            const float2 ei = make_float2(__uint_as_float(e[4 * i + 2]), __uint_as_float(e[4 * i + 3]));
            const float2 fr = make_float2(__uint_as_float(f[4 * i]), __uint_as_float(f[4 * i + 1]));
            const float2 fi = make_float2(__uint_as_float(f[4 * i + 2]), __uint_as_float(f[4 * i + 3]));
            v.re[8 * h + i] = mul2(add2(er, fr), inv);
            v.im[8 * h + i] = mul2(add2(ei, fi), inv);
        }
    }
    return ok;
}

// Addresses of a thread's packed registers in the load mapping under an index mask:
// packed register k holds the true tile indices j and j + 1 (swapped when the mask has
// bit 0), j = (k ^ mr) << (t-4) | (tid ^ mt) << 1. The tile bits map to disjoint bits of
// the state's index, so k's part is an XOR of four offsets and each register costs one XOR.
struct LoadAt {
    uint32_t base;   // the tile's base, the thread's part and the mask's
    uint32_t ho[4];  // index offset of tile bits t-4 .. t-1
    __device__ __forceinline__ uint32_t operator()(int k) const {
        uint32_t i = base;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if ((k >> b) & 1) i ^= ho[b];
        return i;
    }
    __device__ __forceinline__ void mask(uint32_t mr) {
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if ((mr >> b) & 1u) base ^= ho[b];
    }
};
__device__ __forceinline__ LoadAt linear_at(int t, uint32_t tid, uint32_t m) {
    LoadAt at;
    at.base = (tid << 1) ^ (m & ~1u);
#pragma unroll
    for (int b = 0; b < 4; ++b) at.ho[b] = 1u << (t - 4 + b);
    return at;
}
// of a streaming tile: offs the pass's tile-high offsets, c its contiguous low bits
__device__ __forceinline__ LoadAt tile_at(uint32_t base, const uint32_t *__restrict__ offs, int t, int c, uint32_t tid,
                                          uint32_t m) {
    const uint32_t cm = (1u << c) - 1u, j = (tid ^ ((m >> 1) & ((1u << (t - REG_BITS)) - 1u))) << 1;
    LoadAt at;
    at.base = base + __ldg(offs + (j >> c)) + (j & cm);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const uint32_t x = 1u << (t - 4 + b);
        at.ho[b] = __ldg(offs + (x >> c)) + (x & cm);
    }
    at.mask((m >> (t - 4)) & 15u);
    return at;
}

// Criterion partial of one thread's 32 amplitudes, in the load mapping with mask m and
// addresses `at`. Fidelity overlaps and outcome/binning probabilities are summed over
// the 32 registers in FP32 and then added to the FP64 partial (GB300's FP64 rate is a
// small fraction of its FP32 rate; the block and trajectory sums stay FP64); argmax
// compares FP64 probabilities amplitude by amplitude. The FP32 sum is a tree over the
// register bits: the mask only swaps the branches of its nodes, so a score does not
// depend on the checkpoint its trajectory started from. The reference is read two
// neighbours (16 bytes) at a time.
__device__ __forceinline__ void score_registers(Partial &acc, const DCrit &crit, const Amps &v,
                                                const float2 *__restrict__ ref, const LoadAt &at) {
    if (crit.kind == ARSO_CRIT_ARGMAX) {
#pragma unroll
        for (int ri = 0; ri < 32; ++ri)
            accumulate(acc, crit, amp_get(v, ri), ref, (uint64_t)(at(ri >> 1) + (ri & 1)));
        return;
    }
    float2 ta[5], tb[5];  // partial sums of the tree's levels
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t gi = at(k);
        float2 sa, sb = make_float2(0.f, 0.f);
        if (crit.kind == ARSO_CRIT_FIDELITY) {
            const float4 w = __ldg(reinterpret_cast<const float4 *>(ref + gi));
            const float2 rr = make_float2(w.x, w.z), ri = make_float2(w.y, w.w);
            sa = fma2(rr, v.re[k], mul2(ri, v.im[k]));
            sb = fma2(rr, v.im[k], mul2(make_float2(-ri.x, -ri.y), v.re[k]));
        } else {
            uint32_t in;  // bits 0 and 1: whether gi and gi + 1 count
            if (crit.kind == ARSO_CRIT_OUTCOME) in = gi == (crit.target & ~1ull) ? 1u << (crit.target & 1u) : 0u;
            else in = crit.bitmap[gi >> 5] >> (gi & 31);
            sa = fma2(v.re[k], v.re[k], mul2(v.im[k], v.im[k]));
            sa.x = in & 1u ? sa.x : 0.f;
            sa.y = in & 2u ? sa.y : 0.f;
        }
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            if (!((k >> l) & 1)) {
                ta[l] = sa;
                tb[l] = sb;
                break;
            }
            sa = add2(ta[l], sa);
            sb = add2(tb[l], sb);
        }
    }
    acc.a += (double)(ta[4].x + ta[4].y);
    acc.b += (double)(tb[4].x + tb[4].y);
}

// the tile's amplitudes from / to memory, in the load mapping
template <bool L2ONLY>
__device__ __forceinline__ void load_tile(Amps &v, const float2 *__restrict__ src, const LoadAt &at) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float4 *p = reinterpret_cast<const float4 *>(src + at(k));
        const float4 w = L2ONLY ? __ldcg(p) : __ldg(p);
        v.re[k] = make_float2(w.x, w.z);
        v.im[k] = make_float2(w.y, w.w);
    }
}
__device__ __forceinline__ void store_tile(const Amps &v, float2 *dst, const LoadAt &at) {
#pragma unroll
    for (int k = 0; k < 16; ++k)
        *reinterpret_cast<float4 *>(dst + at(k)) = make_float4(v.re[k].x, v.im[k].x, v.re[k].y, v.im[k].y);
}

// v (in the load mapping, masks resolved but for c.m without bit 0) times the frame table (internal.h) and i^gp
__device__ __forceinline__ void apply_frame(Amps &v, TileCtx &c, const float2 *__restrict__ frame, int t) {
    const uint32_t nt = 1u << (t - REG_BITS);
    const float4 *T = reinterpret_cast<const float4 *>(frame + nt);
    float2 F = __ldg(frame + (c.tid ^ ((c.m >> 1) & (nt - 1u))));
    if (c.gp & 1u) F = make_float2(-F.y, F.x);
    if (c.gp & 2u) F = make_float2(-F.x, -F.y);
    c.gp = 0;
    const uint32_t mr = (c.m >> (t - 4)) & 15u;
    const float2 fr = bc2(F.x), fi = bc2(F.y), nfi = bc2(-F.y);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float4 w = __ldg(T + ((uint32_t)k ^ mr));
        const float2 tr = make_float2(w.x, w.y), ti = make_float2(w.z, w.w);
        const float2 gr = fma2(nfi, ti, mul2(fr, tr)), gi = fma2(fi, tr, mul2(fr, ti));
        const float2 ngi = make_float2(-gi.x, -gi.y);
        const float2 r = v.re[k], i = v.im[k];
        v.re[k] = fma2(ngi, i, mul2(gr, r));
        v.im[k] = fma2(gi, r, mul2(gr, i));
    }
}

// the signs of z, then the lanes in true order: what is left of the masks is m without bit 0
__device__ __forceinline__ void resolve_masks(Amps &a, TileCtx &c) {
    uint32_t mask = __popc(c.tpart & c.z) & 1 ? 0xFFFFFFFFu : 0u;
#pragma unroll
    for (int b = 0; b < REG_BITS; ++b)
        if ((c.z >> rbit(c.R, b)) & 1u) mask ^= reg_pattern((uint32_t)b);
    if (mask) negate_masked(a, mask);
    c.z = 0;
    if (c.m & 1u) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            a.re[k] = swp2(a.re[k]);
            a.im[k] = swp2(a.im[k]);
        }
        c.m ^= 1u;
    }
}
// register set of the load/store mapping {0, t-4, ..., t-1}
__device__ __forceinline__ uint32_t load_set(int t) {
    return ((uint32_t)(t - 4) << 5) | ((uint32_t)(t - 3) << 10) | ((uint32_t)(t - 2) << 15) | ((uint32_t)(t - 1) << 20);
}
// the true state up to its mask, in the load mapping
__device__ __forceinline__ void finish_tile(Amps &v, float2 *sm, TileCtx &c, const float2 *__restrict__ frame, int t) {
    if (c.R != load_set(t)) remap(v, sm, c, load_set(t), t);
    resolve_masks(v, c);
    if (frame) apply_frame(v, c, frame, t);
    else apply_global_phase(v, c);
}

// Per-group sums of a criterion partial: `group` threads (a power of two, at least a
// warp) each; the group's first thread gets its sum. Ends with red[] free to reuse only
// after the caller's next barrier.
__device__ __forceinline__ Partial group_reduce_partial(Partial acc, Partial *red, uint32_t group) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double a2 = __shfl_down_sync(0xffffffffu, acc.a, o);
        const double b2 = __shfl_down_sync(0xffffffffu, acc.b, o);
        const double mp = __shfl_down_sync(0xffffffffu, acc.maxp, o);
        const unsigned long long mi = __shfl_down_sync(0xffffffffu, acc.idx, o);
        acc.a += a2;
        acc.b += b2;
        argmax_merge(acc.maxp, acc.idx, mp, mi);
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if ((threadIdx.x & (group - 1)) == 0) {
        const uint32_t w0 = threadIdx.x >> 5, nw = group >> 5;
        for (uint32_t w = w0 + 1; w < w0 + nw; ++w) {
            acc.a += red[w].a;
            acc.b += red[w].b;
            argmax_merge(acc.maxp, acc.idx, red[w].maxp, red[w].idx);
        }
    }
    return acc;
}

// global offset of the tile's first amplitude: the tile index deposited into
// the global bits outside the tile
__device__ __forceinline__ uint64_t tile_base(uint64_t rest_mask, uint64_t tile) {
    uint64_t base = 0;
    for (uint64_t mm = rest_mask; mm; mm &= mm - 1) {
        if (tile & 1) base |= mm & (~mm + 1);
        tile >>= 1;
    }
    return base;
}

// where a slot's tile comes from, and its events from the pass's first gate on; false
// when the slot does not run this pass
__device__ __forceinline__ bool pass_source(const PassArgs &a, uint32_t slot, const float2 *&src, const uint32_t *&ev,
                                            const uint32_t *&ev_end) {
    const uint64_t N = 1ull << a.n;
    ev = ev_end = nullptr;
    if (a.ideal) {
        src = static_cast<const float2 *>(a.ideal_src);
        return true;
    }
    const int start = a.start_pass[slot];
    if (a.pass < start || a.pass > a.end_pass[slot]) return false;
    src = a.pass == start ? static_cast<const float2 *>(a.cache) + (size_t)a.cache_slot[start] * N
                          : static_cast<const float2 *>(a.work) + (size_t)slot * N;
    // binary search for the first key at or after the pass's first gate
    const uint64_t tr = a.slot_traj[slot];
    const uint32_t *lo = a.keys + a.offsets[tr], *hi = a.keys + a.offsets[tr + 1];
    ev_end = hi;
    const uint32_t key_lo = a.gb << 3;
    while (lo < hi) {
        const uint32_t *mid = lo + (hi - lo) / 2;
        if (*mid < key_lo) lo = mid + 1;
        else hi = mid;
    }
    ev = lo;
    return true;
}

// end of a pass: the tile scored against the cached state at the boundary, or stored
__device__ __forceinline__ void pass_finish(const PassArgs &a, Amps &v, TileCtx &c, uint32_t slot, uint32_t tile,
                                            uint32_t base, uint32_t tiles, Partial *red) {
    const uint64_t N = 1ull << a.n;
    resolve_masks(v, c);
    if (a.frame) apply_frame(v, c, a.frame, a.t);
    else apply_global_phase(v, c);
    const LoadAt at = tile_at(base, a.offs, a.t, a.c, c.tid, c.m);
    if (!a.ideal && !a.store_last && a.pass == a.end_pass[slot]) {
        const float2 *ref = static_cast<const float2 *>(a.ref_cache ? a.ref_cache : a.cache) +
                            (size_t)a.cache_slot[a.pass + 1] * N;
        Partial acc = empty_partial();
        score_registers(acc, a.crit, v, ref, at);
        acc = group_reduce_partial(acc, red, c.nthr);
        if (c.tid == 0) a.partials[(size_t)slot * tiles + tile] = acc;
        return;
    }
    store_tile(v, a.ideal ? static_cast<float2 *>(a.ideal_dst) : static_cast<float2 *>(a.work) + (size_t)slot * N, at);
}

// One pass over tiles of 2^t amplitudes: a CTA runs THREADS / 2^(t-5) neighbouring tiles
// of one slot side by side.
// The phase loop holds the 64 amplitude registers; everything needed only
// before or after it (addresses, slot data) is recomputed there instead of
// being kept live.
template <int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) pass_rb_kernel(PassArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Partial red[THREADS / 32];
    __shared__ uint32_t s_base[THREADS / 32];
    __shared__ float2 ubuf[THREADS / 32][16];
    __shared__ uint4 s_ops[2][MAX_PHASE_UNITS];
    const int t = a.t;
    TileCtx c;
    c.m = c.z = 0;
    c.gp = 0;
    c.nthr = 1u << (t - REG_BITS);
    c.tid = threadIdx.x & (c.nthr - 1u);
    const uint32_t sg = threadIdx.x >> (t - REG_BITS), groups = blockDim.x >> (t - REG_BITS);
    float2 *sm = reinterpret_cast<float2 *>(smem_raw) + ((size_t)sg << t);
    Amps v;
    const uint32_t *ev, *ev_end;
    {
        const float2 *src;
        if (!pass_source(a, blockIdx.y, src, ev, ev_end)) return;
        const uint32_t base = (uint32_t)tile_base(a.rest_mask, blockIdx.x * groups + sg);
        if (c.tid == 0) s_base[sg] = base;  // for the store: the phase loop has no register to keep it
        load_tile<false>(v, src, tile_at(base, a.offs, t, a.c, c.tid, 0u));
    }
    set_phase(c, load_set(t), t);
    uint32_t next = ev < ev_end ? *ev : NO_EVENT;
    const float2 *mats = static_cast<const float2 *>(a.mats);
    if (a.pb < a.pe)
        stage_units(s_ops[0], a.prog + a.ph_pg[a.pb], a.ph_pg[a.pb + 1] - a.ph_pg[a.pb], threadIdx.x, blockDim.x);
    for (uint32_t ph = a.pb; ph <= a.pe; ++ph) {  // and back to the load mapping: one copy of the remap's code
        const uint32_t buf = (ph - a.pb) & 1u;
        stage_wait();
        if (ph + 1 < a.pe)
            stage_units(s_ops[buf ^ 1u], a.prog + a.ph_pg[ph + 1], a.ph_pg[ph + 2] - a.ph_pg[ph + 1], threadIdx.x,
                        blockDim.x);
        const uint32_t R = ph < a.pe ? a.ph_R[ph] : load_set(t);
        if (R != c.R) remap<true>(v, sm, c, R, t);
        if (ph == a.pe) break;
        run_prog(v, c, s_ops[buf], s_ops[buf] + (a.ph_pg[ph + 1] - a.ph_pg[ph]), mats, sm, ubuf[sg], t, ev, ev_end, next,
                 a.evs);
    }
    pass_finish(a, v, c, blockIdx.y, blockIdx.x * groups + sg, s_base[sg], gridDim.x * groups, red);
}

// One pass of a probe circuit (kernels.h), or some of its phases, over a state in place: CTAs
// loop over the tiles, so that each warp keeps one row of sums. Bound by instruction issue: a measurement is 64
// packed multiply-adds and about 70 instructions of exchange per warp, next to 64 for the
// gate before it, and a pass reads and writes the state once for some 40 gates. Whole
// single-error analysis, before (one HBM sweep per gate) and after: 24-qubit brickwork, 1,880
// locations, 88.7 -> 33.0 ms for the first call of a handle, which plans and uploads the probe
// circuit, and 23.3 ms for the later ones, which find it there; 20-qubit adder, both states,
// 25.4 -> 1.95 and 0.87 ms.
template <int THREADS, int MINB, bool DUAL>
__global__ void __launch_bounds__(THREADS, MINB) probe_kernel(ProbeArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *sm = reinterpret_cast<float2 *>(smem_raw);
    __shared__ float2 ubuf[16];
    __shared__ uint4 s_ops[2][MAX_PHASE_UNITS];
    const int t = a.t;
    __shared__ uint32_t s_base;
    double *row = a.rows + ((size_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * a.row_len;
    for (uint32_t tile = blockIdx.x; tile < a.tiles; tile += gridDim.x) {
        TileCtx c;
        c.m = c.z = 0;
        c.gp = 0;
        c.nthr = blockDim.x;
        c.tid = threadIdx.x;
        Amps v;
        {
            const uint32_t base = (uint32_t)tile_base(a.rest_mask, tile);
            if (c.tid == 0) s_base = base;
            load_tile<true>(v, a.state, tile_at(base, a.offs, t, a.c, c.tid, 0u));
        }
        set_phase(c, load_set(t), t);
        if (a.pb < a.pe)
            stage_units(s_ops[0], a.prog + a.ph_pg[a.pb], a.ph_pg[a.pb + 1] - a.ph_pg[a.pb], threadIdx.x, blockDim.x);
        for (uint32_t ph = a.pb; ph <= a.pe; ++ph) {
            const uint32_t buf = (ph - a.pb) & 1u;
            stage_wait();
            if (ph + 1 < a.pe)
                stage_units(s_ops[buf ^ 1u], a.prog + a.ph_pg[ph + 1], a.ph_pg[ph + 2] - a.ph_pg[ph + 1], threadIdx.x,
                            blockDim.x);
            const uint32_t R = ph < a.pe ? a.ph_R[ph] : load_set(t);
            if (R != c.R) remap<true>(v, sm, c, R, t);
            if (ph == a.pe) break;
            const uint4 *u = s_ops[buf], *ue = u + (a.ph_pg[ph + 1] - a.ph_pg[ph]);
            while (u < ue) {
                const uint4 h = *u;
                if ((h.x & 255u) == OP_PROBE) run_probe<DUAL>(v, c, h, a.slot0, row);
                else apply_macro(v, c, h, u + 1, a.mats, sm, ubuf, t);
                u += h.x >> 24;  // a probe circuit has no fused runs
            }
        }
        resolve_masks(v, c);
        if (a.frame) apply_frame(v, c, a.frame, t);
        else apply_global_phase(v, c);
        store_tile(v, a.state, tile_at(s_base, a.offs, t, a.c, c.tid, c.m));
        __syncthreads();  // the shared memory is reused by the next tile
    }
}

// rows added in a fixed order: a block sums 32 values, eight rows at a time
__global__ void probe_sum_kernel(const double *__restrict__ rows, uint32_t n_rows, uint32_t row_len, double *out) {
    __shared__ double red[8][32];
    const uint32_t v = blockIdx.x * 32 + (threadIdx.x & 31u), g = threadIdx.x >> 5;
    double x = 0.0;
    if (v < row_len)
        for (uint32_t r = g; r < n_rows; r += 8) x += rows[(size_t)r * row_len + v];
    red[g][threadIdx.x & 31u] = x;
    __syncthreads();
    if (g == 0 && v < row_len) {
        for (int k = 1; k < 8; ++k) x += red[k][threadIdx.x];
        out[v] = x;
    }
}

static const void *probe_fn(int t, bool dual) {
    if (dual) return t <= 12 ? (const void *)probe_kernel<128, 4, true> : (const void *)probe_kernel<512, 1, true>;
    return t <= 12 ? (const void *)probe_kernel<128, 4, false> : (const void *)probe_kernel<512, 1, false>;
}
static uint32_t probe_grid(int t, uint32_t tiles, bool dual) {
    const void *fn = probe_fn(t, dual);
    const int smem = (1 << t) * (int)sizeof(float2);
    ARSO_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    int per_sm = 1, dev = 0, sms = 152;
    ARSO_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 1 << (t - REG_BITS), smem));
    ARSO_CUDA(cudaGetDevice(&dev));
    ARSO_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    return std::min<uint32_t>(tiles, (uint32_t)std::max(per_sm, 1) * (uint32_t)sms);
}
uint32_t probe_rows(int t, uint32_t tiles, bool dual) { return probe_grid(t, tiles, dual) * (1u << (t - REG_BITS - 5)); }

void launch_probe(const ProbeArgs &a, bool dual, cudaStream_t st) {
    ProfScope ps_(ARSO_K_OTHER, 16.0 * (double)(1ull << a.n), st);
    const uint32_t grid = probe_grid(a.t, a.tiles, dual);
    ProbeArgs b = a;
    void *args[] = {&b};
    ARSO_CUDA(cudaLaunchKernel(probe_fn(a.t, dual), dim3(grid), dim3(1u << (a.t - REG_BITS)), args,
                               (size_t(1) << a.t) * sizeof(float2), st));
}

void launch_probe_sum(const double *rows, uint32_t n_rows, uint32_t row_len, double *out, cudaStream_t st) {
    if (!row_len) return;
    ProfScope ps_(ARSO_K_REDUCE, 8.0 * (double)n_rows * row_len, st);
    probe_sum_kernel<<<(row_len + 31) / 32, 256, 0, st>>>(rows, n_rows, row_len, out);
    ARSO_CUDA(cudaGetLastError());
}

// The same for circuits with tensor phases: one tile per CTA, gate records instead of the
// register program, and the contraction above for the phases that qualify.
__global__ void __launch_bounds__(512, 1) pass_tensor_kernel(PassArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *sm = reinterpret_cast<float2 *>(smem_raw);
    __shared__ Partial red[16];
    __shared__ float2 ubuf[16];
    __shared__ uint4 s_ops[2][2 * MAX_PHASE_OPS];
    const int t = a.t;
    TileCtx c;
    c.m = c.z = 0;
    c.gp = 0;
    c.tid = threadIdx.x;
    c.nthr = blockDim.x;
    Amps v;
    const uint32_t *ev, *ev_end;
    {
        const float2 *src;
        if (!pass_source(a, blockIdx.y, src, ev, ev_end)) return;
        load_tile<false>(v, src, tile_at((uint32_t)tile_base(a.rest_mask, blockIdx.x), a.offs, t, a.c, c.tid, 0u));
    }
    set_phase(c, load_set(t), t);
    uint32_t next = ev < ev_end ? *ev : NO_EVENT;
    const float2 *mats = static_cast<const float2 *>(a.mats);
    // tensor memory for D0 and D1 (128 columns per block of 128 rows), one mbarrier
    // for the contractions' completion, and two 16 KiB buffers for the staged B images
    __shared__ uint64_t s_tbar[4];  // one per block of 128 rows
    __shared__ uint32_t s_tmem;
    const uint32_t nblk = blockDim.x / TP_ROWS;
    unsigned char *img = smem_raw + ((size_t)1 << t) * sizeof(float2);
    const unsigned char *tmats = static_cast<const unsigned char *>(a.tmats);
    uint32_t tpar = 0;
    if (threadIdx.x < 32) tmem_alloc(&s_tmem, nblk * 128u);
    if (threadIdx.x < nblk) {
        mbar_init(&s_tbar[threadIdx.x], 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    auto stage = [&](uint32_t ph, uint32_t buf) {
        if (a.ph_t[ph] != NO_TENSOR)
            stage_image(img + buf * TP_IMAGE_BYTES, tmats + (size_t)a.ph_t[ph] * TP_IMAGE_BYTES, threadIdx.x, blockDim.x);
        stage_units(s_ops[buf], a.rops + a.ph_gb[ph], 2 * (a.ph_gb[ph + 1] - a.ph_gb[ph]), threadIdx.x, blockDim.x);
    };
    if (a.pb < a.pe) stage(a.pb, 0);
    for (uint32_t ph = a.pb; ph < a.pe; ++ph) {
        const uint32_t buf = (ph - a.pb) & 1u;
        stage_wait();
        if (ph + 1 < a.pe) stage(ph + 1, buf ^ 1u);
        const uint32_t R = a.ph_R[ph];
        if (R != c.R) remap<true>(v, sm, c, R, t);
        const uint32_t g0 = a.ph_gb[ph], ge = a.ph_gb[ph + 1];
        // the contraction applies U to the true amplitudes: no event of this trajectory in
        // the phase and no mask bit on a register bit (the CTA takes the same branch)
        uint32_t rm = 0;
#pragma unroll
        for (int b = 0; b < REG_BITS; ++b) rm |= 1u << rbit(R, b);
        const bool tp = a.ph_t[ph] != NO_TENSOR && (next == NO_EVENT || ev_pos(next) >= ge) && (c.m & rm) == 0u;
        const int rounds = tp ? 2 : 1;
#pragma unroll 1
        for (int rd = 0; rd < rounds; ++rd) {
            if (rd == 1) {
                __syncthreads();  // every thread's reads of the tile buffer are done
                if (!tensor_apply(v, smem_raw, img + buf * TP_IMAGE_BYTES, nblk, tmem, s_tbar, tpar))
                    atomicOr(a.terr, 1u);
            }
            const uint32_t skip =
                tp ? (rd == 0 ? (1u << TR_CORE) | (1u << TR_AFTER) : (1u << TR_CORE) | (1u << TR_BEFORE)) : 0u;
            run_gates(v, c, g0, ge, reinterpret_cast<const RegOp *>(s_ops[buf]), g0, mats, sm, ubuf, t, ev, ev_end, next,
                      skip);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) {
        tc_fence_after();
        tmem_free(tmem, nblk * 128u);
    }
    if (c.R != load_set(t)) remap(v, sm, c, load_set(t), t);
    pass_finish(a, v, c, blockIdx.y, blockIdx.x, (uint32_t)tile_base(a.rest_mask, blockIdx.x), gridDim.x, red);
}

// ------------------------------------------------------------- resident ---
// Whole state (2^n, 10 <= n <= 13) in one CTA: each trajectory restarts from
// the cached error-free state at the checkpoint (phase boundary) at or before
// its first error and runs the remaining phases; ckpt_every counts phases. The
// checkpoints before the last are in their boundary's frame (RegOpCode, internal.h), so
// that a run from any of them has the bits of a run through it; the last is the true psi_R.

// store the state (mask applied) to dst, times the frame when one is given; without one
// v stays as it is (in the load mapping)
__device__ __forceinline__ void rb_store_linear(Amps &v, float2 *sm, TileCtx &c, float2 *dst, int t,
                                                const float2 *__restrict__ frame) {
    if (c.R != load_set(t)) remap(v, sm, c, load_set(t), t);
    resolve_masks(v, c);
    if (frame) apply_frame(v, c, frame, t);
    else apply_global_phase(v, c);
    store_tile(v, dst, linear_at(t, c.tid, c.m));
}

template <int MODE>
__global__ void __launch_bounds__(512, 1) resident_rb_kernel(ResidentArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *sm = reinterpret_cast<float2 *>(smem_raw);
    __shared__ Partial red[32];
    __shared__ float2 ubuf[16];
    __shared__ uint4 s_ops[2][MAX_PHASE_UNITS];
    const int t = a.n;
    const uint32_t N = 1u << t;
    const float2 *cache = static_cast<const float2 *>(a.cache);
    const float2 *mats = static_cast<const float2 *>(a.mats);
    const uint64_t count = MODE == 2 ? 1 : a.count;
    for (uint64_t b = blockIdx.x; b < count; b += gridDim.x) {
        Amps v;
        TileCtx c;
        c.m = c.z = 0;
        c.gp = 0;
        c.tid = threadIdx.x;
        c.nthr = blockDim.x;
        set_phase(c, load_set(t), t);
        uint32_t ph0 = 0;
        const uint32_t *ev = nullptr, *ev_end = nullptr;
        uint64_t tr = 0;
        if (MODE == 2) {
#pragma unroll
            for (int k = 0; k < 16; ++k) v.re[k] = v.im[k] = make_float2(0.f, 0.f);
            if (threadIdx.x == 0) v.re[0].x = 1.f;
        } else {
            tr = a.ids ? a.ids[b] : a.first_traj + b;
            const uint32_t first = a.first[tr];
            if (MODE == 0 && first == NO_EVENT) {
                if (threadIdx.x == 0) {
                    a.score[tr] = *a.ref_score;
                    if (a.pass_flags) a.pass_flags[tr] = *a.ref_score >= a.crit.threshold;
                }
                continue;
            }
            uint32_t ck;
            if (first == NO_EVENT) {
                ck = a.n_ckpt - 1;
                ph0 = a.n_phases;
            } else {
                ck = a.phase_of_pos[first] / (uint32_t)a.ckpt_every;
                ph0 = ck * (uint32_t)a.ckpt_every;
            }
            load_tile<false>(v, cache + (size_t)ck * N, linear_at(t, c.tid, 0u));
            ev = a.keys + a.offsets[tr];
            ev_end = a.keys + a.offsets[tr + 1];
        }
        uint32_t next = ev && ev < ev_end ? *ev : NO_EVENT;
        if (ph0 < a.n_phases)
            stage_units(s_ops[0], a.prog + a.ph_pg[ph0], a.ph_pg[ph0 + 1] - a.ph_pg[ph0], threadIdx.x, blockDim.x);
        for (uint32_t ph = ph0; ph < a.n_phases; ++ph) {
            const uint32_t buf = (ph - ph0) & 1u;
            stage_wait();
            if (ph + 1 < a.n_phases)
                stage_units(s_ops[buf ^ 1u], a.prog + a.ph_pg[ph + 1], a.ph_pg[ph + 2] - a.ph_pg[ph + 1], threadIdx.x,
                            blockDim.x);
            if (MODE == 2 && ph % (uint32_t)a.ckpt_every == 0) {
                float2 *dst = const_cast<float2 *>(cache) + (size_t)(ph / (uint32_t)a.ckpt_every) * N;
                rb_store_linear(v, sm, c, dst, t, nullptr);
            }
            const uint32_t R = a.ph_R[ph];
            if (R != c.R) remap<MODE != 2>(v, sm, c, R, t);
            run_prog(v, c, s_ops[buf], s_ops[buf] + (a.ph_pg[ph + 1] - a.ph_pg[ph]), mats, sm, ubuf, t, ev, ev_end,
                     next, a.evs);
        }
        // the last checkpoint is the true psi_R, so a trajectory that starts there ends there too
        const float2 *frame_end = ph0 < a.n_phases ? a.frame + (size_t)(a.n_ckpt - 1) * frame_floats2(t) : nullptr;
        if (MODE == 2) {
            rb_store_linear(v, sm, c, const_cast<float2 *>(cache) + (size_t)(a.n_ckpt - 1) * N, t, frame_end);
        } else if (MODE == 1) {
            rb_store_linear(v, sm, c, static_cast<float2 *>(a.states_out) + (size_t)b * N, t, frame_end);
        } else {
            finish_tile(v, sm, c, frame_end, t);
            const float2 *ref = cache + (size_t)(a.n_ckpt - 1) * N;
            Partial acc = empty_partial();
            score_registers(acc, a.crit, v, ref, linear_at(t, c.tid, c.m));
            acc = block_reduce_partial(acc, red);
            if (threadIdx.x == 0) {
                const double sc = finish_score(a.crit, acc);
                a.score[tr] = sc;
                if (a.pass_flags) a.pass_flags[tr] = sc >= a.crit.threshold;
            }
        }
        __syncthreads();  // shared memory and red[] are reused by the next trajectory
    }
}

void launch_resident_rb(const ResidentArgs &a, int mode, double bytes, cudaStream_t st) {
    ProfScope ps_(ARSO_K_RESIDENT, bytes, st);
    const int nt = 1 << (a.n - REG_BITS);
    const size_t smem = (size_t(1) << a.n) * sizeof(float2);
    const void *fn = mode == 0 ? (const void *)resident_rb_kernel<0>
                   : mode == 1 ? (const void *)resident_rb_kernel<1> : (const void *)resident_rb_kernel<2>;
    if (smem > 48 * 1024) ARSO_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 1;
    ARSO_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, nt, smem));
    int dev = 0, sms = 152;
    ARSO_CUDA(cudaGetDevice(&dev));
    ARSO_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const uint64_t want = mode == 2 ? 1 : a.count;
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)std::max(per_sm, 1) * sms));
    if (mode == 0) resident_rb_kernel<0><<<grid, nt, smem, st>>>(a);
    else if (mode == 1) resident_rb_kernel<1><<<grid, nt, smem, st>>>(a);
    else resident_rb_kernel<2><<<grid, nt, smem, st>>>(a);
    ARSO_CUDA(cudaGetLastError());
}

// --------------------------------------------------------- batched resident ---
// Persistent CTAs of 256 threads pull (circuit, trajectory block) items from a
// device counter. A circuit of n qubits needs 2^(n-5) threads per trajectory,
// so one CTA runs 2^(13-n) trajectories of the same circuit side by side: the
// sub-groups share the circuit's phase program (uniform barriers) and keep
// their own registers, shared-memory tile, index mask and error events.
constexpr int BATCH_THREADS = 256;

// One batched resident item (see above) run by the whole CTA.
__device__ __forceinline__ void batch_item(const BatchItem &it, const BatchCircuit &C, const uint64_t *__restrict__ ids,
                                           unsigned char *smem_raw, Partial *red, float2 (*ubuf)[16],
                                           uint4 (*s_ops)[MAX_PHASE_UNITS]) {
    const int t = C.n;
    const uint32_t N = 1u << t, gsize = 1u << (t - REG_BITS), sg = threadIdx.x / gsize;
    float2 *sm = reinterpret_cast<float2 *>(smem_raw) + (size_t)sg * N;
    const bool active = sg < it.count;
    const uint64_t tr = ids[it.off + (active ? sg : 0)];
    TileCtx c;
    c.m = c.z = 0;
    c.gp = 0;
    c.tid = threadIdx.x % gsize;
    c.nthr = gsize;
    set_phase(c, load_set(t), t);
    Amps v;
    load_tile<false>(v, C.cache + (size_t)it.ck * N, linear_at(t, c.tid, 0u));
    const uint32_t *ev = C.keys + C.offsets[tr];
    const uint32_t *ev_end = C.keys + C.offsets[tr + 1];
    uint32_t next = ev < ev_end ? *ev : NO_EVENT;
    const uint32_t ph0 = it.ck * C.ckpt_every;
    if (ph0 < C.n_phases)
        stage_units(s_ops[0], C.prog + C.ph_pg[ph0], C.ph_pg[ph0 + 1] - C.ph_pg[ph0], threadIdx.x, BATCH_THREADS);
    for (uint32_t ph = ph0; ph < C.n_phases; ++ph) {
        const uint32_t buf = (ph - ph0) & 1u;
        stage_wait();
        if (ph + 1 < C.n_phases)
            stage_units(s_ops[buf ^ 1u], C.prog + C.ph_pg[ph + 1], C.ph_pg[ph + 2] - C.ph_pg[ph + 1], threadIdx.x,
                        BATCH_THREADS);
        const uint32_t R = C.ph_R[ph];
        if (R != c.R) remap<true>(v, sm, c, R, t);
        run_prog(v, c, s_ops[buf], s_ops[buf] + (C.ph_pg[ph + 1] - C.ph_pg[ph]), C.mats, sm, ubuf[sg], t, ev, ev_end,
                 next, C.evs);
    }
    finish_tile(v, sm, c, C.frame + (size_t)(C.n_ckpt - 1) * frame_floats2(t), t);
    const float2 *ref = C.cache + (size_t)(C.n_ckpt - 1) * N;
    Partial acc = empty_partial();
    score_registers(acc, C.crit, v, ref, linear_at(t, c.tid, c.m));
    acc = group_reduce_partial(acc, red, gsize);
    if (c.tid == 0 && active) {
        const double sc = finish_score(C.crit, acc);
        C.score[tr] = sc;
        if (C.pass_flags) C.pass_flags[tr] = sc >= C.crit.threshold;
    }
}

__global__ void __launch_bounds__(BATCH_THREADS, 2)
    batch_resident_kernel(const BatchCircuit *__restrict__ circs, const BatchItem *__restrict__ items, uint32_t n_items,
                          uint32_t *counter, const uint64_t *__restrict__ ids) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_item;
    __shared__ Partial red[BATCH_THREADS / 32];
    __shared__ float2 ubuf[8][16];
    __shared__ uint4 s_ops[2][MAX_PHASE_UNITS];
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1u);
        __syncthreads();
        const uint32_t item = s_item;
        if (item >= n_items) return;
        const BatchItem it = items[item];
        batch_item(it, circs[it.circuit], ids, smem_raw, red, ubuf, s_ops);
    }
}

void launch_batch_resident(const BatchCircuit *circs, const BatchItem *items, uint32_t n_items, uint32_t *counter,
                           const uint64_t *ids, double bytes, cudaStream_t st) {
    if (!n_items) return;
    ProfScope ps_(ARSO_K_RESIDENT, bytes, st);
    const size_t smem = (size_t(1) << 13) * sizeof(float2);
    ARSO_CUDA(cudaFuncSetAttribute(batch_resident_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 1, dev = 0, sms = 152;
    ARSO_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_resident_kernel, BATCH_THREADS, smem));
    ARSO_CUDA(cudaGetDevice(&dev));
    ARSO_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const unsigned grid = (unsigned)std::min<uint64_t>(n_items, (uint64_t)std::max(per_sm, 1) * sms);
    batch_resident_kernel<<<grid, BATCH_THREADS, smem, st>>>(circs, items, n_items, counter, ids);
    ARSO_CUDA(cudaGetLastError());
}

// ------------------------------------------------- persistent mixed batch ---
// One launch over every unit of a batch of uneven circuits (MixArgs in kernels.h).
// A CTA of 256 threads takes sub-items from one counter in list order. Streaming
// sub-items wait (thread 0, bounded polls) for their slot's counter of finished
// tiles; since a unit's dependencies always sit earlier in the list, the lowest
// sub-item in progress never waits on a later one and the launch cannot deadlock.
// A wait that gives up sets the error word; every CTA then stops at its next item.
constexpr int MIX_THREADS = BATCH_THREADS;  // one 2^13-amplitude tile: 256 threads x 32 registers

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// thread 0: wait until *ctr >= need + extra (extra is 0 except in the failure-path test);
// false if the wait gave up or another CTA's did
__device__ bool mix_wait(const uint32_t *ctr, uint32_t need, uint32_t extra, uint32_t limit, uint32_t *err) {
    const uint64_t target = (uint64_t)need + extra;
    for (uint32_t it = 0;; ++it) {
        if ((uint64_t)ld_acquire_u32(ctr) >= target) return true;
        if (it >= limit || ld_acquire_u32(err) != 0u) {
            atomicOr(err, 1u);
            return false;
        }
        __nanosleep(256);
    }
}

__device__ __forceinline__ Partial ld_partial_cg(const Partial *p) {
    Partial v;
    v.a = __ldcg(&p->a);
    v.b = __ldcg(&p->b);
    v.maxp = __ldcg(&p->maxp);
    v.idx = __ldcg(&p->idx);
    return v;
}

// First unit u >= lo with unit_end[u] > i (warp 0; unit_end ascending, unit_end[lo - 1] <= i
// by the caller's previous item): 32-way search, each round one load per lane.
__device__ uint32_t mix_find_unit(const uint64_t *__restrict__ unit_end, uint32_t n_units, uint32_t lo, uint64_t i) {
    if (__ldg(unit_end + lo) > i) return lo;
    uint32_t hi = n_units - 1;  // unit_end[hi] = total > i; invariant unit_end[lo] <= i < unit_end[hi]
    const uint32_t lane = threadIdx.x & 31u;
    while (hi - lo > 1) {
        const uint32_t step = (hi - lo + 31) / 32;
        const uint32_t probe = min(lo + step * (lane + 1), hi);
        const unsigned m = __ballot_sync(0xffffffffu, __ldg(unit_end + probe) > i);
        const uint32_t f = (uint32_t)(__ffs(m) - 1);  // lane 31 probes hi, so m != 0
        const uint32_t nhi = min(lo + step * (f + 1), hi);
        lo = f == 0 ? lo : lo + step * f;
        hi = nhi;
    }
    return hi;
}

// MIX_REF: chunk `chunk` of psi_R scored; the last chunk adds the chunk partials in
// order and gives that score to every error-free trajectory of the circuit.
__device__ __noinline__ void mix_ref(const MixRef &R, uint32_t chunk, Partial *red, uint32_t *s_flag, double *s_val) {
    const uint32_t N = 1u << R.n, j0 = chunk << 13, j1 = min(N, j0 + 8192u);
    Partial acc = empty_partial();
    for (uint32_t j = j0 + threadIdx.x; j < j1; j += blockDim.x) accumulate(acc, R.crit, R.psi_R[j], R.psi_R, j);
    acc = block_reduce_partial(acc, red);
    if (threadIdx.x == 0) {
        R.partials[chunk] = acc;
        __threadfence();
        *s_flag = atomicAdd(R.done, 1u) == R.chunks - 1;
    }
    __syncthreads();
    if (!*s_flag) return;
    __threadfence();
    if (threadIdx.x == 0) {
        Partial sum = empty_partial();
        for (uint32_t k = 0; k < R.chunks; ++k) {
            const Partial q = ld_partial_cg(R.partials + k);
            sum.a += q.a;
            sum.b += q.b;
            argmax_merge(sum.maxp, sum.idx, q.maxp, q.idx);
        }
        *s_val = finish_score(R.crit, sum);
    }
    __syncthreads();
    const double sc = *s_val;
    for (uint64_t t = threadIdx.x; t < R.n_traj; t += blockDim.x)
        if (R.first[t] == NO_EVENT) {
            R.score[t] = sc;
            if (R.pass_flags) R.pass_flags[t] = sc >= R.crit.threshold;
        }
}

// MIX_SMALL: up to 32 trajectories of one circuit of n <= 9 qubits side by side in
// shared memory as one state of n + log2(count) qubits (gates touch only the low n
// bits, so one update covers every trajectory); each trajectory's Pauli errors are
// applied to its own block; 8 threads score each trajectory.
__device__ __noinline__ void mix_small(const MixSmall &C, const BatchItem &it, const uint64_t *__restrict__ ids, float2 *s) {
    __shared__ const uint32_t *s_ev[MIX_SMALL_MAX];
    __shared__ const uint32_t *s_end[MIX_SMALL_MAX];
    __shared__ uint32_t s_pe[MIX_SMALL_MAX];
    const int n = C.n;
    const uint32_t N = 1u << n, cnt = it.count;
    int tb = n;
    while ((1u << (tb - n)) < cnt) ++tb;  // n + ceil(log2 cnt) <= 13
    const float2 *src = C.cache + (size_t)it.ck * N;
    for (uint32_t i = threadIdx.x; i < (1u << tb); i += blockDim.x)
        s[i] = (i >> n) < cnt ? src[i & (N - 1)] : make_float2(0.f, 0.f);
    if (threadIdx.x < cnt) {
        const uint64_t tr = ids[it.off + threadIdx.x];
        s_ev[threadIdx.x] = C.keys + C.offsets[tr];
        s_end[threadIdx.x] = C.keys + C.offsets[tr + 1];
    }
    __syncthreads();
    const uint32_t g0 = min(C.G, it.ck * C.ckpt_every);
    for (uint32_t g = g0; g < C.G; ++g) {
        const DGate gate = C.gates[g];
        if (gate.cls != GC_NOP) tile_gate(s, tb, gate, C.mats + gate.mat);
        // this gate's error events of each trajectory: up to two, (valid | qubit << 2 | code) per half
        bool any = false;
        if (threadIdx.x < cnt) {
            const uint32_t *e = s_ev[threadIdx.x], *ee = s_end[threadIdx.x];
            uint32_t pe = 0, sh = 0;
            while (e < ee && ev_pos(*e) == g) {
                const uint32_t q = ev_slot(*e) ? gate.q1 : gate.q0;
                pe |= (0x8000u | (q << 2) | ev_code(*e)) << sh;
                sh = 16;
                ++e;
            }
            s_ev[threadIdx.x] = e;
            s_pe[threadIdx.x] = pe;
            any = pe != 0;
        }
        if (__syncthreads_or(any)) {
            for (int w = 0; w < 2; ++w) {
                for (uint32_t p = threadIdx.x; p < (cnt << (n - 1)); p += blockDim.x) {
                    const uint32_t k = p >> (n - 1), e = (s_pe[k] >> (16 * w)) & 0xFFFFu;
                    if (!(e & 0x8000u)) continue;
                    const uint32_t q = (e >> 2) & 63u, code = e & 3u, bit = 1u << q;
                    const uint32_t i0 = (k << n) | insert_zero(p & ((N >> 1) - 1), q), i1 = i0 | bit;
                    const float2 a0 = s[i0], a1 = s[i1];
                    if (code == 1) {
                        s[i0] = a1;
                        s[i1] = a0;
                    } else if (code == 2) {
                        s[i1] = cneg(a1);
                    } else {  // Y: (a0, a1) -> (-i a1, i a0), Eq. (2)
                        s[i0] = make_float2(a1.y, -a1.x);
                        s[i1] = make_float2(-a0.y, a0.x);
                    }
                }
                __syncthreads();
            }
        }
    }
    // score: 8 threads per trajectory, FP64 sums, shuffles within each group of 8
    const uint32_t k = threadIdx.x >> 3, r = threadIdx.x & 7u;
    const float2 *ref = C.cache + (size_t)(C.n_ckpt - 1) * N;
    Partial acc = empty_partial();
    if (k < cnt)
        for (uint32_t j = r; j < N; j += 8) accumulate(acc, C.crit, s[(k << n) + j], ref, j);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        const double a2 = __shfl_down_sync(0xffffffffu, acc.a, o, 8);
        const double b2 = __shfl_down_sync(0xffffffffu, acc.b, o, 8);
        const double mp = __shfl_down_sync(0xffffffffu, acc.maxp, o, 8);
        const unsigned long long mi = __shfl_down_sync(0xffffffffu, acc.idx, o, 8);
        acc.a += a2;
        acc.b += b2;
        argmax_merge(acc.maxp, acc.idx, mp, mi);
    }
    if (r == 0 && k < cnt) {
        const uint64_t tr = ids[it.off + k];
        const double sc = finish_score(C.crit, acc);
        C.score[tr] = sc;
        if (C.pass_flags) C.pass_flags[tr] = sc >= C.crit.threshold;
    }
}

__device__ __noinline__ void mix_res(const BatchItem &it, const BatchCircuit &C, const uint64_t *__restrict__ ids,
                                    unsigned char *smem_raw, Partial *red, float2 (*ubuf)[16],
                                    uint4 (*s_ops)[MAX_PHASE_UNITS]) {
    batch_item(it, C, ids, smem_raw, red, ubuf, s_ops);
}

// MIX_STR: one tile of pass j of trajectory k of stream S (the body of pass_rb_kernel
// with explicit coordinates), after the slot's dependencies. The item's coordinates live
// in shared memory (`it`) and the stream's descriptor too: read where needed rather than
// held in registers, since the phase loop already uses all 128 (kept in registers they
// spilled into the loop).
struct MixTile {
    uint32_t k, j, tile;
};

__device__ __forceinline__ void mix_tile(const MixArgs &A, const MixStream &S, const MixTile &it,
                                         unsigned char *smem_raw, Partial *red, float2 *ubuf,
                                         uint4 (*s_ops)[MAX_PHASE_UNITS], uint32_t *s_flag) {
    float2 *sm = reinterpret_cast<float2 *>(smem_raw);
    if (threadIdx.x == 0) {
        const MixTraj &T = S.trajs[it.k];
        *s_flag = mix_wait(S.slot_done + T.slot, T.base + (uint32_t)((int)it.j - T.start) * S.tiles,
                           A.stall_extra, A.wait_limit, A.err);
    }
    __syncthreads();  // thread 0's acquire load, then the barrier, order the tile loads after it
    if (!*s_flag) return;
    const int t = S.t;
    Amps v;
    const uint32_t *ev, *ev_end;
    {
        const uint32_t k = it.k, j = it.j;
        const MixTraj &T = S.trajs[k];
        const uint64_t N = 1ull << S.n;
        const bool from_cache = (int)j == T.start;
        const float2 *src = from_cache ? S.cache + (size_t)S.cache_slot[j] * N : S.work + (size_t)T.slot * N;
        // the working slot was written by other CTAs of this launch: read it through L2
        load_tile<true>(v, src, tile_at((uint32_t)tile_base(S.passes[j].rest_mask, it.tile), S.passes[j].offs, t, S.c,
                                        threadIdx.x, 0u));
        // this pass's events: binary search for the first key at or after the pass's first gate
        const uint32_t *lo = S.keys + S.offsets[T.tr], *hi_ = S.keys + S.offsets[T.tr + 1];
        ev_end = hi_;
        const uint32_t key_lo = S.passes[j].gb << 3;
        while (lo < hi_) {
            const uint32_t *mid = lo + (hi_ - lo) / 2;
            if (*mid < key_lo) lo = mid + 1;
            else hi_ = mid;
        }
        ev = lo;
    }
    TileCtx c;
    c.m = c.z = 0;
    c.gp = 0;
    c.tid = threadIdx.x;
    c.nthr = blockDim.x;
    set_phase(c, load_set(t), t);
    uint32_t next = ev < ev_end ? *ev : NO_EVENT;
    {
        const uint32_t pb = S.passes[it.j].pb;
        if (pb < S.passes[it.j].pe)
            stage_units(s_ops[0], S.prog + S.ph_pg[pb], S.ph_pg[pb + 1] - S.ph_pg[pb], threadIdx.x, blockDim.x);
    }
    for (uint32_t ph = S.passes[it.j].pb, buf = 0; ph < S.passes[it.j].pe; ++ph, buf ^= 1u) {
        stage_wait();
        if (ph + 1 < S.passes[it.j].pe)
            stage_units(s_ops[buf ^ 1u], S.prog + S.ph_pg[ph + 1], S.ph_pg[ph + 2] - S.ph_pg[ph + 1], threadIdx.x,
                        blockDim.x);
        const uint32_t R = S.ph_R[ph];
        if (R != c.R) remap<true>(v, sm, c, R, t);
        run_prog(v, c, s_ops[buf], s_ops[buf] + (S.ph_pg[ph + 1] - S.ph_pg[ph]), S.mats, sm, ubuf, t, ev, ev_end, next,
                 S.evs);
    }
    finish_tile(v, sm, c, S.passes[it.j].frame, t);
    const uint32_t k = it.k, j = it.j;
    const MixTraj &T = S.trajs[k];
    const uint64_t N = 1ull << S.n;
    const LoadAt at = tile_at((uint32_t)tile_base(S.passes[j].rest_mask, it.tile), S.passes[j].offs, t, S.c, c.tid, c.m);
    const bool scored = (int)j == T.end;
    if (scored) {
        const float2 *ref = S.ref_cache + (size_t)S.cache_slot[j + 1] * N;
        Partial acc = empty_partial();
        score_registers(acc, S.crit, v, ref, at);
        acc = group_reduce_partial(acc, red, MIX_THREADS);
        if (threadIdx.x == 0) S.partials[(size_t)k * S.tiles + it.tile] = acc;
    } else {
        store_tile(v, S.work + (size_t)T.slot * N, at);
    }
    // publish: the barrier orders every thread's stores before thread 0's fence and
    // counter increments (the release the waiting CTAs acquire)
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(S.slot_done + T.slot, 1u);
        *s_flag = scored && atomicAdd(S.traj_done + k, 1u) == S.tiles - 1 ? 2u : 1u;
    }
    __syncthreads();
    if (*s_flag != 2u) return;
    // last tile of the scored pass: the trajectory's partials added in the order of
    // finish_partials_kernel, so the score equals the one of the per-pass launches
    __threadfence();
    Partial acc = empty_partial();
    for (uint32_t i = threadIdx.x; i < S.tiles; i += blockDim.x) {
        const Partial q = ld_partial_cg(S.partials + (size_t)k * S.tiles + i);
        acc.a += q.a;
        acc.b += q.b;
        argmax_merge(acc.maxp, acc.idx, q.maxp, q.idx);
    }
    acc = block_reduce_partial(acc, red);
    if (threadIdx.x == 0) {
        const double sc = finish_score(S.crit, acc);
        S.score[T.tr] = sc;
        if (S.pass_flags) S.pass_flags[T.tr] = sc >= S.crit.threshold;
    }
}

__global__ void __launch_bounds__(MIX_THREADS, 2) mix_kernel(const __grid_constant__ MixArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned long long s_i;
    __shared__ uint32_t s_u, s_flag;
    __shared__ double s_val;
    __shared__ Partial red[MIX_THREADS / 32];
    __shared__ float2 ubuf[8][16];
    __shared__ uint4 s_ops[2][MAX_PHASE_UNITS];
    // the current streaming circuit's descriptor: read from shared memory in the phase loop
    // instead of being held in registers (the loop already uses all 128)
    __shared__ MixStream s_stream;
    __shared__ uint32_t s_stream_idx;
    __shared__ MixTile s_tile;
    if (threadIdx.x == 0) s_u = 0, s_stream_idx = ~0u;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_i = ld_acquire_u32(a.err) ? a.n_sub : atomicAdd(a.counter, 1ull);
        __syncthreads();
        const unsigned long long i = s_i;
        if (i >= a.n_sub) return;
        if (threadIdx.x < 32) {
            const uint32_t u = mix_find_unit(a.unit_end, a.n_units, s_u, i);
            if (threadIdx.x == 0) s_u = u;
        }
        __syncthreads();
        const uint32_t u = s_u;
        const MixUnit un = a.units[u];
        const uint32_t sub = (uint32_t)(i - (u ? a.unit_end[u - 1] : 0ull));
        if (un.kind == MIX_REF) {
            mix_ref(a.refs[un.idx], sub, red, &s_flag, &s_val);
        } else if (un.kind == MIX_SMALL) {
            const BatchItem it = a.items[un.idx];
            mix_small(a.smalls[it.circuit], it, a.ids, reinterpret_cast<float2 *>(smem_raw));
        } else if (un.kind == MIX_RES) {
            const BatchItem it = a.items[un.idx];
            mix_res(it, a.rcircs[it.circuit], a.ids, smem_raw, red, ubuf, s_ops);
        } else {
            if (threadIdx.x == 0) {
                if (s_stream_idx != un.idx) {
                    s_stream = a.streams[un.idx];
                    s_stream_idx = un.idx;
                }
                s_tile = MixTile{un.a, un.b, sub};
            }
            __syncthreads();
            mix_tile(a, s_stream, s_tile, smem_raw, red, ubuf[0], s_ops, &s_flag);
        }
    }
}

void launch_mix(const MixArgs &a, double bytes, double flops, double smem_bytes, cudaStream_t st) {
    if (!a.n_sub) return;
    ProfScope ps_(ARSO_K_MIX, bytes, st, flops, smem_bytes);
    const size_t smem = (size_t(1) << 13) * sizeof(float2);
    static std::atomic<unsigned long long> set_for{0};  // the context whose attribute was set last
    if (const unsigned long long id = context_id(); set_for.load() != id) {
        ARSO_CUDA(cudaFuncSetAttribute(mix_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        set_for.store(id);
    }
    int per_sm = 1, dev = 0, sms = 152;
    ARSO_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mix_kernel, MIX_THREADS, smem));
    ARSO_CUDA(cudaGetDevice(&dev));
    ARSO_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const unsigned grid = (unsigned)std::min<uint64_t>(a.n_sub, (uint64_t)std::max(per_sm, 1) * sms);
    mix_kernel<<<grid, MIX_THREADS, smem, st>>>(a);
    ARSO_CUDA(cudaGetLastError());
}

// Raise the dynamic shared-memory limit of the pass kernels once a context, before any
// launch (and outside stream capture).
static const auto pass_128 = pass_rb_kernel<128, 5>;  // 96 registers, five CTAs per SM
static const auto pass_256 = pass_rb_kernel<256, 3>;  // 80 registers, three CTAs per SM
static const auto pass_256_wide = pass_rb_kernel<256, 2>;  // 128 registers, two
static const auto pass_512 = pass_rb_kernel<512, 1>;
void prepare_pass_rb() {
    static std::atomic<unsigned long long> set_for{0};  // the context whose attributes were set last
    const unsigned long long id = context_id();
    if (set_for.load() == id) return;
    const int tile = (1 << MAX_TILE_QUBITS) * (int)sizeof(float2);
    ARSO_CUDA(cudaFuncSetAttribute(pass_128, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 256));
    ARSO_CUDA(cudaFuncSetAttribute(pass_256, cudaFuncAttributeMaxDynamicSharedMemorySize, 256 * 256));
    ARSO_CUDA(cudaFuncSetAttribute(pass_256_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, 256 * 256));
    ARSO_CUDA(cudaFuncSetAttribute(pass_512, cudaFuncAttributeMaxDynamicSharedMemorySize, tile));
    ARSO_CUDA(cudaFuncSetAttribute(pass_tensor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   tile + 2 * (int)TP_IMAGE_BYTES));
    set_for.store(id);
}

// Tiles of up to 2^12 amplitudes run in 128-thread CTAs (small tiles several side by side),
// 2^13 in 256 and 2^14 in 512, each compiled for the registers that fill the SM. Measured
// (device time of all pass launches): 12-qubit tiles, 24-qubit brickwork, 177 trajectories:
// five 128-thread CTAs 342 ms, four 353, two tiles in a 256-thread CTA 353 (three per SM) or
// 376 (two); 13-qubit tiles: three CTAs per SM 6.53 ms against 6.87 with two (16-qubit
// brickwork, 2,000 trajectories) and 3.12 against 3.41 (20-qubit adder, 500); both sides
// before the fused runs and the z mask (305 ms, 6.0 ms and 1.7 ms since).
// A full one-qubit matrix does not fit 80 registers: its constants and products spill. Passes
// of 13-qubit tiles with more of them than one gate in 32 take two CTAs per SM; the single ones
// that restore a frame's scale, at most one gate in 80, do not (17 qubits, 400 gates, 200
// trajectories, matrices that have no frame form: 8.72 ms with three CTAs, 3.59 with two; one
// such gate in eleven: 2.36 and 2.08).
void launch_pass_rb(const PassArgs &a, bool last, uint32_t slots, double bytes, cudaStream_t st, double flops,
                    double smem_bytes) {
    ProfScope ps_(last && !a.store_last ? ARSO_K_PASS_LAST : ARSO_K_PASS, bytes, st, flops, smem_bytes);
    prepare_pass_rb();
    const uint32_t tiles = 1u << (a.n - a.t);
    const uint32_t nt = 1u << (a.t - REG_BITS);
    const size_t smem = (size_t(1) << a.t) * sizeof(float2);
    if (a.ph_t) {
        ARSO_REQUIRE(a.t >= 12 && a.t <= MAX_TILE_QUBITS, "tensor phases need 12-14-qubit tiles");
        pass_tensor_kernel<<<dim3(tiles, slots), nt, smem + 2 * TP_IMAGE_BYTES, st>>>(a);
    } else if (nt == 512) {
        pass_512<<<dim3(tiles, slots), nt, smem, st>>>(a);
    } else if (nt == 256 && a.wide) {
        pass_256_wide<<<dim3(tiles, slots), nt, smem, st>>>(a);
    } else if (nt == 256) {
        pass_256<<<dim3(tiles, slots), nt, smem, st>>>(a);
    } else {
        const uint32_t groups = std::min<uint32_t>(tiles, 128 / nt);
        pass_128<<<dim3(tiles / groups, slots), nt * groups, smem * groups, st>>>(a);
    }
    ARSO_CUDA(cudaGetLastError());
}

}  // namespace arso
