// FP32 pencil FFT on pairs of pencils with packed arithmetic (internal).
//
// With one pencil per thread the y and z passes were bound by instruction issue and by loads in
// flight, not by DRAM.  Here a thread owns two neighbouring pencils: every value is a pair (re0, re1)
// or (im0, im1) in a 64-bit register, added and multiplied by the packed FP32 instructions of sm_100
// (add/sub/mul/fma.f32x2: one issue slot for two results, the same FP32 rate), a global access is
// 16 bytes instead of 8, a shared-memory access 16 bytes for two pencils, and a twiddle is read once
// for both.  The tile holds N rows of W / 2 pairs {re0, re1, im0, im1}; eight consecutive lanes read
// 128 contiguous bytes of one row, so no padding is needed.  Same factorisation and order of
// operations as lpp_fft_dev.cuh.
//
// Eight grids of 256^3 to k = 0.995 k_Ny: y pass 414 -> 383 us, z pass 368 -> 320 us; with the bounds of
// ColumnBound and tiles of 16 columns 320 us (1.9 GB, 6.0 TB/s: bound by DRAM) and 246 us (1.4 GB,
// 5.7 TB/s).  512^3 stays bound by the latency of its five steps per tile, 32 warps per SM (y pass 454
// us, z pass 446 us for eight grids of a survey).  Grids below 64^3 keep one pencil per thread: their
// passes take a few microseconds and have too few pencils to pair.
#pragma once

#include "lpp_fft_dev.cuh"

namespace lpp {

typedef unsigned long long f2x;   // two floats

__device__ __forceinline__ f2x pk2(float a, float b) {
    f2x r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpk2(f2x v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2x add2(f2x a, f2x b) {
    f2x r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2x sub2(f2x a, f2x b) {
    f2x r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2x mul2(f2x a, f2x b) {
    f2x r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2x fma2(f2x a, f2x b, f2x c) {
    f2x r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// A complex value of two pencils; as stored in the tile (16 bytes).
struct __align__(16) cpair {
    f2x re, im;
};
__device__ __forceinline__ cpair padd(cpair a, cpair b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ cpair psub(cpair a, cpair b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
// v w, the twiddle stored as {(wx, wx), (-wy, -wy)}
__device__ __forceinline__ cpair pmul(cpair v, cpair w) {
    return {fma2(v.im, w.im, mul2(v.re, w.re)), sub2(mul2(v.im, w.re), mul2(v.re, w.im))};
}
// v f of two complex values as they are
__device__ __forceinline__ cpair pmul_plain(cpair v, cpair f) {
    return {sub2(mul2(v.re, f.re), mul2(v.im, f.im)), fma2(v.re, f.im, mul2(v.im, f.re))};
}

__device__ __forceinline__ void pdft4(cpair* v) {
    const cpair a0 = padd(v[0], v[2]), a1 = psub(v[0], v[2]);
    const cpair b0 = padd(v[1], v[3]), b1 = psub(v[1], v[3]);
    v[0] = padd(a0, b0);
    v[2] = psub(a0, b0);
    // a1 -+ i b1
    v[1] = {add2(a1.re, b1.im), sub2(a1.im, b1.re)};
    v[3] = {sub2(a1.re, b1.im), add2(a1.im, b1.re)};
}

__device__ __forceinline__ void pdft2(cpair* v) {
    const cpair a = v[0];
    v[0] = padd(a, v[1]);
    v[1] = psub(a, v[1]);
}

__device__ __forceinline__ void pdft8(cpair* v) {
    cpair e[4] = {v[0], v[2], v[4], v[6]};
    cpair o[4] = {v[1], v[3], v[5], v[7]};
    pdft4(e);
    pdft4(o);
    const f2x r = pk2(0.70710678118654752440f, 0.70710678118654752440f);
    const cpair t1 = {mul2(add2(o[1].re, o[1].im), r), mul2(sub2(o[1].im, o[1].re), r)};   // * (1 - i)/sqrt2
    const cpair t3 = {mul2(sub2(o[3].im, o[3].re), r), mul2(add2(o[3].re, o[3].im), r)};   // * (-1 - i)/sqrt2, im negated
    v[0] = padd(e[0], o[0]);
    v[4] = psub(e[0], o[0]);
    v[1] = padd(e[1], t1);
    v[5] = psub(e[1], t1);
    v[2] = {add2(e[2].re, o[2].im), sub2(e[2].im, o[2].re)};   // o2 * (-i) = (im, -re)
    v[6] = {sub2(e[2].re, o[2].im), add2(e[2].im, o[2].re)};
    v[3] = {add2(e[3].re, t3.re), sub2(e[3].im, t3.im)};
    v[7] = {sub2(e[3].re, t3.re), add2(e[3].im, t3.im)};
}

// Pass shape: W pencils (128-byte segments; 64 bytes at n = 1024), half as many pencil pairs; one
// butterfly slot (eight values of a pair: 32 registers) per thread, as two would spill at the 64
// registers of 1024 threads per SM.  Small CTAs overlap one tile's stores with another's loads: at
// 256^3, 32 -> 16 columns, y pass 375 -> 320 us, z pass 280 -> 246 us (at 512^3, 16 -> 8 columns, 454 ->
// 465 us: half segments); 64^3 keeps 32 (16: y pass 5.1 -> 5.5 us, its persistent CTAs get no work).
template <int LOGN>
struct PairShape {
    static constexpr int N = 1 << LOGN;
    static constexpr int W = LOGN == 6 ? 32 : (LOGN < 10 ? 16 : 8);
    static constexpr int CP = W / 2;
    static constexpr int LOGC = ilog2(CP);
    static constexpr int IPT = 1;
    static constexpr int THREADS = CP * N / (8 * IPT);
    static constexpr int PER = 8 * IPT;   // operands per thread
    static constexpr size_t SMEM = (size_t)(N + N * CP) * sizeof(cpair);
    // resident CTAs per SM that the registers are budgeted for: 1024 threads (shared memory allows as many)
    static constexpr int MINB = 1024 / THREADS;
};

// FFT of length N along every pencil pair of the tile with operands from load(b, e) in the first stage
// (point e, operand b as in lead_row) and results to store(e, value) in the last; c: the
// thread's pair, u: its first butterfly slot.  The caller reuses the tile only after a barrier.
template <int LOGN, class Load, class Store>
__device__ __forceinline__ void fft_pairs_io(cpair* tile, int c, int u, const cpair* tw, Load&& load, Store&& store) {
    using S = PairShape<LOGN>;
    constexpr int N = S::N, IPT = S::IPT, LD = S::CP, US = N / (8 * IPT), R = LeadRadix<LOGN>::R, Q = 8 / R;
    cpair v[IPT][8];
#pragma unroll
    for (int s = 0; s < IPT; ++s)
#pragma unroll
        for (int k = 0; k < 8; ++k) v[s][k] = load(s * 8 + k, lead_row<LOGN, IPT>(u, s * 8 + k));
#pragma unroll
    for (int s = 0; s < IPT; ++s)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int j = u + s * US + q * (N / 8);
            if (R == 8) pdft8(v[s] + q * R);
            else if (R == 4) pdft4(v[s] + q * R);
            else pdft2(v[s] + q * R);
            cpair* dst = tile + j * R * LD + c;
#pragma unroll
            for (int r = 0; r < R; ++r) dst[r * LD] = v[s][q * R + r];
        }
    __syncthreads();
    // radix-8 stages in the tile
#pragma unroll
    for (int ns = R; ns < N / 8; ns *= 8) {
        const cpair* src = tile + u * LD + c;
#pragma unroll
        for (int s = 0; s < IPT; ++s)
#pragma unroll
            for (int r = 0; r < 8; ++r) v[s][r] = src[(s * US + r * (N / 8)) * LD];
        __syncthreads();
#pragma unroll
        for (int s = 0; s < IPT; ++s) {
            const int j = u + s * US, jm = j & (ns - 1), step = jm * (N / (ns * 8));
#pragma unroll
            for (int r = 1; r < 8; ++r) v[s][r] = pmul(v[s][r], tw[step * r]);
            pdft8(v[s]);
            cpair* dst = tile + ((j - jm) * 8 + jm) * LD + c;
#pragma unroll
            for (int r = 0; r < 8; ++r) dst[r * ns * LD] = v[s][r];
        }
        __syncthreads();
    }
    const cpair* src = tile + u * LD + c;
#pragma unroll
    for (int s = 0; s < IPT; ++s)
#pragma unroll
        for (int r = 0; r < 8; ++r) v[s][r] = src[(s * US + r * (N / 8)) * LD];
#pragma unroll
    for (int s = 0; s < IPT; ++s) {
        const int j = u + s * US;
#pragma unroll
        for (int r = 1; r < 8; ++r) v[s][r] = pmul(v[s][r], tw[j * r]);
        pdft8(v[s]);
#pragma unroll
        for (int r = 0; r < 8; ++r) store(j + r * (N / 8), v[s][r]);
    }
}

}  // namespace lpp
