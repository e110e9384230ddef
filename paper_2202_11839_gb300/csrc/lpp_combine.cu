// k-space combination and FP64 shell sums (Sec. 3.1.2 estimators).
//
// A batch grid Z holds two real fields packed as Z = a + i b: either the two
// interlaced sub-grids of one field, or two different fields.  Their DFTs are
// recovered exactly from the pair of modes (m, -m):
//   A(m) = (Z(m) + conj Z(-m)) / 2,   B(m) = -i (Z(m) - conj Z(-m)) / 2,
//   A(-m) = conj A(m),  B(-m) = conj B(m).
// Interlaced fields become F = (A + e^{-i pi (fx+fy+fz)/n} B) / 2, and every field is
// divided by the assignment window prod_a sinc^p(pi f_a / n) when compensation is on.
//
// A lane owns the up to four mode pairs (+-fx, +-fy, fz) with one |k|: they share the shell, the
// window, Q_L^m(z) and, up to signs, (x + i y)^m.  A warp takes items of 32 consecutive |fx|
// of one (|fy|, fz), so |k| grows monotonically along the warp and equal shells form
// contiguous lane runs.  The lanes' products are reduced by a segmented scan; the lane that ends
// a segment adds it to the warp's own compensated (two-float) or FP64 accumulators in shared
// memory (every shell occurs in one segment of an item: no atomics, no block barrier), which
// the CTA adds to the global FP64 shell sums once at the end.
//
// The channels of one moment enter its shell sums only through sum_n Y_Ln(khat) F_n(k), and
// unpacking, interlacing phase, window and partner are linear in the packed values, so a mode
// pair first contracts its packed values with the harmonics (a run of channels: two real
// multiply-adds per value) and unpacks, phases, multiplies by the partner and reduces once per
// run instead of once per channel.
#include "lpp_internal.h"
#include "lpp_kernels.h"
#include "lpp_reduce.cuh"
#include "lpp_ylm.cuh"

#include <algorithm>

namespace lpp {

// k-space field at m and -m for sub-field `sub` of a slot from its packed values zm, zp: iw the
// inverse window at m and -m, ph the interlacing phase at m, whose mirror is ps conj(ph)
// (ps = -1 for an odd number of indices at the Nyquist frequency, else 1).
template <typename T>
__device__ __forceinline__ void field_of(c2<T> zm, c2<T> zp, int sub, int interlace, T iw, c2<T> ph, T ps, c2<T>& Fm,
                                         c2<T>& Fp) {
    const T h = (T)0.5;
    const c2<T> A = mk<T>(h * (zm.x + zp.x), h * (zm.y - zp.y));
    const c2<T> B = mk<T>(h * (zm.y + zp.y), -h * (zm.x - zp.x));   // -i (zm - conj zp) / 2
    if (interlace) {
        const c2<T> pb = cmul<T>(ph, B);
        Fm = cscale<T>(cadd<T>(A, pb), h * iw);
        Fp = cscale<T>(cconj<T>(cadd<T>(A, cscale<T>(pb, ps))), h * iw);
    } else {
        const c2<T> X = sub ? B : A;
        Fm = cscale<T>(X, iw);
        Fp = cscale<T>(cconj<T>(X), iw);
    }
}

// One (|fx|, |fy|, fz) of a lane: what its four mode pairs share.
template <typename T>
struct Lane {
    Azimuth<T> az;   // of (|kx|, |ky|) / |k|
    T kz, iw, ps;    // fz / |k|, inverse window, mirror sign of the phase (field_of)
    int nyq;         // bits 0, 1, 2: x, y, z sit at the Nyquist frequency (the mirror keeps them)
};

// For the pairs (+|fx|, fy) and (-|fx|, fy), q = 0, 1 (fy < 0: yneg): sum_n Y_n(khat) Z_n(m) and
// sum_n Y_n(khat) Z_n(-m) of a run's channels for the real (s[q][0], s[q][1]) and imaginary
// (s[q][2], s[q][3]) kernel parts; with two fields per grid the sums are those of the unpacked
// fields X at m (s[q][0] and s[q][2] alone).  mirror: with the harmonics of the mirror's own
// vector, which differs from -k in the sign of the Nyquist components.  on[q]: the lane owns
// the pair; im[q], ip[q] its indices.  A unit is the up to four channels n = +-m x (real,
// imaginary part) that share Q_L^m: their packed values are loaded together, ahead of the
// harmonic.
template <typename T>
__device__ __forceinline__ void contract_run(const CombineArgs<T>& a, const CombineRun& run, const Lane<T>& c,
                                             bool yneg, bool mirror, const bool on[2], const unsigned im[2],
                                             const unsigned ip[2], c2<T> s[2][4]) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) s[q][k] = mk<T>((T)0, (T)0);
    for (int ui = run.u0; ui < run.u1; ++ui) {
        const CombineUnit<T>& u = a.unit[ui];
        c2<T> zm[4][2], zp[4][2];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const c2<T>* g = a.grids + (long long)max(u.slot[k], 0) * a.grid_stride;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                zm[k][q] = zp[k][q] = mk<T>((T)0, (T)0);
                if (on[q] && u.slot[k] >= 0) {
                    zm[k][q] = g[im[q]];
                    zp[k][q] = g[ip[q]];
                }
            }
        }
        T yc, ys;
        ylm_pair<T>(u.L, u.m, c.az, c.kz, yc, ys);
        yc *= u.ynorm;
        ys *= u.ynorm;
        const bool odd = u.m & 1;
        if (yneg) ys = -ys;
        if (mirror) {
            // Y(-k') = Y(k') (L even) with k' = k but for the signs of its Nyquist components
            const int nx = c.nyq & 1, ny = (c.nyq >> 1) & 1, nz = c.nyq >> 2;
            if (odd && (nx ^ nz)) { yc = -yc; ys = -ys; }
            if (nx ^ ny) ys = -ys;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (u.slot[k] < 0) continue;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                // (-x + i y)^m = (-1)^m conj (x + i y)^m
                const T yk = (k >> 1) ? ((q == 1 && !odd) ? -ys : ys) : ((q == 1 && odd) ? -yc : yc);
                c2<T> vm = zm[k][q];
                const c2<T> vp = zp[k][q];
                const int o = 2 * (k & 1);
                if (a.interlace) {
                    s[q][o + 1] = mk<T>(s[q][o + 1].x + yk * vp.x, s[q][o + 1].y + yk * vp.y);
                } else {
                    const T h = (T)0.5;
                    // A = (zm + conj zp) / 2 or B = -i (zm - conj zp) / 2
                    vm = u.sub[k] ? mk<T>(h * (vm.y + vp.y), -h * (vm.x - vp.x))
                                  : mk<T>(h * (vm.x + vp.x), h * (vm.y - vp.y));
                }
                s[q][o] = mk<T>(s[q][o].x + yk * vm.x, s[q][o].y + yk * vm.y);
            }
        }
    }
}

// Walks the work list with 8 warps per CTA.  PARTNER: unpack the partner fields and sum their
// own products instead of the channels.
//
// What bounds it: the latency of the scattered rows (both members of every pair, 16 loads in
// flight per lane; DRAM at 37% of its peak) with 16 warps per SM; instruction issue at 42%.
// Eight grids of 256^3 to k = 0.995 k_Ny: 0.40 -> 0.23 ms (one mode pair and one reduction per
// lane and channel before); 1.5 M galaxies on 512^3: 7.1 -> 3.9 ms for the 17 combines.
constexpr int kCombineWarps = 8;
template <typename T>
constexpr int combine_ctas() { return sizeof(T) == 4 ? 2 : 1; }

template <typename T, bool PARTNER>
__global__ void __launch_bounds__(32 * kCombineWarps, combine_ctas<T>()) k_combine(CombineArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n;
    const int nb = a.nb;
    const int nacc = PARTNER ? 2 : a.n_runs;
    const int E = nacc * nb * 2;
    constexpr int W = Owned<T>::words, NW = kCombineWarps;
    T* own = reinterpret_cast<T*>(smem_raw);                       // [NW][words][E] accumulators per warp
    c2<T>* ph = reinterpret_cast<c2<T>*>(own + NW * E * W);        // [n]  (E is even)
    T* iw = reinterpret_cast<T*>(ph + n);                          // [n]
    int* thr = reinterpret_cast<int*>(iw + n);                     // [nb+1]

    const int tid = threadIdx.x;
    constexpr int nthr = 32 * NW;
    const int warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < NW * E * W; i += nthr) own[i] = (T)0;
    for (int i = tid; i < n; i += nthr) { iw[i] = a.inv_w[i]; ph[i] = a.phase[i]; }
    for (int i = tid; i <= nb; i += nthr) thr[i] = a.thr[i];
    __syncthreads();
    T* mine = own + warp * E * W;

    const int na = max(a.nk_pos, a.nk_neg) + 1, nseg = (na + 31) / 32;   // |f| values and their segments
    const int n_work = a.n_items << a.split;
    for (int wi = blockIdx.x * NW + warp; wi < n_work; wi += gridDim.x * NW) {
        // split: the pairs of +fy and of -fy by different warps
        const int it = wi >> a.split;
        const int sy0 = a.split ? wi & 1 : 0, sy1 = a.split ? sy0 : 1;
        int row, seg;
        if (a.items) {
            row = a.items[it] >> 6;
            seg = a.items[it] & 63;
        } else {
            row = it / nseg;
            seg = it - row * nseg;
        }
        const int zi = row / na;
        const int ay = row - zi * na;
        const int ax = 32 * seg + lane;
        const int z = zi <= a.nk_pos ? zi : n / 2;
        const int zp = (n - z) & (n - 1);
        const int fz = z < n / 2 ? z : z - n;
        // the shell of the lane's four pairs (contiguous along the warp)
        const int q2 = ax * ax + ay * ay + fz * fz;
        int bin = -1;
        if (ax < na && q2 > 0 && q2 >= thr[0] && q2 < thr[nb]) {
            int lo = 0, hi = nb;  // thr[lo] <= q2 < thr[hi]
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (q2 >= thr[mid]) lo = mid; else hi = mid;
            }
            bin = lo;
        }
        if (!LPP_IN_BOUNDS(bin < nb && (bin < 0 || (ax <= n / 2 && ay <= n / 2)), a.err)) bin = -1;
        if (!__any_sync(0xffffffffu, bin >= 0)) continue;
        const SegMask segm = seg_mask(bin);
        Lane<T> c;
        const T inv = bin >= 0 ? (T)1 / sqrt((T)q2) : (T)0;
        if constexpr (!PARTNER) c.az.set((T)ax * inv, (T)ay * inv);
        c.kz = (T)fz * inv;
        c.nyq = (ax == n / 2 ? 1 : 0) | (ay == n / 2 ? 2 : 0) | (fz == -n / 2 ? 4 : 0);
        c.ps = (__popc(c.nyq) & 1) ? (T)-1 : (T)1;
        const int x0 = bin >= 0 ? ax : 0;   // index of +ax (and of -ax at the Nyquist frequency)
        const int x1 = (n - x0) & (n - 1);
        c.iw = iw[x0] * iw[ay] * iw[z];
        const c2<T> phx = ph[x0];
        const bool anyq = __any_sync(0xffffffffu, bin >= 0 && c.nyq != 0);
        T dd = 0, gg = 0;
        // the pairs of +fy and of -fy: whether the lane owns those of +-fx, and their indices
        auto side = [&](int sy, bool on[2], unsigned im[2], unsigned ip[2], c2<T> phs[2]) {
            const int y = sy ? (n - ay) & (n - 1) : ay;
            const int yp = (n - y) & (n - 1);
            const bool ey = sy ? (ay >= 1 && ay <= a.nk_neg) : ay <= a.nk_pos;
            // self-conjugate planes: each pair once, from its lexicographically smaller member
            const bool half = z == zp;
            const bool row_on = bin >= 0 && ey && !(half && y > yp);
            on[0] = row_on && ax <= a.nk_pos;
            on[1] = row_on && ax >= 1 && ax <= a.nk_neg && !(half && y == yp && x1 > x0);
            const unsigned rm = ((unsigned)z * n + y) * n, rp = ((unsigned)zp * n + yp) * n;
            im[0] = rm + x0;
            ip[0] = rp + x1;
            im[1] = rm + x1;
            ip[1] = rp + x0;
            const c2<T> pyz = cmul<T>(ph[y], ph[z]);
            phs[0] = cmul<T>(phx, pyz);
            phs[1] = cmul<T>(ax == n / 2 ? phx : cconj<T>(phx), pyz);
        };
        if constexpr (PARTNER) {
            for (int sy = sy0; sy <= sy1; ++sy) {
                bool on[2];
                unsigned im[2], ip[2];
                c2<T> phs[2];
                side(sy, on, im, ip, phs);
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    if (!on[q]) continue;
                    const bool self = im[q] == ip[q];
                    auto field = [&](int slot, int sub, c2<T>& Fm, c2<T>& Fp) {
                        const c2<T>* g = a.grids + (long long)slot * a.grid_stride;
                        field_of<T>(g[im[q]], g[ip[q]], sub, a.interlace, c.iw, phs[q], c.ps, Fm, Fp);
                    };
                    // partner grids: interlaced -> G1 | G2 | D one field per grid;
                    // otherwise (G1, G2) packed in one grid, then (D, -)
                    int slot = 0;
                    if (a.has_g) {
                        c2<T> G1m, G1p, G2m, G2p;
                        field(0, 0, G1m, G1p);
                        field(a.interlace ? 1 : 0, a.interlace ? 0 : 1, G2m, G2p);
                        slot = a.interlace ? 2 : 1;
                        a.pG1[im[q]] = G1m;
                        a.pG1[ip[q]] = G1p;
                        a.pG2[im[q]] = G2m;
                        a.pG2[ip[q]] = G2p;
                        // G = G1 + i G2: the transform of the complex shear field
                        const T gr = G1m.x - G2m.y, gi = G1m.y + G2m.x;
                        gg += gr * gr + gi * gi;
                        if (!self) {
                            const T hr = G1p.x - G2p.y, hi2 = G1p.y + G2p.x;
                            gg += hr * hr + hi2 * hi2;
                        }
                    }
                    if (a.has_d) {
                        c2<T> Dm, Dp;
                        field(slot, 0, Dm, Dp);
                        if (a.pD) {   // null: the caller wants only the shell sums
                            a.pD[im[q]] = Dm;
                            a.pD[ip[q]] = Dp;
                        }
                        dd += Dm.x * Dm.x + Dm.y * Dm.y;
                        if (!self) dd += Dp.x * Dp.x + Dp.y * Dp.y;
                    }
                }
            }
            warp_own_add<T>(dd, (T)0, bin, segm, mine, E);
            warp_own_add<T>(gg, (T)0, bin, segm, mine + 2 * nb, E);
        } else {
            for (int ri = 0; ri < a.n_runs; ++ri) {
                const CombineRun& run = a.run[ri];
                T tre = 0, tim = 0;
                for (int sy = sy0; sy <= sy1; ++sy) {
                    bool on[2];
                    unsigned im[2], ip[2];
                    c2<T> phs[2];
                    side(sy, on, im, ip, phs);
                    if (!__any_sync(0xffffffffu, on[0] || on[1])) continue;   // warp-uniform
                    // partner: delta(-k) = conj D; gamma*(-k) = conj G1 - i conj G2;
                    // gamma(-k) = conj G1 + i conj G2
                    c2<T> Pm[2], Pp[2];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        Pm[q] = Pp[q] = mk<T>((T)0, (T)0);
                        if (!on[q]) continue;
                        if (run.kind == KIND_CROSS || run.kind == KIND_DENS) {
                            Pm[q] = cconj<T>(a.pD[im[q]]);
                            Pp[q] = cconj<T>(a.pD[ip[q]]);
                        } else {
                            const c2<T> G1m = a.pG1[im[q]], G1p = a.pG1[ip[q]], G2m = a.pG2[im[q]], G2p = a.pG2[ip[q]];
                            const T s = run.kind == KIND_PLUS ? (T)-1 : (T)1;
                            // conj(G1) + s i conj(G2)
                            Pm[q] = mk<T>(G1m.x + s * G2m.y, -G1m.y + s * G2m.x);
                            Pp[q] = mk<T>(G1p.x + s * G2p.y, -G1p.y + s * G2p.x);
                        }
                        if (im[q] == ip[q]) Pp[q] = mk<T>((T)0, (T)0);   // its own mirror: counted once
                    }
                    // where the mirror is -k, an even-degree harmonic (every L here is even) takes the
                    // same value at both members of the pair; Nyquist lanes contract their mirror
                    // with its own harmonics in a second pass
                    for (int pass = 0; pass < (anyq ? 2 : 1); ++pass) {
                        c2<T> S[2][4];
                        contract_run<T>(a, run, c, sy != 0, pass == 1, on, im, ip, S);
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            // X = F_re + i F_im at m and at the mirror
                            c2<T> Xm, Xp;
                            if (a.interlace) {
                                c2<T> Hm, Hp;
                                field_of<T>(S[q][0], S[q][1], 0, 1, c.iw, phs[q], c.ps, Xm, Xp);
                                field_of<T>(S[q][2], S[q][3], 0, 1, c.iw, phs[q], c.ps, Hm, Hp);
                                Xm = mk<T>(Xm.x - Hm.y, Xm.y + Hm.x);
                                Xp = mk<T>(Xp.x - Hp.y, Xp.y + Hp.x);
                            } else {
                                Xm = mk<T>(c.iw * (S[q][0].x - S[q][2].y), c.iw * (S[q][0].y + S[q][2].x));
                                Xp = mk<T>(c.iw * (S[q][0].x + S[q][2].y), c.iw * (S[q][2].x - S[q][0].y));
                            }
                            const c2<T> tm = cmul<T>(Xm, Pm[q]), tp = cmul<T>(Xp, Pp[q]);
                            if (pass == 0) {
                                tre += tm.x;
                                tim += tm.y;
                            }
                            if ((c.nyq != 0) == (pass == 1)) {
                                tre += tp.x;
                                tim += tp.y;
                            }
                        }
                    }
                }
                warp_own_add<T>(tre, tim, bin, segm, mine + ri * 2 * nb, E);
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < E; i += nthr) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < NW; ++w) v += Owned<T>::value(own + w * E * W + i, own + w * E * W + (W - 1) * E + i);
        if (v != 0.0) {
            const int ci = i / (2 * nb);
            const int rem = i - ci * 2 * nb;
            const int row_out = PARTNER ? (ci == 0 ? a.row_dd0 : a.row_plus0) : a.run[ci].out_row;
            if (row_out >= 0) atomicAdd(a.out + (long long)row_out * 2 * nb + rem, v);
        }
    }
}

template <typename T, bool PARTNER>
static cudaError_t launch_combine_mode(const CombineArgs<T>& a, int n_sm, cudaStream_t st) {
    const int nacc = PARTNER ? 2 : a.n_runs;
    const int E = nacc * a.nb * 2;
    const size_t smem = (size_t)kCombineWarps * E * Owned<T>::words * sizeof(T) +
                        (size_t)a.n * (sizeof(c2<T>) + sizeof(T)) + (size_t)(a.nb + 1) * sizeof(int);
    CombineArgs<T> c = a;
    const int na = std::max(a.nk_pos, a.nk_neg) + 1;
    if (c.items == nullptr) c.n_items = a.nzi * na * ((na + 31) / 32);   // every segment of every row
    // one resident wave (the launch bounds' CTAs per SM)
    cudaError_t e = allow_shared(k_combine<T, PARTNER>, kMaxShared);
    if (e != cudaSuccess) return e;
    // lists that leave half of the resident warps idle take the two signs of fy as separate items
    // (64^3 to k = 0.8 k_Ny: 530 items for 2432 warps; an estimate 1.43 -> 1.37 ms)
    const int warps = n_sm * combine_ctas<T>() * kCombineWarps;
    c.split = 2 * c.n_items <= warps ? 1 : 0;
    const int work = c.n_items << c.split;
    const int blocks = std::max(1, std::min(n_sm * combine_ctas<T>(), (work + kCombineWarps - 1) / kCombineWarps));
    k_combine<T, PARTNER><<<blocks, 32 * kCombineWarps, smem, st>>>(c);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_combine(const CombineArgs<T>& a, int n_sm, cudaStream_t st) {
    return a.partner_mode ? launch_combine_mode<T, true>(a, n_sm, st) : launch_combine_mode<T, false>(a, n_sm, st);
}

void combine_items(int n, int nk_pos, int nk_neg, int nzi, int q_max, std::vector<int>& items) {
    items.clear();
    const int na = std::max(nk_pos, nk_neg) + 1;
    for (int zi = 0; zi < nzi; ++zi) {
        const int z = zi <= nk_pos ? zi : n / 2;
        const long long fz = z < n / 2 ? z : z - n;
        for (int ay = 0; ay < na; ++ay) {
            const long long rem = (long long)q_max - (long long)ay * ay - fz * fz;
            for (int x0 = 0; x0 < na && (long long)x0 * x0 < rem; x0 += 32) items.push_back((zi * na + ay) << 6 | x0 / 32);
        }
    }
}

template cudaError_t launch_combine<float>(const CombineArgs<float>&, int, cudaStream_t);
template cudaError_t launch_combine<double>(const CombineArgs<double>&, int, cudaStream_t);

}  // namespace lpp
