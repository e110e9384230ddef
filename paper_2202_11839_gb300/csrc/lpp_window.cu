// Window multipoles Q_l(s) (Eq. windowQ_ell with the endpoint line of sight d = x).
//
// With the addition theorem L_l(s.x) = 4 pi / (2l+1) sum_n Y_{l,n}(s) Y_{l,n}(x) (real
// harmonics), Q_l(s) = 4 pi < sum_n Y_{l,n}(s) C_n(s) >_shell / I with the
// cross-correlations C_n(s) = int_x A_n(x) W(x+s) of A_n = W Y_{l,n}(x) and W.  Each C_n is
// IFFT[conj(A_n(k)) W(k)]; two real fields share one complex grid Z = A_a + i A_b.  For real fields
// conj(A_a(k)) + i conj(A_b(k)) = Z(-k), so C_a + i C_b = IFFT[Z(-k) W(k)] = FFT[Z(k) conj(W(k))] / n^3:
// the z pass of Z's transform multiplies its results by conj(W) (deconvolved twice) and a second
// forward transform returns both correlations at once.  (As a kernel of its own over the pairs (k, -k)
// the products took 1.44 of 12.5 ms of kernels of a 256^3 call.)
#include "lpp_internal.h"
#include "lpp_kernels.h"
#include "lpp_reduce.cuh"
#include "lpp_ylm.cuh"

#include <algorithm>

namespace lpp {

template <typename T>
__global__ void k_window_partner(const c2<T>* __restrict__ grid, c2<T>* __restrict__ pD, const T* __restrict__ inv_w,
                                 int n) {
    const long long n3 = (long long)n * n * n;
    for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < n3;
         m += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(m % n), y = (int)((m / n) % n), z = (int)(m / ((long long)n * n));
        const T w = inv_w[x] * inv_w[y] * inv_w[z];
        pD[m] = cscale<T>(cconj<T>(grid[m]), w * w);
    }
}

template <typename T>
cudaError_t launch_window_partner(const c2<T>* grid, c2<T>* pD, const T* inv_w, int n, cudaStream_t st) {
    k_window_partner<T><<<152 * 8, 256, 0, st>>>(grid, pD, inv_w, n);
    return cudaGetLastError();
}

// Shell sums over separations.  A warp takes 32 consecutive sx >= 0 or sx < 0 of one row (sz, sy)
// of the kept cube, so that |s| grows monotonically along it.  The channels of one degree l enter
// Q_l only through sum_n Y_ln(shat) C_n(s): they are contracted separation by separation and
// reduced once per degree (a.run), into the warp's own accumulators (warp_own_add).
// (One reduction, a harmonic with divisions and block barriers per channel and row before: 3.75 ms
// of the 16 ms of kernels of a 256^3 call to 115 grid spacings.)
constexpr int kSbinWarps = 8;

template <typename T>
__global__ void __launch_bounds__(32 * kSbinWarps, sizeof(T) == 4 ? 3 : 2) k_sbin(const __grid_constant__ SbinArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n, nb = a.nb;
    const int E = a.n_runs * nb * 2;
    constexpr int W = Owned<T>::words, NW = kSbinWarps;
    T* own = reinterpret_cast<T*>(smem_raw);                 // [NW][words][E]
    int* thr = reinterpret_cast<int*>(own + NW * E * W);     // [nb+1]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < NW * E * W; i += 32 * NW) own[i] = (T)0;
    for (int i = tid; i <= nb; i += 32 * NW) thr[i] = a.thr[i];
    __syncthreads();
    T* mine = own + warp * E * W;
    const int npos = (a.ns_pos + 32) / 32, nseg = npos + (a.ns_neg + 31) / 32;
    const int items = a.nks * a.nks * nseg;
    for (int it = blockIdx.x * NW + warp; it < items; it += gridDim.x * NW) {
        const int row = it / nseg, seg = it - row * nseg;
        const int zj = row / a.nks, yj = row - zj * a.nks;
        const int z = zj <= a.ns_pos ? zj : n - (a.nks - zj);
        const int y = yj <= a.ns_pos ? yj : n - (a.nks - yj);
        const int fz = z < n / 2 ? z : z - n, fy = y < n / 2 ? y : y - n;
        const bool neg = seg >= npos;
        const int ax = neg ? 32 * (seg - npos) + lane + 1 : 32 * seg + lane;   // |sx|
        const int fx = neg ? -ax : ax;
        const int q2 = fx * fx + fy * fy + fz * fz;
        int bin = -1;
        if (ax <= (neg ? a.ns_neg : a.ns_pos) && q2 > 0 && q2 >= thr[0] && q2 < thr[nb]) {
            int lo = 0, hi = nb;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (q2 >= thr[mid]) lo = mid; else hi = mid;
            }
            bin = lo;
        }
        if (!__any_sync(0xffffffffu, bin >= 0)) continue;
        const SegMask segm = seg_mask(bin);
        const T inv = bin >= 0 ? (T)1 / sqrt((T)q2) : (T)0;
        Azimuth<T> az;
        az.set((T)fx * inv, (T)fy * inv);
        const T sz = (T)fz * inv;
        const unsigned idx = bin >= 0 ? ((unsigned)z * n + y) * n + (fx >= 0 ? fx : n + fx) : 0u;
        for (int ri = 0; ri < a.n_runs; ++ri) {
            T v = 0;
            for (int ci = a.run[ri].c0; ci < a.run[ri].c1; ci += 2) {
                // channels n = +m and -m of one degree (m = 0: one)
                const SbinChan &p = a.ch[ci], &q = a.ch[min(ci + 1, a.run[ri].c1 - 1)];
                T cp = 0, cq = 0;
                if (bin >= 0) {
                    const c2<T> u = a.grids[(long long)p.grid * a.grid_stride + idx];
                    const c2<T> w = a.grids[(long long)q.grid * a.grid_stride + idx];
                    cp = p.sub ? u.y : u.x;
                    cq = q.sub ? w.y : w.x;
                }
                const bool pair = ci + 1 < a.run[ri].c1 && q.m == -p.m && p.m != 0;
                T yc, ys;
                ylm_pair<T>(p.l, p.m < 0 ? -p.m : p.m, az, sz, yc, ys);
                v += (T)p.ynorm * (p.m < 0 ? ys : yc) * cp;
                if (pair) v += (T)q.ynorm * (q.m < 0 ? ys : yc) * cq;
                else --ci;   // one channel this time
            }
            warp_own_add<T>(v * (T)a.scale, (T)0, bin, segm, mine + ri * 2 * nb, E);
        }
    }
    __syncthreads();
    for (int i = tid; i < E; i += 32 * NW) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < NW; ++w) v += Owned<T>::value(own + w * E * W + i, own + w * E * W + (W - 1) * E + i);
        if (v != 0.0) {
            const int ri = i / (2 * nb);
            atomicAdd(a.out + (long long)a.run[ri].out_row * 2 * nb + (i - ri * 2 * nb), v);
        }
    }
}

template <typename T>
cudaError_t launch_sbin(const SbinArgs<T>& a, int n_sm, cudaStream_t st) {
    const int E = a.n_runs * a.nb * 2;
    const size_t smem = (size_t)kSbinWarps * E * Owned<T>::words * sizeof(T) + (size_t)(a.nb + 1) * sizeof(int);
    cudaError_t e = allow_shared(k_sbin<T>, kMaxShared);
    if (e != cudaSuccess) return e;
    const long long items = (long long)a.nks * a.nks * ((a.ns_pos + 32) / 32 + (a.ns_neg + 31) / 32);
    const int blocks = (int)std::max(1LL, std::min<long long>((long long)n_sm * (sizeof(T) == 4 ? 3 : 2),
                                                              (items + kSbinWarps - 1) / kSbinWarps));
    k_sbin<T><<<blocks, 32 * kSbinWarps, smem, st>>>(a);
    return cudaGetLastError();
}

template cudaError_t launch_window_partner<float>(const c2<float>*, c2<float>*, const float*, int, cudaStream_t);
template cudaError_t launch_window_partner<double>(const c2<double>*, c2<double>*, const double*, int, cudaStream_t);
template cudaError_t launch_sbin<float>(const SbinArgs<float>&, int, cudaStream_t);
template cudaError_t launch_sbin<double>(const SbinArgs<double>&, int, cudaStream_t);

}  // namespace lpp
