// Window multipoles by pair counting (Sec. 4.3: the paper measures Q_l(s) from pairs of
// random points in the footprint; Eq. windowQ_ell with the endpoint line of sight).
//
//   Q_l(b) = (2l+1) alpha^2 / (I V_b) sum_{r != r', s_rr' in b} w_r w_r' L_l(shat_rr' . xhat_r)
//
// Every unordered pair {i, j} is visited once and adds w_i w_j [L_l(shat . xhat_i) +
// L_l(shat . xhat_j)] (L_l is even, so the sign of shat does not matter).  A CTA takes a
// tile of 128 points i (one per thread) against a tile of 128 points j staged in shared
// memory; tiles (it, jt) with jt >= it cover the upper triangle, the diagonal tile keeps
// j > i only.  All sums are FP64.  The squared separation that decides the shell is formed
// with explicitly rounded operations (no fused multiply-add), and compared with the smallest
// double whose correctly rounded square root reaches the edge: the shell of every pair is
// exactly the one of the oracle's definition, without a square root per pair.
//
// The Legendre polynomials enter through the power sums p_k = y_i^k + y_j^k, k = 0 .. 4, of
// y = 2 (shat . xhat)^2 - 1 in [-1, 1]; the shells collect w w' p_k and the host forms the five
// multipoles from them.
#include "lpp_internal.h"

#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

namespace {

constexpr int kTile = 128;
constexpr int kWarps = kTile / 32;
constexpr int kEll = 5;   // l = 0, 2, 4, 6, 8, and the powers k = 0 .. 4
constexpr int kMaxShells = 256;

struct PairArgs {
    const double* pos;   // [3][n]
    const double* w;     // [n] or null
    long long n;
    int n_tiles;
    double obs[3];
    double box;          // > 0: minimal image in a periodic box of this side
    const double* thr;   // [nb + 1] thresholds on the squared separation
    double s_max;        // the last edge
    int nb;
    int copies;          // lanes' private copies of a warp's shell sums: 32, 16, 8, 4, 2 or 1
    double* out;         // [nb][5] pair sums of w w' p_k (k = 0: of w w')
};

// d minus the nearest multiple of box: box rint(d / box) with correctly rounded operations.  Away
// from the half boxes, where d / box cannot round across a tie, the multiple is read off by
// comparison (a division costs as much as the rest of the separation).
__device__ __forceinline__ double min_image(double d, double box) {
    if (box > 0.0) {
        const double a = fabs(d), h = 0.5 * box;
        double k;
        if (a < h * (1.0 - 1e-12)) k = 0.0;
        else if (a > h * (1.0 + 1e-12) && a < 1.4 * box) k = copysign(1.0, d);
        else k = rint(__ddiv_rn(d, box));
        d = __dsub_rn(d, __dmul_rn(box, k));
    }
    return d;
}

// tile pair index -> (it, jt) with jt >= it (row-major over the upper triangle)
__device__ __forceinline__ void tile_pair(long long t, int nt, int& it, int& jt) {
    // rows before it hold it nt - it (it - 1) / 2 tiles
    const double m = nt + 0.5;
    long long r = (long long)(m - sqrt(fmax(0.0, m * m - 2.0 * (double)t)));
    if (r > nt - 1) r = nt - 1;
    auto before = [&](long long q) { return q * nt - q * (q - 1) / 2; };
    while (r > 0 && before(r) > t) --r;
    while (before(r + 1) <= t) ++r;
    it = (int)r;
    jt = (int)(r + (t - before(r)));
}

// A non-negative double as an integer of the same order (NaN above infinity), and its truncation
// to a float pattern, which keeps the order up to ties (a double beyond the float range saturates).
// Integer instructions: conversions and comparisons of doubles share the slow FP64 pipe.
__device__ __forceinline__ long long order_bits(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ int float_bits(double v) {
    const int hi = __double2hiint(v);
    if (hi < 0x38100000) return 0;            // below 2^-126
    if (hi >= 0x47f00000) return 0x7f800000;  // 2^128 and beyond
    return ((hi - 0x38000000) << 3) | (int)((unsigned)__double2loint(v) >> 29);
}

// What bounds it: the FP64 rate (1/64 of FP32 on GB300), about 35 operations a pair in range (110
// with a square root, a division and two sets of polynomials per pair).  The sums need no
// atomics (FP64 ones in shared memory are compare-and-swap loops): every lane adds to its own copy
// of its warp's shells, copies[nb][5][32], and with fewer copies the lanes that share one and meet on
// a shell go one after the other (all lanes of a copy in fixed turns: 16.0 ms at 40 shells, 43.0 at
// 256, more than atomics had taken there); 4 warps per SM hide the FP64 latency.  20000 points: 37.9 ->
// 15.0 ms with 40 shells, 34.3 -> 15.8 with 256.
__global__ void __launch_bounds__(kTile) k_pair_sums(PairArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nb = a.nb, C = a.copies;
    double* hist = reinterpret_cast<double*>(smem_raw);            // [kWarps][nb][kEll][C]
    double* xj = hist + (size_t)kWarps * nb * kEll * C;             // [7][kTile]: x, y, z, w, ux, uy, uz
    double* thr = xj + 7 * kTile;                                   // [nb + 1]
    int* thf = reinterpret_cast<int*>(thr + nb + 1);                // [nb + 1] float_bits of thr
    float* xf = reinterpret_cast<float*>(thf + nb + 1);             // [3][kTile] x, y, z rounded
    __shared__ float reach[kWarps];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < kWarps * nb * kEll * C; i += kTile) hist[i] = 0.0;
    for (int i = tid; i <= nb; i += kTile) {
        thr[i] = a.thr[i];
        thf[i] = float_bits(a.thr[i]);
    }
    double* h = hist + (size_t)warp * nb * kEll * C + (lane & (C - 1));
    const long long pairs = (long long)a.n_tiles * (a.n_tiles + 1) / 2;
    const long long n = a.n;
    const double root2 = 1.4142135623730950488;   // (d . root2 u)^2 / s^2 = 2 mu^2
    for (long long t = blockIdx.x; t < pairs; t += gridDim.x) {
        int it, jt;
        tile_pair(t, a.n_tiles, it, jt);
        __syncthreads();   // the previous tile's j points are no longer read
        double xi = 0, yi = 0, zi = 0, wi = 0, ux = 0, uy = 0, uz = 0;
        auto point = [&](long long q, double& x, double& y, double& z, double& w, double& vx, double& vy, double& vz) {
            x = y = z = w = vx = vy = vz = 0.0;
            if (q < n) {
                x = a.pos[q];
                y = a.pos[n + q];
                z = a.pos[2 * n + q];
                w = a.w ? a.w[q] : 1.0;
                const double px = x - a.obs[0], py = y - a.obs[1], pz = z - a.obs[2];
                const double inv = root2 / sqrt(px * px + py * py + pz * pz);
                vx = px * inv;
                vy = py * inv;
                vz = pz * inv;
            }
        };
        point((long long)jt * kTile + tid, xi, yi, zi, wi, ux, uy, uz);
        xj[tid] = xi;
        xj[kTile + tid] = yi;
        xj[2 * kTile + tid] = zi;
        xj[3 * kTile + tid] = wi;
        xj[4 * kTile + tid] = ux;
        xj[5 * kTile + tid] = uy;
        xj[6 * kTile + tid] = uz;
        // the largest |x| + |y| + |z| of the tile bounds the rounding of the FP32 separations below
        float far_j = (float)(fabs(xi) + fabs(yi) + fabs(zi));
        xf[tid] = (float)xi;
        xf[kTile + tid] = (float)yi;
        xf[2 * kTile + tid] = (float)zi;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) far_j = fmaxf(far_j, __shfl_xor_sync(0xffffffffu, far_j, o));
        if (lane == 0) reach[warp] = far_j;
        if (it != jt) point((long long)it * kTile + tid, xi, yi, zi, wi, ux, uy, uz);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kWarps; ++q) far_j = fmaxf(far_j, reach[q]);
        const bool live = (long long)it * kTile + tid < n;
        const int j0 = it == jt ? tid + 1 : 0;
        const long long jn = n - (long long)jt * kTile;
        const int j1 = jn < kTile ? (int)jn : kTile;
        // a pair whose FP32 separation exceeds the last edge by more than every rounding (2^-21 of the
        // coordinates) is out of range; below 1e-16 the squares would round among FP32's denormals and
        // every pair is taken
        const float boxf = (float)a.box, ibox = a.box > 0.0 ? 1.0f / boxf : 0.0f;
        const float xif = (float)xi, yif = (float)yi, zif = (float)zi;
        const float edge = (float)a.s_max * 1.00001f + 4.8e-7f * (far_j + fabsf(xif) + fabsf(yif) + fabsf(zif) + boxf);
        const float far = edge >= 1e-16f ? edge * edge : INFINITY;
        for (int jj = 0; jj < j1; ++jj) {   // warp-uniform: the lanes wait for one another below
            bool in = live && jj >= j0;
            float fx = xf[jj] - xif, fy = xf[kTile + jj] - yif, fz = xf[2 * kTile + jj] - zif;
            if (boxf > 0.f) {
                fx -= boxf * rintf(fx * ibox);
                fy -= boxf * rintf(fy * ibox);
                fz -= boxf * rintf(fz * ibox);
            }
            in = in && !(fx * fx + fy * fy + fz * fz > far);
            if (!__any_sync(0xffffffffu, in)) continue;
            const double dx = min_image(__dsub_rn(xj[jj], xi), a.box);
            const double dy = min_image(__dsub_rn(xj[kTile + jj], yi), a.box);
            const double dz = min_image(__dsub_rn(xj[2 * kTile + jj], zi), a.box);
            const double s2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
            const long long b2 = order_bits(s2);
            in = in && b2 > 0 && b2 >= order_bits(thr[0]) && b2 < order_bits(thr[nb]);
            // the shell by the truncated squares; equal truncations are decided in full
            const int f2 = float_bits(s2);
            int lo = 0, hi = nb;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (f2 >= thf[mid]) lo = mid; else hi = mid;
            }
            while (lo > 0 && f2 == thf[lo] && b2 < order_bits(thr[lo])) --lo;
            const double di = dx * ux + dy * uy + dz * uz;
            const double dj = dx * xj[4 * kTile + jj] + dy * xj[5 * kTile + jj] + dz * xj[6 * kTile + jj];
            // 1 / s2: an FP32 reciprocal and a third-order correction (its error to the third power); beyond
            // FP32's exponents by the cosines themselves, as 1 / s2 and the squares leave FP64's too
            double yi2, yj2;
            if (f2 > 0x0e000000 && f2 < 0x70000000) {   // 2^-99 .. 2^97
                float r;
                asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__int_as_float(f2)));
                const int rb = __float_as_int(r);   // widened by its bits (normal)
                const double rd = __hiloint2double((rb >> 3) + 0x38000000, rb << 29);
                const double e = fma(-s2, rd, 1.0);
                const double inv = fma(rd, fma(e, e, e), rd);
                yi2 = fma(di * di, inv, -1.0);
                yj2 = fma(dj * dj, inv, -1.0);
            } else {
                const double s = sqrt(s2), ci = di / s, cj = dj / s;
                yi2 = fma(ci, ci, -1.0);
                yj2 = fma(cj, cj, -1.0);
            }
            // Newton's identities for the power sums of two numbers
            const double e1 = yi2 + yj2, e2 = yi2 * yj2;
            const double p2 = fma(e1, e1, -2.0 * e2);
            const double p3 = fma(e1, p2, -e2 * e1);
            const double p4 = fma(e1, p3, -e2 * p2);
            const double ww = wi * xj[3 * kTile + jj];
            auto add = [&]() {
                double* q = h + lo * kEll * C;
                q[0] += ww;
                q[C] = fma(ww, e1, q[C]);
                q[2 * C] = fma(ww, p2, q[2 * C]);
                q[3 * C] = fma(ww, p3, q[3 * C]);
                q[4 * C] = fma(ww, p4, q[4 * C]);
            };
            if (C == 32) {
                if (in) add();
            } else {
                // the lanes that meet on one copy of one shell, one after the other
                const unsigned peers = __match_any_sync(0xffffffffu, in ? lo * C + (lane & (C - 1)) : -1 - lane);
                const int rank = __popc(peers & ((1u << lane) - 1u));
                for (int turn = 0; __any_sync(0xffffffffu, in && rank >= turn); ++turn) {
                    if (in && rank == turn) add();
                    __syncwarp();
                }
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < nb * kEll; i += kTile) {
        double v = 0.0;
        for (int wq = 0; wq < kWarps; ++wq)
            for (int c = 0; c < C; ++c) v += hist[((size_t)wq * nb * kEll + i) * C + c];
        if (v != 0.0) atomicAdd(a.out + i, v);
    }
}

__global__ void k_nw2_sum(const double* __restrict__ w, const double* __restrict__ nbar, long long n,
                          double* __restrict__ out) {
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double wi = w ? w[i] : 1.0;
        s += (nbar ? nbar[i] : 1.0) * wi * wi;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, s);
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

extern "C" lpp_status lpp_window_Q_pairs_workspace_size(int n_s, size_t* bytes) {
    if (!bytes || n_s < 1 || n_s > kMaxShells) return LPP_ERR_INVALID_ARG;
    *bytes = align256((size_t)n_s * kEll * sizeof(double)) + align256((size_t)(n_s + 1) * sizeof(double)) +
             align256(sizeof(double));
    return LPP_OK;
}

extern "C" lpp_status lpp_window_Q_pairs(const double* pos, const double* w, const double* nbar, long long n,
                                         const double* observer, double box, double alpha, int n_s,
                                         const double* s_edges, double* q, void* workspace, size_t bytes,
                                         void* stream) {
    size_t need = 0;
    if (lpp_window_Q_pairs_workspace_size(n_s, &need) != LPP_OK) return LPP_ERR_INVALID_ARG;
    if (!observer || !s_edges || !q || n < 0 || (n > 0 && !pos) || box < 0.0 || !(alpha > 0.0))
        return LPP_ERR_INVALID_ARG;
    if (!(s_edges[0] >= 0.0)) return LPP_ERR_INVALID_ARG;
    for (int b = 0; b < n_s; ++b)
        if (!(s_edges[b] < s_edges[b + 1])) return LPP_ERR_INVALID_ARG;
    if (!workspace || ((uintptr_t)workspace & 255) != 0) return LPP_ERR_INVALID_ARG;
    if (bytes < need) return LPP_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    char* ws = static_cast<char*>(workspace);
    double* d_out = reinterpret_cast<double*>(ws);
    double* d_thr = reinterpret_cast<double*>(ws + align256((size_t)n_s * kEll * sizeof(double)));
    double* d_norm = reinterpret_cast<double*>(ws + align256((size_t)n_s * kEll * sizeof(double)) +
                                               align256((size_t)(n_s + 1) * sizeof(double)));
    if (cudaMemsetAsync(d_out, 0, (size_t)n_s * kEll * sizeof(double), st) != cudaSuccess) return LPP_ERR_CUDA;
    if (cudaMemsetAsync(d_norm, 0, sizeof(double), st) != cudaSuccess) return LPP_ERR_CUDA;
    // the smallest double whose rounded square root reaches the edge
    std::vector<double> thr(n_s + 1);
    for (int b = 0; b <= n_s; ++b) {
        const double e = s_edges[b];
        double x = e * e;
        while (x > 0.0 && sqrt(x) >= e) x = nextafter(x, 0.0);
        while (sqrt(x) < e) x = nextafter(x, INFINITY);
        thr[b] = x;
    }
    if (cudaMemcpyAsync(d_thr, thr.data(), (size_t)(n_s + 1) * sizeof(double), cudaMemcpyHostToDevice, st) != cudaSuccess)
        return LPP_ERR_CUDA;
    if (n > 0) {
        long long nbk = (n + 255) / 256;
        if (nbk > 152 * 8) nbk = 152 * 8;
        k_nw2_sum<<<(int)nbk, 256, 0, st>>>(w, nbar, n, d_norm);
        PairArgs a;
        memset(&a, 0, sizeof(a));
        a.pos = pos;
        a.w = w;
        a.n = n;
        a.n_tiles = (int)((n + kTile - 1) / kTile);
        for (int k = 0; k < 3; ++k) a.obs[k] = observer[k];
        a.box = box;
        a.thr = d_thr;
        a.s_max = s_edges[n_s];
        a.nb = n_s;
        a.out = d_out;
        // copies of the shell sums: as many as leave room for two CTAs per SM (40 shells: 16 copies,
        // 20.6 -> 15.9 ms against 32 copies and one CTA, whose four warps do not hide the FP64 latency;
        // 256 shells: two)
        auto smem_of = [&](int c) {
            return ((size_t)kWarps * n_s * kEll * c + 7 * kTile + n_s + 1) * sizeof(double) +
                   ((size_t)(n_s + 1) + 3 * kTile) * sizeof(float);
        };
        a.copies = 32;
        while (a.copies > 1 && smem_of(a.copies) > 112 * 1024) a.copies /= 2;
        const size_t smem = smem_of(a.copies);
        if (lpp::allow_shared(k_pair_sums, lpp::kMaxShared) != cudaSuccess) return LPP_ERR_CUDA;
        const long long tp = (long long)a.n_tiles * (a.n_tiles + 1) / 2;
        int dev = 0, sms = 152;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int per_sm = std::max(1, std::min(4, (int)((227 * 1024) / (smem + 1024))));
        const long long grid = tp < (long long)sms * per_sm ? tp : (long long)sms * per_sm;
        k_pair_sums<<<(int)grid, kTile, smem, st>>>(a);
        if (cudaGetLastError() != cudaSuccess) return LPP_ERR_CUDA;
    }
    std::vector<double> h_out((size_t)n_s * kEll);
    double h_norm = 0.0;
    if (cudaMemcpyAsync(h_out.data(), d_out, h_out.size() * sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return LPP_ERR_CUDA;
    if (cudaMemcpyAsync(&h_norm, d_norm, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess) return LPP_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return LPP_ERR_CUDA;
    // L_l(mu) as a polynomial in y = 2 mu^2 - 1: mu^(2 i) = ((1 + y) / 2)^i
    double leg[kEll][kEll];
    for (int e = 0; e < kEll; ++e) {
        double c[16] = {0};
        lpp::legendre_poly(2 * e, c);
        for (int k = 0; k < kEll; ++k) leg[e][k] = 0.0;
        for (int i = 0; i <= e; ++i) {
            double binom = 1.0;   // i choose k
            for (int k = 0; k <= i; ++k) {
                leg[e][k] += c[2 * i] * binom / (double)(1 << i);
                binom = binom * (i - k) / (k + 1);
            }
        }
    }
    const double I = alpha * h_norm;
    const double pi = 3.14159265358979323846;
    for (int e = 0; e < kEll; ++e)
        for (int b = 0; b < n_s; ++b) {
            const double vol = 4.0 * pi * (s_edges[b + 1] * s_edges[b + 1] * s_edges[b + 1] -
                                           s_edges[b] * s_edges[b] * s_edges[b]) / 3.0;
            const double* p = &h_out[(size_t)b * kEll];
            double sum = 2.0 * leg[e][0] * p[0];   // p_0 = 2 per pair
            // to degree e: the powers beyond are not its own (NaN where a line of sight does not exist)
            for (int k = 1; k <= e; ++k) sum += leg[e][k] * p[k];
            q[e * n_s + b] = I > 0.0 ? (4.0 * e + 1.0) * alpha * alpha * sum / (I * vol) : 0.0;
        }
    return LPP_OK;
}
