// Batched 3D complex FFT of n^3 grids as three pencil passes (x, y, z).
//
// Each CTA transforms a tile of W pencils (n complex points each) with a mixed-radix
// Stockham FFT (radix 8 stages, one leading radix-2 or -4 stage), every thread holding
// 8 points per stage (FP32 grids of 64^3 and more: 8 points of two pencils,
// lpp_fft_pair.cuh), and writes the pencils back in place.  Pencils along y and z are read
// as rows of W consecutive x values, so every global access is a contiguous W-element
// segment; the first stage takes its operands straight from those rows and the last stage
// stores straight to them, so shared memory holds only the stages in between.  x pencils
// are transposed into the same column layout in shared memory.
//
// Passes can be pruned to the frequencies the shell binning needs: with a kept
// range f in [-nk_neg, nk_pos] per axis, the x pass writes only kept x, the y pass
// reads only kept x columns and writes kept y, and the z pass runs only on kept
// (x, y) columns and writes kept z.  With the last shell's bound q_max on |f|^2 the y pass
// writes and the z pass reads only columns with fx^2 + fy^2 < q_max (pi / 4 of the kept square),
// and the z pass writes only modes with |f|^2 < q_max (pi / 6 of the cube).  Values outside are
// left stale.
#include <algorithm>
#include <vector>

#include "lpp_internal.h"
#include "lpp_kernels.h"
#include "lpp_fft_dev.cuh"
#include "lpp_fft_pair.cuh"

namespace lpp {

// MODE 0: pencils along x (W consecutive y lines at fixed z)
// MODE 1: pencils along y (W consecutive kept x columns at fixed z)
// MODE 2: pencils along z (W consecutive kept x columns at a fixed kept y)
// Offsets inside one grid fit in 32 bits (n <= 1024); the tile base is a 64-bit pointer.

// Whether z plane `z` of grid `gi` of the call holds anything for the y pass: false when no
// particle of the grid's roles reaches it (neither the fused assignment nor the y pass stores
// it, and the z pass reads zeros there).  CTA-uniform.
__device__ __forceinline__ bool plane_live(const FftGeom& g, int gi, int z, int n) {
    if (!g.pmask || !g.gmask[gi]) return true;
    int hit = 0;
#pragma unroll
    for (int r = 0; r < 3; ++r)
        if (g.gmask[gi] & (1 << r)) hit |= __ldg(g.pmask + r * n + z);
    return hit != 0;
}

// What a thread moves of a column whose smallest |fx| is fx: nothing for a column outside the kept
// range or (MODE 2: at fy) outside the last shell's circle; of the others the results on kept
// frequencies inside the last shell's sphere.  Nothing else is read by a later pass or the combine.
// Eight grids of 256^3 to k = 0.995 k_Ny, against whole tiles of columns within the kept ranges: y
// pass 383 -> 375 us, z pass 320 -> 280 us.
template <int N>
struct ColumnBound {
    int q, lim;   // |f|^2 of the column at f = 0 of its own axis, and its limit
    bool live;
    __device__ __forceinline__ ColumnBound(const FftGeom& g, bool keep, int fx, int fy) {
        lim = g.q_max > 0 ? g.q_max : 0x3fffffff;
        q = fx * fx + fy * fy;
        live = keep && q < lim;
        if (!live) q = lim;
    }
    __device__ __forceinline__ bool stores(const FftGeom& g, int e) const {
        const int f = e < N / 2 ? e : N - e;
        return kept(e, N, g.nk_pos, g.nk_neg) && q + f * f < lim;
    }
};

// One y (MODE 1) or z (MODE 2) tile of W pencils of one grid.  twg: with it the twiddles are
// loaded into tw here, after the column test and beside the operand loads (they are first
// read after the first stage's barrier); null when tw already holds them.  Every return is
// CTA-uniform; the tile is free again after the caller's next barrier.
template <typename T, int LOGN, int MODE>
__device__ __forceinline__ void pencil_tile(c2<T>* grid, const c2<T>* twg, c2<T>* tw, c2<T>* tile, const FftGeom& g,
                                            int tile_id, int gi) {
    using S = PassShape<LOGN>;
    constexpr int N = S::N, W = S::W, LD = S::LD;
    const int tid = threadIdx.x;
    const unsigned N2 = (unsigned)N * N;
    c2<T>* base = grid;
    const int o = tile_id / g.ntx;
    const int i = tile_id - o * g.ntx;
    const int x0 = (g.ntx == N / W || i < g.nlo) ? i * W : N - (g.ntx - i) * W;
    if (!LPP_IN_BOUNDS(o >= 0 && o < (MODE == 1 ? N : g.nky) && x0 >= 0 && x0 + W <= N, g.err)) return;
    int fy = 0;
    if (MODE == 1) {
        base += (size_t)o * N2 + x0;  // o = z
    } else {
        const int y = (o <= g.nk_pos) ? o : N - (g.nky - o);
        fy = y < N / 2 ? y : N - y;
        if (g.q_max > 0) {
            // columns outside the last shell in (fx, fy) for every fz: nothing to transform
            int m2 = 0x7fffffff;
            for (int c = 0; c < W; ++c) {
                const int x = x0 + c;
                const int fx = x < N / 2 ? x : x - N;
                m2 = min(m2, fx * fx);
            }
            if (m2 + fy * fy >= g.q_max) return;
        }
        base += (size_t)y * N + x0;
    }
    // Thread (c, u) owns pencil c (W consecutive x values per row: 128-byte segments in
    // FP32) and butterfly slot u.  The first FFT stage loads its operands straight from
    // the grid and the last stores its results straight back, so the tile holds only the
    // intermediate stages.
    const int c = tid & (W - 1), u = tid >> S::LOGW;
    constexpr unsigned ES = MODE == 1 ? (unsigned)N : (unsigned)N * N;
    c2<T>* gp = base + c;
    const ColumnBound<N> col(g, kept(x0 + c, N, g.nk_pos, g.nk_neg), min(x0 + c, N - x0 - c), fy);
    static_assert(S::PER == 8 * S::IPT && S::PER <= 32, "one liveness bit per operand");
    // operands on rows that no particle of the grid's roles reaches (y pencils of this z
    // plane for the y pass, z planes for the z pass) are zero and not loaded
    unsigned live = col.live ? 0xffffffffu : 0u;
    const int gm = g.gmask[gi];
    if (col.live && gm && (MODE == 1 ? g.plive != nullptr : g.pmask != nullptr)) {
        const int z = o;   // the y pass's plane
        live = 0u;
#pragma unroll
        for (int b = 0; b < S::PER; ++b) {
            const int e = lead_row<LOGN, S::IPT>(u, b);
            int hit = 0;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                if (gm & (1 << r))
                    hit |= MODE == 1 ? __ldg(g.plive + (size_t)r * N * N + (size_t)z * N + e)
                                     : __ldg(g.pmask + r * N + e);
            }
            live |= (hit ? 1u : 0u) << b;
        }
    }
    if (twg)
        for (int k = tid; k < N; k += S::THREADS) tw[k] = twg[k];
    fft_columns_io<T, LOGN, S::IPT, LD>(
        tile, c, u, tw,
        [&](int b, int e) { return ((live >> b) & 1u) ? gp[(size_t)e * ES] : mk<T>((T)0, (T)0); },
        [&](int e, c2<T> v) {
            if (!col.stores(g, e)) return;
            if (MODE == 2 && g.mult) v = cmul<T>(v, static_cast<const c2<T>*>(g.mult)[(gp - grid) + (size_t)e * ES]);
            gp[(size_t)e * ES] = v;
        });
}

template <typename T, int LOGN, int MODE>
__global__ void __launch_bounds__(PassShape<LOGN>::THREADS, sizeof(T) == 4 ? (LOGN == 9 ? 3 : 2) : 1) k_fft_pass(c2<T>* __restrict__ data,
                                                                      const c2<T>* __restrict__ twg, FftGeom g) {
    using S = PassShape<LOGN>;
    constexpr int N = S::N, W = S::W, LD = S::LD;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c2<T>* tw = reinterpret_cast<c2<T>*>(smem_raw);
    c2<T>* tile = tw + N;
    const int tid = threadIdx.x;
    const unsigned N2 = (unsigned)N * N;
    c2<T>* grid = data + (size_t)blockIdx.y * N2 * N;
    const int tile_id = blockIdx.x;
    if constexpr (MODE == 0) {
        for (int i = tid; i < N; i += S::THREADS) tw[i] = twg[i];
        const int ty = tile_id & (N / W - 1);
        const int z = tile_id >> (LOGN - S::LOGW);
        if (!LPP_IN_BOUNDS(z < N, g.err)) return;
        c2<T>* base = grid + (size_t)z * N2 + (size_t)ty * W * N;
#pragma unroll
        for (int k = 0; k < S::PER; ++k) {
            const int idx = tid + k * S::THREADS;
            const int e = idx & (N - 1), c = idx >> LOGN;
            tile[e * LD + c] = base[e + c * N];
        }
        __syncthreads();
        fft_columns<T, LOGN, S::IPT, LD>(tile, tid & (W - 1), tid >> S::LOGW, tw);
#pragma unroll
        for (int k = 0; k < S::PER; ++k) {
            const int idx = tid + k * S::THREADS;
            const int e = idx & (N - 1), c = idx >> LOGN;
            if (kept(e, N, g.nk_pos, g.nk_neg)) base[e + c * N] = tile[e * LD + c];
        }
    } else {
        // a z plane that no particle of the grid's roles reaches: its pencils are zero;
        // neither the fused assignment nor this pass stores it
        if (MODE == 1 && !plane_live(g, blockIdx.y, tile_id / g.ntx, N)) return;
        pencil_tile<T, LOGN, MODE>(grid, twg, tw, tile, g, tile_id, blockIdx.y);
    }
}

// The y pass as a persistent grid over the (grid, plane, x tile) items of the call, for calls
// that skip unreached planes: the items of unreached planes cost a mask test instead of a
// CTA launch (with its shared memory held), and the twiddles are loaded once per CTA.
template <typename T, int LOGN>
__global__ void __launch_bounds__(PassShape<LOGN>::THREADS, sizeof(T) == 4 ? (LOGN == 9 ? 3 : 2) : 1) k_fft_ypass(c2<T>* __restrict__ data,
                                                                       const c2<T>* __restrict__ twg, FftGeom g, int n_grids) {
    using S = PassShape<LOGN>;
    constexpr int N = S::N;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c2<T>* tw = reinterpret_cast<c2<T>*>(smem_raw);
    c2<T>* tile = tw + N;
    for (int i = threadIdx.x; i < N; i += S::THREADS) tw[i] = twg[i];   // first read after a barrier
    const int per_grid = g.ntx * N;
    const int items = per_grid * n_grids;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int gi = it / per_grid, tile_id = it - gi * per_grid;
        if (!plane_live(g, gi, tile_id / g.ntx, N)) continue;
        pencil_tile<T, LOGN, 1>(data + (size_t)gi * N * N * N, nullptr, tw, tile, g, tile_id, gi);
        __syncthreads();   // the next item's first stage rewrites the tile
    }
}

// ---- FP32 passes on pencil pairs (lpp_fft_pair.cuh), 64 <= n <= 1024
// One y (MODE 1) or z (MODE 2) tile of one grid, as pencil_tile.  MULT: the results take the factors
// g.mult (the window multipoles on 256^3: z passes and products 2.12 -> 1.41 ms for 23 grids).
template <int LOGN, int MODE, bool MULT>
__device__ __forceinline__ void pair_tile(float2* grid, const float2* twg, cpair* tw, cpair* tile, const FftGeom& g,
                                          int tile_id, int gi) {
    using S = PairShape<LOGN>;
    constexpr int N = S::N, W = S::W;
    const int tid = threadIdx.x;
    const unsigned N2 = (unsigned)N * N;
    const int o = tile_id / g.ntx;
    const int i = tile_id - o * g.ntx;
    const int x0 = (g.ntx == N / W || i < g.nlo) ? i * W : N - (g.ntx - i) * W;
    if (!LPP_IN_BOUNDS(o >= 0 && o < (MODE == 1 ? N : g.nky) && x0 >= 0 && x0 + W <= N, g.err)) return;
    float2* base = grid;
    int fy = 0;
    if (MODE == 1) {
        base += (size_t)o * N2 + x0;  // o = z
    } else {
        const int y = (o <= g.nk_pos) ? o : N - (g.nky - o);
        fy = y < N / 2 ? y : N - y;
        if (g.q_max > 0) {
            // columns outside the last shell in (fx, fy) for every fz: nothing to transform
            // the smallest |fx| of the tile: x0 itself or its upper end (tiles do not straddle N / 2)
            const int fx = x0 < N / 2 ? x0 : N - (x0 + W - 1);
            if (fx * fx + fy * fy >= g.q_max) return;
        }
        base += (size_t)y * N + x0;
    }
    const int c = tid & (S::CP - 1), u = tid >> S::LOGC;
    constexpr unsigned ES = MODE == 1 ? (unsigned)N : (unsigned)N * N;
    float4* gp = reinterpret_cast<float4*>(base + 2 * c);   // x0 even: 16-byte aligned
    const int xa = x0 + 2 * c;   // the pair's columns: xa and xa + 1
    const ColumnBound<N> col(g, kept(xa, N, g.nk_pos, g.nk_neg) || kept(xa + 1, N, g.nk_pos, g.nk_neg),
                             min(xa, N - xa - 1), fy);
    static_assert(S::PER <= 32, "one liveness bit per operand");
    // operands on rows that no particle of the grid's roles reaches are zero and not loaded
    unsigned live = col.live ? 0xffffffffu : 0u;
    const int gm = g.gmask[gi];
    if (col.live && gm && (MODE == 1 ? g.plive != nullptr : g.pmask != nullptr)) {
        live = 0u;
#pragma unroll
        for (int b = 0; b < S::PER; ++b) {
            const int e = lead_row<LOGN, S::IPT>(u, b);
            int hit = 0;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                if (gm & (1 << r))
                    hit |= MODE == 1 ? __ldg(g.plive + (size_t)r * N * N + (size_t)o * N + e)
                                     : __ldg(g.pmask + r * N + e);
            }
            live |= (hit ? 1u : 0u) << b;
        }
    }
    auto twiddle = [](float2 w) { return cpair{pk2(w.x, w.x), pk2(-w.y, -w.y)}; };
    if (twg)
        for (int k = tid; k < N; k += S::THREADS) tw[k] = twiddle(twg[k]);
    fft_pairs_io<LOGN>(
        tile, c, u, tw,
        [&](int b, int e) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if ((live >> b) & 1u) v = gp[(size_t)e * (ES / 2)];
            return cpair{pk2(v.x, v.z), pk2(v.y, v.w)};
        },
        [&](int e, cpair v) {
            if (!col.stores(g, e)) return;
            if constexpr (MULT) {
                const float4 f = static_cast<const float4*>(
                    g.mult)[(gp - reinterpret_cast<float4*>(grid)) + (size_t)e * (ES / 2)];
                v = pmul_plain(v, cpair{pk2(f.x, f.z), pk2(f.y, f.w)});
            }
            float4 w;
            unpk2(v.re, w.x, w.z);
            unpk2(v.im, w.y, w.w);
            gp[(size_t)e * (ES / 2)] = w;
        });
}

template <int LOGN, int MODE, bool MULT = false>
__global__ void __launch_bounds__(PairShape<LOGN>::THREADS, PairShape<LOGN>::MINB)
k_fft_pair(float2* __restrict__ data, const float2* __restrict__ twg, const __grid_constant__ FftGeom g) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpair* tw = reinterpret_cast<cpair*>(smem_raw);
    constexpr size_t N = PairShape<LOGN>::N;
    // a z plane that no particle of the grid's roles reaches is neither stored by the fused
    // assignment nor by this pass
    if (MODE == 1 && !plane_live(g, blockIdx.y, blockIdx.x / g.ntx, (int)N)) return;
    // MULT: the grids' CTAs of one tile side by side (they share its factors in L2)
    const int ng = MULT ? (int)gridDim.x / (g.ntx * g.nky) : 1;
    const int gi = MULT ? (int)blockIdx.x % ng : (int)blockIdx.y, tile_id = (int)blockIdx.x / ng;
    pair_tile<LOGN, MODE, MULT>(data + gi * N * N * N, twg, tw, tw + N, g, tile_id, gi);
}

// The y pass as a persistent grid (see k_fft_ypass).
template <int LOGN>
__global__ void __launch_bounds__(PairShape<LOGN>::THREADS, PairShape<LOGN>::MINB)
k_fft_ypair(float2* __restrict__ data, const float2* __restrict__ twg, const __grid_constant__ FftGeom g, int n_grids) {
    using S = PairShape<LOGN>;
    constexpr int N = S::N;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpair* tw = reinterpret_cast<cpair*>(smem_raw);
    for (int i = threadIdx.x; i < N; i += S::THREADS) {   // first read after a barrier
        const float2 w = twg[i];
        tw[i] = cpair{pk2(w.x, w.x), pk2(-w.y, -w.y)};
    }
    const int per_grid = g.ntx * N;
    const int items = per_grid * n_grids;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int gi = it / per_grid, tile_id = it - gi * per_grid;
        if (!plane_live(g, gi, tile_id / g.ntx, N)) continue;
        pair_tile<LOGN, 1, false>(data + (size_t)gi * N * N * N, nullptr, tw, tw + N, g, tile_id, gi);
        __syncthreads();   // the next item's first stage rewrites the tile
    }
}

int fft_tile_width(int n) {
    int w = 8192 / n;
    if (w > 32) w = 32;
    if (w > n) w = n;
    return w;
}

// tiles of w columns over the kept x range
static void set_tiles(FftGeom& g, int n, int w) {
    g.W = w;
    const int tiles = n / w;
    g.nlo = g.nk_pos / w + 1;
    const int nhi = (g.nk_neg + w - 1) / w;
    g.ntx = g.nlo + nhi >= tiles ? tiles : g.nlo + nhi;
    if (g.ntx == tiles) g.nlo = tiles;
}

FftGeom fft_geometry(int n, int nk_pos, int nk_neg) {
    FftGeom g;
    g.nk_pos = nk_pos;
    g.nk_neg = nk_neg;
    set_tiles(g, n, fft_tile_width(n));
    g.nky = (nk_pos + 1 + nk_neg >= n) ? n : nk_pos + 1 + nk_neg;
    return g;
}

template <typename T, int LOGN>
static cudaError_t launch_passes(c2<T>* data, int n_grids, const c2<T>* tw, const FftGeom& geom, bool with_x,
                                 cudaStream_t st, Timer* timer) {
    using S = PassShape<LOGN>;
    constexpr int N = S::N, W = S::W;
    if (geom.W != W) return cudaErrorInvalidConfiguration;
    FftGeom g = geom;
    if (sizeof(T) == 4 && LOGN >= 6) set_tiles(g, N, PairShape<LOGN>::W);
    const size_t smem = (size_t)(N + N * S::LD) * sizeof(c2<T>);
    // the attribute is per device and function: set it on every call (cheap, host-only)
    cudaFuncSetAttribute(k_fft_pass<T, LOGN, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const double es = (double)sizeof(c2<T>);
    const double n3 = (double)N * N * N;
    const double keep = (double)(g.nky) / N;               // kept fraction of one axis
    if (with_x) {
        if (timer) timer->begin(KK_FFT, st);
        k_fft_pass<T, LOGN, 0><<<dim3((N / W) * N, n_grids), S::THREADS, smem, st>>>(data, tw, g);
        if (timer) timer->end(KK_FFT, st, n_grids * n3 * es * (1.0 + keep));
    }
    if (timer) timer->begin(KK_FFT, st);
    bool skip = false;
    for (int i = 0; i < n_grids && i < kMaxSlots; ++i) skip = skip || (g.pmask && g.gmask[i]);
    // one wave of resident CTAs (the occupancy the launch bounds give), at most one per item
    auto wave = [&](auto kernel, int threads, size_t bytes) {
        int dev = 0, sms = 0, ps = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, kernel, threads, bytes);
        return (int)std::min<long long>((long long)g.ntx * N * n_grids, (long long)std::max(ps, 1) * std::max(sms, 1));
    };
    if constexpr (sizeof(T) == 4 && LOGN >= 6) {
        using P = PairShape<LOGN>;
        auto attr = [&](auto kernel) {
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P::SMEM);
        };
        if (skip) {
            attr(k_fft_ypair<LOGN>);
            k_fft_ypair<LOGN><<<wave(k_fft_ypair<LOGN>, P::THREADS, P::SMEM), P::THREADS, P::SMEM, st>>>(
                data, tw, g, n_grids);
        } else {
            attr(k_fft_pair<LOGN, 1>);
            k_fft_pair<LOGN, 1><<<dim3(g.ntx * N, n_grids), P::THREADS, P::SMEM, st>>>(data, tw, g);
        }
    } else if (skip) {
        cudaFuncSetAttribute(k_fft_ypass<T, LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_fft_ypass<T, LOGN><<<wave(k_fft_ypass<T, LOGN>, S::THREADS, smem), S::THREADS, smem, st>>>(
            data, tw, g, n_grids);
    } else {
        cudaFuncSetAttribute(k_fft_pass<T, LOGN, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_fft_pass<T, LOGN, 1><<<dim3(g.ntx * N, n_grids), S::THREADS, smem, st>>>(data, tw, g);
    }
    // the fractions of the grid's columns and modes that the passes move (ColumnBound)
    double circle = keep * keep, sphere = keep * keep * keep;
    if (timer && g.q_max > 0) {
        std::vector<long long> sq(g.nky);
        for (int i = 0; i < g.nky; ++i) {
            const int y = (i <= g.nk_pos) ? i : N - (g.nky - i), f = std::min(y, N - y);
            sq[i] = (long long)f * f;
        }
        std::sort(sq.begin(), sq.end());
        long long cols = 0, modes = 0;
        for (long long a : sq)
            for (long long b : sq) {
                if (a + b >= g.q_max) break;
                ++cols;
                modes += std::lower_bound(sq.begin(), sq.end(), g.q_max - a - b) - sq.begin();
            }
        circle = cols / ((double)N * N);
        sphere = modes / n3;
    }
    // y: only the reached planes are read and written; z: their entries are read, all written
    if (timer) timer->end(KK_FFT, st, n_grids * n3 * es * (keep * (double)g.ylive_frac + (double)g.yread_frac * circle));
    if (timer) timer->begin(KK_FFT, st);
    if constexpr (sizeof(T) == 4 && LOGN >= 6) {
        using P = PairShape<LOGN>;
        auto attr = [&](auto kernel) {
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P::SMEM);
        };
        if (g.mult) {
            attr(k_fft_pair<LOGN, 2, true>);
            k_fft_pair<LOGN, 2, true><<<g.ntx * g.nky * n_grids, P::THREADS, P::SMEM, st>>>(data, tw, g);
        } else {
            attr(k_fft_pair<LOGN, 2>);
            k_fft_pair<LOGN, 2><<<dim3(g.ntx * g.nky, n_grids), P::THREADS, P::SMEM, st>>>(data, tw, g);
        }
    } else {
        cudaFuncSetAttribute(k_fft_pass<T, LOGN, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_fft_pass<T, LOGN, 2><<<dim3(g.ntx * g.nky, n_grids), S::THREADS, smem, st>>>(data, tw, g);
    }
    if (timer) timer->end(KK_FFT, st, n_grids * n3 * es * (circle * (double)g.yread_frac + sphere));
    return cudaGetLastError();
}

template <typename T>
static cudaError_t fft_dispatch(c2<T>* data, int n_grids, int n, const c2<T>* tw, const FftGeom& g,
                                bool with_x, cudaStream_t st, Timer* timer) {
    int logn = 0;
    while ((1 << logn) < n) ++logn;
#define LPP_FFT_CASE(LG)                                                                          \
    case LG:                                                                                      \
        return launch_passes<T, LG>(data, n_grids, tw, g, with_x, st, timer);
    switch (logn) {
        LPP_FFT_CASE(3)
        LPP_FFT_CASE(4)
        LPP_FFT_CASE(5)
        LPP_FFT_CASE(6)
        LPP_FFT_CASE(7)
        LPP_FFT_CASE(8)
        LPP_FFT_CASE(9)
        LPP_FFT_CASE(10)
        default:
            return cudaErrorInvalidValue;
    }
#undef LPP_FFT_CASE
}

template <typename T>
cudaError_t fft3d(c2<T>* data, int n_grids, int n, const c2<T>* tw, const FftGeom& g,
                  cudaStream_t st, Timer* timer) {
    return fft_dispatch<T>(data, n_grids, n, tw, g, true, st, timer);
}

template <typename T>
cudaError_t fft_yz(c2<T>* data, int n_grids, int n, const c2<T>* tw, const FftGeom& g,
                   cudaStream_t st, Timer* timer) {
    return fft_dispatch<T>(data, n_grids, n, tw, g, false, st, timer);
}

template cudaError_t fft3d<float>(c2<float>*, int, int, const c2<float>*, const FftGeom&, cudaStream_t, Timer*);
template cudaError_t fft3d<double>(c2<double>*, int, int, const c2<double>*, const FftGeom&, cudaStream_t, Timer*);
template cudaError_t fft_yz<float>(c2<float>*, int, int, const c2<float>*, const FftGeom&, cudaStream_t, Timer*);
template cudaError_t fft_yz<double>(c2<double>*, int, int, const c2<double>*, const FftGeom&, cudaStream_t, Timer*);

}  // namespace lpp
