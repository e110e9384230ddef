// Template surrogate network: 6 -> [256, GELU] x 4 -> 320, BF16 operands, FP32 accumulation.
//
// Every matrix product runs on the tensor cores (mma.m16n8k16, BF16 in, FP32 accumulate, the
// reduction dimension in ascending steps of 16).  The network is a chain of small products:
// a layer of a 256-row minibatch is 34 MFLOP, less than a microsecond of one launch, so the
// chain is fused by rows.  A cluster of four CTAs carries 16 rows through all layers (and, when
// training, back): each CTA computes a quarter of a layer's columns while its slice of the weight
// matrices streams through a ring of cp.async stages, and writes its activations into the shared
// memory of all four.  Predictions of many rows take one CTA per 32 rows.  A second kernel forms
// every layer's weight gradient and applies Adam in the epilogue.  Adam keeps FP32 master weights
// and refreshes their BF16 copies (and transposes) after every step.  The training loop is native:
// one call runs all steps of a schedule of minibatch indices.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <utility>
#include <vector>

#include "lpp_internal.h"

namespace {

using bf16 = __nv_bfloat16;
constexpr int kLayers = 5;
constexpr int kIn[kLayers] = {6, 256, 256, 256, 256};
constexpr int kInPad[kLayers] = {16, 256, 256, 256, 256};
constexpr int kOut[kLayers] = {256, 256, 256, 256, 320};
constexpr int kNout = 320;
constexpr int kNin = 6;

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void cp16(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Two neighbouring floats of a caller's array, which may start at any float (rows of 320 keep the
// address's remainder: the branch goes one way for a whole call).
__device__ __forceinline__ float2 load2(const float* p) {
    return ((uintptr_t)p & 7) == 0 ? *reinterpret_cast<const float2*>(p) : make_float2(p[0], p[1]);
}
__device__ __forceinline__ void store2(float* p, float a, float b) {
    if (((uintptr_t)p & 7) == 0) {
        *reinterpret_cast<float2*>(p) = make_float2(a, b);
    } else {
        p[0] = a;
        p[1] = b;
    }
}

// ---- weight streaming
// The passes of a row chain: the forward layers 0..4, then (training) the activation gradients
// through layers 4..1.  Pass p multiplies by w[p] [rows][K], K contiguous, in chunks of 32 K
// columns (16 for the padded input layer).
struct Passes {
    const bf16* w[2 * kLayers - 1];
};
__host__ __device__ constexpr int pass_rows(int p) { return p == kLayers - 1 ? kNout : 256; }
__host__ __device__ constexpr int pass_k(int p) { return p == 0 ? 16 : (p == kLayers ? kNout : 256); }

constexpr int kRowThreads = 256;       // 8 warps: warp w owns the output columns 8 (w NT) ..
constexpr int kChunkLd = 40;           // BF16 per chunk row: 32 and padding (conflict-free fragments)
constexpr int kStageElems = kNout * kChunkLd;

// A ring of weight chunks in shared memory: load(c) starts the copy of the c-th chunk of the whole
// chain (the copies run ahead of the layers).
template <int kStages>
struct WeightRing {
    bf16* ring;
    int pass = 0, k = 0, n_pass, put = 0, got = 0;
    __device__ __forceinline__ void load(const Passes& ps) {
        if (pass < n_pass) {
            const int rows = pass_rows(pass), K = pass_k(pass);
            const bf16* w = ps.w[pass];
            bf16* dst = ring + (put % kStages) * kStageElems;
            if (K >= 32) {
                for (int i = threadIdx.x; i < rows * 4; i += kRowThreads)
                    cp16(dst + (i >> 2) * kChunkLd + (i & 3) * 8, w + (size_t)(i >> 2) * K + k + (i & 3) * 8);
            } else {
                for (int i = threadIdx.x; i < rows * 2; i += kRowThreads)
                    cp16(dst + (i >> 1) * kChunkLd + (i & 1) * 8, w + (size_t)(i >> 1) * K + (i & 1) * 8);
            }
            k += 32;
            if (k >= K) { k = 0; ++pass; }
        }
        cp_commit();   // an empty group past the end keeps the count of groups in flight
        ++put;
    }
    // The next chunk, once it has landed and every warp has left the chunk before it; starts the
    // copy that replaces that one.
    __device__ __forceinline__ const bf16* next(const Passes& ps) {
        cp_wait<kStages - 2>();
        __syncthreads();
        load(ps);
        return ring + (got++ % kStages) * kStageElems;
    }
};

// acc[mt][j] += act[16 MT rows][K] . w[columns][K]^T for the warp's NT tiles of 8 columns.
template <int MT, int NT, int K, int LDA, int ST>
__device__ __forceinline__ void row_product(WeightRing<ST>& ring, const Passes& ps, const bf16* act,
                                            float (&acc)[MT][NT][4]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[mt][j][r] = 0.f;
    for (int k0 = 0; k0 < K; k0 += 32) {
        const bf16* w = ring.next(ps);
#pragma unroll
        for (int kk = 0; kk < (K < 32 ? K : 32); kk += 16) {
            uint32_t a[MT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                const bf16* ap = act + (mt * 16 + g) * LDA + k0 + kk + 2 * t;
                a[mt][0] = *reinterpret_cast<const uint32_t*>(ap);
                a[mt][1] = *reinterpret_cast<const uint32_t*>(ap + 8 * LDA);
                a[mt][2] = *reinterpret_cast<const uint32_t*>(ap + 8);
                a[mt][3] = *reinterpret_cast<const uint32_t*>(ap + 8 * LDA + 8);
            }
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                const bf16* bp = w + (8 * (warp * NT + j) + g) * kChunkLd + kk + 2 * t;
                const uint32_t b0 = *reinterpret_cast<const uint32_t*>(bp);
                const uint32_t b1 = *reinterpret_cast<const uint32_t*>(bp + 8);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) mma_bf16(acc[mt][j], a[mt], b0, b1);
            }
        }
    }
}

constexpr int kActLd = 328;   // BF16 per activation row of a cluster: up to 320 and padding (conflict-free fragments)
// Ring stages and BF16 per activation row of a CTA that carries 32 rows (256 and padding); two
// such CTAs share an SM.
constexpr int kPredLd = 264;
constexpr int kPredStages = 3, kPredRows = 32;
constexpr size_t kPredSmem = ((size_t)kPredStages * kStageElems + (size_t)2 * kPredRows * kPredLd) * sizeof(bf16);

// ---- 16 rows on a cluster of kSplit CTAs
// CTA `rank` owns the columns [rank, rank + 1) N / kSplit of every product (64, or 80 of the output
// layer), in tiles of 8 columns: tile w by warp w, tiles 8 and 9 of the output layer by warps 0
// and 1.  Weight chunks are 128 K columns of those rows.
constexpr int kSplit = 4;
constexpr int kSliceStages = 4, kSliceLd = 136, kSliceElems = (kNout / kSplit) * kSliceLd;
__host__ __device__ constexpr int slice_rows(int p) { return pass_rows(p) / kSplit; }
constexpr size_t kSliceSmem = ((size_t)kSliceStages * kSliceElems + (size_t)2 * 16 * kActLd) * sizeof(bf16);

struct SliceRing {
    bf16* ring;
    int n_pass, rank;
    int pass = 0, k = 0, put = 0, got = 0;
    __device__ __forceinline__ void load(const Passes& ps) {
        if (pass < n_pass) {
            const int rows = slice_rows(pass), K = pass_k(pass);
            const int kc = min(128, K - k), sh = kc == 128 ? 4 : (kc == 64 ? 3 : 1);   // kc = 128, 64 or 16
            const bf16* w = ps.w[pass] + (size_t)rank * rows * K + k;
            bf16* dst = ring + (put % kSliceStages) * kSliceElems;
            for (int i = threadIdx.x; i < rows << sh; i += kRowThreads) {
                const int r = i >> sh, c = (i & ((1 << sh) - 1)) * 8;
                cp16(dst + r * kSliceLd + c, w + (size_t)r * K + c);
            }
            k += 128;
            if (k >= K) { k = 0; ++pass; }
        }
        cp_commit();   // an empty group past the end keeps the count of groups in flight
        ++put;
    }
    __device__ __forceinline__ const bf16* next(const Passes& ps) {
        cp_wait<kSliceStages - 2>();
        __syncthreads();
        load(ps);
        return ring + (got++ % kSliceStages) * kSliceElems;
    }
};

__device__ __forceinline__ void ldmatrix_x4(uint32_t a[4], const bf16* p) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(s));
}

// acc[j] = act[16][K] . w[tile warp + 8 j]^T, tiles of this CTA's slice; TILES = 8 or 10 in the slice.
template <int K, int TILES>
__device__ __forceinline__ void slice_product(SliceRing& ring, const Passes& ps, const bf16* act,
                                              float (&acc)[(TILES + 7) / 8][4]) {
    constexpr int NT = (TILES + 7) / 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[j][r] = 0.f;
    const bf16* arow = act + (lane & 15) * kActLd + (lane >> 4) * 8;
    for (int k0 = 0; k0 < K; k0 += 128) {
        const bf16* w = ring.next(ps);
        const int kc = K < 128 ? K : min(128, K - k0);
#pragma unroll
        for (int kk = 0; kk < (K < 128 ? K : 128); kk += 16) {
            if (K % 128 != 0 && kk >= kc) break;
            uint32_t a[4];
            ldmatrix_x4(a, arow + k0 + kk);
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                if (TILES > 8 && warp + 8 * j >= TILES) break;   // warp-uniform
                const bf16* bp = w + (8 * (warp + 8 * j) + g) * kSliceLd + kk + 2 * t;
                mma_bf16(acc[j], a, *reinterpret_cast<const uint32_t*>(bp), *reinterpret_cast<const uint32_t*>(bp + 8));
            }
        }
    }
}

// Two neighbouring values (row r, columns c, c + 1 of the whole layer) into the activation buffer of
// every CTA of the cluster.
__device__ __forceinline__ void share2(bf16* buf, int r, int c, float v0, float v1) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const __nv_bfloat162 v(__float2bfloat16_rn(v0), __float2bfloat16_rn(v1));
#pragma unroll
    for (int q = 0; q < kSplit; ++q)
        *reinterpret_cast<__nv_bfloat162*>(cl.map_shared_rank(buf + r * kActLd + c, q)) = v;
}

// [16 rows][columns c0 .. c0 + cols) of a shared activation tile -> global transpose [column][ld] at
// row r0: 16 rows of one column are 32 contiguous bytes.
__device__ __forceinline__ void store_transposed(const bf16* act, int c0, int cols, bf16* dst, int ld, int r0) {
    for (int c = c0 + threadIdx.x; c < c0 + cols; c += kRowThreads) {
        __align__(16) bf16 v[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) v[r] = act[r * kActLd + c];
        uint4* d = reinterpret_cast<uint4*>(dst + (size_t)c * ld + r0);
        d[0] = reinterpret_cast<const uint4*>(v)[0];
        d[1] = reinterpret_cast<const uint4*>(v)[1];
    }
}

struct TrainRowArgs {
    Passes ps;
    const float* bias[kLayers];
    const float* x;
    const float* y;
    const int* idx;            // minibatch rows of x, y
    int batch;
    bf16* actt[kLayers];       // layer inputs, transposed [kInPad][batch]
    bf16* gt[kLayers];         // gradients of the pre-activations, transposed [kOut][batch]
    float* g32[kLayers];       // and FP32 [batch][kOut]
    double* loss;
};

// One training step's row chain: 16 rows of the minibatch per cluster through the forward layers,
// the loss gradient and the activation gradients, down to every layer's input and pre-activation
// gradient (transposed, for the weight gradients).  The pre-activations stay in registers: the
// backward products place their outputs on the same threads.  The activation buffers alternate,
// and the cluster's barrier after each layer separates a buffer's last reads from its next
// writes two layers later.
//
// What bounds it: the latency of nine dependent products (16 to 20 dependent mma each, the ring's
// and the cluster's barriers).  A step at batch 256 (both kernels): 199 us as 22 launches, 64 us
// with one CTA per 16 rows, 39 us on clusters.
__global__ void __cluster_dims__(kSplit, 1, 1) __launch_bounds__(kRowThreads, 1)
k_train_rows(const __grid_constant__ TrainRowArgs a) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cg::cluster_group cluster = cg::this_cluster();
    SliceRing ring;
    ring.ring = reinterpret_cast<bf16*>(smem_raw);
    ring.n_pass = 2 * kLayers - 1;
    ring.rank = (int)cluster.block_rank();
    bf16* buf[2];
    buf[0] = ring.ring + kSliceStages * kSliceElems;
    buf[1] = buf[0] + 16 * kActLd;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int r0 = (int)(blockIdx.x / kSplit) * 16;
    const int h0 = ring.rank * (256 / kSplit), o0 = ring.rank * (kNout / kSplit);   // this CTA's columns
    for (int c = 0; c < kSliceStages - 1; ++c) ring.load(a.ps);
    {   // inputs: BF16 [16][16], zero padded
        const int r = tid >> 4, c = tid & 15;
        const float v = c < kNin ? a.x[(size_t)a.idx[r0 + r] * kNin + c] : 0.f;
        buf[0][r * kActLd + c] = __float2bfloat16_rn(v);
    }
    cluster.sync();   // every CTA of the cluster runs before its shared memory is written
    if (ring.rank == 0) store_transposed(buf[0], 0, pass_k(0), a.actt[0], a.batch, r0);
    const int c = h0 + 8 * warp + 2 * t;   // the thread's hidden columns c, c + 1
    float z[kLayers - 1][4];
    int cur = 0;
#pragma unroll
    for (int l = 0; l < kLayers - 1; ++l) {
        float acc[1][4];
        if (l == 0) slice_product<16, 8>(ring, a.ps, buf[cur], acc);
        else slice_product<256, 8>(ring, a.ps, buf[cur], acc);
        const float2 b = *reinterpret_cast<const float2*>(a.bias[l] + c);
#pragma unroll
        for (int r = 0; r < 4; ++r) z[l][r] = acc[0][r] + ((r & 1) ? b.y : b.x);
#pragma unroll
        for (int h = 0; h < 2; ++h) share2(buf[cur ^ 1], g + 8 * h, c, gelu(z[l][2 * h]), gelu(z[l][2 * h + 1]));
        cur ^= 1;
        cluster.sync();
        store_transposed(buf[cur], h0, 256 / kSplit, a.actt[l + 1], a.batch, r0);
    }
    // output layer, loss and its gradient 2 (out - y) / (batch * 320)
    {
        float acc[2][4];
        slice_product<256, 10>(ring, a.ps, buf[cur], acc);
        const float sc = 2.0f / (float)(a.batch * kNout);
        double part = 0.0;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (warp + 8 * j >= kNout / kSplit / 8) break;
            const int co = o0 + 8 * (warp + 8 * j) + 2 * t;
            const float2 b = *reinterpret_cast<const float2*>(a.bias[kLayers - 1] + co);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = r0 + g + 8 * h;
                const float2 yv = load2(a.y + (size_t)a.idx[r] * kNout + co);
                const float d0 = (acc[j][2 * h] + b.x) - yv.x, d1 = (acc[j][2 * h + 1] + b.y) - yv.y;
                part += (double)d0 * d0 + (double)d1 * d1;
                const float2 gv = make_float2(sc * d0, sc * d1);
                *reinterpret_cast<float2*>(a.g32[kLayers - 1] + (size_t)r * kNout + co) = gv;
                share2(buf[cur ^ 1], g + 8 * h, co, gv.x, gv.y);
            }
        }
        for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
        if (lane == 0 && part != 0.0) atomicAdd(a.loss, part / (double)(a.batch * kNout));
        cur ^= 1;
        cluster.sync();
        store_transposed(buf[cur], o0, kNout / kSplit, a.gt[kLayers - 1], a.batch, r0);
    }
    // g_{l-1} = (g_l W_l) * GELU'(z_{l-1})
#pragma unroll
    for (int l = kLayers - 1; l > 0; --l) {
        float acc[1][4];
        if (l == kLayers - 1) slice_product<kNout, 8>(ring, a.ps, buf[cur], acc);
        else slice_product<256, 8>(ring, a.ps, buf[cur], acc);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 gv = make_float2(acc[0][2 * h] * gelu_grad(z[l - 1][2 * h]),
                                          acc[0][2 * h + 1] * gelu_grad(z[l - 1][2 * h + 1]));
            *reinterpret_cast<float2*>(a.g32[l - 1] + (size_t)(r0 + g + 8 * h) * 256 + c) = gv;
            share2(buf[cur ^ 1], g + 8 * h, c, gv.x, gv.y);
        }
        cur ^= 1;
        cluster.sync();   // also: no CTA leaves while the others write to it
        store_transposed(buf[cur], h0, 256 / kSplit, a.gt[l - 1], a.batch, r0);
    }
}

struct AdamLayer {
    float *w, *b, *mw, *vw, *mb, *vb, *dw, *db;
    bf16 *w16, *w16t;
    int out, in, inp;
};
struct AdamArgs {
    AdamLayer L[kLayers];
    float lr, b1, b2, eps, bc1, bc2;
};

// The weight and bias gradients of a step and their Adam update.
struct TrainWeightArgs {
    AdamArgs adam;
    const bf16* actt[kLayers];   // layer inputs, transposed [kInPad][batch]
    const bf16* gt[kLayers];     // pre-activation gradients, transposed [kOut][batch]
    const float* g32[kLayers];   // and FP32 [batch][kOut]
    int batch;
    int update;                  // 0: store the gradients (AdamLayer::dw, db) and change nothing else
};

// One Adam step of a parameter: the new value.
__device__ __forceinline__ float adam_step(const AdamArgs& a, float p, float& m, float& v, float gr) {
    const float mm = a.b1 * m + (1.f - a.b1) * gr;
    const float vv = a.b2 * v + (1.f - a.b2) * gr * gr;
    m = mm;
    v = vv;
    const float upd = a.lr * (mm / a.bc1) / (sqrtf(vv / a.bc2) + a.eps);
    return p - upd;
}

// dW_l = g_l^T a_l in tiles of 32 outputs x 64 inputs per CTA (144 CTAs, one wave) with Adam in the
// epilogue, and the bias gradients, 32 columns per CTA: a row's columns by one warp, eight
// partial sums over the rows r = w (mod 8) added in a fixed order.
constexpr int kTileM = 32, kTileN = 64, kPanel = 256, kPanelLd = kPanel + 8;
constexpr int kWeightTiles = 8 + 3 * 8 * 4 + 10 * 4;    // layer 0, layers 1..3, layer 4
constexpr int kBiasTiles = 4 * 8 + 10;
constexpr size_t kWeightSmem = (size_t)(kTileM + kTileN) * kPanelLd * sizeof(bf16);

__global__ void __launch_bounds__(128) k_train_weights(const __grid_constant__ TrainWeightArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int b = blockIdx.x;
    if (b >= kWeightTiles) {
        b -= kWeightTiles;
        const int l = b < 32 ? b >> 3 : kLayers - 1;
        const int c = (b - 8 * l) * 32 + lane, n = kOut[0] + (l == kLayers - 1 ? kNout - 256 : 0);
        float* part = reinterpret_cast<float*>(smem_raw);   // [8][33]
        for (int w = warp; w < 8; w += 4) {
            float s = 0.f;
#pragma unroll 8
            for (int r = w; r < a.batch; r += 8) s += a.g32[l][(size_t)r * n + c];
            part[w * 33 + lane] = s;
        }
        __syncthreads();
        if (warp == 0) {
            float gr = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) gr += part[k * 33 + lane];
            const AdamLayer& L = a.adam.L[l];
            if (a.update) L.b[c] = adam_step(a.adam, L.b[c], L.mb[c], L.vb[c], gr);
            else L.db[c] = gr;
        }
        return;
    }
    int l = 0, tn = 1;
    if (b >= 8) {
        b -= 8;
        l = b < 96 ? 1 + (b >> 5) : kLayers - 1;
        b -= 32 * (l - 1);
        tn = 4;
    }
    const int m0 = (b / tn) * kTileM, n0 = (b % tn) * kTileN;
    const AdamLayer& L = a.adam.L[l];
    const int inp = L.inp, rows_b = min(kTileN, inp - n0);
    bf16* As = reinterpret_cast<bf16*>(smem_raw);
    bf16* Bs = As + kTileM * kPanelLd;
    const int wm = warp >> 1, wn = warp & 1, g = lane >> 2, t = lane & 3;
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[j][r] = 0.f;
    for (int k0 = 0; k0 < a.batch; k0 += kPanel) {
        const int kp = min(kPanel, a.batch - k0);   // a multiple of 32
        const int seg = kp / 8;
        __syncthreads();
        for (int i = tid; i < (kTileM + rows_b) * seg; i += 128) {
            const int r = i / seg, c = (i - r * seg) * 8;
            if (r < kTileM) cp16(As + r * kPanelLd + c, a.gt[l] + (size_t)(m0 + r) * a.batch + k0 + c);
            else cp16(Bs + (r - kTileM) * kPanelLd + c, a.actt[l] + (size_t)(n0 + r - kTileM) * a.batch + k0 + c);
        }
        cp_commit();
        cp_wait<0>();
        __syncthreads();
        for (int k = 0; k < kp; k += 16) {
            const bf16* ap = As + (wm * 16 + g) * kPanelLd + k + 2 * t;
            uint32_t af[4];
            af[0] = *reinterpret_cast<const uint32_t*>(ap);
            af[1] = *reinterpret_cast<const uint32_t*>(ap + 8 * kPanelLd);
            af[2] = *reinterpret_cast<const uint32_t*>(ap + 8);
            af[3] = *reinterpret_cast<const uint32_t*>(ap + 8 * kPanelLd + 8);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (wn * 32 + 8 * j >= rows_b) break;   // warp-uniform (the input layer has 16 columns)
                const bf16* bp = Bs + (wn * 32 + 8 * j + g) * kPanelLd + k + 2 * t;
                mma_bf16(acc[j], af, *reinterpret_cast<const uint32_t*>(bp), *reinterpret_cast<const uint32_t*>(bp + 8));
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (wn * 32 + 8 * j >= rows_b) break;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = m0 + wm * 16 + g + 8 * h, col = n0 + wn * 32 + 8 * j + 2 * t;
            const size_t i = (size_t)row * inp + col;
            if (!a.update) {
                *reinterpret_cast<float2*>(L.dw + i) = make_float2(acc[j][2 * h], acc[j][2 * h + 1]);
                continue;
            }
            if (col >= L.in) continue;   // padded input columns stay zero (L.in is even)
            float2 p = *reinterpret_cast<const float2*>(L.w + i);
            float2 m = *reinterpret_cast<const float2*>(L.mw + i);
            float2 v = *reinterpret_cast<const float2*>(L.vw + i);
            p.x = adam_step(a.adam, p.x, m.x, v.x, acc[j][2 * h]);
            p.y = adam_step(a.adam, p.y, m.y, v.y, acc[j][2 * h + 1]);
            *reinterpret_cast<float2*>(L.w + i) = p;
            *reinterpret_cast<float2*>(L.mw + i) = m;
            *reinterpret_cast<float2*>(L.vw + i) = v;
            const __nv_bfloat162 q(__float2bfloat16_rn(p.x), __float2bfloat16_rn(p.y));
            *reinterpret_cast<__nv_bfloat162*>(L.w16 + i) = q;
            L.w16t[(size_t)col * L.out + row] = q.x;
            L.w16t[(size_t)(col + 1) * L.out + row] = q.y;
        }
    }
}

// BF16 copies of the master weights (after loading parameters)
__global__ void k_refresh(AdamArgs a) {
    const int layer = blockIdx.y;
    const AdamLayer& L = a.L[layer];
    const int nw = L.out * L.inp;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nw; i += gridDim.x * blockDim.x) {
        const int r = i / L.inp, c = i % L.inp;
        const bf16 h = __float2bfloat16_rn(L.w[i]);
        L.w16[i] = h;
        L.w16t[(size_t)c * L.out + r] = h;
    }
}

// parameters -> network inputs and network outputs -> curves (see lpp_surrogate_map)
constexpr int kMaxNodes = 8;
constexpr int kBadExponent = 1 << 20;   // a row or column with an infinity or NaN
struct MapArgs {
    float scale[kNin], shift[kNin];   // x_c = theta_c * scale_c + shift_c (0, 0 when not fed)
    double dscale[kNin], dshift[kNin];
    const double* mu;
    const double* sd;
    const double* shot;
    const double* ref;
    const double* sigma;
    const double* base;               // [nodes^2][320] or null
    int nodes, base_in[2];
    double N[2][3], M[3][3];          // native moments -> derived multipoles
    // the decoding's copy of base: kDigits signed base-256 digits per value relative to 2^column
    // exponent (digit_fragments), the exponents, and the Lobatto nodes with the Lagrange
    // normalisations 1 / prod_{j != i} (x_i - x_j)
    const uint4* digits;
    const int* exponent;    // [kNout]
    double xs[kMaxNodes], cw[kMaxNodes];
};

__global__ void k_encode(const double* __restrict__ theta, int n, float* __restrict__ x, MapArgs m) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * kNin; i += gridDim.x * blockDim.x) {
        const int c = i % kNin;
        x[i] = (float)(theta[i] * (double)m.scale[c] + (double)m.shift[c]);
    }
}

// Lagrange basis at the Chebyshev-Lobatto nodes x_i = -cos(pi i / (n - 1)), evaluated at x
__device__ void lobatto_basis(double x, int n, double* l) {
    double xs[kMaxNodes];
    for (int i = 0; i < n; ++i) xs[i] = -cospi((double)i / (double)(n - 1));
    for (int i = 0; i < n; ++i) {
        double v = 1.0;
        for (int j = 0; j < n; ++j)
            if (j != i) v *= (x - xs[j]) / (xs[i] - xs[j]);
        l[i] = v;
    }
}

// The same Lagrange basis from the map's nodes and normalisations: products only.
__device__ __forceinline__ void lobatto_basis_fast(double x, const MapArgs& a, double* l) {
    for (int i = 0; i < a.nodes; ++i) {
        double v = a.cw[i];
        for (int j = 0; j < a.nodes; ++j)
            if (j != i) v *= x - a.xs[j];
        l[i] = v;
    }
}

// ---- exact products of the baseline on the tensor cores
// The baseline sum_q w_q base_qj cancels: it needs more than the FP32 digits of its terms, and
// GB300 runs FP64 at 1/64 of the FP32 rate.  Both factors are therefore written as signed base-256
// digits of fixed-point numbers: base values with kDigits (48 bits) relative to the column's largest,
// below 2^ec, weights with kWDigits (56 bits) relative to the row's largest, below 2^er.  A digit is
// an integer of at most 128, exact in BF16; a sum of 64 products of digits is an integer below 2^20,
// and one of up to six such sums below 2^23, exact in the FP32 accumulators.  Products of digits i
// and j have weight 2^(-8 (i + j)): the sums of equal i + j <= 6 share an accumulator (27 of the 42
// products), and the seven accumulators are added in float pairs.
// The error is that of the base digits, 2^(ec - 48) sum |w_q|, and at most 2^(er + ec - 45) (64 times the
// weight digits' 2^(er + ec - 56) and the dropped products' 5 x 2^(er + ec - 56), the last orders
// added in one float 2^(er + ec - 46), the pairs).  It is small against the largest terms, not against every
// sum: decode_tile decides output by output whether it is small enough.
constexpr int kDigits = 6, kWDigits = 7, kOrders = 7;
constexpr int kBaseKsteps = kMaxNodes * kMaxNodes / 16;            // 16 baseline terms per mma
constexpr int kDigitWords = kDigits * (kNout / 8) * (kBaseKsteps / 2) * 32;   // uint4 of digit fragments
constexpr int kZeroExponent = -(1 << 20);   // a column of zeros

// v with |v| <= 2^e -> the kDigits digits d_i of v = 2^e sum_i d_i 2^(-8 i - 7) to 2^(e - 48).  One
// FP64 multiply-add: v 2^(47 - e) + 1.5 2^52 holds the rounded integer in its low bits.
__device__ __forceinline__ void fixed_digits(double v, int e, int* d) {
    const double scale = __hiloint2double((47 - e + 1023) << 20, 0);
    long long q = __double_as_longlong(fma(v, scale, 6755399441055744.0)) - 0x4338000000000000LL;
#pragma unroll
    for (int i = kDigits - 1; i > 0; --i) {
        d[i] = (int)((q + 128) & 255) - 128;
        q = (q - d[i]) >> 8;
    }
    d[0] = (int)q;
}
// v with |v| < 2^e -> kWDigits digits of v to 2^(e - 56).
__device__ __forceinline__ void weight_digits(double v, int e, int* d) {
    const double scale = __hiloint2double((55 - e + 1023) << 20, 0);
    long long q = __double2ll_rn(v * scale);
#pragma unroll
    for (int i = kWDigits - 1; i > 0; --i) {
        d[i] = (int)((q + 128) & 255) - 128;
        q = (q - d[i]) >> 8;
    }
    d[0] = (int)q;
}
// The exponent e of the largest of the warp's values (two per lane): |v| < 2^e; kBadExponent for
// an infinity, a NaN or values beyond 2^900; kZeroExponent for zeros (and denormals below 2^-1042); the
// smallest usable exponent for others below it.  Integer instructions on the high words.
__device__ __forceinline__ int warp_exponent(double v0, double v1) {
    int h = max(__double2hiint(v0) & 0x7fffffff, __double2hiint(v1) & 0x7fffffff);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
    const int e = (h >> 20) - 1022;
    return h == 0 ? kZeroExponent : (e > 900 ? kBadExponent : max(e, -900));
}
__device__ __forceinline__ bool usable(int e) { return e >= -900 && e <= 900; }

// base -> digits in the order in which a lane reads its operand fragments: word
// ((digit 40 + column tile) 2 + k half) 32 + lane holds terms q = 32 half + {2t, 2t+1, 2t+8, 2t+9} + {0, 16}
// of column 8 tile + g (g = lane / 4, t = lane % 4); one warp per column.
__global__ void k_base_digits(const double* __restrict__ base, int nn, uint4* __restrict__ digits,
                              int* __restrict__ exponent) {
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (j >= kNout) return;
    double v[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) v[h] = lane + 32 * h < nn ? base[(size_t)(lane + 32 * h) * kNout + j] : 0.0;
    const int e = warp_exponent(v[0], v[1]);
    if (lane == 0) exponent[j] = e;
    bf16* out = reinterpret_cast<bf16*>(digits);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        int d[kDigits];
        fixed_digits(usable(e) ? v[h] : 0.0, usable(e) ? e : 0, d);
        // term q = 32 h + lane: k step of 16, position in it -> fragment register and half
        const int s16 = lane >> 4, p = lane & 15, t = (p & 7) >> 1;
        const int word = 2 * s16 + (p >> 3);   // of the uint4: {b0, b1} of two k steps
        for (int i = 0; i < kDigits; ++i) {
            const size_t w = ((size_t)(i * (kNout / 8) + j / 8) * 2 + h) * 32 + (j & 7) * 4 + t;
            out[w * 8 + word * 2 + (p & 1)] = __float2bfloat16_rn((float)d[i]);
        }
    }
}

// baseline mu_j + sum_ab l_a(x_p) l_b(x_q) base[a n + b][j] for one parameter row
__device__ double baseline(const MapArgs& a, const double* t, int j) {
    double u = a.mu[j];
    if (a.base) {
        double la[kMaxNodes], lb[kMaxNodes];
        lobatto_basis(t[a.base_in[0]] * a.dscale[a.base_in[0]] + a.dshift[a.base_in[0]], a.nodes, la);
        lobatto_basis(t[a.base_in[1]] * a.dscale[a.base_in[1]] + a.dshift[a.base_in[1]], a.nodes, lb);
        for (int p = 0; p < a.nodes; ++p)
            for (int q = 0; q < a.nodes; ++q) u += la[p] * lb[q] * a.base[(size_t)(p * a.nodes + q) * kNout + j];
    }
    return u;
}

// ---- float pairs (hi + lo, |lo| <= ulp(hi) / 2): sums and products to about 2^-46
struct fpair {
    float hi, lo;
};
__device__ __forceinline__ fpair two_sum(float a, float b) {   // exact (Knuth)
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ fpair fast_two_sum(float a, float b) {   // exact for |a| >= |b| (Dekker)
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ fpair pair_of(double v) {
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}
__device__ __forceinline__ fpair pair_add(fpair a, fpair b) {
    fpair s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ fpair pair_mul(fpair a, fpair b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return fast_two_sum(p, e);
}
__device__ __forceinline__ fpair pair_mul(fpair a, float b) {
    const float p = __fmul_rn(a.hi, b);
    return fast_two_sum(p, fmaf(a.lo, b, fmaf(a.hi, b, -p)));
}
__device__ __forceinline__ float exp2i(int e) {   // 2^e for -126 <= e <= 127
    return __int_as_float((e + 127) << 23);
}

constexpr float kTiny = 7.174648137343064e-43f;   // 2^-140: low words may lose up to 2^-149 by underflow

struct PredictArgs {
    Passes ps;
    const float* bias[kLayers];
    const float* x;         // network inputs [n][6], or
    const double* theta;    // parameters [n][6], encoded by the map
    int n;
    float* out;             // [n][320]
    MapArgs map;
    const struct ColumnConst* cols;   // [320] of this call (k_columns), for many rows
};

// The columns' constants of the decoding (float pairs) and the column exponents of the baseline, from
// the map's arrays as they are at this call.  Each column is taken in the power-of-two unit of its baseline (else
// of mu or sd), sigma with it: curves in any unit stay within FP32's exponents (without that 1e30
// took 570 us for 8192 rows, all done again in FP64).
struct ColumnConst {
    float2 mu, sd, shot, ref, isig;
    float tiny;   // kTiny, 0 when shot and ref are zero
    int e;
};
__device__ __forceinline__ ColumnConst column_const(const MapArgs& m, int j) {
    auto as2 = [](fpair p) { return make_float2(p.hi, p.lo); };
    ColumnConst c;
    const int e = m.base ? m.exponent[j] : kZeroExponent;
    const double mu = m.mu[j], sd = m.sd[j];
    int k = e;
    if (!usable(e)) {
        const double big = fmax(fabs(mu), fabs(sd));
        k = big > 1e-270 && big < 1e270 ? ((__double2hiint(big) >> 20) - 1022) : 0;
    }
    const double s = __hiloint2double((1023 - k) << 20, 0);   // 2^-k
    c.mu = as2(pair_of(mu * s));
    c.sd = as2(pair_of(sd * s));
    c.shot = as2(pair_of(m.shot[j] * s));
    c.ref = as2(pair_of(m.ref ? m.ref[j] * s : 0.0));
    c.isig = as2(pair_of(1.0 / (m.sigma ? m.sigma[j] * s : s)));
    c.tiny = m.shot[j] != 0.0 || (m.ref && m.ref[j] != 0.0) ? kTiny : 0.f;
    c.e = usable(e) ? 0 : e;   // relative to the unit
    return c;
}
__global__ void k_columns(MapArgs m, ColumnConst* __restrict__ out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < kNout) out[j] = column_const(m, j);
}

// The rows' constants.
template <int R>
struct RowConst {
    float2 amp[2][R], t5[R];   // A b sigma_8^2 (gE), A^2 sigma_8^2 (EE, BB); shot-noise scale
    float tiny[2][R];          // kTiny, 0 when the amplitude is zero
    int e[R];                  // exponent of the weights' digits
    float wsum[R];             // sum of |w_q|
    double la[R][kMaxNodes], lb[R][kMaxNodes];
};

// The constants of R parameter rows and their Lagrange weights as digit fragments
// wd[kWDigits][R / 16][kBaseKsteps][32]; ends with a barrier.
template <int R>
__device__ __forceinline__ void decode_rows(const MapArgs& m, const double* theta, int r0, int rows, RowConst<R>& rc,
                                            uint4* wd) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int MT = R / 16;
    auto as2 = [](fpair p) { return make_float2(p.hi, p.lo); };
    for (int i = tid; i < 3 * R; i += kRowThreads) {
        const int r = i / 3, k = i - 3 * r;
        if (r >= rows) continue;
        const double* th = theta + (size_t)(r0 + r) * kNin;
        if (k == 0) {
            const double s2 = th[2] * th[2];
            const double amp[2] = {s2 * (th[0] * th[1]), s2 * (th[0] * th[0])};
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                rc.amp[c][r] = as2(pair_of(amp[c]));
                rc.tiny[c][r] = amp[c] != 0.0 ? kTiny : 0.f;
            }
            rc.t5[r] = as2(pair_of(th[5]));
        } else if (m.base) {
            const int c = m.base_in[k - 1];
            lobatto_basis_fast(th[c] * m.dscale[c] + m.dshift[c], m, k == 1 ? rc.la[r] : rc.lb[r]);
        }
    }
    __syncthreads();
    if (!m.base) return;
    const int nn = m.nodes * m.nodes;
    bf16* wo = reinterpret_cast<bf16*>(wd);
    for (int r = warp; r < R; r += kRowThreads / 32) {   // one warp per row
        double v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int q = lane + 32 * h;
            v[h] = (r < rows && q < nn) ? rc.la[r][q / m.nodes] * rc.lb[r][q % m.nodes] : 0.0;
        }
        const int e = warp_exponent(v[0], v[1]);
        float sum = (float)(fabs(v[0]) + fabs(v[1]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) {
            rc.e[r] = e;
            rc.wsum[r] = sum;
        }
        const int mt = r >> 4, rr = r & 15;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int d[kWDigits];
            weight_digits(usable(e) ? v[h] : 0.0, usable(e) ? e : 0, d);
            // term q = 32 h + lane = 16 ks + p: register (rr >> 3) + 2 (p >> 3) of lane 4 (rr & 7) + (p & 7) / 2
            const int ks = 2 * h + (lane >> 4), p = lane & 15;
            const int reg = (rr >> 3) + 2 * (p >> 3), ln = 4 * (rr & 7) + ((p & 7) >> 1);
#pragma unroll
            for (int i = 0; i < kWDigits; ++i)
                wo[((((i * MT + mt) * kBaseKsteps + ks) * 32 + ln) * 4 + reg) * 2 + (p & 1)] =
                    __float2bfloat16_rn((float)d[i]);
        }
    }
    __syncthreads();
}

// One output of a parameter row th in FP64: y the network's output j, la and lb the row's Lagrange
// weights.  WARP: by a whole warp (an FP64 instruction takes as long for one lane as for 32: 40 of them
// instead of 110); else by each calling lane.
template <bool WARP>
__device__ __noinline__ float decode_exact(const MapArgs& m, const double* la, const double* lb, const double* th, int j,
                                           float y) {
    double b = 0.0;
    if (m.base) {
        const double* base = m.base + j;
        if (WARP) {
            for (int q = threadIdx.x & 31; q < m.nodes * m.nodes; q += 32)
                b = fma(la[q / m.nodes] * lb[q % m.nodes], base[(size_t)q * kNout], b);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
        } else {
            for (int p = 0; p < m.nodes; ++p) {
                double row = 0.0;
                for (int q = 0; q < m.nodes; ++q) row = fma(lb[q], base[(size_t)(p * m.nodes + q) * kNout], row);
                b = fma(la[p], row, b);
            }
        }
    }
    const double amp = th[2] * th[2] * (j < 2 * (kNout / 8) ? th[0] * th[1] : th[0] * th[0]);
    double v = amp * (m.mu[j] + b + m.sd[j] * (double)y) + th[5] * m.shot[j];
    if (m.ref) v -= m.ref[j];
    if (m.sigma) v /= m.sigma[j];
    return (float)v;
}

// The decoding of one tile: rows 16 mt + {g, g + 8}, columns 8 tile + {2 t, 2 t + 1}, from the
// network outputs y[4] on the mma accumulator's positions; theta: the first row's parameters.
//
// The digit products and the float pairs bound their error (the terms' magnitudes times 2^-43, the
// digits' bound above, and 2^-140 where a low word may underflow).  An output for which that is more than
// a quarter of its last FP32 place, which is no number or whose exponents leave FP32's range is done
// again in FP64 (decode_exact), one by one by the warp or, when they are more than two, each by its lane:
// the stored value is the FP64 one to 3/4 of a place, whatever the map holds.  Curves of some hundred
// error bars around the reference repeat a fraction of a per cent (8192 rows 98 -> 107 us); where a
// baseline spans 2^17 and more nearly all are repeated (300 us, 280 in float pairs before).
template <int R>
__device__ __forceinline__ void decode_tile(const MapArgs& m, const uint4* wd, const RowConst<R>& rc,
                                            const ColumnConst* cc, int mt, int tile, int rows, const float y[4],
                                            const double* theta, float* out) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    constexpr int MT = R / 16;
    constexpr unsigned full = 0xffffffffu;
    auto pr = [](float2 v) { return fpair{v.x, v.y}; };
    float acc[kOrders][4];
#pragma unroll
    for (int o = 0; o < kOrders; ++o)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[o][r] = 0.f;
    if (m.base) {
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            uint4 bd[kDigits];
#pragma unroll
            for (int i = 0; i < kDigits; ++i) bd[i] = m.digits[((size_t)(i * (kNout / 8) + tile) * 2 + h) * 32 + lane];
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int i = 0; i < kWDigits; ++i) {
                    const uint4 av = wd[((i * MT + mt) * kBaseKsteps + 2 * h + k) * 32 + lane];
                    const uint32_t af[4] = {av.x, av.y, av.z, av.w};
#pragma unroll
                    for (int q = 0; q < kDigits; ++q)
                        if (i + q < kOrders) mma_bf16(acc[i + q], af, k ? bd[q].z : bd[q].x, k ? bd[q].w : bd[q].y);
                }
        }
    }
    ColumnConst cq[2];
    cq[0] = cc[8 * tile + 2 * t];
    cq[1] = cc[8 * tile + 2 * t + 1];
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        const int r = mt * 16 + g + 8 * hh;
        float res[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int v = 2 * hh + q;
            const ColumnConst& c = cq[q];
            bool done = r >= rows;
            if (!done) {
                fpair u = pr(c.mu);
                float mag = fabsf(c.mu.x), eb = 0.f;   // the terms' magnitudes, the digits' error
                bool range = true;
                if (m.base && c.e != kZeroExponent) {
                    // sum_o acc_o 2^(-8 o): the first four orders exactly, the rest in one float
                    const float low = fmaf(acc[6][v], exp2i(-48), fmaf(acc[5][v], exp2i(-40), __fmul_rn(acc[4][v], exp2i(-32))));
                    const fpair s1 = two_sum(acc[0][v], __fmul_rn(acc[1][v], exp2i(-8)));
                    const fpair s2 = two_sum(s1.hi, __fmul_rn(acc[2][v], exp2i(-16)));
                    const fpair s3 = two_sum(s2.hi, __fmul_rn(acc[3][v], exp2i(-24)));
                    fpair b = fast_two_sum(s3.hi, __fadd_rn(s3.lo, __fadd_rn(s2.lo, __fadd_rn(s1.lo, low))));
                    const int er = rc.e[r], ec = c.e;
                    range = er > -50 && er < 50 && ec == 0;   // ec: 0, or kBadExponent
                    const int e = range ? er : 0;
                    b.hi *= exp2i(e - 14);   // the digits' unit: 2^(e_r + e_c) 2^-14
                    b.lo *= exp2i(e - 14);
                    u = pair_add(u, b);
                    mag += fabsf(b.hi);
                    eb = fmaf(rc.wsum[r], exp2i(-48), exp2i(e - 45));
                }
                const int ci = tile < 2 * (kNout / 8) / 8 ? 0 : 1;
                const fpair amp = pr(rc.amp[ci][r]);
                const float tiny = rc.tiny[ci][r];
                const fpair net = pair_mul(pr(c.sd), y[v]), shot = pair_mul(pr(rc.t5[r]), pr(c.shot));
                u = pair_add(u, net);
                mag += fabsf(net.hi);
                u = pair_mul(u, amp);
                u = pair_add(u, shot);
                u = pair_add(u, fpair{-c.ref.x, -c.ref.y});
                const float all = fmaf(fabsf(amp.hi), mag, fabsf(shot.hi) + fabsf(c.ref.x));
                u = pair_mul(u, pr(c.isig));
                res[q] = __fadd_rn(u.hi, u.lo);
                const float err = fmaf(fabsf(amp.hi), eb + tiny, fmaf(all, exp2i(-43), fmaf(mag, tiny, fmaxf(tiny, c.tiny))));
                const float bound = fmaf(fabsf(c.isig.x), err, all * kTiny);
                done = range && bound <= fabsf(res[q]) * exp2i(-26) && fabsf(res[q]) < INFINITY;
            }
            unsigned again = __ballot_sync(full, !done);
            if (__popc(again) > 2) {   // warp-uniform
                if (!done)
                    res[q] = decode_exact<false>(m, rc.la[r], rc.lb[r], theta + (size_t)r * kNin, 8 * tile + 2 * t + q, y[v]);
                again = 0;
            }
            while (again) {
                const int src = __ffs(again) - 1, rs = mt * 16 + (src >> 2) + 8 * hh;
                again &= again - 1;
                const float x = decode_exact<true>(m, rc.la[rs], rc.lb[rs], theta + (size_t)rs * kNin, 8 * tile + 2 * (src & 3) + q,
                                                   __shfl_sync(full, y[v], src));
                if (lane == src) res[q] = x;
            }
        }
        if (r < rows) store2(out + (size_t)r * kNout + 8 * tile + 2 * t, res[0], res[1]);
    }
}

// Network inputs of R rows (encoded by the map, or given), BF16 [R][16], zero padded.
template <int R, bool MAP>
__device__ __forceinline__ void input_rows(const PredictArgs& a, int r0, int rows, bf16* act, int lda) {
    for (int i = threadIdx.x; i < R * 16; i += kRowThreads) {
        const int r = i >> 4, c = i & 15;
        float v = 0.f;
        if (r < rows && c < kNin) {
            if constexpr (MAP) v = (float)(a.theta[(size_t)(r0 + r) * kNin + c] * (double)a.map.scale[c] + (double)a.map.shift[c]);
            else v = a.x[(size_t)(r0 + r) * kNin + c];
        }
        act[r * lda + c] = __float2bfloat16_rn(v);
    }
}

// Forward pass of 32 rows per CTA and, with MAP, the whole prediction: the parameters' encoding
// before it and the decoding after it
//   (pre_c (mu + sum_q w_q base_q + sd y) + theta_5 shot - ref) / sigma,
// the baseline by exact digit products (above), the rest in float pairs, FP64 where those do not decide
// the FP32 result.
//
// What bounds it: the GELUs' instructions and the mma issue.  8192 rows: 287 us as eight launches
// with the decoding's last operations in FP64 -> 98 us (90 us without decode_tile's error bound and the
// seventh weight digit; 107 us near a reference curve, where a per cent of the outputs are done
// again).
template <bool MAP>
__global__ void __launch_bounds__(kRowThreads, 2) k_predict(const __grid_constant__ PredictArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int R = kPredRows, MT = R / 16;
    WeightRing<kPredStages> ring;
    ring.ring = reinterpret_cast<bf16*>(smem_raw);
    ring.n_pass = kLayers;
    bf16* buf[2];
    buf[0] = ring.ring + kPredStages * kStageElems;
    buf[1] = buf[0] + R * kPredLd;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int r0 = blockIdx.x * R, rows = min(R, a.n - r0);
    for (int c = 0; c < kPredStages - 1; ++c) ring.load(a.ps);
    input_rows<R, MAP>(a, r0, rows, buf[0], kPredLd);
    int cur = 0;
    for (int l = 0; l < kLayers - 1; ++l) {
        float acc[MT][4][4];
        if (l == 0) row_product<MT, 4, 16, kPredLd>(ring, a.ps, buf[cur], acc);
        else row_product<MT, 4, 256, kPredLd>(ring, a.ps, buf[cur], acc);
        bf16* nx = buf[cur ^ 1];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = 8 * (warp * 4 + j) + 2 * t;
            const float2 b = *reinterpret_cast<const float2*>(a.bias[l] + c);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    *reinterpret_cast<__nv_bfloat162*>(nx + (mt * 16 + g + 8 * h) * kPredLd + c) =
                        __nv_bfloat162(__float2bfloat16_rn(gelu(acc[mt][j][2 * h] + b.x)),
                                       __float2bfloat16_rn(gelu(acc[mt][j][2 * h + 1] + b.y)));
        }
        cur ^= 1;
    }
    float y[MT][5][4];
    row_product<MT, 5, 256, kPredLd>(ring, a.ps, buf[cur], y);
    cp_wait<0>();
    __syncthreads();   // the ring and the activations are free
    // network outputs in shared memory on their accumulator positions [tile][mt][lane]: the decoding
    // loops over the tiles without unrolling (an unrolled one stalls on instruction fetches)
    uint4* wd = reinterpret_cast<uint4*>(smem_raw);                     // [kWDigits][MT][kBaseKsteps][32]
    float4* ys = reinterpret_cast<float4*>(wd + kWDigits * MT * kBaseKsteps * 32);   // [kNout / 8][MT][32]
    RowConst<R>& rc = *reinterpret_cast<RowConst<R>*>(ys + (kNout / 8) * MT * 32);
    static_assert(sizeof(uint4) * kWDigits * MT * kBaseKsteps * 32 + sizeof(float4) * (kNout / 8) * MT * 32 +
                      sizeof(RowConst<R>) <= kPredSmem, "the decoding fits in the forward pass's shared memory");
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int c = 8 * (warp * 5 + j) + 2 * t;
        const float2 b = *reinterpret_cast<const float2*>(a.bias[kLayers - 1] + c);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            const float4 v = make_float4(y[mt][j][0] + b.x, y[mt][j][1] + b.y, y[mt][j][2] + b.x, y[mt][j][3] + b.y);
            if constexpr (MAP) {
                ys[((warp * 5 + j) * MT + mt) * 32 + lane] = v;
            } else {
                const int r = mt * 16 + g;
                float* o = a.out + (size_t)(r0 + r) * kNout + c;
                if (r < rows) store2(o, v.x, v.y);
                if (r + 8 < rows) store2(o + 8 * kNout, v.z, v.w);
            }
        }
    }
    if constexpr (MAP) {
        decode_rows<R>(a.map, a.theta, r0, rows, rc, wd);   // begins after the stores above: other addresses, and a barrier inside
#pragma unroll 1
        for (int i = warp * 5 * MT; i < (warp + 1) * 5 * MT; ++i) {
            const float4 v = ys[i * 32 + lane];
            const float yv[4] = {v.x, v.y, v.z, v.w};
            decode_tile<R>(a.map, wd, rc, a.cols, i % MT, i / MT, rows, yv, a.theta + (size_t)r0 * kNin,
                           a.out + (size_t)r0 * kNout);
        }
    }
}

// The same for few rows: 16 rows on a cluster of kSplit CTAs, each a quarter of every layer's columns
// and of the outputs.  What bounds it: the latency of the dependent layers.  50 rows: 85 us as eight
// launches, 49 us with one CTA per 16 rows -> 27 us.
template <bool MAP>
__global__ void __cluster_dims__(kSplit, 1, 1) __launch_bounds__(kRowThreads, 1)
k_predict_few(const __grid_constant__ PredictArgs a) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cg::cluster_group cluster = cg::this_cluster();
    SliceRing ring;
    ring.ring = reinterpret_cast<bf16*>(smem_raw);
    ring.n_pass = kLayers;
    ring.rank = (int)cluster.block_rank();
    bf16* buf[2];
    buf[0] = ring.ring + kSliceStages * kSliceElems;
    buf[1] = buf[0] + 16 * kActLd;
    // the decoding's rows and columns are prepared while the first weights arrive
    constexpr int R = 16;
    uint4* wd = reinterpret_cast<uint4*>(smem_raw + kSliceSmem);                     // [kWDigits][1][kBaseKsteps][32]
    RowConst<R>& rc = *reinterpret_cast<RowConst<R>*>(wd + kWDigits * kBaseKsteps * 32);
    ColumnConst* cols = reinterpret_cast<ColumnConst*>(&rc + 1);                     // [kNout / kSplit]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int r0 = (int)(blockIdx.x / kSplit) * R, rows = min(R, a.n - r0);
    const int h0 = ring.rank * (256 / kSplit), o0 = ring.rank * (kNout / kSplit);
    for (int c = 0; c < kSliceStages - 1; ++c) ring.load(a.ps);
    input_rows<R, MAP>(a, r0, rows, buf[0], kActLd);
    if constexpr (MAP) {
        if (tid < kNout / kSplit) cols[tid] = column_const(a.map, o0 + tid);
        decode_rows<R>(a.map, a.theta, r0, rows, rc, wd);
    }
    cluster.sync();   // every CTA of the cluster runs before its shared memory is written
    const int c = h0 + 8 * warp + 2 * t;
    int cur = 0;
    for (int l = 0; l < kLayers - 1; ++l) {
        float acc[1][4];
        if (l == 0) slice_product<16, 8>(ring, a.ps, buf[cur], acc);
        else slice_product<256, 8>(ring, a.ps, buf[cur], acc);
        const float2 b = *reinterpret_cast<const float2*>(a.bias[l] + c);
#pragma unroll
        for (int h = 0; h < 2; ++h)
            share2(buf[cur ^ 1], g + 8 * h, c, gelu(acc[0][2 * h] + b.x), gelu(acc[0][2 * h + 1] + b.y));
        cur ^= 1;
        cluster.sync();   // after the last layer: no CTA leaves while the others write to it
    }
    float y[2][4];
    slice_product<256, 10>(ring, a.ps, buf[cur], y);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        if (warp + 8 * j >= kNout / kSplit / 8) break;   // warp-uniform
        const int tile = o0 / 8 + warp + 8 * j, co = 8 * tile + 2 * t;
        const float2 b = *reinterpret_cast<const float2*>(a.bias[kLayers - 1] + co);
        const float v[4] = {y[j][0] + b.x, y[j][1] + b.y, y[j][2] + b.x, y[j][3] + b.y};
        if constexpr (MAP) {
            decode_tile<R>(a.map, wd, rc, cols - o0, 0, tile, rows, v, a.theta + (size_t)r0 * kNin,
                           a.out + (size_t)r0 * kNout);
        } else {
            float* o = a.out + (size_t)(r0 + g) * kNout + co;
            if (g < rows) store2(o, v[0], v[1]);
            if (g + 8 < rows) store2(o + 8 * kNout, v[2], v[3]);
        }
    }
}
constexpr size_t kFewSmem = kSliceSmem + sizeof(uint4) * kWDigits * kBaseKsteps * 32 + sizeof(RowConst<16>) +
                            sizeof(ColumnConst) * (kNout / kSplit);

// training targets: derived curves u of native template slots [n][LPP_N_MOMENTS][40] (FP64, unit
// amplitude, no shot noise), y = (u - baseline) / sd
__global__ void k_targets(const double* __restrict__ theta, const double* __restrict__ native, int n,
                          float* __restrict__ y, MapArgs a) {
    constexpr int nb = kNout / 8;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * kNout; i += gridDim.x * blockDim.x) {
        const int r = i / kNout, j = i % kNout, c = j / nb, b = j % nb;
        const double* o = native + (size_t)r * LPP_N_MOMENTS * nb;
        double u;
        if (c < 2) {
            u = a.N[c][0] * o[1 * nb + b] + a.N[c][1] * o[2 * nb + b] + a.N[c][2] * o[3 * nb + b];
        } else {
            const int li = (c - 2) % 3;
            const double mm = a.M[li][0] * o[7 * nb + b] + a.M[li][1] * o[8 * nb + b] + a.M[li][2] * o[9 * nb + b];
            u = 0.5 * (o[(4 + li) * nb + b] + (c < 5 ? mm : -mm));
        }
        y[i] = (float)((u - baseline(a, theta + (size_t)r * kNin, j)) / a.sd[j]);
    }
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

struct lpp_surrogate_s {
    int batch = 0;
    long long step = 0;
    char* ws = nullptr;
    size_t need = 0;
    // offsets
    size_t w[kLayers], b[kLayers], mw[kLayers], vw[kLayers], mb[kLayers], vb[kLayers], dw[kLayers], db[kLayers];
    size_t w16[kLayers], w16t[kLayers], actt[kLayers], gt[kLayers], g32[kLayers], loss;
    size_t digits, exponent;          // the decoding's digits of the map's base
    size_t cols;                      // and the columns' constants of a call
    bool has_map = false;
    bool base_split = false;          // digits, exponent hold the current map's base
    MapArgs map;
};

extern "C" lpp_status lpp_surrogate_create(int batch, lpp_surrogate_t* out) {
    if (!out || batch < 32 || batch % 32 != 0 || batch > (1 << 20)) return LPP_ERR_INVALID_ARG;
    lpp_surrogate_t s = new lpp_surrogate_s();
    s->batch = batch;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align256(off + bytes); return o; };
    for (int l = 0; l < kLayers; ++l) {
        const size_t nw = (size_t)kOut[l] * kInPad[l];
        s->w[l] = take(nw * 4);
        s->mw[l] = take(nw * 4);
        s->vw[l] = take(nw * 4);
        s->dw[l] = take(nw * 4);
        s->b[l] = take(kOut[l] * 4);
        s->mb[l] = take(kOut[l] * 4);
        s->vb[l] = take(kOut[l] * 4);
        s->db[l] = take(kOut[l] * 4);
        s->w16[l] = take(nw * 2);
        s->w16t[l] = take(nw * 2);
        s->actt[l] = take((size_t)batch * kInPad[l] * 2);
        s->gt[l] = take((size_t)batch * kOut[l] * 2);
        s->g32[l] = take((size_t)batch * kOut[l] * 4);
    }
    s->loss = take(8);
    s->digits = take((size_t)kDigitWords * sizeof(uint4));
    s->exponent = take((size_t)kNout * sizeof(int));
    s->cols = take((size_t)kNout * sizeof(ColumnConst));
    s->need = off;
    *out = s;
    return LPP_OK;
}

extern "C" void lpp_surrogate_destroy(lpp_surrogate_t s) { delete s; }

extern "C" lpp_status lpp_surrogate_workspace_size(lpp_surrogate_t s, size_t* bytes) {
    if (!s || !bytes) return LPP_ERR_INVALID_ARG;
    *bytes = s->need;
    return LPP_OK;
}

static AdamArgs adam_args(lpp_surrogate_t s) {
    AdamArgs a;
    memset(&a, 0, sizeof(a));
    for (int l = 0; l < kLayers; ++l) {
        AdamLayer& L = a.L[l];
        L.w = (float*)(s->ws + s->w[l]);
        L.b = (float*)(s->ws + s->b[l]);
        L.mw = (float*)(s->ws + s->mw[l]);
        L.vw = (float*)(s->ws + s->vw[l]);
        L.mb = (float*)(s->ws + s->mb[l]);
        L.vb = (float*)(s->ws + s->vb[l]);
        L.dw = (float*)(s->ws + s->dw[l]);
        L.db = (float*)(s->ws + s->db[l]);
        L.w16 = (bf16*)(s->ws + s->w16[l]);
        L.w16t = (bf16*)(s->ws + s->w16t[l]);
        L.out = kOut[l];
        L.in = kIn[l];
        L.inp = kInPad[l];
    }
    return a;
}

// Host params: for every layer W [out][in] then b [out], FP32, unpadded.
extern "C" lpp_status lpp_surrogate_set_workspace(lpp_surrogate_t s, void* dev, size_t bytes, const float* params,
                                                  void* stream) {
    if (!s || !dev || !params) return LPP_ERR_INVALID_ARG;
    if (((uintptr_t)dev & 255) != 0) return LPP_ERR_INVALID_ARG;
    if (bytes < s->need) return LPP_ERR_WORKSPACE;
    s->ws = (char*)dev;
    s->step = 0;
    s->base_split = false;   // the digits of the map's base went with the old contents
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(s->ws, 0, s->need, st) != cudaSuccess) return LPP_ERR_CUDA;
    std::vector<float> wpad;
    size_t p = 0;
    for (int l = 0; l < kLayers; ++l) {
        wpad.assign((size_t)kOut[l] * kInPad[l], 0.f);
        for (int r = 0; r < kOut[l]; ++r)
            for (int c = 0; c < kIn[l]; ++c) wpad[(size_t)r * kInPad[l] + c] = params[p++];
        if (cudaMemcpyAsync(s->ws + s->w[l], wpad.data(), wpad.size() * 4, cudaMemcpyHostToDevice, st) != cudaSuccess)
            return LPP_ERR_CUDA;
        if (cudaMemcpyAsync(s->ws + s->b[l], params + p, kOut[l] * 4, cudaMemcpyHostToDevice, st) != cudaSuccess)
            return LPP_ERR_CUDA;
        p += kOut[l];
        if (cudaStreamSynchronize(st) != cudaSuccess) return LPP_ERR_CUDA;
    }
    AdamArgs a = adam_args(s);
    k_refresh<<<dim3(64, kLayers), 256, 0, st>>>(a);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return LPP_ERR_CUDA;
    return LPP_OK;
}

// Training state (checkpoint): a 32-byte header (magic, version, Adam step, FNV-1a 64-bit
// checksum of the rest, 8 reserved bytes), then per layer the FP32 master W (rows padded to
// kInPad, the device layout), its Adam moments m and v, the bias and its m and v.  The BF16
// copies are derived and rebuilt on load.
constexpr unsigned kStateMagic = 0x5350504Cu;   // "LPPS"
constexpr unsigned kStateVersion = 2u;
constexpr size_t kStateHeader = 32;

static unsigned long long fnv1a64(const unsigned char* p, size_t n) {
    unsigned long long h = 1469598103934665603ull;
    for (size_t i = 0; i < n; ++i) {
        h ^= p[i];
        h *= 1099511628211ull;
    }
    return h;
}

static size_t state_bytes() {
    size_t b = kStateHeader;
    for (int l = 0; l < kLayers; ++l) b += (size_t)3 * ((size_t)kOut[l] * kInPad[l] + kOut[l]) * 4;
    return b;
}

extern "C" lpp_status lpp_surrogate_state_size(lpp_surrogate_t s, size_t* bytes) {
    if (!s || !bytes) return LPP_ERR_INVALID_ARG;
    *bytes = state_bytes();
    return LPP_OK;
}

// The state's device arrays in file order: {offset, bytes} per layer.
static void state_parts(lpp_surrogate_t s, std::vector<std::pair<size_t, size_t>>& parts) {
    parts.clear();
    for (int l = 0; l < kLayers; ++l) {
        const size_t nw = (size_t)kOut[l] * kInPad[l] * 4, nb = (size_t)kOut[l] * 4;
        parts.push_back({s->w[l], nw});
        parts.push_back({s->mw[l], nw});
        parts.push_back({s->vw[l], nw});
        parts.push_back({s->b[l], nb});
        parts.push_back({s->mb[l], nb});
        parts.push_back({s->vb[l], nb});
    }
}

extern "C" lpp_status lpp_surrogate_save_state(lpp_surrogate_t s, void* host, size_t bytes, void* stream) {
    if (!s || !s->ws || !host || bytes < state_bytes()) return LPP_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    unsigned char* p = (unsigned char*)host;
    const unsigned hdr[2] = {kStateMagic, kStateVersion};
    memcpy(p, hdr, 8);
    const long long step = s->step;
    memcpy(p + 8, &step, 8);
    memset(p + 16, 0, 16);
    size_t o = kStateHeader;
    std::vector<std::pair<size_t, size_t>> parts;
    state_parts(s, parts);
    for (const auto& q : parts) {
        if (cudaMemcpyAsync(p + o, s->ws + q.first, q.second, cudaMemcpyDeviceToHost, st) != cudaSuccess)
            return LPP_ERR_CUDA;
        o += q.second;
    }
    if (cudaStreamSynchronize(st) != cudaSuccess) return LPP_ERR_CUDA;
    const unsigned long long sum = fnv1a64(p + kStateHeader, state_bytes() - kStateHeader);
    memcpy(p + 16, &sum, 8);
    return LPP_OK;
}

extern "C" lpp_status lpp_surrogate_load_state(lpp_surrogate_t s, const void* host, size_t bytes, void* stream) {
    if (!s || !s->ws || !host || bytes < state_bytes()) return LPP_ERR_INVALID_ARG;
    const unsigned char* p = (const unsigned char*)host;
    unsigned hdr[2];
    memcpy(hdr, p, 8);
    if (hdr[0] != kStateMagic || hdr[1] != kStateVersion) return LPP_ERR_INVALID_ARG;
    long long step = 0;
    memcpy(&step, p + 8, 8);
    if (step < 0) return LPP_ERR_INVALID_ARG;
    unsigned long long sum = 0;
    memcpy(&sum, p + 16, 8);
    if (sum != fnv1a64(p + kStateHeader, state_bytes() - kStateHeader)) return LPP_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    size_t o = kStateHeader;
    std::vector<std::pair<size_t, size_t>> parts;
    state_parts(s, parts);
    for (const auto& q : parts) {
        if (cudaMemcpyAsync(s->ws + q.first, p + o, q.second, cudaMemcpyHostToDevice, st) != cudaSuccess)
            return LPP_ERR_CUDA;
        o += q.second;
    }
    AdamArgs a = adam_args(s);
    k_refresh<<<dim3(64, kLayers), 256, 0, st>>>(a);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return LPP_ERR_CUDA;
    s->step = step;
    return LPP_OK;
}

extern "C" lpp_status lpp_surrogate_get_params(lpp_surrogate_t s, float* params, void* stream) {
    if (!s || !s->ws || !params) return LPP_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    std::vector<float> wpad;
    size_t p = 0;
    for (int l = 0; l < kLayers; ++l) {
        wpad.resize((size_t)kOut[l] * kInPad[l]);
        if (cudaMemcpyAsync(wpad.data(), s->ws + s->w[l], wpad.size() * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess)
            return LPP_ERR_CUDA;
        if (cudaMemcpyAsync(params + p + (size_t)kOut[l] * kIn[l], s->ws + s->b[l], kOut[l] * 4,
                            cudaMemcpyDeviceToHost, st) != cudaSuccess)
            return LPP_ERR_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) return LPP_ERR_CUDA;
        for (int r = 0; r < kOut[l]; ++r)
            for (int c = 0; c < kIn[l]; ++c) params[p++] = wpad[(size_t)r * kInPad[l] + c];
        p += kOut[l];
    }
    return LPP_OK;
}

static Passes passes(lpp_surrogate_t s) {
    Passes p;
    for (int l = 0; l < kLayers; ++l) p.w[l] = (const bf16*)(s->ws + s->w16[l]);
    for (int l = kLayers - 1; l > 0; --l) p.w[2 * kLayers - 1 - l] = (const bf16*)(s->ws + s->w16t[l]);
    return p;
}

// The fused forward pass (MAP: the whole prediction) of n rows: clusters of four CTAs per 16 rows
// while they fit the SMs at once (608 rows on 152 SMs), one CTA per 32 rows beyond.
template <bool MAP>
static cudaError_t launch_predict(lpp_surrogate_t s, PredictArgs& a, cudaStream_t st) {
    if (a.n == 0) return cudaSuccess;
    a.ps = passes(s);
    for (int l = 0; l < kLayers; ++l) a.bias[l] = (const float*)(s->ws + s->b[l]);
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int groups = (a.n + 15) / 16;
    if (groups * kSplit <= sms) {
        cudaFuncSetAttribute(k_predict_few<MAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewSmem);
        k_predict_few<MAP><<<groups * kSplit, kRowThreads, kFewSmem, st>>>(a);
    } else {
        if (MAP) {
            a.cols = (const ColumnConst*)(s->ws + s->cols);
            k_columns<<<(kNout + 63) / 64, 64, 0, st>>>(a.map, (ColumnConst*)(s->ws + s->cols));
        }
        cudaFuncSetAttribute(k_predict<MAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPredSmem);
        k_predict<MAP><<<(a.n + kPredRows - 1) / kPredRows, kRowThreads, kPredSmem, st>>>(a);
    }
    return cudaGetLastError();
}

extern "C" lpp_status lpp_surrogate_infer(lpp_surrogate_t s, const float* x, int n, float* y, void* stream) {
    if (!s || !s->ws || n < 0 || (n > 0 && (!x || !y))) return LPP_ERR_INVALID_ARG;
    PredictArgs a;
    memset(&a, 0, sizeof(a));
    a.x = x;
    a.n = n;
    a.out = y;
    return launch_predict<false>(s, a, (cudaStream_t)stream) == cudaSuccess ? LPP_OK : LPP_ERR_CUDA;
}

extern "C" lpp_status lpp_surrogate_set_map(lpp_surrogate_t s, const lpp_surrogate_map* m) {
    if (!s || !m || !m->mu || !m->sd || !m->shot) return LPP_ERR_INVALID_ARG;
    MapArgs a;
    memset(&a, 0, sizeof(a));
    for (int c = 0; c < kNin; ++c) {
        if (!m->feed[c]) continue;
        if (!(m->hi[c] > m->lo[c])) return LPP_ERR_INVALID_ARG;
        const double sc = 2.0 / (m->hi[c] - m->lo[c]);
        a.dscale[c] = sc;
        a.dshift[c] = -1.0 - m->lo[c] * sc;
        a.scale[c] = (float)a.dscale[c];
        a.shift[c] = (float)a.dshift[c];
    }
    if (m->base) {
        if (m->base_nodes < 2 || m->base_nodes > kMaxNodes) return LPP_ERR_INVALID_ARG;
        for (int d = 0; d < 2; ++d)
            if (m->base_in[d] < 0 || m->base_in[d] >= kNin || !m->feed[m->base_in[d]]) return LPP_ERR_INVALID_ARG;
        a.base = m->base;
        a.nodes = m->base_nodes;
        a.base_in[0] = m->base_in[0];
        a.base_in[1] = m->base_in[1];
        const double pi = 3.14159265358979323846;
        for (int i = 0; i < a.nodes; ++i) a.xs[i] = -cos(pi * i / (a.nodes - 1));
        for (int i = 0; i < a.nodes; ++i) {
            double d = 1.0;
            for (int k = 0; k < a.nodes; ++k)
                if (k != i) d *= a.xs[i] - a.xs[k];
            a.cw[i] = 1.0 / d;
        }
    }
    a.mu = m->mu;
    a.sd = m->sd;
    a.shot = m->shot;
    a.ref = m->ref;
    a.sigma = m->sigma;
    lpp::eb_matrices(a.N, a.M);
    s->map = a;
    s->has_map = true;
    s->base_split = false;
    return LPP_OK;
}

extern "C" lpp_status lpp_surrogate_targets(lpp_surrogate_t s, const double* theta, const double* native, int n,
                                            float* y, void* stream) {
    if (!s || !s->has_map || n < 0 || (n > 0 && (!theta || !native || !y))) return LPP_ERR_INVALID_ARG;
    if (n == 0) return LPP_OK;
    const long long total = (long long)n * kNout;
    const int blocks = (int)((total + 255) / 256 < 65535 * 8 ? (total + 255) / 256 : 65535 * 8);
    k_targets<<<blocks, 256, 0, (cudaStream_t)stream>>>(theta, native, n, y, s->map);
    return cudaGetLastError() == cudaSuccess ? LPP_OK : LPP_ERR_CUDA;
}

extern "C" lpp_status lpp_surrogate_encode(lpp_surrogate_t s, const double* theta, int n, float* x, void* stream) {
    if (!s || !s->has_map || n < 0 || (n > 0 && (!theta || !x))) return LPP_ERR_INVALID_ARG;
    if (n == 0) return LPP_OK;
    k_encode<<<(n * kNin + 255) / 256, 256, 0, (cudaStream_t)stream>>>(theta, n, x, s->map);
    return cudaGetLastError() == cudaSuccess ? LPP_OK : LPP_ERR_CUDA;
}

extern "C" lpp_status lpp_surrogate_predict(lpp_surrogate_t s, const double* theta, int n, float* out, void* stream) {
    if (!s || !s->ws || !s->has_map || n < 0 || (n > 0 && (!theta || !out))) return LPP_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if (s->map.base) {
        s->map.digits = (const uint4*)(s->ws + s->digits);
        s->map.exponent = (const int*)(s->ws + s->exponent);
        if (!s->base_split) {
            k_base_digits<<<kNout / 8, 256, 0, st>>>(s->map.base, s->map.nodes * s->map.nodes,
                                                     (uint4*)(s->ws + s->digits), (int*)(s->ws + s->exponent));
            if (cudaGetLastError() != cudaSuccess) return LPP_ERR_CUDA;
            // a captured launch has not run yet: the graph forms the digits each time, and so does the
            // next call outside of it
            cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
            if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) return LPP_ERR_CUDA;
            s->base_split = cap == cudaStreamCaptureStatusNone;
        }
    }
    PredictArgs a;
    memset(&a, 0, sizeof(a));
    a.theta = theta;
    a.n = n;
    a.out = out;
    a.map = s->map;
    return launch_predict<true>(s, a, st) == cudaSuccess ? LPP_OK : LPP_ERR_CUDA;
}

// The gradients of the minibatch rows idx[0..batch) of (x, y) and, with update, one Adam step; the
// mean squared error of the minibatch (before the step) is added to *loss_out (device).
static cudaError_t train_step(lpp_surrogate_t s, const float* x, const float* y, const int* idx, float lr,
                              bool update, double* loss_out, cudaStream_t st) {
    TrainRowArgs r;
    memset(&r, 0, sizeof(r));
    TrainWeightArgs w;
    memset(&w, 0, sizeof(w));
    r.ps = passes(s);
    for (int l = 0; l < kLayers; ++l) {
        r.bias[l] = (const float*)(s->ws + s->b[l]);
        r.actt[l] = (bf16*)(s->ws + s->actt[l]);
        r.gt[l] = (bf16*)(s->ws + s->gt[l]);
        r.g32[l] = (float*)(s->ws + s->g32[l]);
        w.actt[l] = r.actt[l];
        w.gt[l] = r.gt[l];
        w.g32[l] = r.g32[l];
    }
    r.x = x;
    r.y = y;
    r.idx = idx;
    r.batch = w.batch = s->batch;
    r.loss = loss_out;
    cudaFuncSetAttribute(k_train_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSliceSmem);
    cudaFuncSetAttribute(k_train_weights, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWeightSmem);
    k_train_rows<<<s->batch / 16 * kSplit, kRowThreads, kSliceSmem, st>>>(r);
    if (update) s->step += 1;
    AdamArgs& a = w.adam;
    a = adam_args(s);
    a.lr = lr;
    a.b1 = 0.9f;
    a.b2 = 0.999f;
    a.eps = 1e-8f;
    a.bc1 = (float)(1.0 - pow(0.9, (double)s->step));
    a.bc2 = (float)(1.0 - pow(0.999, (double)s->step));
    w.update = update ? 1 : 0;
    k_train_weights<<<kWeightTiles + kBiasTiles, 128, kWeightSmem, st>>>(w);
    return cudaGetLastError();
}

extern "C" lpp_status lpp_surrogate_train(lpp_surrogate_t s, const float* x, const float* y, const int* schedule,
                                          int n_steps, float lr, double* losses, void* stream) {
    if (!s || !s->ws || !x || !y || !schedule || n_steps < 0) return LPP_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if (losses && cudaMemsetAsync(losses, 0, (size_t)n_steps * sizeof(double), st) != cudaSuccess) return LPP_ERR_CUDA;
    double* scratch = (double*)(s->ws + s->loss);
    for (int i = 0; i < n_steps; ++i) {
        double* lo = losses ? losses + i : scratch;
        if (train_step(s, x, y, schedule + (size_t)i * s->batch, lr, true, lo, st) != cudaSuccess) return LPP_ERR_CUDA;
    }
    return LPP_OK;
}

// Gradients of the loss of one minibatch without an update (for checks): host dW [out][in], db [out].
extern "C" lpp_status lpp_surrogate_gradients(lpp_surrogate_t s, const float* x, const float* y, const int* idx,
                                              float* grads, double* loss, void* stream) {
    if (!s || !s->ws || !x || !y || !idx || !grads) return LPP_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    double* lo = (double*)(s->ws + s->loss);
    if (cudaMemsetAsync(lo, 0, 8, st) != cudaSuccess) return LPP_ERR_CUDA;
    if (train_step(s, x, y, idx, 0.0f, false, lo, st) != cudaSuccess) return LPP_ERR_CUDA;
    size_t p = 0;
    std::vector<float> dw;
    for (int l = 0; l < kLayers; ++l) {
        const size_t nw = (size_t)kOut[l] * kInPad[l];
        dw.resize(nw);
        cudaMemcpyAsync(dw.data(), s->ws + s->dw[l], nw * 4, cudaMemcpyDeviceToHost, st);
        cudaMemcpyAsync(grads + p + (size_t)kOut[l] * kIn[l], s->ws + s->db[l], kOut[l] * 4, cudaMemcpyDeviceToHost, st);
        if (cudaStreamSynchronize(st) != cudaSuccess) return LPP_ERR_CUDA;
        for (int r = 0; r < kOut[l]; ++r)
            for (int c = 0; c < kIn[l]; ++c) grads[p++] = dw[(size_t)r * kInPad[l] + c];
        p += kOut[l];
    }
    if (loss && cudaMemcpyAsync(loss, lo, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess) return LPP_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return LPP_ERR_CUDA;
    return LPP_OK;
}
