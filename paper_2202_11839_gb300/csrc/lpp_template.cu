// Window-convolved theory templates by FFTLog (Sec. 3.2, Eqs. window_convolution_X_hankel,
// def_of_Q_llp; Appendix D).
//
//   Pt^(L)_X(k) = H_L[ sum_L' Q^X_LL'(r) xi^(L')_X(r) ](k),   xi^(L')_X = H^-1_L'[P^(L')_X]
//
// Both Hankel transforms use the log-Fourier method of Hamilton (2000): A(x) x^-q is
// expanded in a discrete Fourier series in ln x and each term is transformed with the Mellin
// transform of j_l,  int_0^inf x^(s-1) j_l(x) dx = 2^(s-2) sqrt(pi) G((l+s)/2) / G((3+l-s)/2).
// Everything is FP64.
//
// For one window the whole chain, from the model spectrum to the shell averages of the fourteen
// output slots (the estimator's order: the density quadrupole and hexadecapole, whose
// templates are the leakage of the monopole through Q_2 and Q_4, Sec. 4.3, then the minus
// moments L = 10, 12, which the model leaves zero and only the window fills), is one linear
// map of the spectrum on the 2048 grid k.  It is formed once per window (k_operator: one row of
// 2048 weights per slot and shell, by the transposed chain of two to four transforms), and a
// parameter set costs its model spectrum and one product with the rows (k_template, on the
// FP64 tensor cores).
//
// Grid (shared with the tests): 2048 log-spaced k in [1e-4, 10], zero padding to 4096,
// k_0 r_0 = exp(-(N-1) Delta), biases 1.5 (inverse) and 0.5 (forward), the input tapered by
// t - sin(2 pi t)/(2 pi) over the outer 10% of the log-k range at both ends.
#include <math.h>
#include <string.h>

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <complex>
#include <vector>

#include "lpp_internal.h"
#include "lpp_kernels.h"
#include "lpp_fft_dev.cuh"

namespace {

constexpr int kNin = 2048;
constexpr int kNfft = 4096;
constexpr int kLogN = 12;
constexpr double kKmin = 1e-4, kKmax = 10.0, kQinv = 1.5, kQfwd = 0.5, kTaper = 0.1;
constexpr double kPi = 3.14159265358979323846;
constexpr int kSlots = LPP_N_MOMENTS;
// the slots the derived curves read: cross L = 2, 4, 6, plus l = 0, 2, 4, minus L = 4, 6, 8
constexpr unsigned kEbSlots = 0x3FEu;
constexpr int kNfwd = 7;      // forward transforms of order l = 0, 2, ..., 12 (the output slots' L)
constexpr int kMaxTerms = 3;   // model multipoles L' feeding one output slot

struct SlotDesc {
    int kind;      // 0 dd, 1 cross, 2 plus, 3 minus
    int L;
    int n_terms;
    int lp[kMaxTerms];      // L' of each term (0, 2, 4)
    double coef[kMaxTerms]; // model coefficient (power_for_validation, without A and b_g)
    int qx[kMaxTerms];      // row of the mixed window table Q^X_LL'(r_m)
};

struct OperatorArgs {
    const double* ain;      // [2048] k^3 taper k^-q_inv
    const double2* uinv;    // [3][4096] inverse kernels (1/N folded in)
    const double* rinv;     // [4096] r^-q_inv / (2 pi^2)
    const double2* ufwd;    // [7][4096] forward kernels of l = 0, 2, ..., 12 (1/N folded in)
    const double* rfwd;     // [4096] r^(3 - q_fwd)
    const double* kfwd;     // [2048] 4 pi k^-q_fwd
    const double* qx;       // [rows][4096] mixed window Q^X_LL'(r_m)
    const double2* tw;      // [4096] e^{-2 pi i j / N}
    const int* bin_lo;      // [nb] first k_n of each shell
    const int* bin_hi;      // [nb] one past the last
    const double* bin_w;    // [2048] k_n^3
    int nb;
    SlotDesc slots[kSlots];
    double* op;             // [kSlots][nb][2048]
};

struct TemplateArgs {
    const double* params;   // [n][6]: A, b_g, sigma8, tilt, Gamma, shot-noise scale
    int n_templates;
    double* out;            // [n][LPP_N_MOMENTS][nb]
    const double* op;       // [kSlots][nb][2048] the operator's rows
    const uint2* digits;    // their digits (k_op_digits), [kDigits][kSlots nb][512]
    const int* exponent;    // [kSlots nb][8] exponents of the digits per slab
    const double* iref;     // [2048] 1 / reference spectrum
    const double* kin;      // [2048] k_n
    const double* lnk;      // [2048] ln k_n
    const double* ik;       // [2048] 1 / (2.34 k_n)
    const double2* logtab;  // [128] (1 / c, ln c) of log1p_over
    double dlnk;            // ln k_{n+1} - ln k_n
    const double* s8w;      // [2048] sigma_8 quadrature weight w_n k^3 W^2(8k) / (2 pi^2)
    const int* bin_lo;      // [nb] first k_n of each shell
    const int* bin_hi;      // [nb] one past the last
    int nb;
    int bins;               // shells per cluster
    int n_slots;            // slots to compute, in order
    int slot[kSlots];
    double shot_plus;
    // optional derived curves gE_0,2, EE_0,2,4, BB_0,2,4 per shell, standardised as
    // (value - ref) / sigma and stored FP32 [n][8][nb]
    float* eb;
    const double* eb_ref;
    const double* eb_sigma;
    double N[2][3], M[3][3];
    // spin-2 primordial non-Gaussianity (Sec. 5): 12 f_NL^(s=2) delta b_IA and (c / H0)^2 / Omega_m;
    // png_amp = 0: Gaussian initial conditions
    double png_amp, png_len2;
    unsigned slot_mask;     // output slots to compute; the others are written as zeros
};

// wk <- FFT(wk) * u ; FFT again (the log-Fourier transform between the two grids)
__device__ void log_fourier(double2* wk, const double2* __restrict__ u, const double2* __restrict__ tw) {
    const int tid = threadIdx.x;
    lpp::fft_columns<double, kLogN, 1, 1>(wk, 0, tid, tw);
    for (int i = tid; i < kNfft; i += blockDim.x) wk[i] = lpp::cmul<double>(wk[i], u[i]);
    __syncthreads();
    lpp::fft_columns<double, kLogN, 1, 1>(wk, 0, tid, tw);
}

// One row (slot, shell) of the operator: out = sum_n op[n] P(k_n).  Forwards, a spectrum is
// weighted (ain), transformed (T_L' = Re F u F, a real symmetric matrix because u is Hermitian),
// weighted by the window and the radial powers, transformed again (T_L) and averaged over the
// shell; the row applies the transposed steps in reverse order to the shell's weights.
__global__ void __launch_bounds__(512, 1) k_operator(OperatorArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* wk = reinterpret_cast<double2*>(smem_raw);        // [4096]
    double* back = reinterpret_cast<double*>(wk + kNfft);      // [4096]
    double* acc = back + kNfft;                                // [2048]
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int bb = blockIdx.x % a.nb;
    const SlotDesc& sd = a.slots[blockIdx.x / a.nb];
    const int lo = a.bin_lo[bb], hi = a.bin_hi[bb];
    double den = 0.0;
    for (int n = lo; n < hi; ++n) den += a.bin_w[n];
    const double sgn = ((sd.L / 2) & 1) ? -1.0 : 1.0;   // (-i)^L
    for (int m = tid; m < kNfft; m += nthr)
        wk[m] = make_double2(m >= lo && m < hi ? sgn * a.bin_w[m] * a.kfwd[m] / den : 0.0, 0.0);
    for (int m = tid; m < kNin; m += nthr) acc[m] = 0.0;
    __syncthreads();
    log_fourier(wk, a.ufwd + (size_t)(sd.L / 2) * kNfft, a.tw);
    for (int m = tid; m < kNfft; m += nthr) back[m] = wk[m].x * a.rfwd[m] * a.rinv[m];
    __syncthreads();
    for (int j = 0; j < sd.n_terms; ++j) {
        const double c = sd.lp[j] == 2 ? -sd.coef[j] : sd.coef[j];   // i^L'
        for (int m = tid; m < kNfft; m += nthr)
            wk[m] = make_double2(c * a.qx[(size_t)sd.qx[j] * kNfft + m] * back[m], 0.0);
        __syncthreads();
        log_fourier(wk, a.uinv + (size_t)(sd.lp[j] / 2) * kNfft, a.tw);
        for (int m = tid; m < kNin; m += nthr) acc[m] += wk[m].x;
        __syncthreads();
    }
    double* op = a.op + (size_t)blockIdx.x * kNin;
    for (int m = tid; m < kNin; m += nthr) op[m] = acc[m] * a.ain[m];
}

// c[8][8] += a[8][4] b[4][8] (one warp, FP64 tensor cores): lane l holds a[l / 4][l % 4],
// b[l % 4][l / 4] and c[l / 4][2 (l % 4) + {0, 1}].
__device__ __forceinline__ void mma_f64(double c[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};\n"
                 : "+d"(c[0]), "+d"(c[1])
                 : "d"(a), "d"(b));
}

// ln(1 + y) for 0 < y < 2^1000 by Tang's table method (ACM TOMS 16, 378, 1990): 1 + y = 2^e m,
// c the middle of m's 1/128 interval (c = 1 in the first, so that small y keep their relative
// accuracy), r = m / c - 1 with the rounding of 1 + y restored, |r| < 2^-7, and eight terms of
// ln(1 + r).  16 FP64 operations, to 4e-16 relative; log1p takes several times as many, and the
// FP64 rate bounds the spectra.
__device__ __forceinline__ double log1p_table(double y, const double2* tab) {
    const double s = 1.0 + y;
    const double lost = y - (s - 1.0);   // s + lost = 1 + y exactly
    const long long bits = __double_as_longlong(s);
    const int e = (int)(bits >> 52) - 1023;
    const double2 c = tab[(int)(bits >> 45) & 127];
    const double m = __longlong_as_double((bits & 0x000fffffffffffffLL) | 0x3ff0000000000000LL);
    const double w = __longlong_as_double((long long)(1023 - e) << 52);   // 2^-e
    const double r = fma(lost * w, c.x, fma(m, c.x, -1.0));
    double p = -1.0 / 8.0;
    p = fma(p, r, 1.0 / 7.0);
    p = fma(p, r, -1.0 / 6.0);
    p = fma(p, r, 1.0 / 5.0);
    p = fma(p, r, -1.0 / 4.0);
    p = fma(p, r, 1.0 / 3.0);
    p = fma(p, r, -1.0 / 2.0);
    p = fma(p * r, r, r);
    return fma((double)e, 0.69314718055994530942, c.y) + p;
}

// The unnormalised BBKS spectrum (Bardeen, Bond, Kaiser & Szalay 1986) at k: ik = 1 / (2.34 k), ig =
// 1 / Gamma, kt = k^tilt; *transfer receives T(k) when asked for.
__device__ __forceinline__ double bbks_value(double k, double ik, double gam, double ig, double kt,
                                             const double2* logtab, double* transfer) {
    const double q = k * ig, y = 2.34 * q;
    double l;
    if (y > 0.0 && y < 1e300) l = log1p_table(y, logtab) * (ik * gam);
    else l = log1p(y) / y;
    const double x = 1.0 + q * (3.89 + q * (16.1 * 16.1 + q * (5.46 * 5.46 * 5.46 + q * (6.71 * 6.71 * 6.71 * 6.71))));
    const double rs = rsqrt(x);        // T = l x^(-1/4)
    if (transfer) *transfer = l * sqrt(rs);
    return k * kt * (l * l * rs);
}

__device__ __forceinline__ double warp_sum(double s) {
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;
}

__device__ __forceinline__ void mma_bf16(float c[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

constexpr int kCluster = 8, kSets = 8, kSlab = kNin / kCluster, kTiles = 9;
constexpr int kSegs = 4;   // column segments of a slab, each summed by itself

// The end of a cluster of SETS sets: the CTAs' partial sums part[KPARTS][rows][SETS] added over the
// cluster, normalised and written.  val: [SETS][kSlots] of shared memory that is no longer read.
template <int CL, int SETS, int KPARTS>
__device__ __forceinline__ void finish_sets(const TemplateArgs& a, cooperative_groups::cluster_group& cluster,
                                            double* s8part, double* part, double* val, int t0, int sets, int b0,
                                            int nbl, int rows, int rank) {
    const int tid = threadIdx.x;
    cluster.sync();
    // sums over the cluster, normalisation and outputs: CTA `rank` takes the shells rank, rank + CL, ..
    for (int bl = rank; bl < nbl; bl += CL) {
        const int b = b0 + bl;
        for (int i = tid; i < sets * a.n_slots; i += blockDim.x) {
            const int t = i % sets, si = i / sets, sl = a.slot[si];
            const double* th = a.params + 6 * (size_t)(t0 + t);
            double sv[CL], pv[CL][KPARTS];
#pragma unroll
            for (int c = 0; c < CL; ++c) {
                sv[c] = *cluster.map_shared_rank(&s8part[t], c);
                const double* pc = cluster.map_shared_rank(part + (si * nbl + bl) * SETS + t, c);
#pragma unroll
                for (int kp = 0; kp < KPARTS; ++kp) pv[c][kp] = pc[kp * rows * SETS];
            }
            double s2 = 0.0, v = 0.0;
#pragma unroll
            for (int c = 0; c < CL; ++c) {
                s2 += sv[c];
                double slab = pv[c][0];
#pragma unroll
                for (int kp = 1; kp < KPARTS; ++kp) slab += pv[c][kp];
                v += slab;
            }
            const int kind = sl == 0 || sl == 10 || sl == 11 ? 0 : (sl <= 3 ? 1 : 2);
            const double amp = kind == 0 ? th[1] * th[1] : (kind == 1 ? th[0] * th[1] : th[0] * th[0]);
            const bool some = a.bin_lo[b] < a.bin_hi[b];
            v *= amp * (th[2] * th[2] / s2);
            if (sl == 4) v += th[5] * a.shot_plus;
            if (!some) v = 0.0;   // a shell without grid k
            a.out[((size_t)(t0 + t) * kSlots + sl) * a.nb + b] = v;
            val[t * kSlots + sl] = v;
        }
        for (int i = tid; i < sets * kSlots; i += blockDim.x) {
            const int t = i / kSlots, sl = i % kSlots;
            if (!((a.slot_mask >> sl) & 1u)) a.out[((size_t)(t0 + t) * kSlots + sl) * a.nb + b] = 0.0;
        }
        __syncthreads();
        for (int i8 = tid; a.eb && i8 < 8 * sets; i8 += blockDim.x) {
            // Legendre multipoles of P_gE = Re P_gd and P_EE/BB = (P_+ +- P_-)/2 (Sec. 2.4, Eq. relation_pm_EB)
            const int t = i8 >> 3, c = i8 & 7;
            const double* o = val + t * kSlots;
            double v;
            if (c < 2) {
                v = a.N[c][0] * o[1] + a.N[c][1] * o[2] + a.N[c][2] * o[3];
            } else {
                const int li = (c - 2) % 3;
                const double mm = a.M[li][0] * o[7] + a.M[li][1] * o[8] + a.M[li][2] * o[9];
                v = 0.5 * (o[4 + li] + (c < 5 ? mm : -mm));
            }
            const int i = c * a.nb + b;
            const double ref = a.eb_ref ? a.eb_ref[i] : 0.0;
            const double sg = a.eb_sigma ? a.eb_sigma[i] : 1.0;
            a.eb[(size_t)(t0 + t) * 8 * a.nb + i] = (float)((v - ref) / sg);
        }
        __syncthreads();
    }
    cluster.sync();   // the partial sums are read until here
}

// Templates of eight parameter sets on one cluster of eight CTAs (blockIdx.y: a group of a.bins
// shells).  CTA c forms the model spectra on its 256 grid k (one thread per k, the sets in turn)
// and multiplies them with its 256 columns of the operator's rows, 8 sets x 8 rows x 4 columns
// per tensor instruction, the columns split over four groups of warps when the rows are few;
// the cluster then adds the partial sums through distributed shared memory in a fixed order,
// CTA c for every eighth shell, normalises to sigma_8 and writes the slots and derived curves.
//
// What bounds it: the FP64 rate, 0.59 T multiply-adds/s on GB300 (0.52 through the FP64 mma, which
// is no faster here but issues and loads a quarter as much): 6.1 G multiply-adds of the products
// are 11.6 ms of 8192 sets with nine slots and 40 shells, the model spectra (k^tilt from two
// short tables of powers, log1p_table, rsqrt: about 50 operations a value) most of the rest.
// With a non-Gaussian response, whose three spectra only the rows of their families read, 107 -> 15.4
// ms against one CTA per set running its own transforms (FFTs of 4096 points); without one three and more
// sets take k_template_many.  One set, fourteen
// slots: 1.99 ms -> 24 us, the shells spread over the SMs by blockIdx.y; there an mma would idle
// seven of its eight rows, and up to kFewSets sets take plain multiply-adds (FEW).
constexpr int kFewSets = 2;
// sets from which the digit products are used (nine slots, 40 shells, FP64 products -> digits: 4 sets
// 79 -> 46 us, 16 sets 109 -> 81, 64 sets 328 -> 161, 1024 sets 2163 -> 493)
constexpr int kManyFrom = kFewSets + 1;
constexpr int kMaxRows = 8 * 8 * kTiles;   // rows per cluster: 8 warps x kTiles tiles of 8
constexpr int kSlabPad = kSlab + 2;        // the eight sets' rows start in different banks
// the most dynamic shared memory of a launch: three spectra, kMaxRows rows (kSegs parts of at most 64 are fewer)
constexpr size_t kTemplateSmem = ((size_t)3 * kSets * kSlabPad + (size_t)kMaxRows * kSets) * sizeof(double);

// NT: tiles of 8 rows per warp, KPARTS: column segments taken by different warps (1 or kSegs);
// compile-time, so that every tile of a warp is one unconditional product
template <int NT, int KPARTS, bool FEW = false>
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(256, NT <= 6 ? 3 : 2)
k_template(const __grid_constant__ TemplateArgs a) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const bool png = a.png_amp != 0.0;
    const int n_pow = png ? 3 : 1;   // P, P f, P f^2 with the PNG response f
    double* spec = reinterpret_cast<double*>(smem_raw);   // [n_pow][kSets][kSlabPad]
    double* part = spec + n_pow * kSets * kSlabPad;       // [kparts][rows][kSets] partial sums
    __shared__ double s8part[kSets];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int t0 = (int)(blockIdx.x / kCluster) * kSets;
    const int sets = min(kSets, a.n_templates - t0);
    const int b0 = blockIdx.y * a.bins, nbl = min(a.bins, a.nb - b0);
    const int rows = a.n_slots * nbl;

    // per set: k^tilt at every 16th grid k of the slab, the 16 powers between, 1 / Gamma
    __shared__ double pw_hi[kSets][16], pw_lo[kSets][16], igam[kSets];
    __shared__ double2 logtab[128];
    {
        const int t = tid >> 5, i = tid & 15;
        if (t < sets) {
            const double tilt = a.params[6 * (size_t)(t0 + t) + 3];
            const double v = exp(tilt * ((lane & 16) ? a.dlnk * i : a.lnk[rank * kSlab + 16 * i]));
            if (lane & 16) pw_lo[t][i] = v;
            else pw_hi[t][i] = v;
            if (lane == 0) igam[t] = 1.0 / a.params[6 * (size_t)(t0 + t) + 4];
        }
        if (tid < 128) logtab[tid] = a.logtab[tid];
    }
    __syncthreads();
    // model spectra (unnormalised BBKS, Bardeen, Bond, Kaiser & Szalay 1986)
    {
        const int n = rank * kSlab + tid;
        const double k = a.kin[n], ik = a.ik[n];
#pragma unroll 2
        for (int t = 0; t < kSets; ++t) {
            double p = 0.0, f = 0.0, tr = 0.0;
            if (t < sets) {
                p = bbks_value(k, ik, a.params[6 * (size_t)(t0 + t) + 4], igam[t], pw_hi[t][tid >> 4] * pw_lo[t][tid & 15],
                               logtab, png ? &tr : nullptr);
                // Sec. 5: P -> [1 + 12 f_NL delta b_IA / M(k)] P per shape field,
                // M(k) = (2/3) k^2 T(k) D (c/H0)^2 / Omega_m with D = 1 (z = 0)
                if (png) f = 1.0 + a.png_amp / ((2.0 / 3.0) * k * k * tr * a.png_len2);
            }
            spec[t * kSlabPad + tid] = p;
            if (png) {
                spec[(kSets + t) * kSlabPad + tid] = p * f;
                spec[(2 * kSets + t) * kSlabPad + tid] = p * f * f;
            }
        }
    }
    __syncthreads();
    // sigma_8^2 of set `warp` over this slab
    {
        double s = 0.0;
        for (int i = lane; i < kSlab; i += 32) s += a.s8w[rank * kSlab + i] * spec[warp * kSlabPad + i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) s8part[warp] = s;
    }
    if constexpr (FEW) {
        // a warp per row (slot index) nbl + shell: 8 columns per lane, then the lanes' sums
        for (int r = warp; r < rows; r += 8) {
            const int si = r / nbl, sl = a.slot[si];
            const int pw = !png || sl == 0 || sl == 10 || sl == 11 ? 0 : (sl <= 3 ? 1 : 2);   // power of the response
            const double2* op = reinterpret_cast<const double2*>(
                a.op + ((size_t)sl * a.nb + b0 + (r - si * nbl)) * kNin + rank * kSlab);
            double2 o[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i] = op[lane + 32 * i];
            for (int t = 0; t < sets; ++t) {
                const double2* sp = reinterpret_cast<const double2*>(spec + (pw * kSets + t) * kSlabPad);
                double v = 0.0, w = 0.0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const double2 p = sp[lane + 32 * i];
                    v = fma(o[i].x, p.x, v);
                    w = fma(o[i].y, p.y, w);
                }
                v += w;
#pragma unroll
                for (int q = 16; q > 0; q >>= 1) v += __shfl_down_sync(0xffffffffu, v, q);
                if (lane == 0) part[r * kSets + t] = v;
            }
        }
    } else {
    // row r = (slot index) nbl + shell; the warp takes tiles wt, wt + lanes, .. of 8 rows, and all
    // four segments of 64 columns or one.  Every segment is summed by itself and the segments are
    // added in order, so a value does not depend on the split (on the slots and sets of the call).
    constexpr int lanes = 8 / KPARTS;
    const int wt = warp % lanes, kpart = warp / lanes;
    const int rl = lane >> 2, cl = 2 * (lane & 3);
    unsigned brow[NT];   // in double2, from the slab's first column
    const double2* op = reinterpret_cast<const double2*>(a.op + rank * kSlab + cl);
    const double* arow = spec + rl * kSlabPad + cl;
    double acc[NT][2];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        // rows beyond the last repeat it and are not read back
        const int r = max(0, min(8 * (wt + lanes * j) + rl, rows - 1));
        const int si = r / nbl;
        brow[j] = (unsigned)((a.slot[si] * a.nb + b0 + (r - si * nbl)) * (kNin / 2));
    }
    for (int seg = kpart; seg < kSegs; seg += KPARTS) {
        const int k_lo = seg * (kSlab / kSegs), k_hi = k_lo + kSlab / kSegs;
#pragma unroll
        for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = 0.0;
        // the response enters the density rows not at all, the cross rows once and the plus and
        // minus rows twice; a tile may straddle two families: it is multiplied with the spectrum of
        // each, and every row keeps the product with its own (not a sum with the others times
        // zero, which an infinite spectrum would spoil)
        auto power = [&](int r) {   // of row r's family
            const int sl = a.slot[min(r, rows - 1) / nbl];
            return sl == 0 || sl == 10 || sl == 11 ? 0 : (sl <= 3 ? 1 : 2);
        };
        for (int pw = 0; pw < 3; ++pw) {
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                const int r8 = 8 * (wt + lanes * j);
                if (r8 >= rows) break;
                if (!__any_sync(0xffffffffu, power(r8 + rl) == pw)) continue;   // warp-uniform
                double v[2] = {0.0, 0.0};
                for (int k0 = k_lo; k0 < k_hi; k0 += 8) {
                    const double2 av = *reinterpret_cast<const double2*>(arow + pw * kSets * kSlabPad + k0);
                    const double2 bv = op[brow[j] + k0 / 2];
                    mma_f64(v, av.x, bv.x);
                    mma_f64(v, av.y, bv.y);
                }
#pragma unroll
                for (int q = 0; q < 2; ++q)   // accumulator columns are rows of the operator
                    if (power(r8 + cl + q) == pw) acc[j][q] = v[q];
            }
        }
        const bool first = seg < KPARTS;
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            const int r = 8 * (wt + lanes * j) + cl;   // accumulator columns are rows of the operator
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (r + q >= rows) continue;
                double* d = part + (kpart * rows + r + q) * kSets + rl;
                *d = first ? acc[j][q] : *d + acc[j][q];
            }
        }
    }
    }
    finish_sets<kCluster, kSets, KPARTS>(a, cluster, s8part, part, spec, t0, sets, b0, nbl, rows, rank);
}

// ---- many sets: exact products on the BF16 tensor cores
// The products of the spectra with the operator are 11.6 of 15 ms of 8192 sets at the FP64 rate.
// Both factors are written as kDigits signed base-256 digits of a 56-bit fixed-point number
// (Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59, 95, 2012): the spectra relative to a
// reference spectrum and to the largest value of the set's slab of 256 grid k, the operator's
// rows (times the reference) relative to the largest of the row's slab.  A digit is an integer of
// at most 128, exact in BF16; 128 products of digits sum to an integer below 2^21, seven such sums
// to one below 2^24, exact in the FP32 accumulators.  Products of digits i and j have weight
// 2^(-8 (i + j)): those of equal i + j <= 6 share an accumulator (28 mma instead of one FP64 product;
// the dropped ones are below 2^-54 of the slab's largest product), and every 128 columns the
// seven accumulators are added to two 64-bit integers.  The slabs are added in FP64.
// A spectrum that varies by less than 2^kSpread against the reference within its slabs is so held to
// 2^-53 of each of its values, as FP64 holds it; a set that varies more, in any slab, takes FP64
// products there (tilts within 0.2 and Gamma within 0.1 to 0.3 vary by 2^1.5 at most; against the
// magnitudes of the terms the digits of a tilt of 2 lost a factor 10, of 8 a factor 90).
constexpr int kDigits = 7;
constexpr int kManySets = 16;                 // sets per cluster: two column tiles of the mma
constexpr int kManyTiles = 5;                 // row tiles of 16 per warp
constexpr int kManyRows = 8 * 16 * kManyTiles;
constexpr int kSpread = 3;
constexpr size_t kManySmem = (size_t)kDigits * 16 * 2 * 32 * sizeof(uint2) + (size_t)kManyRows * kManySets * sizeof(double);
// groups of sets from which a cluster is four CTAs of two slabs each: clusters of eight leave 40 of the 152
// SMs idle (40 shells, nine slots, eight -> four CTAs: 16 sets 81 -> 153 us, 64 sets 165 -> 161, 256 sets
// 306 -> 197, 8192 sets 4421 -> 3654)
constexpr int kWideFrom = 4;

// v with |v| < 2^e -> digits d_i, v = 2^e sum_i d_i 2^(-8 i - 7) to 2^(e - 56)
__device__ __forceinline__ void digits7(double v, int e, int* d) {
    const double scale = __hiloint2double((55 - e + 1023) << 20, 0);
    long long q = __double2ll_rn(v * scale);
#pragma unroll
    for (int i = kDigits - 1; i > 0; --i) {
        d[i] = (int)((q + 128) & 255) - 128;
        q = (q - d[i]) >> 8;
    }
    d[0] = (int)q;
}
// e with 2^(e - 1) <= |v| < 2^e for the bits of the largest high word h; kBadExp for an infinity or NaN
constexpr int kBadExp = 1 << 20;
__device__ __forceinline__ int high_exponent(int h) {
    const int e = (h >> 20) - 1022;
    return e > 900 ? kBadExp : max(e, -900);
}
__device__ __forceinline__ double pow2(int e) {   // -1022 <= e <= 1023
    return __hiloint2double((e + 1023) << 20, 0);
}

// The operator's rows (times the reference) as digits: one warp per (row, slab).  Within 16 columns
// lane t of a fragment reads the four values 4 t .. 4 t + 3 of its row (one 8-byte word): the order
// of the columns in a product is free as long as both factors share it.
__global__ void __launch_bounds__(256) k_op_digits(const double* __restrict__ op, const double* __restrict__ iref,
                                                   int rows, uint2* __restrict__ digits, int* __restrict__ exponent) {
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= rows * 8) return;
    const int row = w >> 3, slab = w & 7;
    double v[8];
    int h = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {   // eight consecutive columns per lane
        const int n = slab * 256 + lane * 8 + i;
        v[i] = op[(size_t)row * kNin + n] / iref[n];
        h = max(h, __double2hiint(v[i]) & 0x7fffffff);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
    const int e = high_exponent(h);
    if (lane == 0) exponent[row * 8 + slab] = e;
    unsigned short out[kDigits][8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        int d[kDigits];
        digits7(e == kBadExp ? 0.0 : v[i], e == kBadExp ? 0 : e, d);
#pragma unroll
        for (int q = 0; q < kDigits; ++q) out[q][i] = __bfloat16_as_ushort(__float2bfloat16_rn((float)d[q]));
    }
#pragma unroll
    for (int q = 0; q < kDigits; ++q)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint2 u;
            u.x = out[q][4 * i] | (unsigned)out[q][4 * i + 1] << 16;
            u.y = out[q][4 * i + 2] | (unsigned)out[q][4 * i + 3] << 16;
            digits[((size_t)q * rows + row) * (kNin / 4) + slab * 64 + lane * 2 + i] = u;
        }
}

// Templates of sixteen parameter sets per cluster of CL CTAs (8 / CL slabs each in turn), as
// k_template, with the products above: a warp multiplies tiles of 16 rows x 16 sets, the operator's digits straight from L2, the
// spectra's from shared memory in fragment order.
//
// What bounds it: the FP64 spectra (1.4 ms at the FP64 rate for 8192 sets) and the mma issue.
// 8192 sets, nine slots, 40 shells: 15.0 -> 3.7 ms against the FP64 products (78.0 ms with transforms
// per set).
template <int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(256, 1)
k_template_many(const __grid_constant__ TemplateArgs a) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // [kDigits][16 k steps][2 set tiles][32 lanes] B fragments, then [rows][kManySets] partial sums
    uint2* frag = reinterpret_cast<uint2*>(smem_raw);
    double* part = reinterpret_cast<double*>(frag + kDigits * 16 * 2 * 32);
    __shared__ double s8part[kManySets];
    __shared__ int hmax[kManySets], hmin[kManySets];
    __shared__ unsigned exact_sets;        // the sets of this slab that take FP64 products
    __shared__ double exact_spec[kSlab];   // and the spectrum of one of them
    __shared__ double pw_hi[kManySets][16], pw_lo[kManySets][16], igam[kManySets];
    __shared__ double2 logtab[128];
    __shared__ double s8w[8][kManySets];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int t0 = (int)(blockIdx.x / CL) * kManySets;
    const int sets = min(kManySets, a.n_templates - t0);
    const int b0 = blockIdx.y * a.bins, nbl = min(a.bins, a.nb - b0);
    const int rows = a.n_slots * nbl;
    for (int slab = rank * (8 / CL); slab < (rank + 1) * (8 / CL); ++slab) {
        for (int q = tid; q < kManySets * 32; q += 256) {
            const int t = q >> 5, i = q & 15;
            if (t < sets) {
                const double tilt = a.params[6 * (size_t)(t0 + t) + 3];
                const double v = exp(tilt * ((q & 16) ? a.dlnk * i : a.lnk[slab * kSlab + 16 * i]));
                if (q & 16) pw_lo[t][i] = v;
                else pw_hi[t][i] = v;
                if ((q & 31) == 0) igam[t] = 1.0 / a.params[6 * (size_t)(t0 + t) + 4];
            }
        }
        if (tid < 128) logtab[tid] = a.logtab[tid];
        if (tid < kManySets) {
            hmax[tid] = 0;
            hmin[tid] = 0x7fffffff;
        }
        __syncthreads();
        // spectra of the sixteen sets at this thread's grid k, relative to the reference
        const int n = slab * kSlab + tid;
        const double k = a.kin[n], ik = a.ik[n], ir = a.iref[n], sw = a.s8w[n];
        double p[kManySets];
    #pragma unroll
        for (int t = 0; t < kManySets; ++t) {
            p[t] = 0.0;
            if (t < sets) {
                const double gam = a.params[6 * (size_t)(t0 + t) + 4];
                p[t] = bbks_value(k, ik, gam, igam[t], pw_hi[t][tid >> 4] * pw_lo[t][tid & 15], logtab, nullptr);
            }
            const double s = warp_sum(sw * p[t]);
            if (lane == 0) s8w[warp][t] = s;
            p[t] *= ir;
            int h = __double2hiint(p[t]) & 0x7fffffff, l = h;
    #pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
                l = min(l, __shfl_xor_sync(0xffffffffu, l, o));
            }
            if (lane == 0) {
                atomicMax(&hmax[t], h);
                atomicMin(&hmin[t], l);
            }
        }
        __syncthreads();
        if (tid < kManySets) {
            double s = 0.0;
            for (int w = 0; w < 8; ++w) s += s8w[w][tid];
            s8part[tid] = slab == rank * (8 / CL) ? s : s8part[tid] + s;
        }
        if (warp == 0) {
            const int t = lane % kManySets, e = high_exponent(hmax[t]);
            const unsigned b = __ballot_sync(0xffffffffu, lane < sets && (hmax[t] - hmin[t] >= kSpread << 20 || e == kBadExp ||
                                                                          e <= -900));
            if (lane == 0) exact_sets = b;
        }
        {   // column tid = 16 ks + 4 tt + 2 r + lo: register r, half lo of the lanes 4 g + tt
            const int ks = tid >> 4, tt = (tid & 15) >> 2, r = (tid >> 1) & 1, lo = tid & 1;
            unsigned short* f = reinterpret_cast<unsigned short*>(frag);
    #pragma unroll
            for (int t = 0; t < kManySets; ++t) {
                const int e = high_exponent(hmax[t]);
                int d[kDigits];
                digits7(e == kBadExp ? 0.0 : p[t], e == kBadExp ? 0 : e, d);
    #pragma unroll
                for (int q = 0; q < kDigits; ++q)
                    f[((((q * 16 + ks) * 2 + (t >> 3)) * 32 + 4 * (t & 7) + tt) * 2 + r) * 2 + lo] =
                        __bfloat16_as_ushort(__float2bfloat16_rn((float)d[q]));
            }
        }
        __syncthreads();
        const int g = lane >> 2, tt = lane & 3;
        const int all_rows = kSlots * a.nb;
        const unsigned exact = exact_sets;
        for (int tile = warp; tile * 16 < rows; tile += 8) {
            // the operator rows g and g + 8 of the tile (rows beyond the last repeat it and are not read back)
            int orow[2];
    #pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = min(16 * tile + g + 8 * h, rows - 1), si = r / nbl;
                orow[h] = a.slot[si] * a.nb + b0 + (r - si * nbl);
            }
            const uint2* src0 = a.digits + (size_t)orow[0] * (kNin / 4) + slab * 64 + tt;
            const uint2* src1 = a.digits + (size_t)orow[1] * (kNin / 4) + slab * 64 + tt;
            const size_t dstride = (size_t)all_rows * (kNin / 4);
            long long vh[2][4], vl[2][4];
    #pragma unroll
            for (int c = 0; c < 2; ++c)
    #pragma unroll
                for (int q = 0; q < 4; ++q) vh[c][q] = vl[c][q] = 0;
            for (int half = 0; half < 2; ++half) {
                float acc[2][kDigits][4];
    #pragma unroll
                for (int c = 0; c < 2; ++c)
    #pragma unroll
                    for (int o = 0; o < kDigits; ++o)
    #pragma unroll
                        for (int q = 0; q < 4; ++q) acc[c][o][q] = 0.f;
    #pragma unroll 1
                for (int ks = 8 * half; ks < 8 * half + 8; ++ks) {
                    uint2 a0[kDigits], a1[kDigits];
    #pragma unroll
                    for (int i = 0; i < kDigits; ++i) {
                        a0[i] = src0[i * dstride + 4 * ks];
                        a1[i] = src1[i * dstride + 4 * ks];
                    }
    #pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint2 bf[kDigits];
    #pragma unroll
                        for (int j = 0; j < kDigits; ++j) bf[j] = frag[((j * 16 + ks) * 2 + c) * 32 + lane];
    #pragma unroll
                        for (int i = 0; i < kDigits; ++i)
    #pragma unroll
                            for (int j = 0; j + i < kDigits; ++j)
                                mma_bf16(acc[c][i + j], a0[i].x, a1[i].x, a0[i].y, a1[i].y, bf[j].x, bf[j].y);
                    }
                }
    #pragma unroll
                for (int c = 0; c < 2; ++c)
    #pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        long long i[kDigits];
    #pragma unroll
                        for (int o = 0; o < kDigits; ++o) i[o] = (long long)__float2int_rn(acc[c][o][q]);
                        vh[c][q] += (i[0] << 16) + (i[1] << 8) + i[2];
                        vl[c][q] += (i[3] << 24) + (i[4] << 16) + (i[5] << 8) + i[6];
                    }
            }
            // order o has unit 2^(e_row + e_set - 14 - 8 o): vh in orders of 2, vl of 6
    #pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = 16 * tile + g + 8 * h;
                if (r >= rows) continue;
                const int er = a.exponent[orow[h] * 8 + slab];
    #pragma unroll
                for (int c = 0; c < 2; ++c)
    #pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int t = 8 * c + 2 * tt + q, es = high_exponent(hmax[t]);
                        if ((exact >> t) & 1u) continue;
                        double v = fma((double)vh[c][2 * h + q], 4294967296.0, (double)vl[c][2 * h + q]) * pow2(-62);
                        v = er == kBadExp || es == kBadExp ? NAN : v * pow2(er) * pow2(es);
                        double* d = part + r * kManySets + t;
                        *d = slab == rank * (8 / CL) ? v : *d + v;
                    }
            }
        }
        for (unsigned rest = exact; rest; rest &= rest - 1) {   // CTA-uniform
            const int t = __ffs(rest) - 1;
            exact_spec[tid] = bbks_value(k, ik, a.params[6 * (size_t)(t0 + t) + 4], igam[t],
                                         pw_hi[t][tid >> 4] * pw_lo[t][tid & 15], logtab, nullptr);
            __syncthreads();
            for (int r = warp; r < rows; r += 8) {   // a warp per row: 8 columns per lane, then the lanes' sums
                const int si = r / nbl;
                const double* op = a.op + (size_t)(a.slot[si] * a.nb + b0 + (r - si * nbl)) * kNin + slab * kSlab;
                double v = 0.0;
    #pragma unroll
                for (int i = 0; i < kSlab / 32; ++i) v = fma(op[lane + 32 * i], exact_spec[lane + 32 * i], v);
                v = warp_sum(v);
                if (lane == 0) {
                    double* d = part + r * kManySets + t;
                    *d = slab == rank * (8 / CL) ? v : *d + v;
                }
            }
            __syncthreads();   // the next set rewrites the spectrum
        }
        __syncthreads();   // the next slab rewrites the tables and digits
    }
    finish_sets<CL, kManySets, 1>(a, cluster, s8part, part, reinterpret_cast<double*>(frag), t0, sets, b0, nbl, rows, rank);
}

// ------------------------------------------------------------------ host tables
double lfact(int n) { return lgamma((double)n + 1.0); }

// Wigner 3j symbol by the Racah formula.
double wigner3j(int j1, int j2, int j3, int m1, int m2, int m3) {
    if (m1 + m2 + m3 != 0) return 0.0;
    if (j3 < abs(j1 - j2) || j3 > j1 + j2) return 0.0;
    if (abs(m1) > j1 || abs(m2) > j2 || abs(m3) > j3) return 0.0;
    const double ldelta = lfact(j1 + j2 - j3) + lfact(j1 - j2 + j3) + lfact(-j1 + j2 + j3) - lfact(j1 + j2 + j3 + 1);
    const double lpre = 0.5 * (ldelta + lfact(j1 + m1) + lfact(j1 - m1) + lfact(j2 + m2) + lfact(j2 - m2) +
                               lfact(j3 + m3) + lfact(j3 - m3));
    double sum = 0.0;
    for (int k = 0; k <= j1 + j2 + j3; ++k) {
        const int a1 = j3 - j2 + k + m1, a2 = j3 - j1 + k - m2, a3 = j1 + j2 - j3 - k, a4 = j1 - k - m1,
                  a5 = j2 - k + m2;
        if (a1 < 0 || a2 < 0 || a3 < 0 || a4 < 0 || a5 < 0) continue;
        const double term = exp(lpre - lfact(k) - lfact(a1) - lfact(a2) - lfact(a3) - lfact(a4) - lfact(a5));
        sum += (k & 1) ? -term : term;
    }
    const int ph = j1 - j2 - m3;
    return ((ph % 2) != 0 ? -1.0 : 1.0) * sum;
}

// Coefficient of Q_l'' in Q^X_LL' (Eq. def_of_Q_llp).
double mixing(int m, int L, int Lp, int lpp) {
    const double pref = (2.0 * L + 1.0) * exp(0.5 * (lfact(L - m) - lfact(L + m) + lfact(Lp + m) - lfact(Lp - m)));
    return pref * wigner3j(lpp, L, Lp, 0, 0, 0) * wigner3j(lpp, L, Lp, 0, m, -m);
}

// ln Gamma(z) for Re z > 0: upward recurrence to Re z >= 12, then the Stirling series with
// Bernoulli numbers B_2 .. B_14.
std::complex<double> lgamma_c(std::complex<double> z) {
    std::complex<double> shift = 0.0;
    while (z.real() < 12.0) {
        shift -= std::log(z);
        z += 1.0;
    }
    const double B[7] = {1.0 / 6, -1.0 / 30, 1.0 / 42, -1.0 / 30, 5.0 / 66, -691.0 / 2730, 7.0 / 6};
    const std::complex<double> iz = 1.0 / z, iz2 = iz * iz;
    std::complex<double> series = 0.0, pw = iz;
    for (int k = 1; k <= 7; ++k) {
        series += B[k - 1] / (2.0 * k * (2.0 * k - 1.0)) * pw;
        pw *= iz2;
    }
    return shift + (z - 0.5) * std::log(z) - z + 0.5 * log(2.0 * kPi) + series;
}

// u_alpha = (k_0 r_0)^{-i eta} M_l(q + i eta) / N, eta = 2 pi alpha / (N Delta), alpha in DFT order;
// the Nyquist coefficient is kept real.  u_-alpha = conj u_alpha, which halves most of the time that a new
// window's tables take.
void fftlog_kernel(int ell, double q, double delta, double kr0, double2* u) {
    for (int i = 0; i <= kNfft / 2; ++i) {
        const int alpha = i < kNfft / 2 ? i : i - kNfft;
        const double eta = 2.0 * kPi * alpha / (kNfft * delta);
        const std::complex<double> s(q, eta);
        const std::complex<double> lm = (s - 2.0) * log(2.0) + 0.5 * log(kPi) + lgamma_c(0.5 * (double(ell) + s)) -
                                        lgamma_c(0.5 * (3.0 + double(ell) - s));
        std::complex<double> v = std::exp(lm - std::complex<double>(0.0, eta * log(kr0))) / double(kNfft);
        if (i == kNfft / 2) v = std::complex<double>(v.real(), 0.0);
        u[i] = make_double2(v.real(), v.imag());
        if (i > 0 && i < kNfft / 2) u[kNfft - i] = make_double2(v.real(), -v.imag());
    }
}

double top_hat(double x) {
    if (x < 1e-2) return 1.0 - x * x / 10.0 + x * x * x * x / 280.0;
    return 3.0 * (sin(x) - x * cos(x)) / (x * x * x);
}

double taper_at(int n) {
    const double x = double(n) / (kNin - 1);
    double out = 1.0;
    for (double t : {x / kTaper, (1.0 - x) / kTaper}) {
        if (t >= 1.0) continue;
        const double tt = t < 0.0 ? 0.0 : t;
        out *= tt - sin(2.0 * kPi * tt) / (2.0 * kPi);
    }
    return out;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

struct lpp_template_s {
    int nb = 0;
    double shot_plus = 0.0;
    double png_amp = 0.0, png_len2 = 0.0;   // 12 f_NL delta b_IA and (c/H0)^2 / Omega_m
    unsigned slot_mask = (1u << kSlots) - 1u;
    int qx_rows = 0;
    std::vector<double> kin, lnk, ik, iref, s8w, ain, rinv, rfwd, kfwd, qx, bin_w;
    std::vector<double2> uinv, ufwd, tw, logtab;
    double dlnk = 0.0;
    std::vector<int> bin_lo, bin_hi;
    SlotDesc slots[kSlots];
    // device
    char* ws = nullptr;
    size_t ws_need = 0, o_kin, o_lnk, o_ik, o_logtab, o_iref, o_op, o_digits, o_exponent, o_s8w, o_ain, o_uinv, o_rinv, o_ufwd, o_rfwd, o_kfwd, o_qx, o_tw, o_lo, o_hi, o_bw;
    bool ready = false;
};

extern "C" lpp_status lpp_template_create(const double* q, const double* s, int n_s, const double* k_edges,
                                          int n_bins, double shot_plus, lpp_template_t* out) {
    if (!q || !s || !k_edges || !out || n_s < 1 || n_bins < 1 || n_bins > 256) return LPP_ERR_INVALID_ARG;
    for (int i = 0; i + 1 < n_s; ++i)
        if (!(s[i] < s[i + 1])) return LPP_ERR_INVALID_ARG;
    for (int i = 0; i < n_bins; ++i)
        if (!(k_edges[i] < k_edges[i + 1])) return LPP_ERR_INVALID_ARG;
    lpp_template_t t = new lpp_template_s();
    t->nb = n_bins;
    t->shot_plus = shot_plus;
    const double delta = log(kKmax / kKmin) / (kNin - 1);
    const double r0 = exp(-(kNfft - 1) * delta) / kKmin;
    const double kr0 = kKmin * r0;
    t->kin.resize(kNin);
    t->lnk.resize(kNin);
    t->ik.resize(kNin);
    t->iref.resize(kNin);
    t->dlnk = delta;
    t->logtab.resize(128);
    for (int i = 0; i < 128; ++i) {
        // ln c from the rounded 1 / c that divides
        const double ic = i == 0 ? 1.0 : 1.0 / (1.0 + (i + 0.5) / 128.0);
        t->logtab[i] = make_double2(ic, i == 0 ? 0.0 : -log(ic));
    }
    t->s8w.resize(kNin);
    t->ain.resize(kNin);
    t->kfwd.resize(kNin);
    t->bin_w.resize(kNin);
    for (int n = 0; n < kNin; ++n) {
        const double k = kKmin * exp(n * delta);
        const double wtr = (n == 0 || n == kNin - 1) ? 0.5 * delta : delta;
        const double th = top_hat(8.0 * k);
        t->kin[n] = k;
        t->lnk[n] = log(kKmin) + n * delta;
        t->ik[n] = 1.0 / (2.34 * k);
        // the reference of the digit products: the BBKS spectrum of Gamma = 0.2
        const double rq = k / 0.2, rl = log1p(2.34 * rq) / (2.34 * rq);
        const double rx = 1.0 + 3.89 * rq + pow(16.1 * rq, 2) + pow(5.46 * rq, 3) + pow(6.71 * rq, 4);
        t->iref[n] = sqrt(rx) / (k * rl * rl);
        t->s8w[n] = wtr * k * k * k / (2.0 * kPi * kPi) * th * th;
        t->ain[n] = k * k * k * taper_at(n) * pow(k, -kQinv);
        t->kfwd[n] = 4.0 * kPi * pow(k, -kQfwd);
        t->bin_w[n] = k * k * k;
    }
    t->rinv.resize(kNfft);
    t->rfwd.resize(kNfft);
    std::vector<double> r(kNfft);
    for (int m = 0; m < kNfft; ++m) {
        r[m] = r0 * exp(m * delta);
        t->rinv[m] = pow(r[m], -kQinv) / (2.0 * kPi * kPi);
        t->rfwd[m] = pow(r[m], 3.0 - kQfwd);
    }
    t->uinv.resize(3 * kNfft);
    for (int li = 0; li < 3; ++li) fftlog_kernel(2 * li, kQinv, delta, kr0, &t->uinv[li * kNfft]);
    t->ufwd.resize(kNfwd * kNfft);
    for (int li = 0; li < kNfwd; ++li) fftlog_kernel(2 * li, kQfwd, delta, kr0, &t->ufwd[li * kNfft]);
    t->tw.resize(kNfft);
    for (int j = 0; j < kNfft; ++j) t->tw[j] = make_double2(cos(2.0 * kPi * j / kNfft), -sin(2.0 * kPi * j / kNfft));
    // window multipoles on the r grid: linear in s, held below s_0, zero beyond the last s
    std::vector<double> qr(5 * kNfft, 0.0);
    for (int li = 0; li < 5; ++li)
        for (int m = 0; m < kNfft; ++m) {
            const double x = r[m];
            double v;
            if (x <= s[0]) v = q[li * n_s];
            else if (x > s[n_s - 1]) v = 0.0;
            else {
                int j = 0;
                while (j + 1 < n_s && s[j + 1] < x) ++j;
                const double f = (x - s[j]) / (s[j + 1] - s[j]);
                v = q[li * n_s + j] + f * (q[li * n_s + j + 1] - q[li * n_s + j]);
            }
            qr[li * kNfft + m] = v;
        }
    // output slots: kind, L and the model multipoles feeding them
    const int kinds[kSlots] = {0, 1, 1, 1, 2, 2, 2, 3, 3, 3, 0, 0, 3, 3};
    const int Ls[kSlots] = {0, 2, 4, 6, 0, 2, 4, 4, 6, 8, 2, 4, 10, 12};
    const int mX[4] = {0, 2, 0, 4};
    int rows = 0;
    for (int sl = 0; sl < kSlots; ++sl) {
        SlotDesc& sd = t->slots[sl];
        sd.kind = kinds[sl];
        sd.L = Ls[sl];
        sd.n_terms = 0;
        auto add = [&](int lp, double coef) {
            const int j = sd.n_terms++;
            sd.lp[j] = lp;
            sd.coef[j] = coef;
            sd.qx[j] = rows++;
            std::vector<double> mix(5);
            for (int lpp = 0; lpp <= 8; lpp += 2) mix[lpp / 2] = mixing(mX[sd.kind], sd.L, lp, lpp);
            for (int m = 0; m < kNfft; ++m) {
                double v = 0.0;
                for (int li = 0; li < 5; ++li) v += mix[li] * qr[li * kNfft + m];
                t->qx.push_back(v);
            }
        };
        // P_dd^(0) = b^2 P, P_gd^(2) = -A b P / 6, P_+^(0,2,4) = A^2 (2/15, -4/21, 2/35) P,
        // P_-^(4) = A^2 P / 420 (the powers of A and b in k_template)
        if (sd.kind == 0) add(0, 1.0);
        else if (sd.kind == 1) add(2, -1.0 / 6.0);
        else if (sd.kind == 2) { add(0, 2.0 / 15.0); add(2, -4.0 / 21.0); add(4, 2.0 / 35.0); }
        else add(4, 1.0 / 420.0);
    }
    t->qx_rows = rows;
    t->bin_lo.resize(n_bins);
    t->bin_hi.resize(n_bins);
    for (int bb = 0; bb < n_bins; ++bb) {
        int lo = kNin, hi = 0;
        for (int n = 0; n < kNin; ++n)
            if (t->kin[n] >= k_edges[bb] && t->kin[n] < k_edges[bb + 1]) {
                lo = n < lo ? n : lo;
                hi = n + 1;
            }
        t->bin_lo[bb] = lo < hi ? lo : 0;
        t->bin_hi[bb] = lo < hi ? hi : 0;
    }
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align256(off + bytes); return o; };
    t->o_kin = take(kNin * 8);
    t->o_lnk = take(kNin * 8);
    t->o_ik = take(kNin * 8);
    t->o_logtab = take(128 * 16);
    t->o_iref = take(kNin * 8);
    t->o_digits = take((size_t)kDigits * kSlots * n_bins * kNin * 2);
    t->o_exponent = take((size_t)kSlots * n_bins * kCluster * 4);
    t->o_op = take((size_t)kSlots * n_bins * kNin * 8);
    t->o_s8w = take(kNin * 8);
    t->o_ain = take(kNin * 8);
    t->o_uinv = take(3 * kNfft * 16);
    t->o_rinv = take(kNfft * 8);
    t->o_ufwd = take(kNfwd * kNfft * 16);
    t->o_rfwd = take(kNfft * 8);
    t->o_kfwd = take(kNin * 8);
    t->o_qx = take((size_t)rows * kNfft * 8);
    t->o_tw = take(kNfft * 16);
    t->o_lo = take(n_bins * 4);
    t->o_hi = take(n_bins * 4);
    t->o_bw = take(kNin * 8);
    t->ws_need = off;
    *out = t;
    return LPP_OK;
}

extern "C" void lpp_template_destroy(lpp_template_t t) { delete t; }

extern "C" lpp_status lpp_template_workspace_size(lpp_template_t t, size_t* bytes) {
    if (!t || !bytes) return LPP_ERR_INVALID_ARG;
    *bytes = t->ws_need;
    return LPP_OK;
}

extern "C" lpp_status lpp_template_set_workspace(lpp_template_t t, void* dev, size_t bytes, void* stream) {
    if (!t || !dev) return LPP_ERR_INVALID_ARG;
    if (((uintptr_t)dev & 255) != 0) return LPP_ERR_INVALID_ARG;
    if (bytes < t->ws_need) return LPP_ERR_WORKSPACE;
    t->ws = (char*)dev;
    cudaStream_t st = (cudaStream_t)stream;
    auto put = [&](size_t o, const void* src, size_t b) {
        return cudaMemcpyAsync(t->ws + o, src, b, cudaMemcpyHostToDevice, st);
    };
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess) e = put(t->o_kin, t->kin.data(), kNin * 8);
    if (e == cudaSuccess) e = put(t->o_lnk, t->lnk.data(), kNin * 8);
    if (e == cudaSuccess) e = put(t->o_ik, t->ik.data(), kNin * 8);
    if (e == cudaSuccess) e = put(t->o_logtab, t->logtab.data(), 128 * 16);
    if (e == cudaSuccess) e = put(t->o_iref, t->iref.data(), kNin * 8);
    if (e == cudaSuccess) e = put(t->o_s8w, t->s8w.data(), kNin * 8);
    if (e == cudaSuccess) e = put(t->o_ain, t->ain.data(), kNin * 8);
    if (e == cudaSuccess) e = put(t->o_uinv, t->uinv.data(), 3 * kNfft * 16);
    if (e == cudaSuccess) e = put(t->o_rinv, t->rinv.data(), kNfft * 8);
    if (e == cudaSuccess) e = put(t->o_ufwd, t->ufwd.data(), kNfwd * kNfft * 16);
    if (e == cudaSuccess) e = put(t->o_rfwd, t->rfwd.data(), kNfft * 8);
    if (e == cudaSuccess) e = put(t->o_kfwd, t->kfwd.data(), kNin * 8);
    if (e == cudaSuccess) e = put(t->o_qx, t->qx.data(), t->qx.size() * 8);
    if (e == cudaSuccess) e = put(t->o_tw, t->tw.data(), kNfft * 16);
    if (e == cudaSuccess) e = put(t->o_lo, t->bin_lo.data(), t->nb * 4);
    if (e == cudaSuccess) e = put(t->o_hi, t->bin_hi.data(), t->nb * 4);
    if (e == cudaSuccess) e = put(t->o_bw, t->bin_w.data(), kNin * 8);
    if (e == cudaSuccess) {
        // the operator's rows, once per window
        OperatorArgs a;
        memset(&a, 0, sizeof(a));
        a.ain = (const double*)(t->ws + t->o_ain);
        a.uinv = (const double2*)(t->ws + t->o_uinv);
        a.rinv = (const double*)(t->ws + t->o_rinv);
        a.ufwd = (const double2*)(t->ws + t->o_ufwd);
        a.rfwd = (const double*)(t->ws + t->o_rfwd);
        a.kfwd = (const double*)(t->ws + t->o_kfwd);
        a.qx = (const double*)(t->ws + t->o_qx);
        a.tw = (const double2*)(t->ws + t->o_tw);
        a.bin_lo = (const int*)(t->ws + t->o_lo);
        a.bin_hi = (const int*)(t->ws + t->o_hi);
        a.bin_w = (const double*)(t->ws + t->o_bw);
        a.nb = t->nb;
        for (int s = 0; s < kSlots; ++s) a.slots[s] = t->slots[s];
        a.op = (double*)(t->ws + t->o_op);
        const size_t smem = (size_t)kNfft * 16 + (size_t)kNfft * 8 + (size_t)kNin * 8;
        cudaFuncSetAttribute(k_operator, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_operator<<<kSlots * t->nb, 512, smem, st>>>(a);
        k_op_digits<<<kSlots * t->nb, 256, 0, st>>>(a.op, (const double*)(t->ws + t->o_iref), kSlots * t->nb,
                                                    (uint2*)(t->ws + t->o_digits), (int*)(t->ws + t->o_exponent));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return LPP_ERR_CUDA;
    t->ready = true;
    return LPP_OK;
}

static lpp_status convolve(lpp_template_t t, const double* params, int n_templates, double* out, float* eb,
                           const double* eb_ref, const double* eb_sigma, void* stream);

extern "C" lpp_status lpp_template_set_png(lpp_template_t t, double f_nl, double db_ia, double omega_m) {
    if (!t || !(omega_m > 0.0) || !(db_ia == db_ia) || !(f_nl == f_nl)) return LPP_ERR_INVALID_ARG;
    const double c_over_h0 = 2997.92458;   // Mpc/h: c / (100 km/s/Mpc)
    t->png_amp = 12.0 * f_nl * db_ia;
    t->png_len2 = c_over_h0 * c_over_h0 / omega_m;
    return LPP_OK;
}

extern "C" lpp_status lpp_template_set_slots(lpp_template_t t, unsigned mask) {
    if (!t || (mask >> kSlots) != 0u) return LPP_ERR_INVALID_ARG;
    t->slot_mask = mask;
    return LPP_OK;
}

extern "C" lpp_status lpp_convolve_template(lpp_template_t t, const double* params, int n_templates, double* out,
                                            void* stream) {
    return convolve(t, params, n_templates, out, nullptr, nullptr, nullptr, stream);
}

extern "C" lpp_status lpp_convolve_template_eb(lpp_template_t t, const double* params, int n_templates, double* out,
                                               float* eb, const double* eb_ref, const double* eb_sigma, void* stream) {
    if (n_templates > 0 && !eb) return LPP_ERR_INVALID_ARG;
    if (t && (t->slot_mask & kEbSlots) != kEbSlots) return LPP_ERR_INVALID_ARG;
    return convolve(t, params, n_templates, out, eb, eb_ref, eb_sigma, stream);
}

static lpp_status convolve(lpp_template_t t, const double* params, int n_templates, double* out, float* eb,
                           const double* eb_ref, const double* eb_sigma, void* stream) {
    if (!t || (n_templates > 0 && (!params || !out)) || n_templates < 0) return LPP_ERR_INVALID_ARG;
    if (!t->ready) return LPP_ERR_NOT_READY;
    if (n_templates == 0) return LPP_OK;
    TemplateArgs a;
    memset(&a, 0, sizeof(a));
    a.params = params;
    a.n_templates = n_templates;
    a.out = out;
    a.op = (const double*)(t->ws + t->o_op);
    a.digits = (const uint2*)(t->ws + t->o_digits);
    a.exponent = (const int*)(t->ws + t->o_exponent);
    a.iref = (const double*)(t->ws + t->o_iref);
    a.kin = (const double*)(t->ws + t->o_kin);
    a.lnk = (const double*)(t->ws + t->o_lnk);
    a.ik = (const double*)(t->ws + t->o_ik);
    a.logtab = (const double2*)(t->ws + t->o_logtab);
    a.dlnk = t->dlnk;
    a.s8w = (const double*)(t->ws + t->o_s8w);
    a.bin_lo = (const int*)(t->ws + t->o_lo);
    a.bin_hi = (const int*)(t->ws + t->o_hi);
    a.nb = t->nb;
    a.shot_plus = t->shot_plus;
    a.png_amp = t->png_amp;
    a.png_len2 = t->png_len2;
    a.slot_mask = t->slot_mask;
    for (int s = 0; s < kSlots; ++s)
        if ((t->slot_mask >> s) & 1u) a.slot[a.n_slots++] = s;
    a.eb = eb;
    a.eb_ref = eb_ref;
    a.eb_sigma = eb_sigma;
    lpp::eb_matrices(a.N, a.M);
    if (n_templates >= kManyFrom && t->png_amp == 0.0 && a.n_slots > 0) {
        // shells per cluster: at most kManyRows rows, and enough clusters for every SM
        const int many = (n_templates + kManySets - 1) / kManySets;
        const int cl = many >= kWideFrom ? 4 : 8;
        int groups = std::max((t->nb * a.n_slots + kManyRows - 1) / kManyRows, std::min(t->nb, (19 + many - 1) / many));
        a.bins = (t->nb + groups - 1) / groups;
        while (a.bins > 1 && a.bins * a.n_slots > kManyRows) --a.bins;
        groups = (t->nb + a.bins - 1) / a.bins;
        const size_t smem = (size_t)kDigits * 16 * 2 * 32 * sizeof(uint2) +
                            (size_t)a.bins * a.n_slots * kManySets * sizeof(double);
        auto launch = [&](void (*kernel)(TemplateArgs)) {
            if (lpp::allow_shared(kernel, kManySmem) != cudaSuccess) return LPP_ERR_CUDA;
            kernel<<<dim3(many * cl, groups), 256, smem, (cudaStream_t)stream>>>(a);
            return cudaGetLastError() == cudaSuccess ? LPP_OK : LPP_ERR_CUDA;
        };
        return cl == 4 ? launch(k_template_many<4>) : launch(k_template_many<8>);
    }
    // shells per cluster: at most kMaxRows rows, and enough clusters for every SM (2 x 19 clusters of 8)
    const int clusters = (n_templates + kSets - 1) / kSets, ns = a.n_slots > 0 ? a.n_slots : 1;
    int groups = std::max((t->nb * ns + kMaxRows - 1) / kMaxRows, std::min(t->nb, (38 + clusters - 1) / clusters));
    a.bins = (t->nb + groups - 1) / groups;
    while (a.bins > 1 && a.bins * ns > kMaxRows) --a.bins;
    groups = (t->nb + a.bins - 1) / a.bins;
    // few rows: a warp takes one column segment (at most four tiles each, so that all eight warps
    // have work and few loads in a row)
    const int rows = ns * a.bins, kparts = rows <= 64 ? kSegs : 1;
    const int nt = ((rows + 7) / 8 + 8 / kparts - 1) / (8 / kparts);
    const size_t smem = ((size_t)(t->png_amp != 0.0 ? 3 : 1) * kSets * kSlabPad + (size_t)kparts * rows * kSets) *
                        sizeof(double);
    auto launch = [&](void (*kernel)(TemplateArgs)) {
        if (lpp::allow_shared(kernel, kTemplateSmem) != cudaSuccess) return LPP_ERR_CUDA;
        kernel<<<dim3(clusters * kCluster, groups), 256, smem, (cudaStream_t)stream>>>(a);
        return cudaGetLastError() == cudaSuccess ? LPP_OK : LPP_ERR_CUDA;
    };
    if (n_templates <= kFewSets) return launch(k_template<1, 1, true>);
    if (kparts == kSegs) {
        switch (nt) {
            case 1: return launch(k_template<1, kSegs>);
            case 2: return launch(k_template<2, kSegs>);
            case 3: return launch(k_template<3, kSegs>);
            default: return launch(k_template<4, kSegs>);
        }
    }
    switch (nt) {
        case 2: return launch(k_template<2, 1>);
        case 3: return launch(k_template<3, 1>);
        case 4: return launch(k_template<4, 1>);
        case 5: return launch(k_template<5, 1>);
        case 6: return launch(k_template<6, 1>);
        case 7: return launch(k_template<7, 1>);
        case 8: return launch(k_template<8, 1>);
        default: return launch(k_template<9, 1>);
    }
}
