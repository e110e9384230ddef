// Per-particle harmonic weights, catalogue sums and CIC/TSC mass assignment.
//
// Harmonic weights.  For a galaxy at xhat with shear gamma, every LPP kernel is a
// pure degree-L spherical harmonic of khat (Y_L^m(S^-1(x) k) = N Lm_L(k.x) e^{im phi},
// Appendix C):
//   cross: gamma (2 e*_ij k_i k_j) Lm2_L(mu)/(1-mu^2)       (Eq. def_of_Xiij)
//   plus : gamma L_l(mu)                                    (Eq. lpp_estimator_auto_+)
//   minus: gamma (2 e*_ij k_i k_j)^2 Lm4_L(mu)/(1-mu^2)^2   (Eq. def_of_Xiijkl)
// with 2 e*_ij k_i k_j = (k.e_theta - i k.e_phi)^2: up to the factor gamma, the spin-0, 2 and 4
// harmonics of the galaxy's own frame.  Its 2L+1 real-harmonic coefficients are the column of
// the degree-L rotation that takes the grid's frame to the galaxy's, written with three angles:
// the polar angles (theta, phi) of xhat and the angle psi by which (e_theta, e_phi) of the plan's
// pole is turned against the grid's own tangent vectors there,
//   k.et - i k.ep = e^{i psi} (k.e_theta - i k.e_phi),
//   c_{+n} = gamma e^{i s psi} (A_n(theta) cos n phi - i B_n(theta) sin n phi),
//   c_{-n} = gamma e^{i s psi} (A_n(theta) sin n phi + i B_n(theta) cos n phi),
// with A_n, B_n short trigonometric series (kernel_series).  One field per coefficient then
// carries the kernel to the grid: F(k) = sum_n Y_{L,n}(khat) FT[sum_g w_g c_n(g) delta_D](k).
#include "lpp_internal.h"
#include "lpp_kernels.h"

namespace lpp {

// Sky frame about the pole p: e_phi = unit(p x xhat), e_theta = e_phi x xhat.
template <typename T>
__device__ __forceinline__ void sky_frame(const T xh[3], const double pole[3], T et[3], T ep[3], int* err) {
    const T p0 = (T)pole[0], p1 = (T)pole[1], p2 = (T)pole[2];
    T c0 = p1 * xh[2] - p2 * xh[1];
    T c1 = p2 * xh[0] - p0 * xh[2];
    T c2v = p0 * xh[1] - p1 * xh[0];
    T nrm = sqrt(c0 * c0 + c1 * c1 + c2v * c2v);
    if (!(nrm >= (T)1e-6)) {
        atomicOr(err, ERRF_POLE);
        nrm = (T)1;
    }
    ep[0] = c0 / nrm;
    ep[1] = c1 / nrm;
    ep[2] = c2v / nrm;
    et[0] = ep[1] * xh[2] - ep[2] * xh[1];
    et[1] = ep[2] * xh[0] - ep[0] * xh[2];
    et[2] = ep[0] * xh[1] - ep[1] * xh[0];
}

// The coefficients of one kernel (compile-time K) for one galaxy: g = w gamma e^{i s psi},
// ct[j] = cos j theta, st[j] = sin j theta, cp[n], sp[n] of n phi.  The series coefficients are
// kernel parameters at compile-time offsets (constant-bank operands of the multiply-adds).
template <typename T, int K, int LMAX>
__device__ __forceinline__ void project_kernel(const CoeffArgs<T>& a, const CoeffGroup& grp, long long i, T gr, T gi,
                                               const T (&ct)[LMAX + 1], const T (&st)[LMAX + 1],
                                               const T (&cp)[LMAX + 1], const T (&sp)[LMAX + 1]) {
    constexpr int L = kernel_degree(K), O = kernel_offset(K);
    T* re = a.coeff + (long long)(grp.row_re + L) * a.stride + i;
    T* im = grp.has_im ? a.coeff + (long long)(grp.row_im + L) * a.stride + i : nullptr;
#pragma unroll
    for (int n = 0; n <= L; ++n) {
        T A = (T)0, B = (T)0;
#pragma unroll
        for (int j = 0; j <= L; ++j) {
            const T f = (n & 1) ? st[j] : ct[j];
            if ((n & 1) && j == 0) continue;
            if (j & 1) B += a.tab[O + n * (L + 1) + j] * f;
            else A += a.tab[O + n * (L + 1) + j] * f;
        }
        if (n == 0) {
            *re = A * gr;
            if (im) *im = A * gi;
        } else {
            const T ac = A * cp[n], as = A * sp[n], bc = B * cp[n], bs = B * sp[n];
            re[n * a.stride] = ac * gr + bs * gi;
            re[-n * a.stride] = as * gr - bc * gi;
            if (im) {
                im[n * a.stride] = ac * gi - bs * gr;
                im[-n * a.stride] = as * gi + bc * gr;
            }
        }
    }
}

template <typename T>
__device__ __forceinline__ void unit_los(const T* pos, long long count, long long i, const double obs[3], T xh[3],
                                         int* err) {
    T r0 = pos[i] - (T)obs[0];
    T r1 = pos[count + i] - (T)obs[1];
    T r2 = pos[2 * count + i] - (T)obs[2];
    T nrm = sqrt(r0 * r0 + r1 * r1 + r2 * r2);
    if (!(nrm > (T)0)) {
        atomicOr(err, ERRF_OBSERVER);
        nrm = (T)1;
    }
    xh[0] = r0 / nrm;
    xh[1] = r1 / nrm;
    xh[2] = r2 / nrm;
}

template <typename T>
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void block_add(double v, double* dst) {
    __shared__ double part[32];
    v = warp_sum<double>(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) part[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = lane < (int)(blockDim.x >> 5) ? part[lane] : 0.0;
        v = warp_sum<double>(v);
        if (lane == 0 && v != 0.0) atomicAdd(dst, v);
    }
}

// LMAX: the largest degree, 8, or 12 for plans with the minus moments beyond L = 8 (a separate
// instantiation, so that its longer angle arrays leave the usual one unchanged).
//
// What bounds it: about 900 operations per galaxy (21,000 for the projection by quadrature, L + 1
// nodes x 2L + 1 azimuths per kernel, that it replaces) and the stores of its 138 rows.  With
// the statistics of the rows: 2 M galaxies FP32 2.74 -> 0.45 ms, 50,000 FP64 3.47 -> 0.12 ms.
template <typename T, int LMAX>
__global__ void __launch_bounds__(256) k_coeffs(const __grid_constant__ CoeffArgs<T> a) {
    double sw = 0.0, sg = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < a.count;
         i += (long long)gridDim.x * blockDim.x) {
        const long long si = a.perm ? (long long)a.perm[i] : i;  // input index of output particle i
        if (!LPP_IN_BOUNDS(si >= 0 && si < a.count, a.err)) continue;
        T xl[3];
        unit_los(a.pos, a.count, si, a.observer, xl, a.err);
        T xg[3] = {(T)a.los_global[0], (T)a.los_global[1], (T)a.los_global[2]};
        const T* xp = a.los_proj == LPP_LOS_GLOBAL ? xg : xl;
        const T* xe = a.los_est == LPP_LOS_GLOBAL ? xg : xl;
        T etp[3], epp[3], ete[3], epe[3];
        sky_frame(xp, a.pole, etp, epp, a.err);
        if (a.los_proj == a.los_est) {
            for (int d = 0; d < 3; ++d) { ete[d] = etp[d]; epe[d] = epp[d]; }
        } else {
            sky_frame(xe, a.pole, ete, epe, a.err);
        }
        T g1, g2;
        if (a.shape_kind == LPP_SHAPE_TENSOR6) {
            const T* s = a.shape;
            const long long c = a.count;
            const T sxx = s[si], syy = s[c + si], szz = s[2 * c + si], sxy = s[3 * c + si], sxz = s[4 * c + si],
                    syz = s[5 * c + si];
            const T st0 = sxx * etp[0] + sxy * etp[1] + sxz * etp[2];
            const T st1 = sxy * etp[0] + syy * etp[1] + syz * etp[2];
            const T st2 = sxz * etp[0] + syz * etp[1] + szz * etp[2];
            const T sp0 = sxx * epp[0] + sxy * epp[1] + sxz * epp[2];
            const T sp1 = sxy * epp[0] + syy * epp[1] + syz * epp[2];
            const T sp2 = sxz * epp[0] + syz * epp[1] + szz * epp[2];
            const T stt = etp[0] * st0 + etp[1] * st1 + etp[2] * st2;
            const T spp = epp[0] * sp0 + epp[1] * sp1 + epp[2] * sp2;
            const T stp = etp[0] * sp0 + etp[1] * sp1 + etp[2] * sp2;
            g1 = (T)0.5 * (stt - spp);  // gamma = e_ij s_ij (Eq. gamma_def)
            g2 = stp;
        } else {
            g1 = a.shape[si];
            g2 = a.shape[a.count + si];
        }
        const T w = a.w ? a.w[si] : (T)1;
        a.coeff[i] = w * g1;              // row 0: w gamma_1
        a.coeff[a.stride + i] = w * g2;   // row 1: w gamma_2
        sw += (double)w;
        sg += (double)w * (double)w * ((double)g1 * g1 + (double)g2 * g2);
        if (a.n_groups == 0) continue;
        // angles of the estimator's line of sight in the grid's frame (phi = 0 on its z axis, and so
        // close to it that the axis is the same direction to the last digit: there the squares may
        // underflow, and a division by their root would not give a unit vector)
        T ct[LMAX + 1], st[LMAX + 1], cp[LMAX + 1], sp[LMAX + 1];
        ct[0] = cp[0] = (T)1;
        st[0] = sp[0] = (T)0;
        const T rho = sqrt(xe[0] * xe[0] + xe[1] * xe[1]);
        ct[1] = xe[2];
        st[1] = rho;
        const bool off_axis = rho > (T)(sizeof(T) == 4 ? 1e-15 : 1e-100);
        cp[1] = off_axis ? xe[0] / rho : (T)1;
        sp[1] = off_axis ? xe[1] / rho : (T)0;
#pragma unroll
        for (int j = 2; j <= LMAX; ++j) {
            ct[j] = ct[j - 1] * ct[1] - st[j - 1] * st[1];
            st[j] = st[j - 1] * ct[1] + ct[j - 1] * st[1];
            cp[j] = cp[j - 1] * cp[1] - sp[j - 1] * sp[1];
            sp[j] = sp[j - 1] * cp[1] + cp[j - 1] * sp[1];
        }
        // psi: ete = cos psi e_theta + sin psi e_phi
        const T cps = ete[0] * ct[1] * cp[1] + ete[1] * ct[1] * sp[1] - ete[2] * st[1];
        const T sps = ete[1] * cp[1] - ete[0] * sp[1];
        const T c2p = cps * cps - sps * sps, s2p = (T)2 * cps * sps;
        T gr[3], gi[3];   // w gamma e^{i s psi} for s = 0, 2, 4
        gr[0] = w * g1;
        gi[0] = w * g2;
#pragma unroll
        for (int s = 1; s < 3; ++s) {
            gr[s] = gr[s - 1] * c2p - gi[s - 1] * s2p;
            gi[s] = gr[s - 1] * s2p + gi[s - 1] * c2p;
        }
        for (int q = 0; q < a.n_groups; ++q) {
            const CoeffGroup& g = a.groups[q];
            switch (g.kernel) {
#define LPP_KERNEL_CASE(K) \
    case K: project_kernel<T, K, LMAX>(a, g, i, gr[kernel_spin(K) / 2], gi[kernel_spin(K) / 2], ct, st, cp, sp); break;
                LPP_KERNEL_CASE(0) LPP_KERNEL_CASE(1) LPP_KERNEL_CASE(2) LPP_KERNEL_CASE(3) LPP_KERNEL_CASE(4)
                LPP_KERNEL_CASE(5) LPP_KERNEL_CASE(6) LPP_KERNEL_CASE(7)
                default:
                    if constexpr (LMAX > 8) {
                        switch (g.kernel) { LPP_KERNEL_CASE(8) LPP_KERNEL_CASE(9) }
                    }
#undef LPP_KERNEL_CASE
            }
        }
    }
    block_add(sw, a.sums + SUM_W_SHAPES);
    block_add(sg, a.sums + SUM_W2G2_SHAPES);
}

template <typename T>
cudaError_t launch_coeffs(const CoeffArgs<T>& a, cudaStream_t st) {
    if (a.count == 0) return cudaSuccess;
    long long blocks = (a.count + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    bool high = false;
    for (int g = 0; g < a.n_groups; ++g) high = high || kernel_degree(a.groups[g].kernel) > 8;
    if (high) k_coeffs<T, 12><<<(int)blocks, 256, 0, st>>>(a);
    else k_coeffs<T, 8><<<(int)blocks, 256, 0, st>>>(a);
    return cudaGetLastError();
}

template <typename T>
__global__ void __launch_bounds__(256) k_sums(const T* w, const T* nbar, long long count, double* sums, int s_w,
                                              int s_w2, int s_nw2) {
    double a = 0.0, b = 0.0, c = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        const double wi = w ? (double)w[i] : 1.0;
        const double ni = nbar ? (double)nbar[i] : 1.0;
        a += wi;
        b += wi * wi;
        c += ni * wi * wi;
    }
    if (s_w >= 0) block_add(a, sums + s_w);
    if (s_w2 >= 0) block_add(b, sums + s_w2);
    if (s_nw2 >= 0) block_add(c, sums + s_nw2);
}

template <typename T>
cudaError_t launch_sums(const T* w, const T* nbar, long long count, double* sums, int s_w, int s_w2, int s_nw2,
                        cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    long long blocks = (count + 255) / 256;
    if (blocks > 152 * 8) blocks = 152 * 8;
    k_sums<T><<<(int)blocks, 256, 0, st>>>(w, nbar, count, sums, s_w, s_w2, s_nw2);
    return cudaGetLastError();
}

__global__ void k_alpha(double* sums, int has_randoms) {
    sums[SUM_ALPHA] = (has_randoms && sums[SUM_W_RAND] != 0.0) ? sums[SUM_W_DENS] / sums[SUM_W_RAND] : 0.0;
}

cudaError_t launch_alpha(double* sums, int has_randoms, cudaStream_t st) {
    k_alpha<<<1, 1, 0, st>>>(sums, has_randoms);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ assignment
// Node i of sub-grid s sits at origin + (i + s/2) H.  CIC (P = 2): w(d) = 1 - |d|;
// TSC (P = 3): w(d) = 3/4 - d^2 for |d| <= 1/2, (3/2 - |d|)^2 / 2 for 1/2 <= |d| < 3/2.
template <typename T, int P>
__device__ __forceinline__ void stencil(T u, int n, int cells[P], T w[P]) {
    if (P == 2) {
        const T fl = floor(u);
        const T f = u - fl;
        int i0 = (int)fl;
        w[0] = (T)1 - f;
        w[1] = f;
        cells[0] = i0;
        cells[1] = i0 + 1;
    } else {
        const T ic = floor(u + (T)0.5);
        const T d = u - ic;
        const int c = (int)ic;
        const T hm = (T)0.5 - d, hp = (T)0.5 + d;
        w[0] = (T)0.5 * hm * hm;
        w[1] = (T)0.75 - d * d;
        w[2] = (T)0.5 * hp * hp;
        cells[0] = c - 1;
        cells[1] = c;
        cells[2] = c + 1;
    }
#pragma unroll
    for (int k = 0; k < P; ++k) {
        int c = cells[k];
        c = c < 0 ? c + n : (c >= n ? c - n : c);
        cells[k] = c;
    }
}

template <typename T, int P, bool IL>
__global__ void __launch_bounds__(256) k_assign(AssignArgs<T> a) {
    const int n = a.n;
    const T ih = (T)((double)n / a.box);
    const T ox = (T)a.origin[0], oy = (T)a.origin[1], oz = (T)a.origin[2];
    const T alpha = (T)a.sums[SUM_ALPHA];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < a.count;
         i += (long long)gridDim.x * blockDim.x) {
        const T u0 = (a.pos[i] - ox) * ih;
        const T u1 = (a.pos[a.count + i] - oy) * ih;
        const T u2 = (a.pos[2 * a.count + i] - oz) * ih;
        if (!(u0 >= (T)0 && u0 <= (T)n && u1 >= (T)0 && u1 <= (T)n && u2 >= (T)0 && u2 <= (T)n)) {
            atomicOr(a.err, ERRF_DOMAIN);
            continue;
        }
        int cx[P], cy[P], cz[P];
        T wx[P], wy[P], wz[P];
        stencil<T, P>(u0, n, cx, wx);
        stencil<T, P>(u1, n, cy, wy);
        stencil<T, P>(u2, n, cz, wz);
        int dx[P], dy[P], dz[P];
        T vx[P], vy[P], vz[P];
        if (IL) {
            stencil<T, P>(u0 - (T)0.5, n, dx, vx);
            stencil<T, P>(u1 - (T)0.5, n, dy, vy);
            stencil<T, P>(u2 - (T)0.5, n, dz, vz);
        }
        for (int s = 0; s < a.n_slots; ++s) {
            const AssignSlot& sl = a.slots[s];
            T va = sl.unit_a ? (T)1 : static_cast<const T*>(sl.src_a)[i];
            if (sl.scale_alpha) va *= -alpha;
            const bool has_b = !IL && sl.src_b != nullptr;
            const T vb = has_b ? static_cast<const T*>(sl.src_b)[i] : (T)0;
            T* g = reinterpret_cast<T*>(a.grids + sl.grid * a.grid_stride);
#pragma unroll
            for (int kz = 0; kz < P; ++kz)
#pragma unroll
                for (int ky = 0; ky < P; ++ky) {
                    const long long row = ((long long)cz[kz] * n + cy[ky]) * n;
                    const T wzy = wz[kz] * wy[ky];
#pragma unroll
                    for (int kx = 0; kx < P; ++kx) {
                        const long long idx = 2 * (row + cx[kx]);
                        const T ww = wzy * wx[kx];
                        atomicAdd(g + idx, va * ww);
                        if (has_b) atomicAdd(g + idx + 1, vb * ww);
                    }
                }
            if (IL) {
#pragma unroll
                for (int kz = 0; kz < P; ++kz)
#pragma unroll
                    for (int ky = 0; ky < P; ++ky) {
                        const long long row = ((long long)dz[kz] * n + dy[ky]) * n;
                        const T wzy = vz[kz] * vy[ky];
#pragma unroll
                        for (int kx = 0; kx < P; ++kx) atomicAdd(g + 2 * (row + dx[kx]) + 1, va * (wzy * vx[kx]));
                    }
            }
        }
    }
}

template <typename T>
cudaError_t launch_assign(const AssignArgs<T>& a, int scheme, int interlace, cudaStream_t st) {
    if (a.count == 0 || a.n_slots == 0) return cudaSuccess;
    long long blocks = (a.count + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    const int b = (int)blocks;
    if (scheme == LPP_CIC) {
        if (interlace) k_assign<T, 2, true><<<b, 256, 0, st>>>(a);
        else k_assign<T, 2, false><<<b, 256, 0, st>>>(a);
    } else {
        if (interlace) k_assign<T, 3, true><<<b, 256, 0, st>>>(a);
        else k_assign<T, 3, false><<<b, 256, 0, st>>>(a);
    }
    return cudaGetLastError();
}

// Per-row statistics of the coefficients: rstat[2r] = max |c| (atomicMax on the float's
// bits: non-negative floats order like ints) and rstat[2r + 1] = rms c, from a grid-stride
// loop per row (blockIdx.y), warp reductions and FP64 sums of squares in rsq.
__global__ void __launch_bounds__(256) k_rowstat(const float* __restrict__ coeff, long long stride, long long count,
                                                 float* __restrict__ rstat, double* __restrict__ rsq) {
    const float* row = coeff + (long long)blockIdx.y * stride;
    float m = 0.f, qf = 0.f;   // per-thread sums cover count / (64 * 256) values: FP32 is plenty
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        const float v = row[i];
        m = fmaxf(m, fabsf(v));
        qf = fmaf(v, v, qf);
    }
    double q = (double)qf;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, o));
        q += __shfl_down_sync(0xffffffffu, q, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (m > 0.f) atomicMax(reinterpret_cast<int*>(rstat) + 2 * blockIdx.y, __float_as_int(m));
        if (q > 0.0) atomicAdd(rsq + blockIdx.y, q);
    }
}

__global__ void k_rowrms(const double* __restrict__ rsq, long long count, int rows, float* __restrict__ rstat) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < rows) rstat[2 * r + 1] = count > 0 ? (float)sqrt(rsq[r] / (double)count) : 0.f;
}

cudaError_t launch_rowstat(const float* coeff, long long stride, long long count, int rows, float* rstat,
                           double* rsq, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(rstat, 0, (size_t)rows * 2 * sizeof(float), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(rsq, 0, (size_t)rows * sizeof(double), st);
    if (e != cudaSuccess || count == 0 || rows == 0) return e;
    long long bx = (count + 2047) / 2048;   // at least eight values per thread
    if (bx > 64) bx = 64;
    k_rowstat<<<dim3((unsigned)bx, (unsigned)rows), 256, 0, st>>>(coeff, stride, count, rstat, rsq);
    k_rowrms<<<(rows + 127) / 128, 128, 0, st>>>(rsq, count, rows, rstat);
    return cudaGetLastError();
}

template cudaError_t launch_coeffs<float>(const CoeffArgs<float>&, cudaStream_t);
template cudaError_t launch_coeffs<double>(const CoeffArgs<double>&, cudaStream_t);
template cudaError_t launch_sums<float>(const float*, const float*, long long, double*, int, int, int, cudaStream_t);
template cudaError_t launch_sums<double>(const double*, const double*, long long, double*, int, int, int,
                                         cudaStream_t);
template cudaError_t launch_assign<float>(const AssignArgs<float>&, int, int, cudaStream_t);
template cudaError_t launch_assign<double>(const AssignArgs<double>&, int, int, cudaStream_t);

}  // namespace lpp
