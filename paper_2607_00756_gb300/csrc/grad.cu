// Reverse pass of a map loss through the contraction (the matrices as a
// forward model, Sec. 5): given g(rho) = dL/dI(rho), the derivatives with
// respect to the site occupancies, the transition potentials H and the
// probe aberrations.  Per site tau, f = f_y f_x:
//   R_tau     = f o_tau sum_{rho in crop} g(rho) c(rho) c(rho)^H     [B x B]
//   Mbar_n    = M_n R_tau            (stored as GMt = conj(R) Mt, Mt[b][(n, d)])
//   T_n(b, r) = sum_d Mbar_n(d, b) conj S2_d(r)
//   dL/dH_n(r) (as dL/dRe + i dL/dIm) = 2 sum_b conj S1_b(r) T_n(b, r)
//   D_b      += (Q_tau R_tau)_bb,  dL/dtheta = -2 sum_b chi'_b Im D_b
//   dL/do_tau = sum_rho g(rho) I_tau(rho)
//
// The contractions run in cgemm_f32.cu (or gemm_tc.cu in split BF16); here:
//   crop_weight_kernel, hgrad_kernel, aberr_kernel, aberr_sum_kernel,
//   occ_grad_kernel
#include "bip_device.cuh"
#include "bip_internal.h"
#include "fft_smem.cuh"

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float2 conjf2(float2 a) { return make_float2(a.x, -a.y); }

// w[bs][rho] = f o_tau g(rho) inside the site's crop window, else 0
__global__ void crop_weight_kernel(GradArgs a, int nb, const int32_t* ids, float* w) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x, bs = blockIdx.y;
    if (p >= a.P) return;
    const int site = ids[bs];
    const SiteDev st = a.sites[site];
    float v = 0.f;
    if (in_crop(a.scans[2 * p], a.scans[2 * p + 1], st.ty, st.tx, a.ny, a.nx, a.fy, a.fx)) {
        const double o = a.occ ? a.occ[site] : 1.0;
        v = (float)(a.scale * o * a.dL_dI[p]);
    }
    w[(size_t)bs * a.P + p] = v;
}

// dL/dH_n(r) = 2 sum_b conj S1_b(r) T_n(b, r); thread = pixel, block row =
// (site, channel)
__global__ void hgrad_kernel(GradArgs a, const int32_t* ids, const float2* S1, int64_t s1_site, const float2* T,
                             int64_t t_site, int64_t t_ch, float2* dH) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    const int bs = blockIdx.y, n = blockIdx.z;
    if (r >= a.K) return;
    const SiteDev st = a.sites[ids[bs]];
    if (n >= st.nch) return;
    const float2* s1 = S1 + (int64_t)bs * s1_site + r;
    const float2* t = T + (int64_t)bs * t_site + (int64_t)n * t_ch + r;
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll 8                     // eight beams' loads in flight: few blocks, a long sum each
    for (int b = 0; b < a.B; ++b) {
        const float2 x = conjf2(__ldg(&s1[(int64_t)b * a.K]));
        const float2 y = __ldg(&t[(int64_t)b * a.K]);
        acc.x = fmaf(x.x, y.x, fmaf(-x.y, y.y, acc.x));
        acc.y = fmaf(x.x, y.y, fmaf(x.y, y.x, acc.y));
    }
    dH[(size_t)st.h_off + (size_t)n * a.K + r] = make_float2(2.f * acc.x, 2.f * acc.y);
}

// D[bs][b] = sum_b' Q[b][b'] R[b'][b]
__global__ void aberr_kernel(int B, int Bpad, const float2* Q, int64_t q_site, const float2* R, int64_t r_site,
                             double2* D) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x, bs = blockIdx.y;
    if (b >= B) return;
    const float2* q = Q + (int64_t)bs * q_site + (int64_t)b * Bpad;
    const float2* rr = R + (int64_t)bs * r_site + b;
    double sx = 0.0, sy = 0.0;
    for (int k = 0; k < B; ++k) {
        const float2 x = q[k], y = rr[(int64_t)k * Bpad];
        sx += (double)x.x * y.x - (double)x.y * y.y;
        sy += (double)x.x * y.y + (double)x.y * y.x;
    }
    D[(size_t)bs * B + b] = make_double2(sx, sy);
}

// Dsum[b] += sum over the batch's sites of D[bs][b], in site order
__global__ void aberr_sum_kernel(int B, int nb, const double2* D, double2* Dsum) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    double2 s = Dsum[b];
    for (int bs = 0; bs < nb; ++bs) {
        s.x += D[(size_t)bs * B + b].x;
        s.y += D[(size_t)bs * B + b].y;
    }
    Dsum[b] = s;
}

// dL/do_tau = sum_rho g(rho) I_tau(rho); block per site
__global__ void occ_grad_kernel(const float* partial, int P, const double* g, double* out) {
    __shared__ double red[kThreads / 32];
    const int k = blockIdx.x;
    double s = 0.0;
    for (int p = threadIdx.x; p < P; p += kThreads) s += g[p] * (double)partial[(size_t)k * P + p];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) t += red[w];
        out[k] = t;
    }
}

// x rounded to BF16 in the upper half (the lower half holds rubbish)
__device__ __forceinline__ uint32_t bf16_rn_u(float x) {
    const uint32_t u = __float_as_uint(x);
    return u + 0x7fffu + ((u >> 16) & 1u);
}
// two values as a pair of BF16 (hi) and their rests as another (lo)
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
    const uint32_t hx = bf16_rn_u(x), hy = bf16_rn_u(y);
    hi = __byte_perm(hx, hy, 0x7632);
    lo = __byte_perm(bf16_rn_u(x - __uint_as_float(hx & 0xffff0000u)),
                     bf16_rn_u(y - __uint_as_float(hy & 0xffff0000u)), 0x7632);
}
__device__ __forceinline__ void put2(uint16_t* dst, uint32_t v, bool pair, bool second) {
    if (pair) {
        *reinterpret_cast<uint32_t*>(dst) = v;
    } else {
        dst[0] = (uint16_t)v;
        if (second) dst[1] = (uint16_t)(v >> 16);
    }
}

// complex64 -> split-BF16 planes, block = 32 rows i x 64 columns k of the
// destination, a lane two adjacent k of a row: a warp writes 128 bytes of
// each plane at a time and reads 512 bytes of a row (the source's k
// contiguous) or 256 bytes of a column (its rows contiguous, turned in shared
// memory).  Bound by memory: 8 bytes read, 8 written per element.  With 32 x 32
// blocks and one element per lane the 2-byte stores bound it (64 bytes of a
// plane per warp); a reverse pass of 64 sites of 64^2 pixels, 80 launches, went
// from 28.8 to 27.1 ms in all.
template <bool TURN>
__global__ void __launch_bounds__(256) split_planes_kernel(SplitArgs a, bool src16, bool dst4) {
    __shared__ float2 tile[TURN ? 32 : 1][TURN ? 65 : 1];
    const int k0 = blockIdx.x * 64, i0 = blockIdx.y * 32, z = blockIdx.z;
    const int tx = threadIdx.x, ty = threadIdx.y;           // 32 x 8
    const float2* src = a.src + (int64_t)z * a.s_batch;
    const int k = k0 + 2 * tx;
    float2 v[8];                                            // (row ty + 8 j, k and k + 1) or (row tx, column ty + 8 j)
#pragma unroll
    for (int j = 0; j < (TURN ? 8 : 4); ++j) {
        if (TURN) {
            const int i = i0 + tx, kk = k0 + ty + 8 * j;
            v[j] = make_float2(0.f, 0.f);
            if (i < a.rows && kk < a.cols) v[j] = __ldg(&src[i + (int64_t)kk * a.s_col]);
        } else {
            const int i = i0 + ty + 8 * j;
            v[2 * j] = v[2 * j + 1] = make_float2(0.f, 0.f);
            if (i >= a.rows) continue;
            const float2* q = src + (int64_t)i * a.s_row + k;
            if (src16 && k + 1 < a.cols) {
                const float4 f = __ldg(reinterpret_cast<const float4*>(q));
                v[2 * j] = make_float2(f.x, f.y);
                v[2 * j + 1] = make_float2(f.z, f.w);
            } else {
                if (k < a.cols) v[2 * j] = __ldg(q);
                if (k + 1 < a.cols) v[2 * j + 1] = __ldg(q + 1);
            }
        }
    }
    if (TURN) {
#pragma unroll
        for (int j = 0; j < 8; ++j) tile[tx][ty + 8 * j] = v[j];
        __syncthreads();
    }
    const int64_t plane = (int64_t)a.d_rows * a.d_cols;
    uint16_t* dst = a.dst + (int64_t)z * a.d_batch + a.dcol0 + k;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int i = i0 + ty + 8 * j;
        if (i >= a.rows || k >= a.cols) continue;
        float2 p = TURN ? tile[ty + 8 * j][2 * tx] : v[2 * j], q = TURN ? tile[ty + 8 * j][2 * tx + 1] : v[2 * j + 1];
        if (a.conj) {
            p.y = -p.y;
            q.y = -q.y;
        }
        uint32_t rh, rl, ih, il;
        split2(p.x, q.x, rh, rl);
        split2(p.y, q.y, ih, il);
        const bool second = k + 1 < a.cols, pair = dst4 && second;
        uint16_t* o = dst + (int64_t)i * a.d_cols;
        put2(o, rh, pair, second);
        put2(o + plane, rl, pair, second);
        put2(o + 2 * plane, ih, pair, second);
        put2(o + 3 * plane, il, pair, second);
    }
}

}  // namespace

cudaError_t bip_split_planes(const SplitArgs& a, cudaStream_t s) {
    if (a.rows < 1 || a.cols < 1 || a.batch < 1 || a.rows > a.d_rows || (int64_t)a.dcol0 + a.cols > a.d_cols)
        return cudaErrorInvalidValue;
    if (a.s_col != 1 && a.s_row != 1) return cudaErrorInvalidValue;
    const dim3 grid((a.cols + 63) / 64, (a.rows + 31) / 32, a.batch);
    if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidValue;
    // pairs of elements in one access, where the addresses allow it
    const bool src16 = ((uintptr_t)a.src & 15) == 0 && ((a.s_row | a.s_batch) & 1) == 0;
    const bool dst4 = ((uintptr_t)a.dst & 3) == 0 && ((a.d_cols | a.dcol0 | a.d_batch) & 1) == 0;
    if (a.s_col == 1)
        split_planes_kernel<false><<<grid, dim3(32, 8), 0, s>>>(a, src16, dst4);
    else
        split_planes_kernel<true><<<grid, dim3(32, 8), 0, s>>>(a, src16, dst4);
    return cudaGetLastError();
}

cudaError_t bip_grad_crop_weights(const GradArgs& a, int nb, const int32_t* ids, float* w, cudaStream_t s) {
    if (nb < 1 || a.P < 1) return cudaErrorInvalidValue;
    crop_weight_kernel<<<dim3((a.P + 255) / 256, nb), 256, 0, s>>>(a, nb, ids, w);
    return cudaGetLastError();
}

cudaError_t bip_grad_h(const GradArgs& a, int nb, const int32_t* ids, int nch, const float2* S1, int64_t s1_site,
                       const float2* T, int64_t t_site, int64_t t_ch, float2* dH, cudaStream_t s) {
    if (nb < 1 || nch < 1 || nch > 9) return cudaErrorInvalidValue;
    hgrad_kernel<<<dim3((a.K + 255) / 256, nb, nch), 256, 0, s>>>(a, ids, S1, s1_site, T, t_site, t_ch, dH);
    return cudaGetLastError();
}

cudaError_t bip_grad_aberr(int B, int Bpad, int nb, const float2* Q, int64_t q_site, const float2* R, int64_t r_site,
                           double2* D, double2* Dsum, cudaStream_t s) {
    if (nb < 1 || B < 1) return cudaErrorInvalidValue;
    aberr_kernel<<<dim3((B + 127) / 128, nb), 128, 0, s>>>(B, Bpad, Q, q_site, R, r_site, D);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    aberr_sum_kernel<<<(B + 127) / 128, 128, 0, s>>>(B, nb, D, Dsum);
    return cudaGetLastError();
}

cudaError_t bip_grad_occ(const float* partial, int n_sites, int P, const double* g, double* out, cudaStream_t s) {
    if (n_sites < 1) return cudaSuccess;
    occ_grad_kernel<<<n_sites, kThreads, 0, s>>>(partial, P, g, out);
    return cudaGetLastError();
}
