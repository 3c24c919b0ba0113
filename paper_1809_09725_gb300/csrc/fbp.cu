// fbp.cu -- filtered back-projection initial guess (Sec. 5 starts the
// iterations from an FBP reconstruction with the Shepp-Logan filter).
//
//   1. q[z][k][.] = h * g[z][k][.]   discrete Shepp-Logan kernel at unit bin
//      spacing, h(n) = -2 / (pi^2 (4 n^2 - 1)), linear (zero-padded)
//      convolution along s (shepp_logan_kernel below).
//   2. Projection k belongs to time window w(k) = clamp(floor(t_k nw)); the FBP
//      image of window w is f_w = (pi / K_w) sum_{k in w} R*_k q_k.  The
//      coefficients are the least-squares fit over the acquisition times,
//      u = argmin sum_k || sum_j phi_j(t_k) u_j - f_{w(k)} ||^2, i.e.
//      u_j = sum_w A[j][w] f_w with A = Phi^+ S (minimum-norm least squares,
//      (Phi^T Phi)^{-1} Phi^T S for functions independent over the times).
//      Both steps are linear in q, so u_j = sum_k Psi[k][j] R*_k q_k with
//      Psi[k][j] = (pi / K_{w(k)}) A[j][w(k)]: one dynamic back-projection
//      with the table Psi in place of Phi (either projector variant).
#include <algorithm>
#include <cmath>
#include <vector>

#include "dr_device.cuh"

namespace dr {

// Filter.  A task is R rows by four consecutive outputs of each, in registers: a
// step of four inputs takes four new taps (one vector, the lanes of a warp read
// consecutive ones) and four inputs of each row (one broadcast vector a row) for
// 16 R multiply-adds, where a thread with one output read a tap and an input for
// each.  The lanes of a row's task run along the outputs; short rows put several
// groups of R rows into one CTA, long ones are cut into tiles of at most 512
// outputs, and the inputs are staged kFbpChunk at a time.  Each output sums its
// row in ascending order, as one thread would by itself.
//
// Bound by the multiply-adds (ns per output).  7200 rows of 512: 0.32 -> 0.11 ms,
// half of the FP32 rate; the rest is the staging of inputs and the last wave
// (900 CTAs, five per SM).
constexpr int kFbpThreads = 128;
constexpr int kFbpChunk = 512;

template <typename S, typename T, int R>
__global__ void __launch_bounds__(kFbpThreads)
    shepp_logan_kernel(const S *__restrict__ g, T *__restrict__ q, const T *__restrict__ taps, long long rows,
                       int ns, int tb, int groups, int tiles) {
    struct alignas(4 * sizeof(T)) V4 { T v[4]; };
    extern __shared__ __align__(32) unsigned char fbp_smem[];
    const int clen = min(kFbpChunk, (ns + 3) & ~3);        // inputs staged at a time, padded with zeros
    V4 *h = reinterpret_cast<V4 *>(fbp_smem);               // [tb + clen / 4]
    T *row = reinterpret_cast<T *>(h + tb + clen / 4);      // [groups R][clen]
    const int tile = blockIdx.x % tiles;
    const long long r0 = (long long)(blockIdx.x / tiles) * groups * R;
    const int grp = threadIdx.x / tb, bt = threadIdx.x - grp * tb, B0 = tile * tb * 4;
    const bool on = grp < groups;
    T acc[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[r][i] = T(0);
    for (int c0 = 0; c0 < ns; c0 += clen) {
        const int n4 = (min(clen, ns - c0) + 3) >> 2;  // steps of this chunk
        __syncthreads();  // previous chunk consumed
        // h[k] = taps 4 (k + k0) - 3 .. 4 (k + k0)
        const int k0 = (B0 - c0) / 4 - (n4 - 1);
        for (int i = threadIdx.x; i < 4 * (tb + n4); i += blockDim.x) {
            const int d = 4 * k0 - 3 + i;
            reinterpret_cast<T *>(h)[i] = d > -ns && d < ns ? taps[d + ns - 1] : T(0);
        }
        for (int k = threadIdx.x; k < groups * R * 4 * n4; k += blockDim.x) {
            const int rr = k / (4 * n4), i = k - rr * (4 * n4);
            row[rr * clen + i] = r0 + rr < rows && c0 + i < ns ? ldc<T>(g + (r0 + rr) * ns + c0 + i) : T(0);
        }
        __syncthreads();
        if (!on) continue;
        const T *rg = row + grp * R * clen;
        V4 up = h[bt + n4];
#pragma unroll 2
        for (int s = 0; s < n4; ++s) {
            const V4 lo = h[bt + n4 - 1 - s];
            // w[3 + e] = h(b0 - b' + e)
            const T w[7] = {lo.v[0], lo.v[1], lo.v[2], lo.v[3], up.v[0], up.v[1], up.v[2]};
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const V4 x = reinterpret_cast<const V4 *>(rg + r * clen)[s];
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[r][i] = fma(w[3 + i - j], x.v[j], acc[r][i]);
            }
            up = lo;
        }
    }
    const int b = B0 + 4 * bt;
    if (!on) return;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const long long rr = r0 + grp * R + r;
        if (rr >= rows) break;
        T *o = q + rr * ns + b;
        if ((ns & 3) == 0 && b < ns) {
            *reinterpret_cast<V4 *>(o) = V4{{acc[r][0], acc[r][1], acc[r][2], acc[r][3]}};
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (b + i < ns) o[i] = acc[r][i];
        }
    }
}

__global__ void fbp_to_bf16_kernel(const float *__restrict__ x, bf16 *__restrict__ y, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16_rn(x[i]);
}

template <typename S, typename T, int R>
static dr_status launch_filter_t(dr_plan *P, const void *g, cudaStream_t st) {
    const long long rows = (long long)P->nz * P->K, rg = (rows + R - 1) / R;
    const int nb4 = (P->ns + 3) / 4, tiles = (nb4 + 127) / 128, tb = (nb4 + tiles - 1) / tiles;
    // as many groups per CTA as its threads hold, while every SM gets two CTAs; in
    // whole warps (idle lanes cost as much)
    const int unit = std::max(1, 32 / tb);
    const long long fill = std::max<long long>(rg * tiles / (2 * P->num_sms) / unit, 1) * unit;
    const int groups = (int)std::min<long long>(std::min<long long>(kFbpThreads / tb, fill), rg);
    const int clen = std::min(kFbpChunk, 4 * nb4);
    const size_t smem = sizeof(T) * (4 * tb + clen + (size_t)groups * R * clen);
    auto kern = shepp_logan_kernel<S, T, R>;
    const dr_status s = allow_dynamic_smem((const void *)kern, smem);
    if (s != DR_OK) return s;
    const long long grid = (rg + groups - 1) / groups * tiles;
    if (grid > 0x7fffffffll) return fail(DR_EINVAL, "dr_fbp_init: too many projection rows");
    kern<<<(unsigned)grid, (groups * tb + 31) / 32 * 32, smem, st>>>((const S *)g, (T *)P->d_fbp_q,
                                                                     (const T *)P->d_fbp_taps, rows, P->ns, tb, groups,
                                                                     tiles);
    DR_CUDA_TRY(cudaGetLastError());
    return DR_OK;
}

// One row per CTA (grid-stride), one output per thread: shared memory holds the taps
// h(n), n = -(ns - 1) .. ns - 1, and the row.
constexpr int kFbpRowThreads = 256;
template <typename S, typename T>
__global__ void __launch_bounds__(kFbpRowThreads)
    shepp_logan_row_kernel(const S *__restrict__ g, T *__restrict__ q, const T *__restrict__ taps, long long rows,
                           int ns) {
    extern __shared__ __align__(32) unsigned char fbp_smem[];
    T *h = reinterpret_cast<T *>(fbp_smem);  // [2 ns - 1], h[i] = h(i - (ns - 1))
    T *row = h + (2 * ns - 1);                // [ns]
    for (int i = threadIdx.x; i < 2 * ns - 1; i += kFbpRowThreads) h[i] = taps[i];
    for (long long r = blockIdx.x; r < rows; r += gridDim.x) {
        __syncthreads();  // previous row consumed
        for (int i = threadIdx.x; i < ns; i += kFbpRowThreads) row[i] = ldc<T>(g + r * ns + i);
        __syncthreads();
        for (int b = threadIdx.x; b < ns; b += kFbpRowThreads) {
            const T *hb = h + b + (ns - 1);  // hb[-b'] = h(b - b')
            T acc = T(0);
#pragma unroll 8
            for (int bp = 0; bp < ns; ++bp) acc = fma(hb[-bp], row[bp], acc);
            q[r * ns + b] = acc;
        }
    }
}

template <typename S, typename T>
static dr_status launch_filter_row(dr_plan *P, const void *g, cudaStream_t st) {
    const long long rows = (long long)P->nz * P->K;
    const size_t smem = sizeof(T) * (size_t)(3 * P->ns - 1);
    auto kern = shepp_logan_row_kernel<S, T>;
    const dr_status s = allow_dynamic_smem((const void *)kern, smem);
    if (s != DR_OK) return s;
    int per_sm = 0;
    DR_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kFbpRowThreads, smem));
    const long long grid = std::min<long long>(rows, (long long)P->num_sms * std::max(per_sm, 1));
    kern<<<(unsigned)grid, kFbpRowThreads, smem, st>>>((const S *)g, (T *)P->d_fbp_q, (const T *)P->d_fbp_taps, rows,
                                                       P->ns);
    DR_CUDA_TRY(cudaGetLastError());
    return DR_OK;
}

// Eight rows per thread, unless that leaves SMs without a warp; then two.  One output
// per thread in FP64, whose pipe (59 clocks per warp instruction) is the bound, so
// that no register tile pays and its idle lanes and uneven CTAs cost (300 rows of
// 257: 1.08 against 1.35 ms), and for a row per SM or fewer, where the longer chain
// of four outputs would be all there is (30 rows of 128: 30 against 34 us).
template <typename S, typename T>
static dr_status launch_filter(dr_plan *P, const void *g, cudaStream_t st) {
    const long long rows = (long long)P->nz * P->K;
    if constexpr (sizeof(T) == 8) {
        return launch_filter_row<S, T>(P, g, st);
    } else {
        if (rows <= P->num_sms && P->ns <= 512) return launch_filter_row<S, T>(P, g, st);
        return rows * ((P->ns + 3) / 4) / 8 >= 32ll * P->num_sms ? launch_filter_t<S, T, 8>(P, g, st)
                                                                  : launch_filter_t<S, T, 2>(P, g, st);
    }
}

template <typename T>
static dr_status upload_as(void *dst, const std::vector<double> &src) {
    std::vector<T> tmp(src.begin(), src.end());
    DR_CUDA_TRY(cudaMemcpy(dst, tmp.data(), sizeof(T) * tmp.size(), cudaMemcpyHostToDevice));
    return DR_OK;
}

// Eigen-decomposition of a symmetric n x n matrix by cyclic Jacobi rotations
// (Jacobi's method; Golub and Van Loan, Matrix Computations, Sec. 8.5):
// A = V diag(lam) V^T, V[i][e] = component i of eigenvector e.
static void sym_eig(std::vector<double> A, int n, std::vector<double> &V, std::vector<double> &lam) {
    V.assign((size_t)n * n, 0.0);
    for (int i = 0; i < n; ++i) V[(size_t)i * n + i] = 1.0;
    for (int sweep = 0; sweep < 64; ++sweep) {
        double off = 0.0, diag = 0.0;
        for (int p = 0; p < n; ++p) {
            diag += A[(size_t)p * n + p] * A[(size_t)p * n + p];
            for (int q = p + 1; q < n; ++q) off += A[(size_t)p * n + q] * A[(size_t)p * n + q];
        }
        if (off <= 1e-32 * diag) break;
        for (int p = 0; p < n; ++p)
            for (int q = p + 1; q < n; ++q) {
                const double apq = A[(size_t)p * n + q];
                if (apq == 0.0) continue;
                const double th = (A[(size_t)q * n + q] - A[(size_t)p * n + p]) / (2.0 * apq);
                const double t = (th >= 0.0 ? 1.0 : -1.0) / (std::fabs(th) + std::sqrt(th * th + 1.0));
                const double c = 1.0 / std::sqrt(t * t + 1.0), s = t * c;
                for (int k = 0; k < n; ++k) {  // columns p, q
                    const double akp = A[(size_t)k * n + p], akq = A[(size_t)k * n + q];
                    A[(size_t)k * n + p] = c * akp - s * akq;
                    A[(size_t)k * n + q] = s * akp + c * akq;
                }
                for (int k = 0; k < n; ++k) {  // rows p, q
                    const double apk = A[(size_t)p * n + k], aqk = A[(size_t)q * n + k];
                    A[(size_t)p * n + k] = c * apk - s * aqk;
                    A[(size_t)q * n + k] = s * apk + c * aqk;
                }
                for (int k = 0; k < n; ++k) {
                    const double vkp = V[(size_t)k * n + p], vkq = V[(size_t)k * n + q];
                    V[(size_t)k * n + p] = c * vkp - s * vkq;
                    V[(size_t)k * n + q] = s * vkp + c * vkq;
                }
            }
    }
    lam.assign(n, 0.0);
    for (int i = 0; i < n; ++i) lam[i] = A[(size_t)i * n + i];
}

// Psi[k][j] (row stride MP, zero padded) for nw windows.
static dr_status fbp_table(const dr_plan *P, int nw, std::vector<double> &psi) {
    const int K = P->K, m = P->m;
    std::vector<int> win(K);
    std::vector<long long> cnt(nw, 0);
    for (int k = 0; k < K; ++k) {
        const double x = std::floor(P->t[k] * nw);
        const int w = x < 0.0 ? 0 : (x > nw - 1 ? nw - 1 : (int)x);
        win[k] = w;
        ++cnt[w];
    }
    // Gram matrix Phi^T Phi = V diag(lam) V^T (cyclic Jacobi rotations)
    std::vector<double> G((size_t)m * m, 0.0), V, lam;
    for (int k = 0; k < K; ++k)
        for (int i = 0; i < m; ++i)
            for (int j = 0; j < m; ++j) G[(size_t)i * m + j] += P->Phi[(size_t)k * m + i] * P->Phi[(size_t)k * m + j];
    sym_eig(G, m, V, lam);
    double lmax = 0.0;
    for (double l : lam) lmax = std::max(lmax, l);
    if (!(lmax > 0.0)) return fail(DR_EINVAL, "dr_fbp_init: the basis vanishes at every acquisition time");
    // A[:, w] = G^+ (sum_{k in w} Phi[k][:]): the minimum-norm least-squares
    // fit; eigenvalues below 1e-12 lam_max (singular values of Phi below
    // 1e-6 of the largest) count as zero
    std::vector<double> A((size_t)m * nw, 0.0), y(m);
    for (int w = 0; w < nw; ++w) {
        std::vector<double> rhs(m, 0.0);
        for (int k = 0; k < K; ++k)
            if (win[k] == w)
                for (int j = 0; j < m; ++j) rhs[j] += P->Phi[(size_t)k * m + j];
        for (int e = 0; e < m; ++e) {  // y = diag(1/lam) V^T rhs
            double v = 0.0;
            for (int j = 0; j < m; ++j) v += V[(size_t)j * m + e] * rhs[j];
            y[e] = lam[e] > 1e-12 * lmax ? v / lam[e] : 0.0;
        }
        for (int i = 0; i < m; ++i) {
            double v = 0.0;
            for (int e = 0; e < m; ++e) v += V[(size_t)i * m + e] * y[e];
            A[(size_t)i * nw + w] = v;
        }
    }
    psi.assign((size_t)K * P->MP, 0.0);
    for (int k = 0; k < K; ++k) {
        const int w = win[k];
        const double sc = M_PI / (double)cnt[w];
        for (int j = 0; j < m; ++j) psi[(size_t)k * P->MP + j] = sc * A[(size_t)j * nw + w];
    }
    return DR_OK;
}

static dr_status ensure(void **p, size_t bytes, size_t &acc) {
    if (*p) return DR_OK;
    cudaError_t e = cudaMalloc(p, std::max<size_t>(bytes, 16));
    if (e != cudaSuccess) {
        *p = nullptr;
        return cuda_fail(e, "dr_fbp_init: scratch allocation");
    }
    acc += bytes;
    return DR_OK;
}

}  // namespace dr

using namespace dr;

extern "C" dr_status dr_fbp_init(dr_plan *P, const void *g, void *u, int n_windows) {
    clear_error();
    if (!P || !g || !u) return fail(DR_EINVAL, "dr_fbp_init: NULL argument");
    if (n_windows < 1 || n_windows > P->K) return fail(DR_EINVAL, "dr_fbp_init: n_windows must be in [1, K]");
    const size_t cs = calc_size(P->prec);
    const size_t ng = (size_t)P->nz * P->K * P->ns, nu = (size_t)P->nx * P->ny * P->nz * P->m;
    std::vector<double> psi;
    dr_status s = fbp_table(P, n_windows, psi);
    if (s != DR_OK) return s;

    // scratch (kept by the plan): taps, Psi, filtered data, FP32 result for BF16 plans
    const bool fresh_taps = P->d_fbp_taps == nullptr;
    if ((s = ensure(&P->d_fbp_taps, cs * (2 * (size_t)P->ns - 1), P->fbp_bytes)) != DR_OK) return s;
    if ((s = ensure(&P->d_fbp_phi, cs * (size_t)P->K * P->MP, P->fbp_bytes)) != DR_OK) return s;
    if ((s = ensure(&P->d_fbp_q, cs * ng, P->fbp_bytes)) != DR_OK) return s;
    if (P->prec == DR_BF16_F32ACC && (s = ensure(&P->d_fbp_u, sizeof(float) * nu, P->fbp_bytes)) != DR_OK) return s;

    // the tables may still be read by a previous call's kernels on this stream
    DR_CUDA_TRY(cudaStreamSynchronize(P->stream));
    if (fresh_taps) {
        std::vector<double> taps(2 * (size_t)P->ns - 1);
        for (int i = 0; i < 2 * P->ns - 1; ++i) {
            const double n = (double)(i - (P->ns - 1));
            taps[i] = -2.0 / (M_PI * M_PI * (4.0 * n * n - 1.0));
        }
        s = P->prec == DR_F64 ? upload_as<double>(P->d_fbp_taps, taps) : upload_as<float>(P->d_fbp_taps, taps);
        if (s != DR_OK) return s;
    }
    s = P->prec == DR_F64 ? upload_as<double>(P->d_fbp_phi, psi) : upload_as<float>(P->d_fbp_phi, psi);
    if (s != DR_OK) return s;

    cudaStream_t st = P->stream;
    switch (P->prec) {
        case DR_F32: s = launch_filter<float, float>(P, g, st); break;
        case DR_BF16_F32ACC: s = launch_filter<bf16, float>(P, g, st); break;
        case DR_F64: s = launch_filter<double, double>(P, g, st); break;
    }
    if (s != DR_OK) return s;

    // back-project with Psi in place of Phi (kernels take the table pointer at launch)
    void *phi = P->d_PhiP;
    P->d_PhiP = P->d_fbp_phi;
    if (P->prec == DR_BF16_F32ACC) s = launch_adj(P, P->d_fbp_q, P->d_fbp_u, 1.0, 0.0, true, st, true);
    else s = launch_adj(P, P->d_fbp_q, u, 1.0, 0.0, false, st);
    P->d_PhiP = phi;
    if (s != DR_OK) return s;
    if (P->prec == DR_BF16_F32ACC) {
        const int grid = P->num_sms * 8;
        fbp_to_bf16_kernel<<<grid, 256, 0, st>>>((const float *)P->d_fbp_u, (bf16 *)u, nu);
        DR_CUDA_TRY(cudaGetLastError());
    }
    return DR_OK;
}
