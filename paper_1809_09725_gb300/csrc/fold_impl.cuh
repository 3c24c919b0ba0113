// fold_impl.cuh -- half-turn folded projector pair (Sec. 4).
//
// With theta = n pi + theta0, theta0 in [0, pi), the static transform obeys
// R f(n pi + theta0, s) = R f(theta0, (-1)^n s) (exact for the Joseph
// discretisation on the symmetric bin grid).  Projections that share theta0
// (one per half-turn in a continuous scan) therefore need the static
// transform of each coefficient volume only once:
//
//   forward  g[k](s) = sum_j phi_j(t_k) (R u_j)(theta0_k, (-1)^{n_k} s)
//   adjoint  u_j = sum_{theta0} R*( gt_j(theta0) ),
//            gt_j(theta0, s) = sum_{k: theta0_k = theta0} phi_j(t_k) g[k]((-1)^{n_k} s)
//
// The forward marches the Joseph rays of each unique angle through a strip
// of the m-vector image staged in shared memory (all m coefficient sums per
// ray in registers) and distributes every ray to all projections of its
// angle in the epilogue.  The adjoint first folds the data per unique angle
// (fold_data_kernel, HBM bound), then back-projects the m folded sinograms
// with the voxel-driven exact transpose: per unique angle a TMA tile load of
// the footprint window (Wb bins x MS coefficients), mbarrier pipeline.
// Work per application drops from K (m + c) to U (2m + c') per voxel, U the
// number of unique angles.
#pragma once
#include <type_traits>

#include "chan.cuh"

namespace dr {

constexpr int kFoldThreads = 256;
constexpr int kFoldAdjStages = 2;
constexpr int kFoldAdjWin = 26 * 1024;  // bytes of windows per stage, at most, by default (four CTAs per SM)
constexpr int kFoldAdjSmem = 227 * 1024;  // bytes of all stages where the caller chose the angles per stage

// Padded coefficient stride in shared memory and in the folded data:
// multiples of 4 floats (16-byte vectors, TMA rows) whose pattern of
// 16-byte slots repeats only every 8 pixels (no bank conflicts between
// neighbouring pixels).
__host__ __device__ constexpr int fold_ms(int M) { return M <= 4 ? 4 : ((M % 8 == 0) ? M + 4 : M); }
__host__ __device__ constexpr int fold_rpt(int M) { return M <= 4 ? 8 : 32 / M; }

// Static-transform CTAs of the two-kernel forward (configurations in
// dr_internal.cuh): 1024 to 4096 rays per CTA.  The more rays a CTA carries,
// the more samples share each staged line.
// Strip element stride of a static group: 4 or 12 floats (bf16: 4 or 8).
__host__ __device__ constexpr int fold_static_ps(int MC, bool bf16) {
    return bf16 ? (MC == 4 ? 4 : 8) : (MC == 4 ? 4 : 12);
}

// Element stride of one pixel's coefficient vector in the forward strip.
// Float strips use fold_ms.  BF16 plans stage the stored bf16 values as they
// are (exact; the march widens them to float in registers), which halves the
// shared-memory bytes per ray step: 8-byte vectors for M <= 4, otherwise an
// odd number of 16-byte slots per pixel (no bank conflicts between
// neighbouring pixels).
__host__ __device__ constexpr int fold_bf16_ps(int M) {
    return M <= 4 ? 4 : 8 * (((M + 7) / 8) % 2 == 1 ? (M + 7) / 8 : (M + 7) / 8 + 1);
}
template <typename S, typename T, int M>
__host__ __device__ constexpr int fold_strip_ps() {
    return sizeof(S) == 2 ? fold_bf16_ps(M) : fold_ms(M);
}

// M bf16 coefficients of one strip pixel (PS-element slots), widened to float.
template <int M, int PS>
__device__ __forceinline__ void load_vec_bf16(const bf16 *p, float (&v)[M]) {
    if constexpr (PS == 4) {
        const uint2 a = *reinterpret_cast<const uint2 *>(p);
        const unsigned w[2] = {a.x, a.y};
#pragma unroll
        for (int j = 0; j < M; ++j) v[j] = __uint_as_float((j & 1) ? (w[j >> 1] & 0xffff0000u) : (w[j >> 1] << 16));
    } else {
#pragma unroll
        for (int c = 0; c < (M + 7) / 8; ++c) {
            const uint4 a = reinterpret_cast<const uint4 *>(p)[c];
            const unsigned w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int h = 0; h < 8; ++h) {
                const int j = 8 * c + h;
                if (j < M) v[j] = __uint_as_float((h & 1) ? (w[h >> 1] & 0xffff0000u) : (w[h >> 1] << 16));
            }
        }
    }
}

template <typename T, int M>
__device__ __forceinline__ void load_vec(const T *p, T (&v)[M]) {
    if constexpr (sizeof(T) == 4 && (M % 4) == 0) {
#pragma unroll
        for (int j = 0; j < M / 4; ++j) {
            const float4 a = reinterpret_cast<const float4 *>(p)[j];
            v[4 * j] = a.x;
            v[4 * j + 1] = a.y;
            v[4 * j + 2] = a.z;
            v[4 * j + 3] = a.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < M; ++j) v[j] = p[j];
    }
}

// Copy the coefficients j0 .. j0+count-1 of one pixel (src points at j0) into
// the forward strip: bf16 strips keep the stored values, float strips hold
// the compute type; slots >= count are zero.  vec: src is 16-byte aligned
// and count == M, so whole 16-byte vectors may be moved (async_stage: with
// cp.async).
template <typename S, typename T, int M, typename ST>
__device__ __forceinline__ void stage_pixel(ST *dst, const S *__restrict__ src, int count, bool vec,
                                            int async_stage) {
    if constexpr (sizeof(S) == 2 && sizeof(ST) == 2) {
        if constexpr ((M % 8) == 0) {
            if (vec) {
                if (async_stage) {
#pragma unroll
                    for (int j = 0; j < M / 8; ++j) cp_async_16(dst + 8 * j, src + 8 * j);
                } else {
#pragma unroll
                    for (int j = 0; j < M / 8; ++j)
                        reinterpret_cast<uint4 *>(dst)[j] = __ldg(reinterpret_cast<const uint4 *>(src) + j);
                }
                return;
            }
        }
#pragma unroll
        for (int j = 0; j < M; ++j) dst[j] = j < count ? src[j] : S(0.0f);
    } else {
        T v[M];
        if constexpr (sizeof(S) == 4 && (M % 4) == 0) {
            if (vec) {
                if (async_stage) {
#pragma unroll
                    for (int j = 0; j < M / 4; ++j) cp_async_16(dst + 4 * j, src + 4 * j);
                    return;
                }
#pragma unroll
                for (int j = 0; j < M / 4; ++j) {
                    const float4 a = __ldg(reinterpret_cast<const float4 *>(src) + j);
                    v[4 * j] = a.x;
                    v[4 * j + 1] = a.y;
                    v[4 * j + 2] = a.z;
                    v[4 * j + 3] = a.w;
                }
            } else {
#pragma unroll
                for (int j = 0; j < M; ++j) v[j] = j < count ? ldc<T>(src + j) : T(0);
            }
        } else {
#pragma unroll
            for (int j = 0; j < M; ++j) v[j] = j < count ? ldc<T>(src + j) : T(0);
        }
        if constexpr (sizeof(T) == 4 && (M % 4) == 0) {
#pragma unroll
            for (int j = 0; j < M / 4; ++j)
                reinterpret_cast<float4 *>(dst)[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < M; ++j) dst[j] = v[j];
        }
    }
}

// ===========================================================================
// Forward
// ===========================================================================
// Resident CTAs per SM the folded forward asks the compiler for: the march is
// latency bound, and at M = 8 three CTAs (<= 85 registers) beat two.
__host__ __device__ constexpr int fold_fwd_min_blocks(int M) { return M == 8 ? 3 : 1; }

// STATIC = false: M covers all coefficients and the epilogue distributes each
// ray to the projections of its angle.  STATIC = true: the CTA handles the
// coefficient group j0 = (blockIdx.y % ngroups) * M .. j0 + M - 1 and writes
// the scaled static transforms (R u_j)(theta0_a, s_b) to
// ru[((z U + a) ns + b) ms_ru + j]; fold_dist_kernel distributes them.  With
// nsplit > 1 the march is split into nsplit chunks of image lines
// (blockIdx.z); chunk c writes its partial sums at ru + c * split_stride.
template <typename S, typename T, int M, bool STATIC, int THREADS = kFoldThreads, int RPTS = 0, int MINB = 1,
          bool TMA = false>
__global__ void __launch_bounds__(THREADS, THREADS == kFoldThreads ? fold_fwd_min_blocks(M) : MINB)
    fold_fwd_kernel(const S *__restrict__ u, S *__restrict__ out, const S *__restrict__ gm,
                    const FwdProj *__restrict__ uproj, const int *__restrict__ start, const int *__restrict__ member,
                    const T *__restrict__ phip, const int *__restrict__ blocks, int nx, int ny, int ns, int K,
                    int m, int MP, int P, int R, int nchunk, int mode, T sigma, int async_stage, int ngroups,
                    T *__restrict__ ru, int U, int ms_ru, int nsplit, size_t split_stride,
                    const __grid_constant__ CUtensorMap tm_rows, const __grid_constant__ CUtensorMap tm_cols,
                    int *status) {
    // strip element: stored bf16 for bf16 storage, else the compute type
    constexpr bool BF16_STRIP = sizeof(S) == 2;
    using ST = std::conditional_t<BF16_STRIP, S, T>;
    // TMA (static transforms of float coefficient groups of 4 or 8, staging
    // mode 3): strips staged by TMA into two buffers on mbarriers, in the TMA
    // line layout, each 4-coefficient plane of a group a line layout of its
    // own (16-byte entries: the even/odd halves stay conflict free); a
    // separate instantiation, so the other kernels carry none of its code
    constexpr bool TMA_CAP = TMA && STATIC && !BF16_STRIP && (M == 4 || M == 8);
    constexpr int NP = TMA_CAP ? M / 4 : 1;  // 16-byte planes per pixel (TMA strips)
    constexpr int MS = TMA_CAP ? 4 : (STATIC ? fold_static_ps(M, BF16_STRIP) : fold_strip_ps<S, T, M>());
    constexpr int RPT = STATIC ? RPTS : fold_rpt(M);
    constexpr int VW = 16 / (int)sizeof(S);  // elements per 16-byte vector
    extern __shared__ __align__(16) unsigned char fold_smem[];
    T *scale_s = reinterpret_cast<T *>(fold_smem);                       // [64]

    const int tid = threadIdx.x;
    const int z = blockIdx.y / ngroups;
    const int j0 = (blockIdx.y - z * ngroups) * M;
    const int count = min(M, m - j0);
    const bool vec = count == M && (m % VW) == 0 && (j0 % VW) == 0;
    const int blk_id = blockIdx.x / nchunk, chunk = blockIdx.x - blk_id * nchunk;
    const int *blk = blocks + (size_t)blk_id * P;
    const int branch = uproj[blk[0]].branch;
    const int W = branch ? ny : nx;
    const int H = branch ? nx : ny;
    constexpr bool tma = TMA_CAP;
    // line stride, zero entries before the even half, offset of the odd half
    // (TMA strips: a line is NP planes of fold_tma_line(W) entries each)
    const int ls = tma ? NP * fold_tma_line(W) : fold_line_elems(W);
    const int kg = tma ? 8 : kFoldGuardE;
    const int ooff = tma ? fold_tma_half(W) + 8 : fold_odd_off(W);
    ST *strip = reinterpret_cast<ST *>(
        tma ? fold_smem + 768 + ((128u - ((smem_u32(fold_smem) + 768u) & 127u)) & 127u) : fold_smem + 768);
    // image lines of this CTA's march: all, or chunk blockIdx.z of nsplit
    const int L0 = STATIC ? (int)(((long long)blockIdx.z * H) / nsplit) : 0;
    const int L1 = STATIC ? (int)(((long long)(blockIdx.z + 1) * H) / nsplit) : H;

    for (int p = tid; p < P; p += THREADS) {
        const int a = blk[p];
        const FwdProj f = uproj[a >= 0 ? a : blk[0]];
        scale_s[p] = (T)f.scale;
    }
    // strip buffers: 1 (synchronous staging), 2 (async_stage 1) or 3 (async_stage 2, 3)
    const int nbuf = tma ? kFoldTmaStages : async_stage + 1;
    if (tma) {
        // zero the guard entries only: TMA writes every data entry of a strip
        // (zero beyond the image), so no entry is written by both proxies
        const int wh = fold_tma_half(W), lp = fold_tma_line(W);  // plane line: 24 guard entries
        for (int i = tid; i < nbuf * R * NP * 24; i += THREADS) {
            const int pl = i / 24, g = i - pl * 24;  // pl: (buffer, line, plane)
            const int e = g < 8 ? g : (g < 16 ? kg + wh + (g - 8) : kg + ooff + wh + (g - 16));
            reinterpret_cast<float4 *>(strip)[(size_t)pl * lp + e] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    } else {
        for (int i = tid; i < nbuf * R * ls * MS; i += THREADS) strip[i] = ST(0.0f);
    }

    // Ray slots: thread t marches RPT rays of one distinct angle p_t of the
    // block, the bins l_t + tpa q (q = 0 .. RPT-1), so the rays of a thread
    // share their per-line step and consecutive threads take consecutive
    // bins; a single angle whose bins exceed one CTA (nchunk > 1) is cut into
    // chunks of THREADS * RPT bins, bins chunk * THREADS * RPT + t + THREADS q.
    const int tpa = nchunk > 1 ? THREADS : (ns + RPT - 1) / RPT;
    const int pt = nchunk > 1 ? 0 : tid / tpa;
    const int bt0 = nchunk > 1 ? chunk * THREADS * RPT + tid : tid - pt * tpa;
    const int at = pt < P ? blk[pt] : -1;
    long long xq[RPT];  // 32.32 position of each ray on its next line
    long long bfx = 0;  // per-line step of this thread's angle
    int lo[RPT], hi[RPT];
    unsigned rng[RPT];
    T acc[RPT][M];
    FwdProj f{};
    if (at >= 0) {
        f = uproj[at];
        bfx = f.B_fx;
    }
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        lo[q] = 1;
        hi[q] = 0;
        xq[q] = 0;
#pragma unroll
        for (int j = 0; j < M; ++j) acc[q][j] = T(0);
        const int b = bt0 + tpa * q;
        if (at >= 0 && b < ns) {
            xq[q] = f.C_fx + (long long)b * f.A_fx + (long long)L0 * bfx;
            const float xf = f.Cf + (float)b * f.Af;
            const float Bf = f.Bf;
            if (fabsf(Bf) < 1e-2f) {
                lo[q] = 0;
                hi[q] = H - 1;
            } else {
                const float r1 = (-1.0f - xf) / Bf, r2 = ((float)W - xf) / Bf;
                float rmin = fminf(r1, r2), rmax = fmaxf(r1, r2);
                rmin = fmaxf(rmin, -4.0f);
                rmax = fminf(rmax, (float)H + 4.0f);
                lo[q] = max(0, (int)floorf(rmin) - 1);
                hi[q] = min(H - 1, (int)ceilf(rmax) + 1);
            }
            lo[q] = max(lo[q], L0);
            hi[q] = min(hi[q], L1 - 1);
        }
        // the TMA kernel keeps each ray's line range in one register (lines < 2^16)
        rng[q] = (unsigned)lo[q] | ((unsigned)hi[q] << 16);
    }
    __syncthreads();

    const size_t zoff = (size_t)z * ny * nx;
    // Stage lines [r0, r0+nl) of the m-vector image into buffer `buf`:
    // asynchronously (cp.async, 16-byte chunks) when the coefficients are
    // 16-byte float vectors, else through registers.
    auto stage = [&](ST *buf, int r0, int nl) {
        const int npx = nl * W;
        for (int qq = tid; qq < npx; qq += THREADS) {
            int rl, i;
            size_t pix;
            if (branch == 0) {
                rl = qq / W;
                i = qq - rl * W;
                pix = zoff + (size_t)(r0 + rl) * nx + i;
            } else {
                i = qq / nl;
                rl = qq - i * nl;
                pix = zoff + (size_t)i * nx + (r0 + rl);
            }
            stage_pixel<S, T, M>(buf + ((size_t)rl * ls + (i & 1) * ooff + kg + (i >> 1)) * MS,
                                 u + pix * m + j0, count, vec, async_stage);
        }
    };
    const size_t buf_elems = (size_t)R * ls * MS;  // buffer b starts at strip + b * buf_elems
    if (!TMA_CAP && async_stage == 1 && L0 < L1) {
        stage(strip, L0, min(R, L1 - L0));
        cp_async_commit();
    }
    if (!TMA_CAP && async_stage == 2) {
        // three buffers: strips s+1 and s+2 are copied while strip s is marched,
        // and one barrier per strip suffices (the buffer refilled after the
        // barrier of strip s held strip s-1, which every thread has finished);
        // one commit group per strip, empty ones included, so that waiting for
        // all but the newest group always means strip s has landed
        if (L0 < L1) stage(strip, L0, min(R, L1 - L0));
        cp_async_commit();
        if (L0 + R < L1) stage(strip + buf_elems, L0 + R, min(R, L1 - L0 - R));
        cp_async_commit();
    }
    // ---- march the rays of lines [r0, r0 + nl) staged at cur: all m coefficient
    // sums per ray, line by line, the thread's RPT rays side by side
    // (independent chains); each ray still adds its lines in increasing order
    const int pstride = tma ? fold_tma_line(W) : 0;  // entries between the planes of a TMA line
    auto march = [&](const ST *cur, int r0, int nl) {
#pragma unroll 1
        for (int rl = 0; rl < nl; ++rl) {
            const int r = r0 + rl;
            const ST *row = cur + ((size_t)rl * ls + kg) * MS;
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                const int lq = TMA_CAP ? (int)(rng[q] & 0xffffu) : lo[q], hq = TMA_CAP ? (int)(rng[q] >> 16) : hi[q];
                if (r >= lq && r <= hq) {
                    const long long x = xq[q];
                    int i0 = (int)(x >> 32);
                    i0 = min(max(i0, -2), W);
                    const float w = __uint_as_float(0x3F800000u | ((unsigned)x >> 9)) - 1.0f;
                    const float w1m = 1.0f - w;
                    // pixels i0 and i0 + 1: the even one from the even half, the
                    // odd one from the odd half, each with its interpolation weight
                    const bool odd = i0 & 1;
                    const float we = odd ? w : w1m, wo = odd ? w1m : w;
                    const ST *pe = row + ((i0 + 1) >> 1) * MS, *po = row + (ooff + (i0 >> 1)) * MS;
                    T t0[M], t1[M];
                    if constexpr (BF16_STRIP) {
                        load_vec_bf16<M, MS>(pe, t0);
                        load_vec_bf16<M, MS>(po, t1);
                    } else if constexpr (NP > 1) {
                        // 4 coefficients per plane; plane p of the line pstride entries on
#pragma unroll
                        for (int pl = 0; pl < NP; ++pl) {
                            const float4 a = *reinterpret_cast<const float4 *>(pe + (size_t)pl * pstride * MS);
                            const float4 c = *reinterpret_cast<const float4 *>(po + (size_t)pl * pstride * MS);
                            t0[4 * pl] = a.x; t0[4 * pl + 1] = a.y; t0[4 * pl + 2] = a.z; t0[4 * pl + 3] = a.w;
                            t1[4 * pl] = c.x; t1[4 * pl + 1] = c.y; t1[4 * pl + 2] = c.z; t1[4 * pl + 3] = c.w;
                        }
                    } else {
                        load_vec<T, M>(pe, t0);
                        load_vec<T, M>(po, t1);
                    }
#pragma unroll
                    for (int j = 0; j < M; ++j) acc[q][j] = fmaf(wo, t1[j], fmaf(we, t0[j], acc[q][j]));
                }
                xq[q] += bfx;
            }
        }
    };
    if constexpr (TMA_CAP) {
        // Two strip buffers; full[b] completes when a strip's TMA copies have
        // landed (expect_tx).  One CTA barrier per strip: thread 0 waits for
        // strip s, the barrier then also says every thread has finished strip
        // s - 1, whose buffer the copies of strip s + 1 refill while strip s is
        // marched.  The copies of a strip are spread over the CTA's threads.
        // Waits are bounded: on a give-up the status word
        // is set and the CTA leaves in order.
        __shared__ __align__(8) uint64_t full[kFoldTmaStages];
        const int nstrips = L1 > L0 ? (L1 - L0 + R - 1) / R : 0;
        const size_t buf_elems = (size_t)R * ls * MS;
        if (tid == 0) {
            for (int b = 0; b < kFoldTmaStages; ++b) mbar_init(&full[b], 1);
            fence_mbar_init();
        }
        __syncthreads();
        // strip sidx into buffer sidx % 2: copy c of its 2 * nbox * nl by thread c (mod THREADS)
        auto issue = [&](int sidx) {
            const int b = sidx % kFoldTmaStages, r0s = L0 + sidx * R, nls = min(R, L1 - r0s);
            const int bw = fold_tma_bw(W), nbox = fold_tma_nbox(W), per_line = NP * 2 * nbox;
            if (tid == 0) mbar_arrive_expect_tx(&full[b], (unsigned)(nls * per_line * (bw / 2) * 16));
            for (int c = tid; c < nls * per_line; c += THREADS) {
                // copy c: line rl, plane pl (coefficients j0 + 4 pl ..), half, box bx
                const int rl = c / per_line, rem = c - rl * per_line, pl = rem / (2 * nbox),
                          rem2 = rem - pl * 2 * nbox, half = rem2 / nbox, bx = rem2 - half * nbox;
                const uint32_t dst = smem_u32(strip + b * buf_elems) +
                                     (uint32_t)(rl * ls + pl * pstride + kg + half * ooff + bx * (bw / 2)) * 16u;
                const int line = r0s + rl, p0 = bx * bw + half;
                if (branch == 0) tma_load_4d(dst, &tm_rows, j0 + 4 * pl, p0, line, z, &full[b]);
                else tma_load_4d(dst, &tm_cols, j0 + 4 * pl, line, p0, z, &full[b]);
            }
        };
        if (nstrips > 0) issue(0);
        for (int sidx = 0; sidx < nstrips; ++sidx) {
            const int b = sidx % kFoldTmaStages;
            int ok = 1;
            if (tid == 0) ok = mbar_wait_bounded_any(&full[b], (unsigned)((sidx / kFoldTmaStages) & 1), status,
                                                     2000000000ull);
            if (__syncthreads_or(!ok)) {
                // strip sidx did not land in time; let no copy of it outlive the CTA
                if (tid == 0)
                    mbar_wait_bounded(&full[b], (unsigned)((sidx / kFoldTmaStages) & 1), status, 100000000ull);
                return;
            }
            if (sidx + 1 < nstrips) issue(sidx + 1);
            const int r0 = L0 + sidx * R;
            march(strip + b * buf_elems, r0, min(R, L1 - r0));
        }
    }
    if constexpr (!TMA_CAP) {
        int s_idx = 0;
        for (int r0 = L0; r0 < L1; r0 += R, ++s_idx) {
            const int nl = min(R, L1 - r0);
            ST *cur;
            if (async_stage == 2) {
                cp_async_wait<1>();
                __syncthreads();
                if (r0 + 2 * R < L1) stage(strip + ((s_idx + 2) % 3) * buf_elems, r0 + 2 * R, min(R, L1 - r0 - 2 * R));
                cp_async_commit();
                cur = strip + (s_idx % 3) * buf_elems;
            } else if (async_stage) {
                // prefetch the next strip into the other buffer, then wait for this one
                if (r0 + R < L1) {
                    stage(strip + ((s_idx + 1) & 1) * buf_elems, r0 + R, min(R, L1 - r0 - R));
                    cp_async_commit();
                    cp_async_wait<1>();
                } else {
                    cp_async_wait<0>();
                }
                __syncthreads();
                cur = strip + (s_idx & 1) * buf_elems;
            } else {
                stage(strip, r0, nl);
                __syncthreads();
                cur = strip;
            }
            march(cur, r0, nl);
            if (async_stage != 2) __syncthreads();
        }
        if (async_stage == 2) cp_async_wait<0>();  // no copy outlives the CTA
    }

    if constexpr (STATIC) {
        // ---- epilogue: the scaled static transforms of this coefficient group ----
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int b = bt0 + tpa * q;
            const int a = at;
            if (a < 0 || b >= ns) continue;
            const T sc = scale_s[pt];
            T *dst = ru + blockIdx.z * split_stride + (((size_t)z * U + a) * ns + b) * ms_ru + j0;
#pragma unroll
            for (int j = 0; j < M; ++j)
                if (j < count) dst[j] = sc * acc[q][j];
        }
        return;
    }
    // ---- epilogue: distribute each ray to every projection of its angle ----
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int b = bt0 + tpa * q;
        const int a = at;
        if (a < 0 || b >= ns) continue;
        const T sc = scale_s[pt];
        const int e = start[a + 1];
        for (int idx = start[a]; idx < e; ++idx) {
            const int mem = member[idx];
            const int k = mem >> 1;
            const int bb = (mem & 1) ? (ns - 1 - b) : b;
            const T *ph = phip + (size_t)k * MP;
            T val = T(0);
#pragma unroll
            for (int j = 0; j < M; ++j) val = fmaf(__ldg(ph + j), acc[q][j], val);
            val *= sc;
            const size_t o = ((size_t)z * K + k) * ns + bb;
            if (mode == 0) {
                stc<T>(out + o, val);
            } else if (mode == 1) {
                stc<T>(out + o, val - ldc<T>(gm + o));
            } else {
                const T h = ldc<T>(out + o);
                stc<T>(out + o, (h + sigma * val - sigma * ldc<T>(gm + o)) / (T(1) + sigma));
            }
        }
    }
}

// ===========================================================================
// Forward, two-kernel form, step 2: distribute the static transforms
//   g[z][k][b] = sum_j phi_j(t_k) ru[z][a(k)][flip_k(b)][j]
// with the forward epilogue modes (store, minus gm, CP dual update).  Line
// chunks of a split march are added first, in chunk order.  A thread takes
// one row (z, a, b) of the static transforms, reads it once, and writes the
// bins of every projection k of angle a (at b, or ns-1-b for odd half-turns):
// consecutive threads write consecutive bins of the same projection.
// ===========================================================================
// (BLK: rows of several slices side by side, whose addresses take divisions; without
// them a row is the i-th.  The divisions cost 1 us of the 37 of 6 x 128^2, m = 8, bf16.)
template <typename S, typename T, int M, bool BLK>
__global__ void __launch_bounds__(kRedThreads)
    fold_dist_kernel(const T *__restrict__ ru, S *__restrict__ out, const S *__restrict__ gm,
                     const int *__restrict__ start, const int *__restrict__ member, const T *__restrict__ phip,
                     int nz, int K, int ns, int U, RowMap rows, int m, int MP, int mode, T sigma, int nsplit,
                     size_t split_stride) {
    // rows and table rows are multiples of 4 floats from 16-byte aligned bases
    constexpr bool V4 = sizeof(T) == 4;
    const size_t n = (size_t)nz * U * ns;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int b = (int)(i % ns);
        const size_t za = i / ns;
        const int a = (int)(za % U), z = (int)(za / U);
        const T *r = ru + (BLK ? row_at(rows, z, (size_t)a * ns + b) : i * rows.C);
        T rv[M];
        if constexpr (V4 && M % 4 == 0) {
#pragma unroll
            for (int q = 0; q < M / 4; ++q) {
                if (4 * q < m) {
                    float4 v = *reinterpret_cast<const float4 *>(r + 4 * q);
                    for (int c = 1; c < nsplit; ++c) {
                        const float4 w = *reinterpret_cast<const float4 *>(r + c * split_stride + 4 * q);
                        v.x += w.x;
                        v.y += w.y;
                        v.z += w.z;
                        v.w += w.w;
                    }
                    rv[4 * q] = v.x;
                    rv[4 * q + 1] = v.y;
                    rv[4 * q + 2] = v.z;
                    rv[4 * q + 3] = v.w;
                } else {
                    rv[4 * q] = rv[4 * q + 1] = rv[4 * q + 2] = rv[4 * q + 3] = T(0);
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < M; ++j) {
                T rj = T(0);
                if (j < m) {
                    rj = r[j];
                    for (int c = 1; c < nsplit; ++c) rj += r[c * split_stride + j];
                }
                rv[j] = rj;
            }
        }
        const int e = __ldg(start + a + 1);
        for (int idx = __ldg(start + a); idx < e; ++idx) {
            const int mem = __ldg(member + idx);
            const int k = mem >> 1;
            const int bb = (mem & 1) ? ns - 1 - b : b;
            const T *ph = phip + (size_t)k * MP;
            T val = T(0);
            if constexpr (V4 && M % 4 == 0) {
#pragma unroll
                for (int q = 0; q < M / 4; ++q) {
                    if (4 * q >= m) break;
                    const float4 f = __ldg(reinterpret_cast<const float4 *>(ph) + q);
                    const float fv[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        if (4 * q + t < m) val = fma(fv[t], rv[4 * q + t], val);
                }
            } else {
#pragma unroll
                for (int j = 0; j < M; ++j)
                    if (j < m) val = fma(__ldg(ph + j), rv[j], val);
            }
            const size_t o = ((size_t)z * K + k) * ns + bb;
            if (mode == 0) {
                stc<T>(out + o, val);
            } else if (mode == 1) {
                stc<T>(out + o, val - ldc<T>(gm + o));
            } else {
                const T h = ldc<T>(out + o);
                stc<T>(out + o, (h + sigma * val - sigma * ldc<T>(gm + o)) / (T(1) + sigma));
            }
        }
    }
}

// ===========================================================================
// Adjoint, step 1: fold the data per unique angle
//   gt[z][a][b][j] = sum_{k in group(a)} phi_j(t_k) g[z][k][flip_k(b)]
// ===========================================================================
// wild[slot] = 1 if a folded row holds an infinity or a NaN: the back-projection
// that follows then takes each voxel's bins by themselves (0 x infinity would
// spread).  The launches of a plan take two slots in turn, and each clears the one
// of the next.  (A recorded launch keeps its slot: a note left in it by an earlier
// replay costs time, not bits.)
template <typename T, int N>
__device__ __forceinline__ void note_wild(const T (&v)[N], int *wild, int slot) {
    T f = T(0);
#pragma unroll
    for (int j = 0; j < N; ++j) f = fma(v[j], T(0), f);
    if (f != T(0)) *(volatile int *)(wild + slot) = 1;
}
__device__ __forceinline__ void clear_next_wild(int *wild, int slot) {
    if (blockIdx.x == 0 && threadIdx.x == 0) wild[1 - slot] = 0;
}

template <typename S, typename T, int M>
__global__ void __launch_bounds__(kRedThreads)
    fold_data_kernel(const S *__restrict__ g, T *__restrict__ gt, const int *__restrict__ start,
                     const int *__restrict__ member, const T *__restrict__ phip, int nz, int U, int ns, int K, int MP,
                     int *wild, int slot) {
    constexpr int MS = fold_ms(M);
    clear_next_wild(wild, slot);
    const size_t n = (size_t)nz * U * ns;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int b = (int)(i % ns);
        const size_t r = i / ns;
        const int a = (int)(r % U);
        const int z = (int)(r / U);
        T acc[M];
#pragma unroll
        for (int j = 0; j < M; ++j) acc[j] = T(0);
        const int e = __ldg(start + a + 1);
        // members in groups of 4: their data loads are issued together (the
        // accumulation keeps the member order)
        constexpr int G = 4;
        for (int idx0 = __ldg(start + a); idx0 < e; idx0 += G) {
            int kq[G];
            T gv[G];
#pragma unroll
            for (int q = 0; q < G; ++q) {
                const int idx = idx0 + q;
                const int mem = idx < e ? __ldg(member + idx) : 0;
                kq[q] = mem >> 1;
                const int bb = (mem & 1) ? (ns - 1 - b) : b;
                gv[q] = idx < e ? ldc<T>(g + ((size_t)z * K + kq[q]) * ns + bb) : T(0);
            }
#pragma unroll
            for (int q = 0; q < G; ++q) {
                if (idx0 + q >= e) break;
                const T *ph = phip + (size_t)kq[q] * MP;
                if constexpr (sizeof(T) == 4 && M % 4 == 0) {
#pragma unroll
                    for (int c = 0; c < M / 4; ++c) {
                        const float4 f = __ldg(reinterpret_cast<const float4 *>(ph) + c);
                        acc[4 * c] = fmaf(f.x, gv[q], acc[4 * c]);
                        acc[4 * c + 1] = fmaf(f.y, gv[q], acc[4 * c + 1]);
                        acc[4 * c + 2] = fmaf(f.z, gv[q], acc[4 * c + 2]);
                        acc[4 * c + 3] = fmaf(f.w, gv[q], acc[4 * c + 3]);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < M; ++j) acc[j] = fmaf(__ldg(ph + j), gv[q], acc[j]);
                }
            }
        }
        note_wild(acc, wild, slot);
        T *dst = gt + i * MS;
        if constexpr ((MS % 4) == 0 && sizeof(T) == 4) {
            float v[MS];
#pragma unroll
            for (int j = 0; j < MS; ++j) v[j] = j < M ? acc[j] : 0.0f;
#pragma unroll
            for (int j = 0; j < MS / 4; ++j)
                reinterpret_cast<float4 *>(dst)[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < MS; ++j) dst[j] = j < M ? acc[j] : T(0);
        }
    }
}

// ===========================================================================
// Adjoint, step 2: voxel-driven exact transpose of the folded sinograms
// ===========================================================================
// A thread holds a patch of 2 x 2 voxels for MC coefficients (all M up to 16 and
// half of them above, or half of that on small grids; other threads hold the rest)
// of ZS slices (the weights, about as many instructions as 8 coefficients' sums,
// serve all of them).  The
// patch projects |cos| + |sin| <= sqrt 2 bins wide, so its eight taps lie in
// four consecutive bins b .. b + 3 counted from the voxel that projects lowest:
// that voxel takes bins 0 and 1, the two beside it two of bins 0 to 2, the one
// across two of bins 1 to 3.  Four bin reads serve four voxels (pairs of voxels
// took three for two), and the 11 weights, each with its exact zero where a
// voxel has three candidates, multiply two coefficients per instruction
// (fma.rn.f32x2, each half rounded by itself).  An added term 0 x value leaves
// a sum of finite data as it is, so each voxel's sum is the two-tap sum, bin by
// bin and angle by angle (ADMM amplifies any other rounding).  Angles whose sine
// or cosine exceeds 0.99999, where the rounding of two positions could put
// neighbouring taps two bins apart, read each voxel's two bins by themselves (a
// CTA-uniform test per angle), and so do all angles when the kernel that wrote
// the folded data found an infinity or a NaN in it (*wild).
// A quarter warp's lanes are 4 x 2 patches: their lowest bins span at most
// 6 |cos| + 2 |sin| < 8 bins, and rows of an odd number of 16-byte slots then
// never collide (lanes on the same bin share one broadcast).
//
// Positions are floats relative to the middle of a subtile of SX x 16 voxels
// (|position| <= 18 bins: the weights are exact to about 1e-6); a tile is one
// or two of them.
//
// Measured (data fold included): 16 x 256^2, K = 1800, m = 8: 0.351 -> 0.293 ms;
// 8 x 1024^2, K = 6000, m = 16: 7.83 -> 6.64 ms.  Shared memory, 90 % busy with
// pairs, is at 61 % (m = 8) and 69 % (m = 16); what bounds it now is issue (59 and
// 62 % of the slots) together with the skew of a CTA's warps at the stage barrier (a
// quarter of the stalls; three stages on mbarriers without it measured 0.300 and
// 6.62 ms).
struct alignas(16) FoldPrm {
    float c, s, c16, e0;  // cos, sin, 16 cos, 1/cm - 1/(2 cm^2)  (cm = max(|c|, |s|))
    float inv_c2;           // 1/cm^2
    float pad_[3];
    struct {
        float qb;  // fraction of a subtile's middle, less 1/2
        int idx;   // its bin in the window, less the float magic
    } sub[2];
};

//
// NG threads share a patch's coefficients (a warp or more apart): one or two, or
// twice as many where that many CTAs would leave the chip to a few long ones.
template <int M>
constexpr int kFoldAdjNG = M <= 16 ? 1 : 2;
template <int M, int NG_>
struct FoldAdjShape {
    static constexpr int NG = NG_;
    static constexpr int MC = M / NG;
    static constexpr int TX = 32 / NG;  // tile: TX x 16 voxels per CTA of 128 threads
    static constexpr int SX = M <= 8 ? 32 : (M <= 16 ? 16 : 8);  // subtile
    // a row's position from the row above it (else from the subtile's middle)
    static constexpr bool STEP = M <= 16;
    // bins of a window: the tile's extent at any angle (35, 22 or 17), the patch's
    // fourth bin and a margin for the rounding of the first
    static constexpr int WB = NG == 1 ? 41 : (NG == 2 ? 28 : 24);
    // A window is one run of WB bins x MS floats of a sinogram row, copied in
    // boxes of at most 256 floats and whole 128-byte lines, one box row each (a
    // box of WB rows of MS floats fetched 2.7 times the bytes from L2).
    static constexpr int NBOX = (WB * fold_ms(M) + 255) / 256;
    static constexpr int BOX = ((WB * fold_ms(M) + NBOX - 1) / NBOX + 31) / 32 * 32;
    static constexpr int WIN = NBOX * BOX;  // floats
};

// Resident CTAs asked for: 4 ZS MC sums, 11 weight pairs and 4 bins per thread.
// (With five for m = 5 to 8 smaller grids are 4 to 6 % faster, but 761 to 912 CTAs
// take a second round: 7 x 256^2, m = 8, U = 120 0.126 ms, with six 0.119; the same
// holds of two threads a patch at m = 16: 2 x 327^2, U = 258 0.256 and 0.229 ms.)
__host__ __device__ constexpr int fold_adj_min_blocks(int M, int NG, int ZS) {
    const int sums = ZS * M / NG;
    return sums <= 4 ? 7 : (sums <= 8 ? (M <= 8 || M == 16 ? 6 : 5) : 4);
}

template <typename S, typename T, int M, int NG_, int ZS>
__global__ void __launch_bounds__(kAdjThreads, fold_adj_min_blocks(M, NG_, ZS))
    fold_adj_kernel(const __grid_constant__ CUtensorMap tm_gt, const FoldAng *__restrict__ ang,
                    S *__restrict__ u_s, T *__restrict__ u_c, int nx, int ny, int nz, int U, int U1, int m, T alpha,
                    T beta, int *status, const int *wild, int PP, int vec) {
    using Sh = FoldAdjShape<M, NG_>;
    constexpr int TX = Sh::TX, TY = kAdjTY, SX = Sh::SX, NG = Sh::NG, MC = Sh::MC;
    constexpr int NST = kFoldAdjStages;
    constexpr int MS = fold_ms(M);
    constexpr float kMag = 12582912.0f;  // 1.5 * 2^23: adding it rounds to an integer
    constexpr int kMagI = 0x4B400000;
    constexpr bool PK = MC % 2 == 0;        // coefficient pairs
    constexpr int NC = PK ? MC / 2 : MC;    // sums per voxel
    constexpr int CH = MC % 4 == 0 ? 2 : (PK ? 1 : MC);  // sums per chunk of bin reads (16, 8 or 4 bytes)
    using A = std::conditional_t<PK, unsigned long long, float>;

    extern __shared__ __align__(128) unsigned char fadj_smem_raw[];
    // round up to 128 B by pointer arithmetic on the __shared__ array, so the
    // compiler keeps addressing it as shared memory (LDS, not generic loads)
    unsigned char *smem_raw = fadj_smem_raw + ((128u - (smem_u32(fadj_smem_raw) & 127u)) & 127u);
    constexpr int WIN = Sh::WIN;  // floats of one slice's window of one angle
    const int win_bytes = PP * ZS * WIN * (int)sizeof(T);
    const int stage_bytes = win_bytes + 128 * ((PP * (int)sizeof(FoldPrm) + 127) / 128);
    __shared__ __align__(8) uint64_t full[NST];
    auto win_s = [&](int st, int p) { return reinterpret_cast<T *>(smem_raw + st * stage_bytes) + p * ZS * WIN; };
    auto prm_s = [&](int st) { return reinterpret_cast<FoldPrm *>(smem_raw + st * stage_bytes + win_bytes); };

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ntx = (nx + TX - 1) / TX;
    const int x0 = (blockIdx.x % ntx) * TX, y0 = (blockIdx.x / ntx) * TY;
    const int z0 = blockIdx.y * ZS;
    // patch of this thread: a warp covers 8 x 4 patches (tiles of 8 columns: 4 x 8),
    // a quarter of it 4 x 2
    const int vw = warp % (4 / NG), cg = warp / (4 / NG);
    const int px = NG == 4 ? (lane & 3) : (lane & 3) + 4 * ((lane >> 3) & 1) + (NG == 1 ? 8 * (vw & 1) : 0);
    const int py = NG == 4 ? lane >> 2 : ((lane >> 2) & 1) + 2 * (lane >> 4) + 4 * (NG == 1 ? vw >> 1 : vw);
    const int dx = 2 * px, dy = 2 * py;
    // blocks of PP angles: those with cos >= 0 (the first U1), then the others
    const int nk1 = (U1 + PP - 1) / PP, nkb = nk1 + (U - U1 + PP - 1) / PP;
    auto first = [&](int kb) { return kb < nk1 ? kb * PP : U1 + (kb - nk1) * PP; };
    auto past = [&](int kb) { return kb < nk1 ? U1 : U; };

    // One lane per angle: window and constants, TMA copies.
    auto issue = [&](int st, int kb) {
        int wb0 = 0, aa = 0;
        if (lane < PP) {
            aa = min(first(kb) + lane, past(kb) - 1);
            const FoldAng pj = ang[aa];
            FoldPrm pr;
            pr.c = pj.cf;
            pr.s = pj.sf;
            pr.c16 = pj.c16;
            pr.e0 = pj.e0;
            pr.inv_c2 = pj.inv_c2;
            const int yo = y0 + TY / 2;
#pragma unroll
            for (int k = 0; k < TX / SX; ++k) {
                const int xo = x0 + k * SX + SX / 2;
                // (written out, so that every tile shape rounds a subtile's middle alike)
                const double posO = fma((double)xo, pj.c, yo * pj.s) + pj.C0, fl = floor(posO);
                if (k == 0)  // the tile's lowest position, less a bin for rounding
                    wb0 = (int)fl - 1 + (int)floorf(fminf((-SX / 2) * pj.cf, (TX - 1 - SX / 2) * pj.cf) +
                                                    fminf((-TY / 2) * pj.sf, (TY / 2 - 1) * pj.sf));
                pr.sub[k].qb = (float)(posO - fl) - 0.5f;
                pr.sub[k].idx = (int)fl - wb0 - kMagI;
            }
            prm_s(st)[lane] = pr;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive_expect_tx(&full[st], (unsigned)win_bytes);
        __syncwarp();
        if (lane < PP) {
#pragma unroll
            for (int k = 0; k < ZS; ++k)  // (slices beyond the volume: the last one again, not stored)
                for (int i = 0; i < Sh::NBOX; ++i)
                    tma_load_2d(win_s(st, lane) + k * WIN + i * Sh::BOX, &tm_gt, wb0 * MS + i * Sh::BOX,
                                min(z0 + k, nz - 1) * U + aa, &full[st]);
        }
        if (lane != 0) mbar_arrive(&full[st]);
    };

    const bool solo = __ldg(wild) != 0;
    if (tid == 0) {
        for (int s = 0; s < NST; ++s) mbar_init(&full[s], 32);
        fence_mbar_init();
    }
    __syncthreads();
    if (warp == 0)
        for (int s = 0; s < NST && s < nkb; ++s) issue(s, s);

    // sums of voxel (x + i, y + j) at [j][i]; for the angles with c < 0 the
    // columns are swapped, so that column 0 is always the lower one on the detector
    A acc[ZS][2][2][NC];
#pragma unroll
    for (int k = 0; k < ZS; ++k)
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int q = 0; q < NC; ++q) acc[k][v >> 1][v & 1][q] = 0;
    // x of the lower (dA) and the upper column from the subtile's middle, and the
    // half of a 32-wide subtile that they lie in
    const int sub = dx / SX, sx = dx - sub * SX;
    float dA = (float)((sx & 15) - SX / 2), dB = dA + 1.0f;
    const bool far = sx >= 16;
    const float dyf = (float)(dy - TY / 2);
    auto flip = [&]() {
        const float t = dA;
        dA = dB;
        dB = t;
#pragma unroll
        for (int j = 0; j < 2 * ZS; ++j)
#pragma unroll
            for (int q = 0; q < NC; ++q) {
                const A t = acc[j >> 1][j & 1][0][q];
                acc[j >> 1][j & 1][0][q] = acc[j >> 1][j & 1][1][q];
                acc[j >> 1][j & 1][1][q] = t;
            }
    };
    auto dup = [](float w) -> A {
        if constexpr (PK) return pack_f2(w, w);
        else return w;
    };
    auto mad = [](A w, A b, A r) {
        if constexpr (PK) return fma_f2(w, b, r);
        else return fmaf(w, b, r);
    };

    for (int kb = 0; kb < nkb; ++kb) {
        const int st = kb % NST;
        const bool bad = !mbar_wait_bounded(&full[st], (unsigned)((kb / NST) & 1), status, 2000000000ull);
        const FoldPrm *prm = prm_s(st);
        const int np = bad ? 0 : min(PP, past(kb) - first(kb));
        if (kb == nk1) flip();
        for (int p = 0; p < np; ++p) {
            const float4 h = *reinterpret_cast<const float4 *>(prm + p);  // c, s, c16, e0
            const float ac = h.x, as = h.y, ic2 = prm[p].inv_c2, qb = prm[p].sub[sub].qb;
            const int idx = prm[p].sub[sub].idx;
            // positions of the patch's voxels: lower and upper column, two rows
            float qA = fmaf(dyf, as, fmaf(dA, ac, qb)), qB = fmaf(dyf, as, fmaf(dB, ac, qb));
            float qC, qD;
            if constexpr (Sh::STEP) {
                if (SX == 32) {
                    const float e = far ? h.z : 0.0f;
                    qA += e;
                    qB += e;
                }
                qC = qA + as;
                qD = qB + as;
            } else {
                qC = fmaf(dyf + 1.0f, as, fmaf(dA, ac, qb));
                qD = fmaf(dyf + 1.0f, as, fmaf(dB, ac, qb));
            }
            // a voxel's lower bin and the weights of its two bins
            auto taps = [&](float q, float &w0, float &w1) {
                const float t = q + kMag, d = q - (t - kMag);
                w0 = fmaxf(0.0f, fmaf(-d, ic2, h.w));
                w1 = fmaxf(0.0f, fmaf(d, ic2, h.w));
                return __float_as_int(t) + idx;
            };
            if (solo || fabsf(ac) > 0.99999f || fabsf(as) > 0.99999f) {
                // close to an axis, or bins that are not finite: each voxel's two bins by themselves
                const float qv[4] = {qA, qB, qC, qD};
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    float w0, w1;
                    const T *r0 = win_s(st, p) + taps(qv[v], w0, w1) * MS + cg * MC;
                    const A p0 = dup(w0), p1 = dup(w1);
#pragma unroll
                    for (int k = 0; k < ZS; ++k)
#pragma unroll
                        for (int q = 0; q < NC; ++q) {
                            const A *r = reinterpret_cast<const A *>(r0 + k * WIN) + q;
                            A &t = acc[k][v >> 1][v & 1][q];
                            t = mad(p1, *reinterpret_cast<const A *>(r0 + k * WIN + MS + q * (PK ? 2 : 1)), mad(p0, *r, t));
                        }
                }
                continue;
            }
            float w0, w1;
            const int b0 = taps(qA, w0, w1);
            const T *w = win_s(st, p) + b0 * MS + cg * MC;
            const A p00 = dup(w0), p01 = dup(w1);
            A p1[3], p2[3], p3[3];
            // weights on three candidate bins, the first of them lim - 1 bins on
            auto three = [&](float q, int lim, A (&o)[3]) {
                const bool on = taps(q, w0, w1) - b0 >= lim;
                o[0] = dup(on ? 0.0f : w0);
                o[1] = dup(on ? w0 : w1);
                o[2] = dup(on ? w1 : 0.0f);
            };
            three(qB, 1, p1);
            three(qC, 1, p2);
            three(qD, 2, p3);
#pragma unroll
            for (int k = 0; k < ZS; ++k) {
                const T *ws = w + k * WIN;
#pragma unroll
                for (int q0 = 0; q0 < NC; q0 += CH) {
                    A bin[4][CH];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const T *r = ws + i * MS + q0 * (PK ? 2 : 1);
                        if constexpr (PK && CH == 2) {
                            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(r);
                            bin[i][0] = v.x;
                            bin[i][1] = v.y;
                        } else if constexpr (PK) {
                            bin[i][0] = *reinterpret_cast<const unsigned long long *>(r);
                        } else {
#pragma unroll
                            for (int q = 0; q < CH; ++q) bin[i][q] = r[q];
                        }
                    }
#pragma unroll
                    for (int q = 0; q < CH; ++q) {
                        A &r0 = acc[k][0][0][q0 + q], &r1 = acc[k][0][1][q0 + q], &r2 = acc[k][1][0][q0 + q],
                          &r3 = acc[k][1][1][q0 + q];
                        r0 = mad(p01, bin[1][q], mad(p00, bin[0][q], r0));
                        r1 = mad(p1[2], bin[2][q], mad(p1[1], bin[1][q], mad(p1[0], bin[0][q], r1)));
                        r2 = mad(p2[2], bin[2][q], mad(p2[1], bin[1][q], mad(p2[0], bin[0][q], r2)));
                        r3 = mad(p3[2], bin[3][q], mad(p3[1], bin[2][q], mad(p3[0], bin[1][q], r3)));
                    }
                }
            }
        }
        if (__syncthreads_or(bad)) {
            if (tid == 0)
                for (int s = kb; s < nkb && s < kb + NST; ++s)
                    mbar_wait_bounded(&full[s % NST], (unsigned)((s / NST) & 1), status, 100000000ull);
            return;
        }
        // (the warps refill in turn: the others are already at the next stage)
        if (warp == (kb & 3) && kb + NST < nkb) issue(st, kb + NST);
    }
    if (nk1 < nkb) flip();

#pragma unroll
    for (int v = 0; v < 4 * ZS; ++v) {
        const int x = x0 + dx + (v & 1), y = y0 + dy + ((v >> 1) & 1), z = z0 + (v >> 2);
        if (x >= nx || y >= ny || z >= nz) continue;
        const size_t base = (((size_t)z * ny + y) * nx + x) * m + cg * MC;
        float r[MC];
        if constexpr (PK) {
#pragma unroll
            for (int q = 0; q < NC; ++q) unpack_f2(acc[v >> 2][(v >> 1) & 1][v & 1][q], r[2 * q], r[2 * q + 1]);
        } else {
#pragma unroll
            for (int q = 0; q < NC; ++q) r[q] = acc[v >> 2][(v >> 1) & 1][v & 1][q];
        }
#pragma unroll
        for (int j = 0; j < MC; ++j) r[j] *= alpha;
        if constexpr (sizeof(S) == 4 && MC % 4 == 0) {
            if (vec) {  // rows of whole 16-byte vectors
                float4 *d = reinterpret_cast<float4 *>((u_c ? u_c : (T *)u_s) + base);
#pragma unroll
                for (int q = 0; q < MC / 4; ++q) {
                    float4 o = make_float4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
                    if (beta != T(0)) {
                        const float4 b = d[q];
                        o.x += beta * b.x;
                        o.y += beta * b.y;
                        o.z += beta * b.z;
                        o.w += beta * b.w;
                    }
                    d[q] = o;
                }
                continue;
            }
        }
#pragma unroll
        for (int j = 0; j < MC; ++j)
            if (cg * MC + j < m) {
                if (u_c) {
                    if (beta != T(0)) r[j] += beta * u_c[base + j];
                    u_c[base + j] = r[j];
                } else {
                    if (beta != T(0)) r[j] += beta * ldc<T>(u_s + base + j);
                    stc<T>(u_s + base + j, r[j]);
                }
            }
    }
}

// ===========================================================================
// Host launchers
// ===========================================================================
template <typename S, typename T, int M>
dr_status fold_fwd_launch_t(dr_plan *P, const void *u, void *out, const void *gm, int mode, double sigma,
                            cudaStream_t st) {
    using ST = std::conditional_t<sizeof(S) == 2, S, T>;
    constexpr int MS = fold_strip_ps<S, T, M>();
    const int ls = fold_line_elems_max(P->nx, P->ny);
    // strip height and staging mode: the autotuned choice (cp.async double
    // buffering needs whole 16-byte coefficient vectors)
    const int async_ok = (P->m == M && ((sizeof(S) == 4 && (M % 4) == 0) || (sizeof(S) == 2 && (M % 8) == 0))) ? 1 : 0;
    const bool bf16_strip = sizeof(S) == 2;
    const int async_stage = async_ok && (bf16_strip ? P->fold_async_st : P->fold_async);
    const int R = std::max(1, bf16_strip ? P->fold_lines_st : P->fold_lines);
    const size_t smem = 768 + sizeof(ST) * (size_t)(async_stage + 1) * R * ls * MS;
    auto kern = fold_fwd_kernel<S, T, M, false>;
    {
        dr_status s = allow_dynamic_smem((const void *)kern, smem);
        if (s != DR_OK) return s;
    }
    dim3 grid(P->n_fold_blocks * P->fold_nchunk, P->nz);
    kern<<<grid, kFoldThreads, smem, st>>>((const S *)u, (S *)out, (const S *)gm, P->d_fold_fwd, P->d_fold_start,
                                           P->d_fold_member, (const T *)P->d_PhiP, P->d_fold_blocks, P->nx, P->ny,
                                           P->ns, P->K, P->m, P->MP, P->fold_P, R, P->fold_nchunk, mode,
                                           (T)sigma, async_stage, 1, (T *)nullptr, 0, 0, 1, (size_t)0, CUtensorMap{},
                                           CUtensorMap{}, P->d_status);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DR_OK : cuda_fail(e, "fold_fwd_kernel launch");
}

// Static transforms of the two-kernel forward (step 1) in coefficient groups
// of MC (4 or 8): into the folded-data scratch (one march) or the split
// scratch (line chunks); `rs` says where.
template <typename S, typename T, int M, int GI>
dr_status fold_static_launch(dr_plan *P, const void *u, cudaStream_t st, StaticOut &rs) {
    constexpr int MC = fold_static_mc(GI), THREADS = fold_static_threads(GI), RPT = fold_static_rpt_gi(GI),
                  MINB = fold_static_min_blocks(GI);
    constexpr bool BF16_STRIP = sizeof(S) == 2;
    using ST = std::conditional_t<BF16_STRIP, S, T>;
    constexpr int MS = fold_static_ps(MC, BF16_STRIP);
    constexpr int VW = 16 / (int)sizeof(S);
    const int gi = GI;
    const int ngroups = (P->m + MC - 1) / MC;
    const int ls = fold_line_elems_max(P->nx, P->ny);
    const bool bf16_kernel = sizeof(S) == 2;
    const int async_req = bf16_kernel ? P->fold2_async_st : P->fold2_async;
    const int R0 = std::max(1, std::min(bf16_kernel ? P->fold2_lines_st : P->fold2_lines,
                                        async_req == 3 && !bf16_kernel && P->fold2_Rt[gi] > 0 ? P->fold2_Rt[gi]
                                                                                              : P->fold2_R[gi]));
    if ((size_t)P->nz * ngroups > 65535) return fail(DR_EINVAL, "two-kernel folded forward: too many slice groups");
    // async 1: two strip buffers, the next strip copied with cp.async while the
    // current one is marched (groups of whole 16-byte vectors; other pixels
    // are staged through registers); async 2: three buffers, two strips ahead
    (void)VW;
    int async = bf16_kernel ? P->fold2_async_st : P->fold2_async;
    int R = R0;
    // async 3: TMA-staged strips (4-float groups of a float plan whose rows
    // of coefficients are whole 16-byte vectors); otherwise three cp.async buffers
    CUtensorMap tm_rows{}, tm_cols{};
    constexpr int NPT = MC / 4;  // 16-byte planes per pixel of a TMA strip
    if (async == 3) {
        bool ok = !BF16_STRIP && (P->m % 4) == 0 && ((uintptr_t)u % 16) == 0;
        if (ok) {
            const uint64_t dims[4] = {(uint64_t)P->m, (uint64_t)P->nx, (uint64_t)P->ny, (uint64_t)P->nz};
            const uint64_t strides[3] = {(uint64_t)P->m * 4, (uint64_t)P->nx * P->m * 4,
                                         (uint64_t)P->ny * P->nx * P->m * 4};
            const uint32_t box_r[4] = {4, (uint32_t)fold_tma_bw(P->nx), 1, 1}, es_r[4] = {1, 2, 1, 1};
            const uint32_t box_c[4] = {4, 1, (uint32_t)fold_tma_bw(P->ny), 1}, es_c[4] = {1, 1, 2, 1};
            ok = encode_tensor_map(&tm_rows, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void *>(u), dims,
                                   strides, box_r, es_r) &&
                 encode_tensor_map(&tm_cols, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void *>(u), dims,
                                   strides, box_c, es_c);
        }
        if (ok) {
            const long long line = 16LL * NPT * std::max(fold_tma_line(P->nx), fold_tma_line(P->ny));
            R = std::max(1, std::min(R, (int)((2LL * kFoldStripBudget) / (kFoldTmaStages * line))));
        } else {
            async = 2;
        }
    }
    if (async == 2) {
        // three buffers within twice the strip budget (below the 227 KB a CTA
        // may hold); where even one line does not fit, two buffers (same march)
        const long long line = (long long)sizeof(ST) * ls * MS;
        const int r3 = (int)((2LL * kFoldStripBudget) / (3 * line));
        if (r3 >= 1) R = std::min(R, r3);
        else async = 1;
    }
    const size_t smem = async == 3 ? 768 + 128 + 16 * (size_t)kFoldTmaStages * R * NPT *
                                               std::max(fold_tma_line(P->nx), fold_tma_line(P->ny))
                                   : 768 + sizeof(ST) * (size_t)(async + 1) * R * ls * MS;
    auto kern = fold_fwd_kernel<S, T, MC, true, THREADS, RPT, MINB>;
    if constexpr (!BF16_STRIP) {
        if (async == 3) kern = fold_fwd_kernel<S, T, MC, true, THREADS, RPT, MINB, true>;
    }
    {
        dr_status s = allow_dynamic_smem((const void *)kern, smem);
        if (s != DR_OK) return s;
    }
    // one march: static transforms into the folded-data scratch (row stride
    // fold_ms(M)); a march split into line chunks: partial sums into the
    // split scratch (row stride m rounded up to 4), one chunk after another
    const int nsplit = P->split_off ? 1 : std::max(1, P->fold2_split);
    T *ru;
    int ms_ru;
    size_t split_stride = 0;
    if (nsplit == 1) {
        dr_status s = ensure_fold_scratch(P);
        if (s != DR_OK) return s;
        ru = (T *)P->d_gt;
        ms_ru = fold_ms(M);
    } else {
        ms_ru = (P->m + 3) / 4 * 4;
        split_stride = (size_t)P->nz * P->fold_U * P->ns * ms_ru;
        dr_status s = ensure_split_scratch(P, sizeof(T) * split_stride * nsplit);
        if (s != DR_OK) return s;
        ru = (T *)P->d_ru_split;
    }
    const int bv = P->d_fold2_blocks[gi][P->fold2_bv] ? P->fold2_bv : 0;
    dim3 grid(P->fold2_nblocks[gi][bv] * P->fold2_nchunk[gi], P->nz * ngroups, nsplit);
    kern<<<grid, THREADS, smem, st>>>((const S *)u, (S *)nullptr, (const S *)nullptr, P->d_fold_fwd, P->d_fold_start,
                                           P->d_fold_member, (const T *)P->d_PhiP, P->d_fold2_blocks[gi][bv],
                                           P->nx, P->ny, P->ns, P->K, P->m, P->MP, P->fold2_P[gi][bv], R,
                                           P->fold2_nchunk[gi],
                                           0, (T)0, async, ngroups, ru, P->fold_U, ms_ru, nsplit,
                                           split_stride, tm_rows, tm_cols, P->d_status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "fold_fwd_kernel (static) launch");
    rs = StaticOut{ru, slice_rows((size_t)P->fold_U * P->ns, ms_ru), nsplit, split_stride};
    return DR_OK;
}

template <typename S, typename T, int M>
dr_status fold_static_dispatch(dr_plan *P, const void *u, cudaStream_t st, StaticOut &rs) {
    if (!P->fold2_ok) return fail(DR_EINVAL, "two-kernel folded forward unavailable for this plan");
    if constexpr (M >= 4) {
        switch (sizeof(S) == 2 ? P->fold2_gi_st : P->fold2_gi) {
            case 0: return fold_static_launch<S, T, M, 0>(P, u, st, rs);
            case 2: return fold_static_launch<S, T, M, 2>(P, u, st, rs);
            case 4: return fold_static_launch<S, T, M, 4>(P, u, st, rs);
            case 6: return fold_static_launch<S, T, M, 6>(P, u, st, rs);
            case 1:
                if constexpr (M >= 8) return fold_static_launch<S, T, M, 1>(P, u, st, rs);
                break;
            case 3:
                if constexpr (M >= 8) return fold_static_launch<S, T, M, 3>(P, u, st, rs);
                break;
            case 5:
                if constexpr (M >= 8) return fold_static_launch<S, T, M, 5>(P, u, st, rs);
                break;
            case 7:
                if constexpr (M >= 8) return fold_static_launch<S, T, M, 7>(P, u, st, rs);
                break;
        }
    }
    return fail(DR_EINVAL, "two-kernel folded forward: unsupported coefficient group");
}

// The forward in two steps: static transforms (chan: of the channel kernel,
// 2 in the order of the thread-per-ray ones), then the distribution.
template <typename S, typename T, int M>
dr_status fold_fwd2_launch_t(dr_plan *P, const void *u, void *out, const void *gm, int mode, double sigma,
                             cudaStream_t st, int chan) {
    StaticOut rs{};
    {
        dr_status s = chan ? chan_static(P, u, sizeof(S) == 2, chan == 2, chan == 2 ? fold2_chunks(P) : P->chan.nsplit,
                                         st, rs)
                           : fold_static_dispatch<S, T, M>(P, u, st, rs);
        if (s != DR_OK) return s;
    }
    auto dist = rs.rows.spb > 1 ? fold_dist_kernel<S, T, M, true> : fold_dist_kernel<S, T, M, false>;
    dist<<<red_grid((size_t)P->nz * P->fold_U * P->ns), kRedThreads, 0, st>>>(
        (const T *)rs.ru, (S *)out, (const S *)gm, P->d_fold_start, P->d_fold_member, (const T *)P->d_PhiP, P->nz,
        P->K, P->ns, P->fold_U, rs.rows, P->m, P->MP, mode, (T)sigma, rs.nsplit, rs.split_stride);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DR_OK : cuda_fail(e, "fold_dist_kernel launch");
}

// gt: where the folded data live (nz U ns MS floats); nullptr: the plan's
// scratch buffer.
template <typename S, typename T, int M>
dr_status fold_backproject(dr_plan *P, void *u, double alpha, double beta, bool u_calc, cudaStream_t st,
                           void *gt = nullptr);

template <typename S, typename T, int M>
dr_status fold_adj_launch_t(dr_plan *P, const void *g, void *u, double alpha, double beta, bool u_calc,
                            cudaStream_t st, void *gt = nullptr) {
    constexpr int MS = fold_ms(M);
    if (!gt) gt = P->d_gt;
    // step 1: fold the data into the scratch buffer
    fold_data_kernel<S, T, M><<<red_grid((size_t)P->nz * P->fold_U * P->ns), kRedThreads, 0, st>>>(
        (const S *)g, (T *)gt, P->d_fold_start, P->d_fold_member, (const T *)P->d_PhiP, P->nz, P->fold_U, P->ns,
        P->K, P->MP, P->d_status + 1, P->wild_slot ^= 1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "fold_data_kernel launch");
    return fold_backproject<S, T, M>(P, u, alpha, beta, u_calc, st, gt);
}

// Back-project the folded sinograms (step 2 of the folded adjoint):
// u = alpha R*(folded) + beta u.
template <typename S, typename T, int M, int NG, int ZS>
dr_status fold_backproject_t(dr_plan *P, void *u, double alpha, double beta, bool u_calc, cudaStream_t st, void *gt) {
    using Sh = FoldAdjShape<M, NG>;
    constexpr int MS = fold_ms(M);
    CUtensorMap tm{};
    if (!encode_tensor_map_2d(&tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, gt, (uint64_t)P->ns * MS, (uint64_t)P->nz * P->fold_U,
                              (uint64_t)P->ns * MS * sizeof(T), (uint32_t)Sh::BOX, 1))
        return fail(DR_ECUDA, "fold adj: tensor map encode failed");
    // angles per pipeline stage: fewer shrink the windows' shared memory so that
    // more CTAs fit on an SM (the angles are summed in the same order)
    constexpr int row_bytes = Sh::WIN * (int)sizeof(T);
    const auto bytes = [&](int pp) {
        return kFoldAdjStages * ((size_t)pp * ZS * row_bytes + 128 * ((pp * sizeof(FoldPrm) + 127) / 128)) + 128;
    };
    int pp = std::max(1, std::min(32, P->fold_adj_pp));
    if (P->fold_adj_pp_set) {
        while (pp > 1 && bytes(pp) > kFoldAdjSmem) --pp;
    } else {
        pp = std::max(1, std::min(pp, kFoldAdjWin / (ZS * row_bytes)));
    }
    P->fold_adj_pp_used = pp;
    const size_t smem = bytes(pp);
    auto kern = fold_adj_kernel<S, T, M, NG, ZS>;
    {
        dr_status s = allow_dynamic_smem((const void *)kern, smem);
        if (s != DR_OK) return s;
    }
    const int ntx = (P->nx + Sh::TX - 1) / Sh::TX, nty = (P->ny + kAdjTY - 1) / kAdjTY;
    dim3 grid(ntx * nty, (P->nz + ZS - 1) / ZS);
    kern<<<grid, kAdjThreads, smem, st>>>(tm, P->d_fold_ang, u_calc ? nullptr : (S *)u, u_calc ? (T *)u : nullptr,
                                          P->nx, P->ny, P->nz, P->fold_U, P->fold_U1, P->m, (T)alpha, (T)beta, P->d_status,
                                          P->d_status + 1 + P->wild_slot, pp,
                                          P->m == M && ((uintptr_t)u & 15u) == 0);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DR_OK : cuda_fail(e, "fold_adj_kernel launch");
}

// Which form, by the CTAs it makes (bits do not depend on it).
//   m <= 8: several slices per thread once that leaves every SM two CTAs and is less
//     work in all: a CTA of four slices (m <= 4) takes up to 2.3 times as long as one
//     of one, of two up to 1.7, so neither a volume's last, partly empty group nor a
//     longer last round per SM may eat the gain.  U = 120, one : several slices:
//     m = 4: 4 x 512^2 0.160 : 0.126 ms, 2 x 700 x 512 0.118 : 0.172; m = 8:
//     4 x 512^2 0.218 : 0.206, 3 x 400^2 0.122 : 0.163.
//   m > 8: twice as many threads per patch while the CTAs are few (U = 120: 64^2,
//     m = 16 0.078 -> 0.058 ms, m = 32 0.082 -> 0.063; above the lines the second
//     reads of the bins' weights cost more, 4 x 256^2, m = 12 0.087 -> 0.135).  At
//     m = 16 the two are within 7 % of one another, and what the last round of CTAs
//     per SM costs decides: times for n CTAs on an SM, in us of U = 120, are those
//     below (462 CTAs, 2 x 327^2, U = 258: 0.259 -> 0.229 ms; 640, 10 x 256^2, U = 120:
//     0.216 -> 0.181).
template <typename S, typename T, int M>
dr_status fold_backproject(dr_plan *P, void *u, double alpha, double beta, bool u_calc, cudaStream_t st, void *gt) {
    if (!gt) gt = P->d_gt;
    constexpr int NG = kFoldAdjNG<M>;
    const long long nty = (P->ny + kAdjTY - 1) / kAdjTY, sms = P->num_sms;
    const auto tiles = [&](int tx) { return (P->nx + tx - 1) / tx * nty; };
    const auto up = [](long long a, long long b) { return (a + b - 1) / b; };
    if constexpr (M <= 8) {
        constexpr int ZS = M <= 4 ? 4 : 2, R = M <= 4 ? 23 : 17;
        const long long one = tiles(32) * P->nz, many = tiles(32) * up(P->nz, ZS);
        if (many >= 2 * sms && R * many < 10 * one && R * up(many, sms) < 10 * up(one, sms))
            return fold_backproject_t<S, T, M, NG, ZS>(P, u, alpha, beta, u_calc, st, gt);
    } else {
        const long long c = tiles(32 / NG) * P->nz, c2 = tiles(16 / NG) * P->nz;
        bool fine;
        if constexpr (M == 16) {
            // all coefficients: full rounds of 103 and a last one of 1 to 4 CTAs; half: one
            // round of up to 6 CTAs, then 13.6 each
            constexpr int last[4] = {78, 86, 104, 135}, once[6] = {60, 67, 73, 82, 101, 118};
            const long long n = up(c, sms), n2 = up(c2, sms);
            fine = (n2 <= 6 ? 10 * once[n2 - 1] : 420 + 136 * n2) <= 1030 * ((n - 1) / 4) + 10 * last[(n - 1) % 4];
        } else {
            constexpr int few = M == 12 ? 4 : (M == 24 ? 6 : 8);  // quarters of CTAs per SM
            fine = 4 * c <= few * sms;
        }
        if (fine)
            return fold_backproject_t<S, T, M, 2 * NG, 1>(P, u, alpha, beta, u_calc, st, gt);
    }
    return fold_backproject_t<S, T, M, NG, 1>(P, u, alpha, beta, u_calc, st, gt);
}

// ===========================================================================
// Normal operator R*R of the folded pair, as the CG steps use it.  Per
// distinct angle a, forward then adjoint give
//   (R*R u)_i = sum_a R_a* [ sum_j G_a[i][j] (R_a u_j) ],
//   G_a = sum_{k in a} phi(t_k) phi(t_k)^T,
// because the bin reversal of an odd half-turn is undone by its adjoint.  So
// the static transforms are mixed by G_a per (slice, angle, bin) and
// back-projected, without the K projections in between.
// ===========================================================================
template <typename T, int M, bool BLK>
__global__ void __launch_bounds__(kRedThreads)
    fold_gram_kernel(const T *ru, T *gt, const T *__restrict__ gram, int nz, int U, int ns, RowMap rin, int m,
                     int nsplit, size_t split_stride, int *wild, int slot) {
    clear_next_wild(wild, slot);
    // ru and gt may be the same buffer (one chunk): each thread reads its row
    // whole before writing it, so they are not declared __restrict__
    constexpr int MS = fold_ms(M);
    constexpr bool V4 = sizeof(T) == 4;
    const size_t n = (size_t)nz * U * ns;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int a = (int)((i / ns) % U);
        const T *r = ru + i * rin.C;
        if constexpr (BLK) {
            const int z = (int)(i / ((size_t)U * ns));
            r = ru + row_at(rin, z, i - (size_t)z * U * ns);
        }
        T rv[M];
        if constexpr (V4 && M % 4 == 0) {
            // rows are multiples of 4 floats from 16-byte aligned bases
#pragma unroll
            for (int q = 0; q < M / 4; ++q) {
                if (4 * q < m) {
                    float4 v = *reinterpret_cast<const float4 *>(r + 4 * q);
                    for (int c = 1; c < nsplit; ++c) {
                        const float4 w = *reinterpret_cast<const float4 *>(r + c * split_stride + 4 * q);
                        v.x += w.x;
                        v.y += w.y;
                        v.z += w.z;
                        v.w += w.w;
                    }
                    // slots at or beyond m: zero (the G rows and columns there are zero)
                    rv[4 * q] = v.x;
                    rv[4 * q + 1] = 4 * q + 1 < m ? v.y : T(0);
                    rv[4 * q + 2] = 4 * q + 2 < m ? v.z : T(0);
                    rv[4 * q + 3] = 4 * q + 3 < m ? v.w : T(0);
                } else {
                    rv[4 * q] = rv[4 * q + 1] = rv[4 * q + 2] = rv[4 * q + 3] = T(0);
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < M; ++j) {
                T rj = T(0);
                if (j < m) {
                    rj = r[j];
                    for (int c = 1; c < nsplit; ++c) rj += r[c * split_stride + j];
                }
                rv[j] = rj;
            }
        }
        const T *G = gram + (size_t)a * M * M;
        T ov[MS];
#pragma unroll
        for (int q = 0; q < MS; ++q) ov[q] = T(0);
#pragma unroll
        for (int q = 0; q < M; ++q) {
            T acc = T(0);
            if constexpr (V4 && M % 4 == 0) {
#pragma unroll
                for (int c = 0; c < M / 4; ++c) {
                    const float4 gq = __ldg(reinterpret_cast<const float4 *>(G + q * M) + c);
                    acc = fma(gq.x, rv[4 * c], acc);
                    acc = fma(gq.y, rv[4 * c + 1], acc);
                    acc = fma(gq.z, rv[4 * c + 2], acc);
                    acc = fma(gq.w, rv[4 * c + 3], acc);
                }
            } else {
#pragma unroll
                for (int j = 0; j < M; ++j) acc = fma(__ldg(G + q * M + j), rv[j], acc);
            }
            ov[q] = acc;
        }
        note_wild(ov, wild, slot);
        T *dst = gt + i * MS;
        if constexpr (V4 && MS % 4 == 0) {
#pragma unroll
            for (int q = 0; q < MS / 4; ++q)
                reinterpret_cast<float4 *>(dst)[q] = make_float4(ov[4 * q], ov[4 * q + 1], ov[4 * q + 2], ov[4 * q + 3]);
        } else {
#pragma unroll
            for (int q = 0; q < MS; ++q) dst[q] = ov[q];
        }
    }
}

template <typename S, typename T, int M>
dr_status fold_normal_launch_t(dr_plan *P, const void *x, void *y, cudaStream_t st, bool chan) {
    if (!P->d_fold_gram) return fail(DR_EINVAL, "folded normal operator unavailable for this plan");
    StaticOut rs{};
    {
        dr_status s = chan ? chan_static(P, x, false, true, fold2_chunks(P), st, rs)
                           : fold_static_dispatch<S, T, M>(P, x, st, rs);
        if (s != DR_OK) return s;
    }
    {
        dr_status s = ensure_fold_scratch(P);
        if (s != DR_OK) return s;
    }
    auto gram = rs.rows.spb > 1 ? fold_gram_kernel<T, M, true> : fold_gram_kernel<T, M, false>;
    gram<<<red_grid((size_t)P->nz * P->fold_U * P->ns), kRedThreads, 0, st>>>(
        (const T *)rs.ru, (T *)P->d_gt, (const T *)P->d_fold_gram, P->nz, P->fold_U, P->ns, rs.rows, P->m,
        rs.nsplit, rs.split_stride, P->d_status + 1, P->wild_slot ^= 1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "fold_gram_kernel launch");
    return fold_backproject<S, T, M>(P, y, 1.0, 0.0, true, st);
}

template <typename S, typename T>
struct FoldOps {
    static dr_status fwd(dr_plan *P, const void *u, void *out, const void *gm, int mode, double sigma,
                         cudaStream_t st);
    static dr_status fwd2(dr_plan *P, const void *u, void *out, const void *gm, int mode, double sigma,
                          cudaStream_t st, int chan = 0);
    static dr_status adj(dr_plan *P, const void *g, void *u, double alpha, double beta, bool u_calc,
                         cudaStream_t st);
    // y = R*R x on compute-typed buffers (static transforms, Gram mix, back-projection)
    static dr_status normal(dr_plan *P, const void *x, void *y, cudaStream_t st, bool chan = false);
};

#define DR_FOLD_DISPATCH(FN, S, T, ...)                   \
    switch (P->M) {                                       \
        case 1: return FN<S, T, 1>(__VA_ARGS__);          \
        case 2: return FN<S, T, 2>(__VA_ARGS__);          \
        case 4: return FN<S, T, 4>(__VA_ARGS__);          \
        case 8: return FN<S, T, 8>(__VA_ARGS__);          \
        case 12: return FN<S, T, 12>(__VA_ARGS__);        \
        case 16: return FN<S, T, 16>(__VA_ARGS__);        \
        case 24: return FN<S, T, 24>(__VA_ARGS__);        \
        case 32: return FN<S, T, 32>(__VA_ARGS__);        \
        default: return fail(DR_EINVAL, "unsupported m"); \
    }

template <typename S, typename T>
dr_status FoldOps<S, T>::fwd(dr_plan *P, const void *u, void *out, const void *gm, int mode, double sigma,
                             cudaStream_t st) {
    DR_FOLD_DISPATCH(fold_fwd_launch_t, S, T, P, u, out, gm, mode, sigma, st)
}

template <typename S, typename T>
dr_status FoldOps<S, T>::fwd2(dr_plan *P, const void *u, void *out, const void *gm, int mode, double sigma,
                              cudaStream_t st, int chan) {
    DR_FOLD_DISPATCH(fold_fwd2_launch_t, S, T, P, u, out, gm, mode, sigma, st, chan)
}

template <typename S, typename T>
dr_status FoldOps<S, T>::adj(dr_plan *P, const void *g, void *u, double alpha, double beta, bool u_calc,
                             cudaStream_t st) {
    DR_FOLD_DISPATCH(fold_adj_launch_t, S, T, P, g, u, alpha, beta, u_calc, st)
}

template <typename S, typename T>
dr_status FoldOps<S, T>::normal(dr_plan *P, const void *x, void *y, cudaStream_t st, bool chan) {
    DR_FOLD_DISPATCH(fold_normal_launch_t, S, T, P, x, y, st, chan)
}

extern template struct FoldOps<float, float>;
extern template struct FoldOps<bf16, float>;

}  // namespace dr
