// chan_fwd.cu -- static transforms of the half-turn folded forward (Sec. 4)
// with channels on the lanes of a warp (chan.cuh).
//
// The volume is first packed into blocks of C = 32 V channels,
// uc[block][y][x][C] (pack_kernel: one pass over u, which also widens bf16 and
// pads m), so that a pixel of a block is one contiguous run.  A CTA of 16
// compute warps and one copy warp takes a block of n neighbouring distinct
// angles and a run of bins: warp w marches RW consecutive bins of angle w / g,
// all image lines, its RW V sums per lane in registers.  Per line the copy
// warp brings the band of pixels the CTA's rays touch (their positions shift
// by the angle's step from line to line; neighbouring angles fan out slowly)
// into a ring of line buffers with TMA boxes, zero beyond the image, completing
// on mbarriers; there is no CTA barrier in the march.  Along a line the rays
// of a warp are 1 to sqrt 2 pixels apart: the next ray's lower pixel is this
// ray's upper one, or (the carry of the position's fraction) one pixel
// further, which is then read too.
//
// Bound by issue and shared memory together (ncu: 64 % of the issue slots and 61 % of
// the shared-memory pipe on 16 x 256^2, m = 8, 180 distinct angles; 80 and 67 % on
// 4 x 1024^2, m = 16; the thread-per-ray kernels reach 90 % of that pipe with 1.7
// times the bytes).
// Forward of 16 x 256^2, K = 1800, m = 8: 0.500 -> 0.373 ms; 8 x 1024^2,
// K = 6000, m = 16: 16.3 -> 7.25 ms (0.13 -> 0.28 of the FP32 multiply-add
// rate).  Tried and slower: packed multiply-adds (0.405 ms: the copies that
// pair the weights), a real branch instead of the predicated read (0.387 ms),
// two lines at a time (0.390 ms with 16 warps, against 0.396 ms).
//
// EO: the same march in the order of the thread-per-ray kernels (a sample's even
// pixel is added before its odd one): the even and the odd pixel keep their own
// registers, and the lanes work out weights and steps of a line's rays side by
// side.  Bit for bit the fold in two kernels, so the solvers can run on it, in that
// fold's line chunks: 0.54 ms with its one on the first volume above (0.44 with three,
// which would round differently) and 8.5 ms on the second.
#include <algorithm>
#include <cmath>
#include <vector>

#include "chan.cuh"

namespace dr {

// V floats of a lane at a shared-memory address.  (Inline PTX: the loads of a
// march must become predicated loads into the registers that already hold the
// other candidate, without a branch or a copy.)
template <int V>
__device__ __forceinline__ void chan_ld(uint32_t p, float (&v)[V]) {
    if constexpr (V == 1) asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[0]) : "r"(p));
    else if constexpr (V == 2) asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(p));
    else
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                     : "r"(p));
}
// frac += a; on a carry p += step and v = [p + off], else v stays.
template <int V>
__device__ __forceinline__ void chan_advance(unsigned &frac, unsigned a, uint32_t &p, float (&v)[V], int step, int off) {
    const unsigned f = frac + a;
    if constexpr (V == 1)
        asm volatile(
            "{\n\t.reg .pred c;\n\t.reg .u32 t;\n\tsetp.lt.u32 c, %2, %3;\n\t@c add.u32 %0, %0, %4;\n\t"
            "add.u32 t, %0, %5;\n\t@c ld.shared.f32 %1, [t];\n\t}"
            : "+r"(p), "+f"(v[0])
            : "r"(f), "r"(frac), "r"(step), "r"(off));
    else if constexpr (V == 2)
        asm volatile(
            "{\n\t.reg .pred c;\n\t.reg .u32 t;\n\tsetp.lt.u32 c, %3, %4;\n\t@c add.u32 %0, %0, %5;\n\t"
            "add.u32 t, %0, %6;\n\t@c ld.shared.v2.f32 {%1, %2}, [t];\n\t}"
            : "+r"(p), "+f"(v[0]), "+f"(v[1])
            : "r"(f), "r"(frac), "r"(step), "r"(off));
    else
        asm volatile(
            "{\n\t.reg .pred c;\n\t.reg .u32 t;\n\tsetp.lt.u32 c, %5, %6;\n\t@c add.u32 %0, %0, %7;\n\t"
            "add.u32 t, %0, %8;\n\t@c ld.shared.v4.f32 {%1, %2, %3, %4}, [t];\n\t}"
            : "+r"(p), "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3])
            : "r"(f), "r"(frac), "r"(step), "r"(off));
    frac = f;
}

// One step along a line in even / odd order: where bit K of the mask is set,
// a += step and v = [a].
template <int V, int K>
__device__ __forceinline__ void chan_step(unsigned mask, uint32_t &a, int step, float (&v)[V]) {
    if constexpr (V == 1)
        asm volatile(
            "{\n\t.reg .pred c;\n\t.reg .u32 t;\n\tand.b32 t, %2, %4;\n\tsetp.ne.u32 c, t, 0;\n\t"
            "@c add.u32 %0, %0, %3;\n\t@c ld.shared.f32 %1, [%0];\n\t}"
            : "+r"(a), "+f"(v[0])
            : "r"(mask), "r"(step), "n"(1u << K));
    else if constexpr (V == 2)
        asm volatile(
            "{\n\t.reg .pred c;\n\t.reg .u32 t;\n\tand.b32 t, %3, %5;\n\tsetp.ne.u32 c, t, 0;\n\t"
            "@c add.u32 %0, %0, %4;\n\t@c ld.shared.v2.f32 {%1, %2}, [%0];\n\t}"
            : "+r"(a), "+f"(v[0]), "+f"(v[1])
            : "r"(mask), "r"(step), "n"(1u << K));
    else
        asm volatile(
            "{\n\t.reg .pred c;\n\t.reg .u32 t;\n\tand.b32 t, %5, %7;\n\tsetp.ne.u32 c, t, 0;\n\t"
            "@c add.u32 %0, %0, %6;\n\t@c ld.shared.v4.f32 {%1, %2, %3, %4}, [%0];\n\t}"
            : "+r"(a), "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3])
            : "r"(mask), "r"(step), "n"(1u << K));
}
// Rays K, K + 1, .. of a line: the even pixel of each in e, the odd one in o.
template <int V, int RW, int K>
__device__ __forceinline__ void chan_line(unsigned me, unsigned mo, uint32_t &pe, uint32_t &po, const float4 *rec,
                                          float4 &w, float (&e)[V], float (&o)[V], float (&acc)[RW][V]) {
    if constexpr (K < RW) {
        if constexpr (K > 0) {
            chan_step<V, K>(me, pe, 2 * 128 * V, e);
            chan_step<V, K>(mo, po, 2 * 128 * V, o);
        }
        if constexpr ((K & 3) == 0) w = rec[K >> 2];
        // (a weight is a multiple of 2^-23: the other one is exactly 1 less it)
        const float we = (K & 3) == 0 ? w.x : (K & 3) == 1 ? w.y : (K & 3) == 2 ? w.z : w.w, wo = 1.0f - we;
#pragma unroll
        for (int v = 0; v < V; ++v) acc[K][v] = fmaf(wo, o[v], fmaf(we, e[v], acc[K][v]));
        chan_line<V, RW, K + 1>(me, mo, pe, po, rec, w, e, o, acc);
    }
}

// ---------------------------------------------------------------------------
// uc[block][pixel][C] <- u[z][pixel][m]: channel zi ms + j of block c is
// coefficient j of slice c spb + zi (zero for j >= m and beyond the volume).
// A thread moves 4 channels.  VEC: rows of float vectors at 16-byte aligned
// addresses (m a multiple of 4).  Bound by HBM (one read, one write of u).
// ---------------------------------------------------------------------------
template <typename S, bool VEC>
__global__ void __launch_bounds__(256)
    pack_kernel(const S *__restrict__ u, float *__restrict__ uc, size_t npix, int nz, int m, int ms, int spb, int C,
                int c0) {
    const int q = C / 4;
    const size_t n = npix * q;
    const int cb = blockIdx.y;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t pix = i / q;
        const int ch = 4 * (int)(i - pix * q), zi = ch / ms, j = ch - zi * ms, z = (c0 + cb) * spb + zi;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (zi < spb && z < nz) {
            const S *p = u + ((size_t)z * npix + pix) * m + j;
            if constexpr (VEC) {
                v = __ldg(reinterpret_cast<const float4 *>(p));
            } else {
                v.x = ldc<float>(p);
                if (j + 1 < m) v.y = ldc<float>(p + 1);
                if (j + 2 < m) v.z = ldc<float>(p + 2);
                if (j + 3 < m) v.w = ldc<float>(p + 3);
            }
        }
        reinterpret_cast<float4 *>(uc)[(size_t)cb * n + i] = v;
    }
}

struct ChanFwdArgs {
    const FwdProj *uproj;
    const int *blocks;  // [nblocks][kChanWarps] distinct angles (-1: none)
    float *ru;
    RowMap rows;
    size_t split_stride;
    int *status;
    int n, g, nx, ny, ns, nz, c0, ms, spb, ring_bytes;
};

template <int V, int RW, int NW, bool EO>
__global__ void __launch_bounds__(32 * (NW + 1), NW == 8 ? 2 : 1)
    chan_fwd_kernel(const __grid_constant__ CUtensorMap tm_rows, const __grid_constant__ CUtensorMap tm_cols,
                    const __grid_constant__ ChanFwdArgs P) {
    constexpr int PXB = 128 * V;              // bytes of a pixel (32 V channels)
    constexpr int BOXB = kChanBox * PXB;      // bytes of one TMA box (kChanBox pixels of a line)
    extern __shared__ __align__(128) unsigned char chan_smem[];
    unsigned char *ring = chan_smem + ((128u - (smem_u32(chan_smem) & 127u)) & 127u);
    __shared__ __align__(8) uint64_t full[kChanSlots], empty[kChanSlots];
    __shared__ int base_s[kChanSlots];  // byte offset of pixel 0 of a buffered line (of its band's first pixel less s0)
    __shared__ long long x_s[NW], e_s[NW], b_s[NW];  // first / last ray, step per line
    __shared__ int lo_s[NW], hi_s[NW];
    __shared__ __align__(16) float rec_s[EO ? NW : 1][2][32];  // weights of the even pixel

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cb = blockIdx.y, chunk = blockIdx.z;
    const int nbx = (P.ns + RW * P.g - 1) / (RW * P.g);
    // bins of the middle of the detector first: their rays are the longest, and
    // the short ones at the edges then fill the last wave
    const int nblk = gridDim.x / nbx, bi = blockIdx.x / nblk, blk = blockIdx.x - bi * nblk;
    const int bx = nbx / 2 + ((bi & 1) ? -((bi + 1) / 2) : bi / 2);
    const int *ang = P.blocks + (size_t)blk * kChanWarps;
    const int branch = P.uproj[ang[0]].branch;
    const int W = branch ? P.ny : P.nx, H = branch ? P.nx : P.ny;
    const int L0 = (int)(((long long)chunk * H) / gridDim.z), L1 = (int)(((long long)(chunk + 1) * H) / gridDim.z);

    // ---- this warp's rays: RW bins of one angle, ordered by increasing position ----
    const int pa = warp / P.g, b0 = bx * RW * P.g + (warp - pa * P.g) * RW;
    const int a = (warp < NW && pa < P.n) ? ang[pa] : -1;
    long long x = 0, bstep = 0;
    unsigned afrac = 0;
    int wlo = 1 << 30, whi = -1;
    bool rev = false;
    float scale = 0.f;
    if (a >= 0) {
        const FwdProj f = P.uproj[a];
        rev = f.A_fx < 0;
        const long long A = rev ? -f.A_fx : f.A_fx;  // 2^32 (1 + afrac / 2^32), 1 <= A < sqrt 2
        afrac = (unsigned)A;
        x = f.C_fx + (long long)(rev ? b0 + RW - 1 : b0) * f.A_fx;
        bstep = f.B_fx;
        scale = f.scale;
        const long long xe = x + (RW - 1) * A;
        // lines on which some sample of the run can touch the image (in float,
        // with a line to spare on both sides; the band is zero filled beyond it)
        const float xf = (float)((double)x * (1.0 / 4294967296.0)), ef = (float)((double)xe * (1.0 / 4294967296.0));
        if (fabsf(f.Bf) < 1e-2f) {
            wlo = L0;
            whi = L1 - 1;
        } else {
            const float r1 = (-1.0f - ef) / f.Bf, r2 = ((float)W - xf) / f.Bf, r3 = (-1.0f - xf) / f.Bf,
                        r4 = ((float)W - ef) / f.Bf;
            const float rmin = fmaxf(fminf(fminf(r1, r2), fminf(r3, r4)), -4.0f);
            const float rmax = fminf(fmaxf(fmaxf(r1, r2), fmaxf(r3, r4)), (float)H + 4.0f);
            wlo = max(L0, (int)floorf(rmin) - 1);
            whi = min(L1 - 1, (int)ceilf(rmax) + 1);
            if (whi < wlo) {
                wlo = 1 << 30;
                whi = -1;
            }
        }
        if (lane == 0) {
            x_s[warp] = x;
            e_s[warp] = xe;
            b_s[warp] = bstep;
        }
    }
    if (warp < NW && lane == 0) {
        lo_s[warp] = wlo;
        hi_s[warp] = whi;
    }
    if (tid == 0) {
        for (int s = 0; s < kChanSlots; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], NW);
        }
        fence_mbar_init();
    }
    __syncthreads();
    // ---- the CTA's lines, and its widest band: the bounds of the band are a
    // minimum and a maximum of functions linear in the line, so its width is
    // largest on the first or the last line ----
    int rlo = 1 << 30, rhi = -1;
    for (int w = 0; w < NW; ++w) {
        rlo = min(rlo, lo_s[w]);
        rhi = max(rhi, hi_s[w]);
    }
    int wide = 1;
    for (int e = 0; e < 2 && rhi >= 0; ++e) {
        const long long r = e ? rhi : rlo;
        int lo = 1 << 30, hi = -(1 << 30);
        for (int w = 0; w < NW; ++w)
            if (hi_s[w] >= 0) {
                lo = min(lo, (int)((x_s[w] + r * b_s[w]) >> 32));
                hi = max(hi, (int)((e_s[w] + r * b_s[w]) >> 32) + 1);
            }
        wide = max(wide, chan_boxes(hi - lo + 2));  // one pixel for the rounding of both ends
    }
    const int ring_boxes = P.ring_bytes / BOXB;
    if (wide > ring_boxes) {  // excluded by the host's rule; the ring could not make progress
        if (tid == 0) atomicOr(P.status, kStatusTimeout);
        return;
    }

    if (warp == NW) {
        // ---- copy warp: lane w knows warp w's band.  Lines take as many boxes
        // of the ring as they need, in order, never wrapping inside a line ----
        long long xl = 0, el = 0, bl = 0;
        int lo_l = 1 << 30, hi_l = -1;
        if (lane < NW) {
            lo_l = lo_s[lane];
            hi_l = hi_s[lane];
            if (hi_l >= 0) {
                bl = b_s[lane];
                xl = x_s[lane] + (long long)rlo * bl;
                el = e_s[lane] + (long long)rlo * bl;
            }
        }
        int k = 0, oldest = 0, head = 0, start = 0;  // start: of line k in lane k % kChanSlots
        bool ok = true;
        for (int r = rlo; r <= rhi && ok; ++r, ++k) {
            const bool on = r >= lo_l && r <= hi_l;
            const int lo = __reduce_min_sync(0xffffffffu, on ? (int)(xl >> 32) : (1 << 30));
            const int hi = __reduce_max_sync(0xffffffffu, on ? (int)(el >> 32) + 1 : -(1 << 30));
            const int nb = hi >= lo ? chan_boxes(hi - lo + 1) : 0, need = max(nb, 1);
            for (;;) {
                bool fits = false;
                if (k - oldest < kChanSlots) {
                    if (oldest == k) {
                        head = 0;
                        fits = true;
                    } else {
                        const int tail = __shfl_sync(0xffffffffu, start, oldest % kChanSlots);
                        if (head > tail) {
                            if (head + need <= ring_boxes) fits = true;
                            else if (need <= tail) {
                                head = 0;
                                fits = true;
                            }
                        } else {
                            fits = head + need <= tail;
                        }
                    }
                }
                if (fits) break;
                if (!mbar_wait_bounded_any(&empty[oldest % kChanSlots], (unsigned)((oldest / kChanSlots) & 1), P.status,
                                           2000000000ull)) {
                    ok = false;
                    break;
                }
                ++oldest;
            }
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const int slot = k % kChanSlots;
            if (lane == slot) start = head;
            if (lane == 0) {
                base_s[slot] = head * BOXB - lo * PXB;
                mbar_arrive_expect_tx(&full[slot], (unsigned)(nb * BOXB));
            }
            __syncwarp();
            for (int i = lane; i < nb; i += 32) {
                const uint32_t dst = smem_u32(ring) + (uint32_t)((head + i) * BOXB);
                const int px = lo + i * kChanBox;
                if (branch == 0) tma_load_4d(dst, &tm_rows, 0, px, r, cb, &full[slot]);
                else tma_load_4d(dst, &tm_cols, 0, r, px, cb, &full[slot]);
            }
            head += need;
            xl += bl;
            el += bl;
        }
        // No copy of this CTA may outlive it: the compute warps leave as soon as any
        // CTA's wait gave up, also after this warp has issued its last line.
        for (int i = oldest; i < k; ++i)
            mbar_wait_bounded(&full[i % kChanSlots], (unsigned)((i / kChanSlots) & 1), P.status, 100000000ull);
        return;
    }

    // ---- compute warps ----
    float acc[RW][V];
#pragma unroll
    for (int q = 0; q < RW; ++q)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[q][v] = 0.0f;
    x += (long long)rlo * bstep;
    const uint32_t mine = smem_u32(ring) + lane * (4 * V);
    int slot = 0;
    unsigned phase = 0;
    // even / odd order: the lanes work out the rays of one line (RW = 32) or two
    // (RW = 16) side by side: weights to shared memory, and in two masks the rays
    // at which the even and the odd pixel change
    constexpr int NL = 32 / RW;
    const int rq = lane % RW;
    const long long roff = (lane / RW) * bstep + rq * ((1ll << 32) + afrac);
    unsigned me = 0, mo = 0;
    int eb = 0, ob = 0, buf = 0;
    for (int r = rlo; r <= rhi; ++r) {
        const int hl = EO ? (r - rlo) % NL : 0;
        if (EO && hl == 0) {
            const long long xr = x + roff;
            const int i0 = (int)(xr >> 32);
            const float w = __uint_as_float(__funnelshift_r((unsigned)xr, 0x7Fu, 9)) - 1.0f, w1m = 1.0f - w;
            buf ^= 1;
            rec_s[EO ? warp : 0][buf][lane] = (i0 & 1) ? w : w1m;
            eb = (i0 + 1) & ~1;
            ob = i0 | 1;
            const int pe = __shfl_up_sync(0xffffffffu, eb, 1), po = __shfl_up_sync(0xffffffffu, ob, 1);
            me = __ballot_sync(0xffffffffu, eb != pe);
            mo = __ballot_sync(0xffffffffu, ob != po);
            __syncwarp();
        }
        if (!mbar_wait_bounded_any(&full[slot], phase, P.status, 2000000000ull)) return;
        if (EO && r >= wlo && r <= whi) {
            uint32_t pe = mine + base_s[slot] + __shfl_sync(0xffffffffu, eb, hl * RW) * PXB;
            uint32_t po = mine + base_s[slot] + __shfl_sync(0xffffffffu, ob, hl * RW) * PXB;
            float e[V], o[V];
            float4 w;
            chan_ld<V>(pe, e);
            chan_ld<V>(po, o);
            chan_line<V, RW, 0>(NL > 1 ? me >> (hl * RW) : me, NL > 1 ? mo >> (hl * RW) : mo, pe, po,
                                reinterpret_cast<const float4 *>(&rec_s[EO ? warp : 0][buf][hl * RW]), w, e, o, acc);
        }
        if (!EO && r >= wlo && r <= whi) {
            // one line: the two pixels of a ray in t[q & 1] and t[(q + 1) & 1]
            uint32_t p = mine + base_s[slot] + (int)(x >> 32) * PXB;
            unsigned frac = (unsigned)x;
            float t[2][V];
            chan_ld<V>(p, t[0]);
#pragma unroll
            for (int q = 0; q < RW; ++q) {
                float(&lo)[V] = t[q & 1];
                float(&hi)[V] = t[(q + 1) & 1];
                chan_ld<V>(p + (q + 1) * PXB, hi);
                const float w = __uint_as_float(__funnelshift_r(frac, 0x7Fu, 9)) - 1.0f;
                const float w1m = 1.0f - w;
#pragma unroll
                for (int v = 0; v < V; ++v) acc[q][v] = fmaf(w, hi[v], fmaf(w1m, lo[v], acc[q][v]));
                // the next ray's lower pixel is hi, or with a carry the one after it
                if (q + 1 < RW) chan_advance<V>(frac, afrac, p, hi, PXB, (q + 1) * PXB);
            }
        }
        x += bstep;
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[slot]);
        if (++slot == kChanSlots) {
            slot = 0;
            phase ^= 1u;
        }
    }
    // ---- the scaled static transforms ----
    const int ch = lane * V, zl = ch / P.ms, j = ch - zl * P.ms, z = (P.c0 + cb) * P.spb + zl;
    if (a < 0 || zl >= P.spb || z >= P.nz) return;
    float *ru = P.ru + (size_t)chunk * P.split_stride;
#pragma unroll
    for (int q = 0; q < RW; ++q) {
        const int b = rev ? b0 + RW - 1 - q : b0 + q;
        if (b >= P.ns) continue;
        float *dst = ru + row_at(P.rows, z, (size_t)a * P.ns + b) + j;
        if constexpr (V == 1) *dst = scale * acc[q][0];
        else if constexpr (V == 2) *reinterpret_cast<float2 *>(dst) = make_float2(scale * acc[q][0], scale * acc[q][1]);
        else
            *reinterpret_cast<float4 *>(dst) =
                make_float4(scale * acc[q][0], scale * acc[q][1], scale * acc[q][2], scale * acc[q][3]);
    }
}

// ===========================================================================
// Host side
// ===========================================================================
namespace {

// The rays of one warp of the kernel above, in pixels (its own arithmetic).
struct Run {
    double x, e, b;
    int lo, hi;  // lines
};
Run run_of(const FwdProj &f, int b0, int RW, int W, int H) {
    Run r{};
    const double A = std::fabs(f.A);
    r.x = f.C + (f.A < 0.0 ? b0 + RW - 1 : b0) * f.A;
    r.e = r.x + (RW - 1) * A;
    r.b = f.B;
    r.lo = 0;
    r.hi = H - 1;
    if (std::fabs(f.B) >= 1e-2) {
        const double r1 = (-1.0 - r.e) / f.B, r2 = (W - r.x) / f.B, r3 = (-1.0 - r.x) / f.B, r4 = (W - r.e) / f.B;
        const double mn = std::max(std::min(std::min(r1, r2), std::min(r3, r4)), -4.0);
        const double mx = std::min(std::max(std::max(r1, r2), std::max(r3, r4)), H + 4.0);
        r.lo = std::max(0, (int)std::floor(mn) - 1);
        r.hi = std::min(H - 1, (int)std::ceil(mx) + 1);
    }
    return r;
}

// Angles of the blocks: every segment (angles of one stepping axis and one
// direction, ascending) in as few blocks of at most n angles as hold it, of
// even size.
std::vector<int> make_blocks(const std::vector<std::vector<int>> &segs, int n) {
    std::vector<int> out;
    for (const auto &s : segs) {
        const int nb = ((int)s.size() + n - 1) / n;
        for (int i = 0; i < nb; ++i) {
            const size_t a0 = s.size() * i / nb, a1 = s.size() * (i + 1) / nb;
            for (int q = 0; q < kChanWarps; ++q) out.push_back(a0 + q < a1 ? s[a0 + q] : -1);
        }
    }
    return out;
}

struct Band {
    double clocks = 0.0;  // shared-memory pixel reads and writes over all lines
    int wide = 0;         // widest band in boxes
};
Band band_of(const dr_plan *P, const std::vector<FwdProj> &fw, const int *ang, int nw, int n, int g, int RW, int bx,
             int samples) {
    Band o;
    const int branch = fw[ang[0]].branch, W = branch ? P->ny : P->nx, H = branch ? P->nx : P->ny;
    Run runs[kChanWarps];
    int nr = 0, lo = 1 << 30, hi = -1;
    for (int w = 0; w < nw; ++w) {
        const int a = w / g < n ? ang[w / g] : -1;
        if (a < 0) continue;
        const Run r = run_of(fw[a], bx * RW * g + (w % g) * RW, RW, W, H);
        if (r.hi < r.lo) continue;
        runs[nr++] = r;
        lo = std::min(lo, r.lo);
        hi = std::max(hi, r.hi);
    }
    if (!nr) return o;
    for (int i = 0; i < samples; ++i) {
        const int r = samples == 1 ? lo : lo + (int)((long long)(hi - lo) * i / (samples - 1));
        const bool end = i == 0 || i == samples - 1;
        double p0 = 1e30, p1 = -1e30, q0 = 1e30, q1 = -1e30, reads = 0.0;
        for (int k = 0; k < nr; ++k) {
            const double x = runs[k].x + r * runs[k].b, e = runs[k].e + r * runs[k].b;
            q0 = std::min(q0, x);
            q1 = std::max(q1, e);
            if (r < runs[k].lo || r > runs[k].hi) continue;
            p0 = std::min(p0, x);
            p1 = std::max(p1, e);
            reads += e - x + 2.0;
        }
        if (end) o.wide = std::max(o.wide, chan_boxes((int)std::ceil(q1 - q0) + 4));
        if (p1 >= p0) o.clocks += (reads + kChanBox * std::ceil((p1 - p0 + 2.0) / kChanBox)) * (hi - lo + 1) / samples;
    }
    return o;
}

}  // namespace

// Channels per lane: the least padded work, a block of 64 or 32 channels
// costing about 0.52 and 0.36 of one of 128 (measured per pass; fewer channels
// amortise the index arithmetic over less work).
static void chan_width(const dr_plan *P, ChanPlan &c) {
    c.ms = (P->m + 3) / 4 * 4;
    double best = 1e30;
    for (int V : {4, 2, 1}) {
        const int C = 32 * V, spb = C / c.ms;
        if (spb < 1) continue;
        const int ncb = (P->nz + spb - 1) / spb;
        const double cost = ncb * (V == 4 ? 1.0 : (V == 2 ? 0.52 : 0.36));
        if (cost < best) {
            best = cost;
            c.V = V;
            c.C = C;
            c.spb = spb;
            c.ncb = ncb;
        }
    }
}

dr_status chan_setup(dr_plan *P, const std::vector<FwdProj> &fw) {
    ChanPlan &c = P->chan;
    c = ChanPlan();
    const int U = (int)fw.size();
    if (P->m < 4 || U < 1 || P->nz * ((P->m + 3) / 4 * 4) < kChanMin) return DR_OK;
    chan_width(P, c);
    if (c.V == 0) return DR_OK;
    const int RW = chan_rw(c.V);
    std::vector<std::vector<int>> segs;
    for (int a = 0; a < U; ++a) {
        if (a == 0 || fw[a].branch != fw[a - 1].branch || (fw[a].A < 0.0) != (fw[a - 1].A < 0.0)) segs.emplace_back();
        segs.back().push_back(a);
    }
    // n angles by g runs of RW bins per CTA: the split with the least shared-memory
    // traffic (many angles share a band until they fan out) whose widest band
    // fits the ring twice
    struct Cand {
        double cost;
        int nw, n;
    };
    std::vector<Cand> cands;
    for (int nw : {8, 16})
        for (int n = 1; n <= nw; n *= 2) {
            const int g = nw / n, nbx = (P->ns + RW * g - 1) / (RW * g);
            const std::vector<int> blocks = make_blocks(segs, n);
            const int nblk = (int)(blocks.size() / kChanWarps), step = std::max(1, nblk / 12), bstep = std::max(1, nbx / 6);
            double cost = 0.0;
            int cnt = 0;
            for (int b = 0; b < nblk; b += step)
                for (int bx = 0; bx < nbx; bx += bstep, ++cnt)
                    cost += band_of(P, fw, &blocks[(size_t)b * kChanWarps], nw, n, g, RW, bx, 5).clocks;
            // (two CTAs of 8 warps per SM hide one another's start and end: measured 6 %
            // faster than one of 16 at equal traffic)
            cands.push_back(Cand{cost / std::max(cnt, 1) * nblk * nbx * (nw == 16 ? 1.08 : 1.0), nw, n});
        }
    std::sort(cands.begin(), cands.end(), [](const Cand &p, const Cand &q) { return p.cost < q.cost; });
    for (const Cand &cd : cands) {
        const int g = cd.nw / cd.n, nbx = (P->ns + RW * g - 1) / (RW * g);
        const std::vector<int> blocks = make_blocks(segs, cd.n);
        const int nblk = (int)(blocks.size() / kChanWarps);
        int wide = 0;
        for (int b = 0; b < nblk; ++b)
            for (int bx = 0; bx < nbx; ++bx)
                wide = std::max(wide, band_of(P, fw, &blocks[(size_t)b * kChanWarps], cd.nw, cd.n, g, RW, bx, 2).wide);
        if (2 * wide > chan_ring(cd.nw) / (kChanBox * c.C * 4)) continue;
        c.nw = cd.nw;
        c.n = cd.n;
        c.g = g;
        c.nblocks = nblk;
        c.nbx = nbx;
        DR_CUDA_TRY(cudaMalloc(&c.d_blocks, sizeof(int) * blocks.size()));
        P->table_bytes += sizeof(int) * blocks.size();
        DR_CUDA_TRY(cudaMemcpy(c.d_blocks, blocks.data(), sizeof(int) * blocks.size(), cudaMemcpyHostToDevice));
        break;
    }
    if (!c.d_blocks) {
        c.V = 0;
        return DR_OK;
    }
    // line chunks: fill the last wave, against the partial sums that every chunk
    // writes and the distribution adds
    c.gt_bytes = sizeof(float) * (size_t)c.ncb * c.C * U * P->ns;
    double best = 1e30;
    for (int s = 1; s <= 4; ++s) {
        if (s > 1 && (!chan_split_fits(P, s) || std::min(P->nx, P->ny) < 16 * s)) break;
        const double ctas = (double)c.nblocks * c.nbx * c.ncb * s;
        const double cost = std::ceil(ctas / (P->num_sms * (c.nw == 8 ? 2 : 1))) / s * (1.0 + 0.04 * (s - 1));
        if (cost < best - 1e-9) {
            best = cost;
            c.nsplit = s;
        }
    }
    c.rows = RowMap{c.spb, c.C, c.ms, (size_t)U * P->ns * c.C};
    // The packed volume, as many blocks at a time as the scratch cap and the
    // memory a serving job is counted for leave (with few projections per
    // distinct angle there is none: the other kernels then)
    const size_t blk = sizeof(float) * (size_t)P->nx * P->ny * c.C, held = P->gt_bytes + c.gt_bytes;
    const size_t budget = fold_budget(P->nz, P->K, P->ns, P->M);
    const size_t room = std::min(kChanScratchMax, budget > held ? budget - held : 0);
    c.cb_pass = (int)std::min<size_t>(c.ncb, room / blk);
    c.uc_bytes = blk * c.cb_pass;
    if (c.cb_pass < 1) c.V = 0;
    return DR_OK;
}

// Scratch buffers: never allocated while the stream is being captured; the
// caller then falls back to the kernels that need none.
static bool chan_alloc(void **p, size_t &held, size_t bytes, cudaStream_t st) {
    if (*p && held >= bytes) return true;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return false;
    }
    if (*p) cudaFree(*p);
    *p = nullptr;
    held = 0;
    if (cudaMalloc(p, std::max<size_t>(bytes, 16)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return false;
    }
    held = bytes;
    return true;
}

// Partial sums of nsplit line chunks within what a serving job is counted for (rows
// padded to whole channel blocks are up to twice the thread-per-ray kernels').
bool chan_split_fits(const dr_plan *P, int nsplit) {
    return nsplit == 1 || P->chan.gt_bytes * nsplit <= split_budget(P->nz, P->K, P->ns, P->m);
}

bool chan_fwd_ready(dr_plan *P, int nsplit, cudaStream_t st) {
    ChanPlan &c = P->chan;
    if (!c.V || P->split_off) return false;  // (a slab's memory is budgeted without this scratch)
    if (!chan_split_fits(P, nsplit)) return false;
    if (!chan_alloc(&c.d_uc, c.uc_held, c.uc_bytes, st) || !chan_alloc(&c.d_gt, c.gt_held, c.gt_bytes, st)) return false;
    if (nsplit == 1) return true;
    // (the buffer of partial sums is shared with the thread-per-ray kernels: never moved from here)
    const size_t need = c.gt_bytes * nsplit;
    if (P->d_ru_split) return P->ru_split_bytes >= need;
    return chan_alloc(&P->d_ru_split, P->ru_split_bytes, std::max(need, split_bytes(P)), st);
}

template <typename S>
static dr_status pack(dr_plan *P, const void *u, int c0, int nc, cudaStream_t st) {
    const ChanPlan &c = P->chan;
    const size_t npix = (size_t)P->nx * P->ny, n = npix * (c.C / 4);
    const dim3 grid((unsigned)std::min<size_t>((n + 255) / 256, 1u << 20), nc);
    const bool vec = sizeof(S) == 4 && P->m % 4 == 0 && ((uintptr_t)u & 15u) == 0;
    if (vec)
        pack_kernel<S, sizeof(S) == 4><<<grid, 256, 0, st>>>((const S *)u, (float *)c.d_uc, npix, P->nz, P->m, c.ms,
                                                             c.spb, c.C, c0);
    else
        pack_kernel<S, false><<<grid, 256, 0, st>>>((const S *)u, (float *)c.d_uc, npix, P->nz, P->m, c.ms, c.spb,
                                                    c.C, c0);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DR_OK : cuda_fail(e, "pack_kernel launch");
}

template <int V, int NW, bool EO>
static dr_status launch_t(dr_plan *P, float *ru, const RowMap &rows, size_t split_stride, int nsplit, int c0, int nc,
                          cudaStream_t st) {
    const ChanPlan &c = P->chan;
    constexpr int RW = chan_rw(V);
    CUtensorMap tr{}, tc{};
    const uint64_t dims[4] = {(uint64_t)c.C, (uint64_t)P->nx, (uint64_t)P->ny, (uint64_t)nc};
    const uint64_t str[3] = {(uint64_t)c.C * 4, (uint64_t)P->nx * c.C * 4, (uint64_t)P->nx * P->ny * c.C * 4};
    const uint32_t br[4] = {(uint32_t)c.C, kChanBox, 1, 1}, bc[4] = {(uint32_t)c.C, 1, kChanBox, 1};
    if (!encode_tensor_map(&tr, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, c.d_uc, dims, str, br) ||
        !encode_tensor_map(&tc, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, c.d_uc, dims, str, bc))
        return fail(DR_ECUDA, "chan_fwd: tensor map encode failed");
    auto kern = chan_fwd_kernel<V, RW, NW, EO>;
    const size_t smem = chan_ring(NW) + 128;
    const dr_status s = allow_dynamic_smem((const void *)kern, smem);
    if (s != DR_OK) return s;
    const ChanFwdArgs a{P->d_fold_fwd, c.d_blocks, ru, rows, split_stride, P->d_status, c.n, c.g, P->nx, P->ny,
                        P->ns, P->nz, c0, c.ms, c.spb, chan_ring(NW)};
    const dim3 grid(c.nblocks * c.nbx, nc, nsplit);
    kern<<<grid, 32 * (NW + 1), smem, st>>>(tr, tc, a);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DR_OK : cuda_fail(e, "chan_fwd_kernel launch");
}

template <bool EO>
static dr_status launch_v(dr_plan *P, float *ru, size_t stride, int nsplit, int c0, int nc, cudaStream_t st) {
    const ChanPlan &c = P->chan;
    switch (c.V + (c.nw == 8 ? 0 : 8)) {
        case 1: return launch_t<1, 8, EO>(P, ru, c.rows, stride, nsplit, c0, nc, st);
        case 2: return launch_t<2, 8, EO>(P, ru, c.rows, stride, nsplit, c0, nc, st);
        case 4: return launch_t<4, 8, EO>(P, ru, c.rows, stride, nsplit, c0, nc, st);
        case 9: return launch_t<1, 16, EO>(P, ru, c.rows, stride, nsplit, c0, nc, st);
        case 10: return launch_t<2, 16, EO>(P, ru, c.rows, stride, nsplit, c0, nc, st);
        default: return launch_t<4, 16, EO>(P, ru, c.rows, stride, nsplit, c0, nc, st);
    }
}

// Static transforms of all channels: into the channel-layout table, or the
// split scratch when the march is cut into line chunks (the caller adds them).
dr_status chan_static(dr_plan *P, const void *u, bool bf, bool eo, int nsplit, cudaStream_t st, StaticOut &rs) {
    ChanPlan &c = P->chan;
    float *ru = (float *)(nsplit > 1 ? P->d_ru_split : c.d_gt);
    const size_t stride = c.gt_bytes / sizeof(float);
    for (int c0 = 0; c0 < c.ncb; c0 += c.cb_pass) {
        const int nc = std::min(c.cb_pass, c.ncb - c0);
        dr_status s = bf ? pack<bf16>(P, u, c0, nc, st) : pack<float>(P, u, c0, nc, st);
        if (s != DR_OK) return s;
        s = eo ? launch_v<true>(P, ru, stride, nsplit, c0, nc, st) : launch_v<false>(P, ru, stride, nsplit, c0, nc, st);
        if (s != DR_OK) return s;
    }
    rs = StaticOut{ru, c.rows, nsplit, stride};
    return DR_OK;
}

// Scratch of trials whose kernel was not chosen.
void chan_release(dr_plan *P) {
    ChanPlan &c = P->chan;
    if (c.fwd || c.fwd_st || c.eo) return;
    for (void **p : {&c.d_uc, &c.d_gt}) {
        if (*p) cudaFree(*p);
        *p = nullptr;
    }
    c.uc_held = c.gt_held = 0;
}

void chan_free(dr_plan *P) {
    for (void *p : {(void *)P->chan.d_blocks, P->chan.d_uc, P->chan.d_gt})
        if (p) cudaFree(p);
    P->chan = ChanPlan();
}

}  // namespace dr

// For the parity tests (not part of the public header): run the automatic
// forward of this plan on the channel kernel whatever the timing says (the
// operator calls; admm: the solvers', in place of the fold in two kernels).  Returns DR_EINVAL where the kernel does not take the plan.
extern "C" dr_status dr_internal_use_channels(dr_plan *P, int admm) {
    if (!P || !P->chan.V) return dr::fail(DR_EINVAL, "no channel kernel for this plan");
    if (admm) {
        P->chan.eo = 1;
        P->sel_fwd = 2;
        P->sel_adj = P->solver_adj = 1;
    } else {
        P->chan.fwd = P->chan.fwd_st = 1;
    }
    P->tuned = true;
    return DR_OK;
}
