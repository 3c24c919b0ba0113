// chan.cuh -- shared declarations of the channel-lane folded forward
// (chan_fwd.cu).
//
// A volume of nz slices with m coefficients is nz m independent images that
// all see the same ray geometry.  The kernels of fold_impl.cuh give a thread
// whole rays and let the lanes of a warp differ in geometry; every Joseph
// sample then reads two pixel vectors from shared memory, 4 bytes per
// multiply-add, and pays its own index arithmetic.  Here the lanes of a warp
// are 32 V of those images ("channels", V = 1, 2 or 4 per lane) and the
// geometry is uniform across the warp: a warp streams along an image line,
// keeps the two current pixels in registers and reads each pixel once for all
// the rays it takes part in, so a sample costs about 1.2 reads instead of 2,
// without bank conflicts, and the index arithmetic is paid once per 32 V
// channels.
#pragma once

#include "dr_device.cuh"

namespace dr {

__host__ __device__ __forceinline__ size_t row_at(const RowMap &r, int z, size_t ab) {
    return (size_t)(z / r.spb) * r.blk + ab * r.C + (size_t)(z % r.spb) * r.ms;
}
// Static transforms: where they are, their rows, and the line chunks whose
// partial sums (split_stride floats apart) the consumer adds.
struct StaticOut {
    void *ru;
    RowMap rows;
    int nsplit;
    size_t split_stride;
};

// forward variant of automatic operator calls, where the autotuner found it faster
constexpr int kVarChan = 3;
// the same kernel in the summation order, and with the line chunks, of the fold
// in two kernels, whose values it then gives bit for bit (the solvers)
constexpr int kVarChanEO = 4;
inline int fold2_chunks(const dr_plan *P) { return P->split_off ? 1 : (P->fold2_split > 1 ? P->fold2_split : 1); }
constexpr int kChanWarps = 16;  // compute warps per CTA, at most (8: two CTAs per SM); one more copies
constexpr int kChanSlots = 8;   // line buffers in flight, at most
constexpr int kChanBox = 8;     // pixels per TMA box
// bytes of line buffers of a CTA of nw compute warps
__host__ __device__ constexpr int chan_ring(int nw) { return (nw == 8 ? 108 : 216) * 1024; }
constexpr int kChanMin = 32;                // least channels (nz times m rounded up to 4) that the kernels take
constexpr size_t kChanScratchMax = size_t(1) << 30;  // packed volume held at a time
// rays per warp: 64 sums per lane at V = 2 and 4, 32 at V = 1
__host__ __device__ constexpr int chan_rw(int V) { return V == 4 ? 16 : 32; }
__host__ __device__ constexpr int chan_boxes(int px) { return (px + kChanBox - 1) / kChanBox; }

size_t split_bytes(const dr_plan *P);  // partial sums that the plan's choices need (projector.cu)
dr_status chan_setup(dr_plan *P, const std::vector<FwdProj> &fw);
bool chan_split_fits(const dr_plan *P, int nsplit);
bool chan_fwd_ready(dr_plan *P, int nsplit, cudaStream_t st);
// static transforms of u (bf: stored bf16, else float); chan_fwd_ready must hold
// (eo: each sample's even pixel first, the order of the thread-per-ray kernels)
dr_status chan_static(dr_plan *P, const void *u, bool bf, bool eo, int nsplit, cudaStream_t st, StaticOut &rs);
void chan_release(dr_plan *P);
void chan_free(dr_plan *P);

inline RowMap slice_rows(size_t rows_per_slice, int ms) { return RowMap{1, ms, ms, rows_per_slice * ms}; }

}  // namespace dr
