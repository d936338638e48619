// od_kernels.h -- launch wrappers for libod's device kernels (host side).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "od_internal.h"

namespace od {

// Tile kernels exist for (threads, cells per thread) in {128}x{2,4,8},
// {256}x{1,2,4,8}, {512}x{1,2}, arithmetic modes 0..15 (and 16, mode 12 over
// fixed-point field words) and both stencils
// (OD_STENCIL_3D7, OD_STENCIL_2D5) (od_tile.cuh).
bool tile_shape_supported(int threads, int cpt, int amode, int stencil);

// Raise the dynamic shared-memory limit of the tile kernels of one shape.
cudaError_t prepare_tile_kernels(int threads, int cpt, int amode, int smem_bytes, int stencil);

// The tiles [a.tile_begin, a.tile_begin + tiles) of stencil a.stencil (so for
// launch_persistent), one CTA per tile; the kernels over fixed-point words
// take several tiles per CTA when there are more than `resident` CTAs (what
// the GPU holds at once; 0: one per tile).  push = 1: a fused step, whose
// tiles read the faces of their neighbours' arrays.
cudaError_t launch_tiles(const KArgs &a, int tiles, int threads, int cpt, int amode, bool push, int smem_bytes,
                         int resident, cudaStream_t s);

// One fused step of several jobs (continuous batching): jobs[j] (device
// array) is job j's KArgs with its source parity, first[j] its first block
// (device array of njobs+1 prefix sums, first[njobs] = grid); geom (host)
// carries the launch's ring geometry and wait limit: stages, stage_doubles
// (at least every job's) and spin_ns.
cudaError_t launch_tiles_multi(const KArgs *jobs, const int32_t *first, int32_t njobs, const KArgs &geom, int grid,
                               int threads, int cpt, int amode, int smem_bytes, int stencil, cudaStream_t s);

// Several fused steps of several jobs in one persistent launch: jobs[j]
// (device array) carries job j's tables, its absolute first step (t0) and
// its steps in this launch (iters <= steps); first[] as for
// launch_tiles_multi; queue a zeroed device counter.
cudaError_t launch_persistent_multi(const KArgs *jobs, const int32_t *first, int32_t njobs, int32_t steps,
                                    int32_t *queue, const KArgs &geom, int grid, int threads, int cpt, int amode,
                                    int smem_bytes, int stencil, cudaStream_t s);

// Persistent ticket kernel over a.iters steps.
cudaError_t launch_persistent(const KArgs &a, int grid, int threads, int cpt, int amode, int smem_bytes,
                              cudaStream_t s);
cudaError_t persistent_occupancy(int threads, int cpt, int amode, int smem_bytes, int stencil,
                                 int *blocks_per_sm);
cudaError_t tiles_occupancy(int threads, int cpt, int amode, int smem_bytes, int stencil, int *blocks_per_sm);
cudaError_t persistent_multi_occupancy(int threads, int cpt, int amode, int smem_bytes, int stencil,
                                       int *blocks_per_sm);

// The tiles' records for the sweep over words, from the tables (TileRec).
cudaError_t launch_tile_recs(const ChareDev *ch, const TileDev *tiles, int64_t ntiles, const int32_t *dep_ptr,
                             const int32_t *dep_idx, TileRec *rec, int stencil, cudaStream_t s);

// Every call below that moves field values between a context's arrays and a
// buffer of doubles takes the context's format word (FmtDev).

// The initial field, written in format `base` (0: plain doubles), of a shard at offset (gx0, gy0, gz0) of a global grid
// gnx x gny x gnz (the whole grid: offsets 0, global = local extents).
cudaError_t launch_init(const ChareDev *ch, int nch, int64_t gnx, int64_t gny, int64_t gnz, int64_t gx0,
                        int64_t gy0, int64_t gz0, uint64_t seed, int mode, int stencil, uint32_t base,
                        cudaStream_t s);
// Domain-face exchange of a shard (od_face_copy) of px x py x pz chares: dir 0
// copies the boundary layer of parity p on face f into buf, dir 1 buf into the
// ghost layer.  vmax (null: the context never holds fixed-point words): an
// import raises it to the face's largest value; *wider (mapped host memory) is
// set to 1 when the field should take another format (launch_refit).
cudaError_t launch_face_copy(const ChareDev *ch, int px, int py, int pz, int parity, int face, int dir, double *buf,
                             int64_t nx, int64_t ny, int64_t nz, uint64_t *vmax, FmtDev *fmt, uint32_t *wider,
                             cudaStream_t s);
cudaError_t launch_pack(const ChareDev *ch, int c, int parity, int elems, cudaStream_t s);
cudaError_t launch_unpack(const ChareDev *ch, int c, int parity, int slot, int elems, cudaStream_t s);
// out[i] = *addr[i] for n device addresses (od_read_cells).
cudaError_t launch_read_cells(const double *const *addr, int64_t n, double *out, const FmtDev *fmt, cudaStream_t s);
// Export; with err (device record, may be null) only if no launch before it failed.
cudaError_t launch_gather(const ChareDev *ch, int nch, int parity, int64_t nx, int64_t ny, double *g,
                          const FmtDev *fmt, const ErrDev *err, cudaStream_t s);
// Arithmetic self-test over device arrays (op: 0 div6, 1 add on the integer
// pipes; 2 division by 6, 3 add on the FP64 pipe).
cudaError_t launch_arith(int op, const double *a, const double *b, double *out, int64_t n, cudaStream_t s);
// Import (od_write): also raises *vmax (device word, may be null) to the
// bit pattern of the largest positive finite value written; words = true
// (the context may hold fixed-point words): the field then takes a wider
// format if that value asks for it.
cudaError_t launch_scatter(const ChareDev *ch, int nch, int parity, int64_t nx, int64_t ny, int64_t nz,
                           const double *g, uint64_t *vmax, FmtDev *fmt, bool words, cudaStream_t s);
// The field takes the format that *vmax asks for, if it has another.
cudaError_t launch_refit(const ChareDev *ch, int nch, int parity, int64_t nx, int64_t ny, const uint64_t *vmax,
                         FmtDev *fmt, cudaStream_t s);
// Internal ghost layers of parity `parity` from the neighbours' boundaries.
cudaError_t launch_ghost_refresh(const ChareDev *ch, int nch, int parity, cudaStream_t s);

}  // namespace od
