// od_noalloc.cu -- od_jacobi_noalloc: Jacobi iterations on a caller's padded
// field without allocating any device memory.
//
// Some callers cannot allocate device memory where they call this library: a
// host framework that owns every byte of device memory through its own pool
// and forbids allocations it does not track, or a latency-critical loop in
// which cudaMalloc / cudaFree would synchronise the device.  This entry point
// serves them: the caller passes the input field and the output field, and the
// one piece of scratch the iteration needs -- the second buffer of the double
// buffer -- is a file-scope static device array of fixed size that the
// module holds on every GPU that loads this library, until the process exits.
//
// It is a variant of the fused step kernel (one chare covering the whole
// grid, the same update, so the same bits), over the caller's plain padded
// layout instead of the context arena.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "od.h"
#include "od_arith.cuh"
#include "od_words.cuh"

namespace od {
od_status set_last_error(od_status s, const std::string &msg);  // od_api.cu
}  // namespace od

namespace {

// 64 MiB of doubles: padded grids up to 8 Mi cells, e.g. 200^3 interior.
constexpr int64_t kScratchDoubles = OD_NOALLOC_MAX_PADDED_CELLS;
static __device__ __align__(256) double g_scratch[kScratchDoubles];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
double *g_scratch_ptr[kMaxDevices] = {nullptr};
od_status set_error(od_status s, const std::string &m) { return od::set_last_error(s, m); }

// One step over the interior of a padded field (x fastest, row length nx+2):
// the same update as the fused tile kernel (arithmetic mode 2).  The padded
// grid holds at most OD_NOALLOC_MAX_PADDED_CELLS (2^23) cells, so every index
// fits 32 bits; threads run along x, blocks along y (grid y) and z (grid z),
// striding when a grid axis is shorter than the field's, so no index needs
// a division.
__global__ void k_noalloc_step(const double *__restrict__ src, double *__restrict__ dst, uint32_t nx, uint32_t ny,
                               uint32_t nz) {
    const uint32_t sx = nx + 2u, sxy = sx * (ny + 2u);
    for (uint32_t k = blockIdx.z; k < nz; k += gridDim.z)
        for (uint32_t j = blockIdx.y; j < ny; j += gridDim.y) {
            const uint32_t row = (k + 1u) * sxy + (j + 1u) * sx + 1u;
            for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nx; i += gridDim.x * blockDim.x) {
                const uint32_t c = row + i;
                dst[c] = od::jacobi_update<2>(src[c - 1u], src[c + 1u], src[c - sx], src[c + sx], src[c - sxy],
                                              src[c + sxy]);
            }
        }
}

// The same over fixed-point words (od_arith.cuh), for calls of several steps:
// the field is turned into words once (two passes over it) and the last step
// writes doubles.  A thread owns two cells of the plane, 256 apart in row-major
// order, and sweeps them through a chunk of planes, so neighbouring planes are
// found in L1; consecutive threads take consecutive cells whatever the row
// length, so no lane is lost to ragged rows.  Bound by the integer ALU and L1:
// 198^3, 20 steps: 1.52 ms with k_noalloc_step, 0.84 with this, whole calls (35 us
// a step, 219 G updates/s).  Four cells a thread measured 0.94, one 0.98.
constexpr int kCells = 2, kBlock = 256;

__device__ unsigned long long g_vmax;  // bit pattern of the input's largest positive finite value

__global__ void k_noalloc_reset() { g_vmax = 0; }

__global__ void k_noalloc_max(const double *__restrict__ u, uint32_t n) {
    unsigned long long m = 0;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const unsigned long long b = od::f64_bits(u[i]);
        if (b < 0x7FF0000000000000ull && b > m) m = b;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xFFFFFFFFu, m, o);
        m = w > m ? w : m;
    }
    if ((threadIdx.x & 31) == 0 && m) atomicMax(&g_vmax, m);
}

// Words of the whole input into `all` and of its Dirichlet shell into `shell`.
__global__ void k_noalloc_encode(const double *__restrict__ u, double *__restrict__ all, double *__restrict__ shell,
                                 uint32_t nx, uint32_t ny, uint32_t nz) {
    const uint32_t base = od::fx_anchor(g_vmax), sx = nx + 2u, rows = (ny + 2u) * (nz + 2u);
    for (uint32_t r = blockIdx.x; r < rows; r += gridDim.x) {
        const uint32_t j = r % (ny + 2u), k = r / (ny + 2u);
        const bool edge = j == 0u || j == ny + 1u || k == 0u || k == nz + 1u;
        for (uint32_t i = threadIdx.x; i < sx; i += blockDim.x) {
            const uint32_t c = r * sx + i;
            const double w = od::f64_from(od::fx_encode(u[c], base));
            all[c] = w;
            if (edge || i == 0u || i == sx - 1u) shell[c] = w;
        }
    }
}

__global__ void __launch_bounds__(kBlock, 4)
    k_noalloc_words(const double *__restrict__ src, double *__restrict__ dst, uint32_t nx, uint32_t cells, uint32_t sx,
                    uint32_t sxy, uint32_t nz, uint32_t chunk) {
    const uint32_t base = od::fx_anchor(g_vmax);
    int rf[kCells];
#pragma unroll
    for (int m = 0; m < kCells; ++m) {
        const uint32_t q0 = blockIdx.x * (kCells * kBlock) + m * kBlock + threadIdx.x;
        const uint32_t q = q0 < cells ? q0 : 0u;  // past the end: cell 0 again, the same value to the same place
        rf[m] = (int)((q / nx + 1u) * sx + q % nx + 1u);
    }
    const uint32_t k0 = blockIdx.y * chunk, k1 = min(k0 + chunk, nz);
    for (uint32_t k = k0; k < k1; ++k) {
        const double *p = src + (size_t)k * sxy;
        od::tile::words_plane<kCells, OD_STENCIL_3D7, false>(p, p + sxy, p + 2u * sxy, dst + (size_t)(k + 1u) * sxy, rf,
                                                      (int)sx, base);
    }
}

// The result's words to doubles, its shell from the input.
__global__ void k_noalloc_decode(const double *__restrict__ u, double *__restrict__ out, uint32_t nx, uint32_t ny,
                                 uint32_t nz) {
    const uint32_t base = od::fx_anchor(g_vmax), sx = nx + 2u, rows = (ny + 2u) * (nz + 2u);
    for (uint32_t r = blockIdx.x; r < rows; r += gridDim.x) {
        const uint32_t j = r % (ny + 2u), k = r / (ny + 2u);
        const bool edge = j == 0u || j == ny + 1u || k == 0u || k == nz + 1u;
        for (uint32_t i = threadIdx.x; i < sx; i += blockDim.x) {
            const uint32_t c = r * sx + i;
            out[c] = edge || i == 0u || i == sx - 1u ? u[c] : od::fx_decode(od::f64_bits(out[c]), base);
        }
    }
}

// Device address of the static scratch array on the current device, looked
// up once per device (the symbol's name is only a host-side stand-in).
od_status scratch_for_current_device(double **out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return set_error(OD_ECUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return set_error(OD_EINVAL, "device ordinal out of range");
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_scratch_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_scratch);
        if (e != cudaSuccess || !p)
            return set_error(OD_ECUDA, std::string("cudaGetSymbolAddress(scratch): ") + cudaGetErrorString(e));
        g_scratch_ptr[dev] = (double *)p;
    }
    *out = g_scratch_ptr[dev];
    return OD_OK;
}


od_status noalloc_words(const double *u_in, double *u_out, double *scratch, int64_t nx, int64_t ny, int64_t nz,
                        int32_t iters, cudaStream_t st) {
    const uint32_t sx = (uint32_t)nx + 2u, sxy = sx * ((uint32_t)ny + 2u), n = sxy * ((uint32_t)nz + 2u);
    const uint32_t cells = (uint32_t)(nx * ny);
    // step t writes u_out when iters-1-t is even, so the last step lands there;
    // the input's words start in the buffer that step 0 reads
    double *first = (iters - 1) % 2 == 0 ? u_out : scratch, *start = first == u_out ? scratch : u_out;
    const uint32_t rows = ((uint32_t)ny + 2u) * ((uint32_t)nz + 2u);
    const uint32_t row_block = sx >= 256u ? 256u : sx > 64u ? 128u : 64u, row_grid = std::min<uint32_t>(rows, 65535u);
    k_noalloc_reset<<<1, 1, 0, st>>>();
    k_noalloc_max<<<std::min<uint32_t>((n + 1023u) / 1024u, 1216u), 256, 0, st>>>(u_in, n);
    k_noalloc_encode<<<row_grid, row_block, 0, st>>>(u_in, start, first, (uint32_t)nx, (uint32_t)ny, (uint32_t)nz);
    // chunks of planes: about four blocks for every one resident (4 per SM,
    // 152 SMs); half, twice and four times as many measured slower
    const uint32_t bx = (cells + kCells * kBlock - 1u) / (kCells * kBlock);
        const uint32_t want = std::max<uint32_t>(1u, 2432u / bx);
    const uint32_t chunk = ((uint32_t)nz + want - 1u) / want;
    const dim3 grid(bx, ((uint32_t)nz + chunk - 1u) / chunk);
    const double *src = start;
    for (int32_t t = 0; t < iters; ++t) {
        double *dst = ((iters - 1 - t) % 2 == 0) ? u_out : scratch;
        k_noalloc_words<<<grid, kBlock, 0, st>>>(src, dst, (uint32_t)nx, cells, sx, sxy, (uint32_t)nz, chunk);
        src = dst;
    }
    k_noalloc_decode<<<row_grid, row_block, 0, st>>>(u_in, u_out, (uint32_t)nx, (uint32_t)ny, (uint32_t)nz);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(OD_ECUDA, std::string("od_jacobi_noalloc: ") + cudaGetErrorString(e));
    return OD_OK;
}

}  // namespace

extern "C" OD_API od_status od_jacobi_noalloc(const double *u_in, double *u_out, int64_t nx, int64_t ny,
                                                int64_t nz, int32_t iters, void *stream) {
    if (!u_in || !u_out) return set_error(OD_EINVAL, "od_jacobi_noalloc: null field pointer");
    if (nx < 1 || ny < 1 || nz < 1 || iters < 0)
        return set_error(OD_EINVAL, "od_jacobi_noalloc: extents must be >= 1 and iters >= 0");
    if (nx > kScratchDoubles || ny > kScratchDoubles || nz > kScratchDoubles ||
        (nx + 2) * (ny + 2) > kScratchDoubles || (nx + 2) * (ny + 2) * (nz + 2) > kScratchDoubles)
        return set_error(OD_EINVAL, "od_jacobi_noalloc: padded grid (nx+2)(ny+2)(nz+2) exceeds the static scratch "
                                    "of " + std::to_string(kScratchDoubles) + " cells");
    const int64_t npad = (nx + 2) * (ny + 2) * (nz + 2);
    const size_t bytes = (size_t)npad * sizeof(double);
    const uintptr_t a0 = (uintptr_t)u_in, b0 = (uintptr_t)u_out;
    if (a0 < b0 + bytes && b0 < a0 + bytes)
        return set_error(OD_EINVAL, "od_jacobi_noalloc: input and output fields overlap");
    double *scratch = nullptr;
    od_status s = scratch_for_current_device(&scratch);
    if (s != OD_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    // Calls of several steps on a field that fills the GPU sweep words.  A step
    // takes 4.6 ps a cell then instead of 9.4, the conversions 6 ps a cell and
    // four launches; below a million cells a step is latency either way.
    // Measured, us: 198^3 x 2 208 with words, 211 without, x 3 243 / 284, x 20
    // 844 / 1520; 500 x 100 x 100 x 3 162 / 177; 64^3 x 20 151 / 144.
    const int64_t cells = nx * ny * nz;
    if (iters >= 3 && cells >= (1 << 20) && cells * (iters - 1) >= 6000000)
        return noalloc_words(u_in, u_out, scratch, nx, ny, nz, iters, st);
    // Both buffers start as the input, so both hold the Dirichlet shell and
    // nothing of an earlier call survives in the scratch.
    cudaError_t e = cudaMemcpyAsync(u_out, u_in, bytes, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess && iters > 1) e = cudaMemcpyAsync(scratch, u_in, bytes, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return set_error(OD_ECUDA, std::string("cudaMemcpyAsync: ") + cudaGetErrorString(e));
    const int block = 128;
    const dim3 grid((unsigned)std::min<int64_t>((nx + block - 1) / block, 64), (unsigned)std::min<int64_t>(ny, 65535),
                    (unsigned)std::min<int64_t>(nz, 65535));
    // step t writes u_out when iters-1-t is even, so the last step lands there
    const double *src = u_in;
    for (int32_t t = 0; t < iters; ++t) {
        double *dst = ((iters - 1 - t) % 2 == 0) ? u_out : scratch;
        k_noalloc_step<<<grid, block, 0, st>>>(src, dst, (uint32_t)nx, (uint32_t)ny, (uint32_t)nz);
        e = cudaGetLastError();
        if (e != cudaSuccess) return set_error(OD_ECUDA, std::string("k_noalloc_step: ") + cudaGetErrorString(e));
        src = dst;
    }
    return OD_OK;
}
