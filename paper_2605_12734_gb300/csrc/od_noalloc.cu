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
struct Statics {  // device addresses of the static arrays of a device
    double *scratch;
    uint32_t *chosen, *base;
};
Statics g_statics[kMaxDevices] = {};
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
// writes doubles.  The planes are cut into chunks, and the cells of a plane are
// dealt over threads in order, two 256 apart to each, which it sweeps through a
// chunk, so neighbouring planes are found in L1; consecutive threads take
// consecutive cells whatever the row length, and planes that would not fill
// their blocks' lanes share them, so few are lost.  Bound by the integer ALU
// and L1: 198^3, 20 steps: 1.52 ms with k_noalloc_step, 0.86 with this, whole
// calls (36 us a step, 216 G updates/s).  Four cells a thread measured 0.94, one
// 0.98.  Planes of 3 cells (3 x 1 x 400000, 20 steps) 2.27 ms with
// k_noalloc_step, 0.40 with this; with a chunk to each block 14.2.
constexpr int kCells = 2, kBlock = 256;
constexpr uint32_t kSms = od::kSms;

// Of a call, beside the static scratch: the bit pattern of the input's largest
// positive finite value and the blocks that have looked for it, both left at
// zero for the next call, and the format the sweep runs in, a base exponent or 0
// for doubles: chosen into g_base, copied to c_base, from which the sweep reads it
// through the constant cache (a load from g_base at the head of every block cost
// 198^3 a microsecond a step).
__device__ unsigned long long g_vmax;
__device__ uint32_t g_done, g_base;
__constant__ uint32_t c_base;

// 256 updates spread over the field (a Weyl sequence of the golden ratio): the
// lowest exponent of the six operands and the result in the low half (0xFFFF: all
// zero), whether one of them is no positive finite value, and whether the update
// stays in a window of its own.
constexpr uint32_t kNoWord = 1u << 31, kOwnWindow = 1u << 30;
__device__ uint32_t g_sample[256];

__device__ uint32_t sample_update(const double *u, uint32_t t, uint32_t nx, uint32_t ny, uint32_t nz) {
    const uint32_t sx = nx + 2u, sxy = sx * (ny + 2u), cells = nx * ny * nz;
    const uint32_t q = (uint32_t)(((uint64_t)((t + 1u) * 0x9E3779B9u) * cells) >> 32), r = q / nx;
    const double *c = u + (size_t)(r / ny + 1u) * sxy + (r % ny + 1u) * sx + (q - r * nx) + 1u;
    double x[7] = {c[-1], c[1], *(c - sx), c[sx], *(c - sxy), c[sxy], 0.0};
    bool own;
    od::jacobi_update_fast<2>(x[0], x[1], x[2], x[3], x[4], x[5], own);
    x[6] = od::jacobi_update_ieee<true>(x[0], x[1], x[2], x[3], x[4], x[5]);
    uint32_t low = 0xFFFFu, flags = own ? kOwnWindow : 0u;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        const uint64_t b = od::f64_bits(x[i]);
        const uint32_t e = (uint32_t)(b >> 52);
        if (b != 0u) low = min(low, e);
        if (e >= 0x7FFu) flags |= kNoWord;
    }
    return low | flags;
}

__global__ void __launch_bounds__(256) k_noalloc_max(const double *__restrict__ u, uint32_t nx, uint32_t ny, uint32_t nz) {
    const uint32_t n = (nx + 2u) * (ny + 2u) * (nz + 2u);
    if (blockIdx.x == 0) g_sample[threadIdx.x] = sample_update(u, threadIdx.x, nx, ny, nz);
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
    // The last block to finish chooses the format.  Words have one window for the
    // whole field and an update outside it costs about 2.6 times one inside;
    // doubles take a window for each update, the six operands within 8 binades, at
    // twice the cost, and 7.7 times where they are not (198^3, us a step: 36, 94,
    // 73, 277).  So a smooth field over many binades, or one with a single large
    // value, sweeps doubles, and a signed one words.  (20 steps of 198^3 from such a
    // field: 1.74 ms over words, 1.45 this way, 1.49 by k_noalloc_step.)
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&g_done, 1u) == gridDim.x - 1u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const uint32_t base = od::fx_anchor(*(volatile unsigned long long *)&g_vmax);
    const uint32_t sample = *(volatile uint32_t *)&g_sample[threadIdx.x];
    const int words = __syncthreads_count((sample & kNoWord) == 0u && (sample & 0xFFFFu) >= base);
    const int own = __syncthreads_count((sample & kOwnWindow) != 0u);
    if (threadIdx.x == 0) {
        g_base = 73 * own + 277 * (256 - own) < 36 * words + 94 * (256 - words) ? 0u : base;
        g_vmax = 0ull;
        g_done = 0u;
    }
}

// Every cell of the padded field: f(index, whether it is of the shell).  A row to
// a block at a time, or, where rows are short or few, the cells in order (FLAT).
template <bool FLAT, typename F>
__device__ __forceinline__ void each_cell(uint32_t sx, uint32_t sy, uint32_t sz, F f) {
    const uint32_t rows = sy * sz;
    auto edge = [&](uint32_t r) {
        const uint32_t j = r % sy, k = r / sy;
        return j == 0u || j == sy - 1u || k == 0u || k == sz - 1u;
    };
    if (FLAT) {
        for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < rows * sx; c += gridDim.x * blockDim.x) {
            const uint32_t r = c / sx, i = c - r * sx;
            f(c, i == 0u || i == sx - 1u || edge(r));
        }
        return;
    }
    for (uint32_t r = blockIdx.x; r < rows; r += gridDim.x) {
        const bool e = edge(r);
        for (uint32_t i = threadIdx.x; i < sx; i += blockDim.x) f(r * sx + i, e || i == 0u || i == sx - 1u);
    }
}

// Words of the whole input into `all` and of its Dirichlet shell into `shell`.
template <bool FLAT>
__global__ void k_noalloc_encode(const double *__restrict__ u, double *__restrict__ all, double *__restrict__ shell,
                                 uint32_t nx, uint32_t ny, uint32_t nz) {
    const uint32_t base = c_base;
    each_cell<FLAT>(nx + 2u, ny + 2u, nz + 2u, [&](uint32_t c, bool edge) {
        const double w = od::f64_from(od::fx_encode(u[c], base));
        all[c] = w;
        if (edge) shell[c] = w;
    });
}

// OWN: a block has one chunk of planes (block y) of `planes`, the last one fewer.
// Otherwise the cells of a plane times the chunks are dealt over the blocks in
// order, and the last chunk begins early enough for `planes` of them (planes that
// two chunks sweep get the same values from both).
template <bool OWN>
__global__ void __launch_bounds__(kBlock, 4)
    k_noalloc_words(const double *__restrict__ src, double *__restrict__ dst, uint32_t nx, uint32_t cells, uint32_t sx,
                    uint32_t sxy, uint32_t nz, uint32_t planes, uint32_t slots) {
    const uint32_t base = c_base;
    int rf[kCells];
#pragma unroll
    for (int m = 0; m < kCells; ++m) {
        const uint32_t s0 = blockIdx.x * (kCells * kBlock) + m * kBlock + threadIdx.x;
        const uint32_t s = s0 < slots ? s0 : 0u;  // past the end: slot 0 again, the same value to the same place
        const uint32_t c = OWN ? 0u : s / cells, q = OWN ? s : s - c * cells;
        rf[m] = (int)((q / nx + 1u) * sx + q % nx + 1u);
        if (!OWN) rf[m] += (int)(min(c * planes, nz - planes) * sxy);
    }
    const uint32_t k0 = OWN ? blockIdx.y * planes : 0u, k1 = OWN ? min(k0 + planes, nz) : planes;
    if (base == 0u) {  // doubles, as k_noalloc_step
#pragma unroll 1
        for (uint32_t k = k0; k < k1; ++k)
#pragma unroll
            for (int m = 0; m < kCells; ++m) {
                const double *c = src + (size_t)(k + 1u) * sxy + rf[m];
                dst[(size_t)(k + 1u) * sxy + rf[m]] =
                    od::jacobi_update<2>(c[-1], c[1], *(c - sx), c[sx], *(c - sxy), c[sxy]);
            }
        return;
    }
#pragma unroll 1
    for (uint32_t k = k0; k < k1; ++k) {
        const double *p = src + (size_t)k * sxy;
        od::tile::words_plane<kCells, OD_STENCIL_3D7, false>(p, p + sxy, p + 2u * sxy, dst + (size_t)(k + 1u) * sxy, rf,
                                                      (int)sx, base);
    }
}

// The result's words to doubles, its shell from the input.
template <bool FLAT>
__global__ void k_noalloc_decode(const double *__restrict__ u, double *__restrict__ out, uint32_t nx, uint32_t ny,
                                 uint32_t nz) {
    const uint32_t base = c_base;
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // (again: calls that overlapped, against the rules, may have left them)
        g_vmax = 0ull;
        g_done = 0u;
    }
    if (base == 0u) return;  // doubles, and the shell is there from the start
    each_cell<FLAT>(nx + 2u, ny + 2u, nz + 2u, [&](uint32_t c, bool edge) {
        out[c] = edge ? u[c] : od::fx_decode(od::f64_bits(out[c]), base);
    });
}

// Device addresses of the static arrays on the current device, looked up once
// per device (a symbol's name is only a host-side stand-in).
od_status statics_for_current_device(Statics *out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return set_error(OD_ECUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return set_error(OD_EINVAL, "device ordinal out of range");
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_statics[dev].scratch) {
        void *p[3] = {nullptr, nullptr, nullptr};
        e = cudaGetSymbolAddress(&p[0], g_scratch);
        if (e == cudaSuccess) e = cudaGetSymbolAddress(&p[1], g_base);
        if (e == cudaSuccess) e = cudaGetSymbolAddress(&p[2], c_base);
        if (e != cudaSuccess || !p[0] || !p[1] || !p[2])
            return set_error(OD_ECUDA, std::string("cudaGetSymbolAddress(scratch): ") + cudaGetErrorString(e));
        g_statics[dev] = {(double *)p[0], (uint32_t *)p[1], (uint32_t *)p[2]};
    }
    *out = g_statics[dev];
    return OD_OK;
}

od_status noalloc_words(const double *u_in, double *u_out, const Statics &dev, int64_t nx, int64_t ny, int64_t nz,
                        int32_t iters, cudaStream_t st) {
    const uint32_t sx = (uint32_t)nx + 2u, sxy = sx * ((uint32_t)ny + 2u), n = sxy * ((uint32_t)nz + 2u);
    const uint32_t cells = (uint32_t)(nx * ny);
    // step t writes u_out when iters-1-t is even, so the last step lands there;
    // the input's words start in the buffer that step 0 reads
    double *const scratch = dev.scratch;
    double *first = (iters - 1) % 2 == 0 ? u_out : scratch, *start = first == u_out ? scratch : u_out;
    const uint32_t rows = ((uint32_t)ny + 2u) * ((uint32_t)nz + 2u);
    // (100000 x 3 x 5, 35 rows: 20 steps 0.57 ms by rows, 0.30 in order; 1 x 5003 x
    // 211, rows of 3 cells: 0.62, 0.30)
    const bool flat = sx < 64u || rows < 8u * kSms;
    const uint32_t io_block = flat || sx >= 256u ? 256u : 128u;
    const uint32_t io_grid = flat ? std::min<uint32_t>((n + 255u) / 256u, 64u * kSms) : std::min<uint32_t>(rows, 65535u);
    k_noalloc_max<<<std::min<uint32_t>((n + 1023u) / 1024u, 8u * kSms), 256, 0, st>>>(u_in, (uint32_t)nx, (uint32_t)ny,
                                                                                      (uint32_t)nz);
    cudaError_t e = cudaMemcpyAsync(dev.base, dev.chosen, sizeof(uint32_t), cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return set_error(OD_ECUDA, std::string("cudaMemcpyAsync: ") + cudaGetErrorString(e));
    auto encode = flat ? k_noalloc_encode<true> : k_noalloc_encode<false>;
    auto decode = flat ? k_noalloc_decode<true> : k_noalloc_decode<false>;
    encode<<<io_grid, io_block, 0, st>>>(u_in, start, first, (uint32_t)nx, (uint32_t)ny, (uint32_t)nz);
    // chunks of planes: about four blocks for every one resident (4 per SM); half,
    // twice and four times as many measured slower.  A block has a chunk of its
    // own unless that leaves a sixteenth of the lanes idle (dealt in order, planes
    // of 4000 to 40000 cells ran up to 7 % slower).
    auto blocks = [](uint32_t m) { return (m + kCells * kBlock - 1u) / (kCells * kBlock); };
    const bool own = blocks(cells) * (kCells * kBlock) <= cells + cells / 16u;
    const uint32_t want = std::max<uint32_t>(1u, own ? 16u * kSms / blocks(cells) : 16u * kSms * kCells * kBlock / cells);
    const uint32_t planes = ((uint32_t)nz + want - 1u) / want, chunks = ((uint32_t)nz + planes - 1u) / planes;
    const uint32_t slots = own ? cells : cells * chunks;
    const dim3 grid(blocks(slots), own ? chunks : 1u);
    const double *src = start;
    for (int32_t t = 0; t < iters; ++t) {
        double *dst = ((iters - 1 - t) % 2 == 0) ? u_out : scratch;
        if (own)
            k_noalloc_words<true>
                <<<grid, kBlock, 0, st>>>(src, dst, (uint32_t)nx, cells, sx, sxy, (uint32_t)nz, planes, slots);
        else
            k_noalloc_words<false>
                <<<grid, kBlock, 0, st>>>(src, dst, (uint32_t)nx, cells, sx, sxy, (uint32_t)nz, planes, slots);
        src = dst;
    }
    decode<<<io_grid, io_block, 0, st>>>(u_in, u_out, (uint32_t)nx, (uint32_t)ny, (uint32_t)nz);
    e = cudaGetLastError();
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
    Statics dev = {};
    od_status s = statics_for_current_device(&dev);
    if (s != OD_OK) return s;
    double *const scratch = dev.scratch;
    cudaStream_t st = (cudaStream_t)stream;
    // Calls of several steps on a field that fills the GPU sweep words.  A step
    // takes 4.6 ps a cell then instead of 9.4, the conversions 6 ps a cell and
    // four launches; below a million cells a step is latency either way.
    // Measured, us: 198^3 x 2 208 with words, 211 without, x 3 234 / 283, x 20
    // 858 / 1506; 500 x 100 x 100 x 3 162 / 177; 64^3 x 20 151 / 144.  One plane
    // or two are mostly shell and find no plane again: 1100 x 1000 x 1 x 20 296 /
    // 280, 1400 x 1400 x 2 x 3 181 / 169, x 6 260 / 274.
    const int64_t cells = nx * ny * nz;
    if (iters >= (nz == 2 ? 6 : 3) && nz > 1 && cells >= (1 << 20) && cells * (iters - 1) >= 6000000)
        return noalloc_words(u_in, u_out, dev, nx, ny, nz, iters, st);
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
