// kernels.cu -- launcher of the tiled BMMC pass kernel for sm_103a.
//
// The tiled pass of Sec. 4.1-4.3 (the tiled BMMC of Sec. 5.1, and each of the
// two passes of Sec. 5.2).  One thread block moves 2^it tiles of one pass; the body (cp.async tile
// load into swizzled shared memory, barrier, 16-byte gathers and stores) is
// dev::run_tile in tile_body.cuh, shared with the persistent batch kernel.
// KEY selects an optional comparator epilogue (a column of compare-exchanges
// on output pairs, for sorting networks built from permutations).
#include <cuda.h>  // CUtensorMap and its encoding function's types
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "pass_desc.h"
#include "tile_body.cuh"

namespace bmmc {

namespace {

// Element size 2^E_LOG bytes; one block per thread-block index of the pass and
// per row: row r of the launch is the array `r * row_bytes` bytes further on.
// A count of rows that is a power of two is better folded into the pass
// (bmmc_plan_lift: whole tiles even where a row is small); the odd factor of
// any other count is gridDim.y.  24 rows of 2^16 floats, permuted there and
// back (parm): 636 us with a launch per row, 60 us with one launch
// each way.
template <int E_LOG, int KEY>
__global__ void __launch_bounds__(256)
    bmmc_tiled_pass(const __grid_constant__ PassDesc d, const uint8_t *__restrict__ in,
                    uint8_t *__restrict__ out, uint64_t row_bytes)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    const uint64_t row = blockIdx.y * row_bytes;
    dev::run_tile<E_LOG, KEY>(d, blockIdx.x, in + row, out + row, sbase);
}

// Bounded waits of the tensor-copy kernel that gave up (read by
// bmmc_device_wait_timeouts).
__device__ unsigned long long g_wait_timeouts;

// The same pass with phase 1 by tensor copies (PassDesc::tma): one copy per
// input segment through `tmap`, a 2-D map of the input array as 128-byte lines
// with the hardware 128-byte swizzle.  The tile starts on a 1 KiB boundary
// (the swizzle pattern repeats every 1 KiB of shared memory) and the mbarrier
// of the copies follows it.  If the copies have not all landed after about a
// second the block counts a timeout, waits once more and returns without
// writing (no trap, no endless wait).
template <int E_LOG, int KEY>
__global__ void __launch_bounds__(256)
    bmmc_tiled_pass_tma(const __grid_constant__ PassDesc d,
                        const __grid_constant__ CUtensorMap tmap, uint8_t *__restrict__ out)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sraw = (uint32_t)__cvta_generic_to_shared(smem);
    const uint32_t sbase = (sraw + 1023u) & ~1023u;
    const uint32_t bar = sbase + d.smem_bytes;
    const dev::TileAddr a = dev::tile_addr(d, blockIdx.x);
    if (threadIdx.x == 0) dev::mbar_init(bar, 1);
    __syncthreads();
    dev::grid_dependency_wait();
    dev::allow_dependent_launch();
    if (!dev::tile_load_tma<E_LOG>(d, &tmap, blockIdx.x, sbase, bar)) {
        if (threadIdx.x == 0) atomicAdd(&g_wait_timeouts, 1ull);
        dev::mbar_wait_bounded(bar, 0);
        return;
    }
    dev::tile_store<E_LOG, KEY>(d, a, out, sbase);
}

// Arrays under 1 KiB: one block per row, one thread per element, direct index
// map.
template <int E_LOG, int KEY>
__global__ void bmmc_naive_pass(const __grid_constant__ PassDesc d,
                                const uint8_t *__restrict__ in, uint8_t *__restrict__ out,
                                uint64_t row_bytes)
{
    dev::grid_dependency_wait();
    dev::allow_dependent_launch();
    const uint64_t row = blockIdx.x * row_bytes;
    dev::run_naive<E_LOG, KEY>(d, in + row, out + row);
}

constexpr int kMaxDevices = 64;
constexpr uint64_t kMaxRows = 65535;  // gridDim.y
constexpr int kSmemLimit = 128 * 1024;
constexpr int kSmemLimitTma = kSmemLimit + 2048;  // 1 KiB alignment + mbarrier
// Per device, element size and key: the kernel's shared-memory limit has
// been raised.  Atomic because plans may be executed from several threads;
// two threads raising it at once both set the same value.
std::atomic<bool> g_attr_set[kMaxDevices][3][7];
std::atomic<bool> g_attr_set_tma[kMaxDevices][3][7];

// cuTensorMapEncodeTiled, from the driver through the runtime (no link
// against the driver library); NULL if unavailable.
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                   const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                   const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

// The input array as a 2-D tensor of 128-byte lines (32 words each), boxes
// of one segment (seg_lines lines), 128-byte swizzle.
bool encode_lines_map(CUtensorMap *m, const void *in, uint64_t bytes, uint32_t seg_lines)
{
    const EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {32, bytes / 128};
    const cuuint64_t strides[1] = {128};
    const cuuint32_t box[2] = {32, seg_lines};
    const cuuint32_t elem_strides[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<void *>(in), dims, strides, box,
              elem_strides, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Every launch allows programmatic dependent launch: the kernels wait on the
// grid dependency before their first global memory access, so a pass may be
// scheduled while the previous kernel of the stream drains.
template <typename... Args>
cudaError_t launch_pdl(void (*kernel)(Args...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t s, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// rows <= kMaxRows (1 for tensor copies, whose map covers one array).
template <int E_LOG, int KEY>
cudaError_t launch_typed(const PassDesc &d, const void *in, void *out, uint32_t rows,
                         cudaStream_t s)
{
    const uint8_t *src = static_cast<const uint8_t *>(in);
    uint8_t *dst = static_cast<uint8_t *>(out);
    const uint64_t row_bytes = ((uint64_t)1 << d.n) << E_LOG;
    if (d.naive)
        return launch_pdl(bmmc_naive_pass<E_LOG, KEY>, dim3(rows), dim3(1u << d.n), 0, s, d, src,
                          dst, row_bytes);
    // Tiles within the default 48 KiB of dynamic shared memory (the default
    // 16 KiB ones) need no attribute, and so no device lookup per launch.
    constexpr uint32_t kDefaultSmem = 48 * 1024;
    int dev = 0;
    cudaError_t err = cudaSuccess;
    const bool needs_attr = d.smem_bytes + (d.tma ? 1024u + 16u : 0u) > kDefaultSmem;
    if (needs_attr) {
        err = cudaGetDevice(&dev);
        if (err != cudaSuccess) return err;
    }
    if (d.tma) {
        CUtensorMap tmap;
        if (encode_lines_map(&tmap, in, row_bytes, 1u << (d.k + E_LOG - 7))) {
            if (needs_attr && dev >= 0 && dev < kMaxDevices &&
                !g_attr_set_tma[dev][E_LOG - 2][KEY].load(std::memory_order_acquire)) {
                err = cudaFuncSetAttribute(bmmc_tiled_pass_tma<E_LOG, KEY>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           kSmemLimitTma);
                if (err != cudaSuccess) return err;
                g_attr_set_tma[dev][E_LOG - 2][KEY].store(true, std::memory_order_release);
            }
            return launch_pdl(bmmc_tiled_pass_tma<E_LOG, KEY>, dim3(1u << d.n_cta),
                              dim3(1u << d.thread_bits), (size_t)d.smem_bytes + 1024 + 16, s, d,
                              tmap, dst);
        }
        // no tensor-map encoder: the same tables through 16-byte copies
    }
    if (needs_attr && dev >= 0 && dev < kMaxDevices &&
        !g_attr_set[dev][E_LOG - 2][KEY].load(std::memory_order_acquire)) {
        err = cudaFuncSetAttribute(bmmc_tiled_pass<E_LOG, KEY>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
        if (err != cudaSuccess) return err;
        g_attr_set[dev][E_LOG - 2][KEY].store(true, std::memory_order_release);
    }
    return launch_pdl(bmmc_tiled_pass<E_LOG, KEY>, dim3(1u << d.n_cta, rows),
                      dim3(1u << d.thread_bits), d.smem_bytes, s, d, src, dst, row_bytes);
}

}  // namespace

// key: 0 (plain permutation) or a bmmc_key_type value matching the element
// size (1..3 for 4-byte, 4..6 for 8-byte elements).  rows: arrays one after
// another, each permuted alike.
cudaError_t launch_pass(const PassDesc &d, const void *in, void *out, cudaStream_t s, int key,
                        uint64_t rows)
{
    using namespace dev;
    auto launch = [&](const void *src, void *dst, uint32_t r) {
        switch (d.e_log) {
        case 2:
            switch (key) {
            case kKeyNone: return launch_typed<2, kKeyNone>(d, src, dst, r, s);
            case kKeyI32: return launch_typed<2, kKeyI32>(d, src, dst, r, s);
            case kKeyU32: return launch_typed<2, kKeyU32>(d, src, dst, r, s);
            case kKeyF32: return launch_typed<2, kKeyF32>(d, src, dst, r, s);
            default: return cudaErrorInvalidValue;
            }
        case 3:
            switch (key) {
            case kKeyNone: return launch_typed<3, kKeyNone>(d, src, dst, r, s);
            case kKeyI64: return launch_typed<3, kKeyI64>(d, src, dst, r, s);
            case kKeyU64: return launch_typed<3, kKeyU64>(d, src, dst, r, s);
            case kKeyF64: return launch_typed<3, kKeyF64>(d, src, dst, r, s);
            default: return cudaErrorInvalidValue;
            }
        case 4:
            if (key != kKeyNone) return cudaErrorInvalidValue;
            return launch_typed<4, kKeyNone>(d, src, dst, r, s);
        default: return cudaErrorInvalidValue;
        }
    };
    const uint64_t row_bytes = ((uint64_t)1 << d.n) << d.e_log;
    const uint64_t step = d.tma ? 1 : kMaxRows;
    for (uint64_t r = 0; r < rows; r += step) {
        const cudaError_t err =
            launch(static_cast<const uint8_t *>(in) + r * row_bytes,
                   static_cast<uint8_t *>(out) + r * row_bytes,
                   (uint32_t)(rows - r < step ? rows - r : step));
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

// Number of bounded waits of tensor-copy kernels that gave up on the current
// device since the library was loaded (0 when nothing went wrong).
cudaError_t device_wait_timeouts(unsigned long long *count)
{
    return cudaMemcpyFromSymbol(count, g_wait_timeouts, sizeof(*count));
}

}  // namespace bmmc
