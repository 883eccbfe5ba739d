// Launches of the FP32 pass kernels of one radius; the radii are built in
// several translation units (compile time).
#pragma once

#include "pass_impl.cuh"

namespace rpiv {

template <int RC, int GC>
static cudaError_t launch_shape(const PassArgs &a, dim3 grid, int smem, cudaStream_t st)
{
    pass_kernel<RC, PREC_FP32, GC><<<grid, PASS_THREADS, smem, st>>>(a);
    return cudaGetLastError();
}

template <int RC, int GC>
static cudaError_t launch_strip(const PassArgs &a, dim3 grid, int smem, cudaStream_t st)
{
    strip_kernel<RC, GC><<<grid, PASS_THREADS, smem, st>>>(a);
    return cudaGetLastError();
}

// Opts a kernel in to the full shared-memory carve-out (done once, outside any
// stream capture).
template <int RC, int GC>
static void prepare_shape()
{
    cudaFuncSetAttribute(pass_kernel<RC, PREC_FP32, GC>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

// Specialised shapes: 50 % overlap with blocks of 8, 12, 16, 24 or 32 pixels
// (16 to 64 px windows), whose window, step and block loops unroll.  Two 8 MP
// pairs at r = 6 against the kernel of any shape: 48 px windows 506 -> 445 us,
// 24 px 540 -> 427 us (306 and 293 M instead of 340 and 368 M warp instructions).
template <int RC>
cudaError_t launch_radius(const PassArgs &a, dim3 grid, int smem, cudaStream_t st);
template <int RC>
void prepare_radius();

#define RPIV_PASS_DECLARE(RC)                                                                \
    template <>                                                                              \
    cudaError_t launch_radius<RC>(const PassArgs &a, dim3 grid, int smem, cudaStream_t st);  \
    template <>                                                                              \
    void prepare_radius<RC>();
RPIV_PASS_DECLARE(1)
RPIV_PASS_DECLARE(2)
RPIV_PASS_DECLARE(3)
RPIV_PASS_DECLARE(4)
RPIV_PASS_DECLARE(6)
RPIV_PASS_DECLARE(8)

// strips are planned only for radii 1 and 4 with 16 and 32 px blocks
template <int RC>
constexpr bool has_strips() { return RC == 1 || RC == 4; }

#define RPIV_PASS_RADIUS(RC)                                                                             \
    template <>                                                                                          \
    cudaError_t launch_radius<RC>(const PassArgs &a, dim3 grid, int smem, cudaStream_t st)               \
    {                                                                                                    \
        return launch_radius_impl<RC>(a, grid, smem, st);                                                \
    }                                                                                                    \
    template <>                                                                                          \
    void prepare_radius<RC>()                                                                            \
    {                                                                                                    \
        prepare_radius_impl<RC>();                                                                       \
    }

template <int RC>
static cudaError_t launch_radius_impl(const PassArgs &a, dim3 grid, int smem, cudaStream_t st)
{
    const int G = a.plan.G;
    if (a.plan.strip_rows > 0) {
        if constexpr (has_strips<RC>()) {
            if (G == 16) return launch_strip<RC, 16>(a, grid, smem, st);
            if (G == 32) return launch_strip<RC, 32>(a, grid, smem, st);
        }
        return cudaErrorInvalidValue;
    }
    if (a.w == 2 * G && a.s == G) {
        switch (G) {
        case 8: return launch_shape<RC, 8>(a, grid, smem, st);
        case 12: return launch_shape<RC, 12>(a, grid, smem, st);
        case 16: return launch_shape<RC, 16>(a, grid, smem, st);
        case 24: return launch_shape<RC, 24>(a, grid, smem, st);
        case 32: return launch_shape<RC, 32>(a, grid, smem, st);
        default: break;
        }
    }
    // the unrolled loops of the usual blocks apart from the rest: in one kernel they spilled, and
    // blocks of 4 px paid 3 to 7 % for them and their order of the units (16 px at 75 %, r = 4,
    // 16 pairs of 1 MP: 1110 us apart, 1159 in one)
    if (fp32_usual_blocks(G)) return launch_shape<RC, BLOCKS_USUAL>(a, grid, smem, st);
    return launch_shape<RC, BLOCKS_ANY>(a, grid, smem, st);
}

template <int RC>
static void prepare_radius_impl()
{
    prepare_shape<RC, BLOCKS_ANY>();
    prepare_shape<RC, BLOCKS_USUAL>();
    prepare_shape<RC, 8>();
    prepare_shape<RC, 12>();
    prepare_shape<RC, 16>();
    prepare_shape<RC, 24>();
    prepare_shape<RC, 32>();
    if constexpr (has_strips<RC>()) {
        cudaFuncSetAttribute(strip_kernel<RC, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        cudaFuncSetAttribute(strip_kernel<RC, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    }
}

}  // namespace rpiv
