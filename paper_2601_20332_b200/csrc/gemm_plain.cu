// CUDA-core GEMM: y[rows, n] = x[rows, k] * w[n, k]^T for any dtype, fp32 multiply and accumulate.  The fp32 models run
// on it entirely; for bf16 it is the cross-check of the tensor-core kernels.  Up to three weight matrices that share
// the input (q/k/v; gate/up) go in one launch, their outputs side by side.
#include <algorithm>
#include <type_traits>

#include "wd_internal.h"
#include "device_utils.cuh"

namespace {

using namespace wdk;

struct Segs {
    const void* w[3];
    int end[3];                     // output columns up to and including matrix i
};

template <typename T> __device__ __forceinline__ float4 ld4(const T* p);
template <> __device__ __forceinline__ float4 ld4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <> __device__ __forceinline__ float4 ld4<__nv_bfloat16>(const __nv_bfloat16* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ float ld1(const float* p) { return *p; }
__device__ __forceinline__ float ld1(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// one element's bits (zero where !ok), and the float they are.  Loads by hand: written as a conditional load of 16 bits, the value
// was merged with the zero at once, which waits for it.
template <typename T> struct Raw;
template <> struct Raw<float> {
    using type = uint32_t;
    static __device__ __forceinline__ type load(const float* p, bool ok) {
        type v;
        asm volatile("{\n.reg .pred q;\nsetp.ne.u32 q, %2, 0;\nmov.b32 %0, 0;\n@q ld.global.b32 %0, [%1];\n}" : "=r"(v) : "l"(p), "r"(ok ? 1u : 0u));
        return v;
    }
    static __device__ __forceinline__ float value(type v) { return __uint_as_float(v); }
};
template <> struct Raw<__nv_bfloat16> {
    using type = uint16_t;
    static __device__ __forceinline__ type load(const __nv_bfloat16* p, bool ok) {
        type v;
        asm volatile("{\n.reg .pred q;\nsetp.ne.u32 q, %2, 0;\nmov.b16 %0, 0;\n@q ld.global.b16 %0, [%1];\n}" : "=h"(v) : "l"(p), "r"(ok ? 1u : 0u));
        return v;
    }
    static __device__ __forceinline__ float value(type v) { return __uint_as_float((uint32_t)v << 16); }
};

// row of the concatenated weights that makes output column c
template <typename T>
__device__ __forceinline__ const T* weight_row(const Segs& s, int c, int k) {
    if (c < s.end[0]) return (const T*)s.w[0] + (size_t)c * k;
    if (c < s.end[1]) return (const T*)s.w[1] + (size_t)(c - s.end[0]) * k;
    return (const T*)s.w[2] + (size_t)(c - s.end[1]) * k;
}

// four elements from position kk of a row of k (zeros beyond); kVec: the row is aligned for one vector load
template <typename T, bool kVec>
__device__ __forceinline__ float4 ld_row4(const T* p, int kk, int k) {
    if (kVec) return kk < k ? ld4<T>(p + kk) : make_float4(0.f, 0.f, 0.f, 0.f);
    return make_float4(kk < k ? ld1(p + kk) : 0.f, kk + 1 < k ? ld1(p + kk + 1) : 0.f, kk + 2 < k ? ld1(p + kk + 2) : 0.f,
                       kk + 3 < k ? ld1(p + kk + 3) : 0.f);
}

// Few rows: the product is as long as its chain of memory round trips, so there is no shared memory, no barrier and no
// loop over K tiles that waits for each.  A warp makes a [8 rows x 4 columns] piece of the result: its lanes split K
// (four consecutive elements each, NC * 128 elements at a time), so every load is a full line, and the 32 sums of a
// lane are reduced over the warp by halving (31 shuffles leave one finished value in each lane).  The weights of the
// first NC * 128 elements are in registers before the dependency wait.  Bound by latency up to about a hundred rows, then by
// the loads from L1 (17 TFLOP/s).  Measured, 768 columns, k = 256: 2.3 us at 9 rows, 2.9 at 64; a [32 x 64]-tile kernel with
// K tiles of 32 through shared memory, a barrier on either side of each, took 19 us at 9 rows.
template <typename T, int NC, bool kVec>
__global__ void __launch_bounds__(128)
gemm_rows_kernel(const T* __restrict__ x, const Segs segs, float* __restrict__ y, int rows, int n, int k, int ldy, int w_static) {
    constexpr int kC = 4, kR = 8;
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, col0 = (int)(blockIdx.x * 4 + (threadIdx.x >> 5)) * kC, row0 = (int)blockIdx.y * kR;
    if (col0 >= n) return;
    const T* wp[kC];
#pragma unroll
    for (int c = 0; c < kC; ++c) wp[c] = weight_row<T>(segs, min(col0 + c, n - 1), k);
    float4 w[NC][kC];
    auto load_w = [&](int kb) {
#pragma unroll
        for (int i = 0; i < NC; ++i)
#pragma unroll
            for (int c = 0; c < kC; ++c) w[i][c] = ld_row4<T, kVec>(wp[c], kb + 128 * i + 4 * lane, k);
    };
    if (!w_static) pdl_wait();
    load_w(0);
    if (w_static) pdl_wait();
    float acc[kR * kC];
#pragma unroll
    for (int i = 0; i < kR * kC; ++i) acc[i] = 0.f;
    for (int kb = 0; kb < k; kb += 128 * NC) {
        if (kb > 0) load_w(kb);
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const int kk = kb + 128 * i + 4 * lane;
            float4 xv[kR];
#pragma unroll
            for (int r = 0; r < kR; ++r) xv[r] = ld_row4<T, kVec>(x + (size_t)min(row0 + r, rows - 1) * k, kk, k);
#pragma unroll
            for (int r = 0; r < kR; ++r)
#pragma unroll
                for (int c = 0; c < kC; ++c) {
                    float& a = acc[r * kC + c];
                    a = fmaf(xv[r].x, w[i][c].x, a);
                    a = fmaf(xv[r].y, w[i][c].y, a);
                    a = fmaf(xv[r].z, w[i][c].z, a);
                    a = fmaf(xv[r].w, w[i][c].w, a);
                }
        }
    }
    // after the step over lane bit b a lane keeps the values whose index has bit b equal to its own
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float send = up ? acc[i] : acc[i + o], keep = up ? acc[i + o] : acc[i];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    const int r = row0 + (lane >> 2), c = col0 + (lane & 3);
    if (r < rows && c < n) y[(size_t)r * ldy + c] = acc[0];
}

// Many rows: [128 x 64] tiles, 256 threads with 8 x 4 results each (bound by the multiply-adds then: 12 shared-memory loads of
// four elements per 128 of them).  K in steps of 16.  kAsync (fp32, aligned rows): a ring of four cp.async stages; otherwise two
// stages filled through registers, one element per load, sixteen lanes along a row, so that rows of any type and alignment are
// read in whole sectors (in the rows kernel a lane's four neighbours are four loads, each of every fourth element: 1024 x 2048, k =
// 255, fp32 131 us there).  Rows of 16 floats 20 apart: eight neighbouring rows' float4 fall on different banks.  Rows and columns
// beyond the end are not read: clamped to the last one, 126 threads of every tile asked the L2 for the same line, and 130 rows of
// 8000 columns, k = 256 took 113 us instead of 31.
constexpr int kTileR = 128, kTileC = 64, kTileK = 16, kTileLd = 20, kTileStages = 4;
constexpr int kTileStage = (kTileR + kTileC) * kTileLd;                      // floats

template <typename T, bool kAsync>
__global__ void __launch_bounds__(256, 2)
gemm_tile_kernel(const T* __restrict__ x, const Segs segs, float* __restrict__ y, int rows, int n, int k, int ldy) {
    extern __shared__ float smem[];
    pdl_launch_dependents();
    pdl_wait();
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, row0 = (int)blockIdx.y * kTileR, col0 = (int)blockIdx.x * kTileC;
    const int n_rows = rows - row0;             // (16 rows at a time are left out where none of them is there)
    float acc[8][4] = {};
    auto multiply_rows = [&](int stage, auto full) {
        const float* xs = smem + stage * kTileStage;
        const float* ws = xs + kTileR * kTileLd;
#pragma unroll
        for (int kk = 0; kk < kTileK; kk += 4) {
            float4 b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(ws + (tx + 16 * j) * kTileLd + kk);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (!decltype(full)::value && 16 * i >= n_rows) break;
                const float4 a = *reinterpret_cast<const float4*>(xs + (ty + 16 * i) * kTileLd + kk);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float& v = acc[i][j];
                    v = fmaf(a.x, b[j].x, v);
                    v = fmaf(a.y, b[j].y, v);
                    v = fmaf(a.z, b[j].z, v);
                    v = fmaf(a.w, b[j].w, v);
                }
            }
        }
    };
    auto multiply = [&](int stage) {
        if (n_rows >= kTileR) multiply_rows(stage, std::true_type());
        else multiply_rows(stage, std::false_type());
    };
    if constexpr (kAsync) {
        // this thread's pieces of a stage: four K elements of rows lr and lr + 64 of x and of weight row lr
        const int lr = threadIdx.x >> 2, lk = (threadIdx.x & 3) * 4;
        const T* src[3] = {x + (size_t)min(row0 + lr, rows - 1) * k, x + (size_t)min(row0 + lr + 64, rows - 1) * k,
                           weight_row<T>(segs, min(col0 + lr, n - 1), k)};
        const bool there[3] = {row0 + lr < rows, row0 + lr + 64 < rows, col0 + lr < n};
        const uint32_t dst = smem_u32(smem + lr * kTileLd + lk);
        auto fetch = [&](int step) {                                         // (one commit group per step, empty beyond the end)
            const int kk = step * kTileK + lk;
            if (step * kTileK < k) {
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const uint32_t d = dst + (uint32_t)(((step % kTileStages) * kTileStage + 64 * i * kTileLd) * 4);
                    const bool ok = there[i] && kk < k;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src[i] + (ok ? kk : 0)), "r"(ok ? 16 : 0) : "memory");
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        for (int i = 0; i < kTileStages - 1; ++i) fetch(i);
        for (int step = 0; step * kTileK < k; ++step) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kTileStages - 2) : "memory");
            __syncthreads();                    // this step's stage is complete, and everyone has left the stage refilled next
            fetch(step + kTileStages - 1);
            multiply(step % kTileStages);
        }
    } else {
        constexpr int kN = (kTileR + kTileC) / 16;
        const T* src[kN];                       // element tx of rows ty, ty + 16, ... of x, then of the weights; null: not there
#pragma unroll
        for (int i = 0; i < kN; ++i) {
            const int r = ty + 16 * i;
            if (i < kTileR / 16) src[i] = row0 + r < rows ? x + (size_t)(row0 + r) * k + tx : nullptr;
            else src[i] = col0 + r - kTileR < n ? weight_row<T>(segs, col0 + r - kTileR, k) + tx : nullptr;
        }
        typename Raw<T>::type v[kN];            // as loaded: converted when stored, or the loads would be waited for before the multiplies
        auto load = [&](int kk) {
#pragma unroll
            for (int i = 0; i < kN; ++i) v[i] = Raw<T>::load(src[i] + kk, src[i] && kk + tx < k);
        };
        auto store = [&](int stage) {
#pragma unroll
            for (int i = 0; i < kN; ++i) smem[stage * kTileStage + (ty + 16 * i) * kTileLd + tx] = Raw<T>::value(v[i]);
        };
        load(0);
        store(0);
        for (int step = 0; step * kTileK < k; ++step) {
            __syncthreads();                    // this step's stage is complete, and everyone has left the other one
            load((step + 1) * kTileK);
            multiply(step & 1);
            store((step + 1) & 1);
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = row0 + ty + 16 * i;
        if (r >= rows) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (col0 + tx + 16 * j < n) y[(size_t)r * ldy + col0 + tx + 16 * j] = acc[i][j];
    }
}

template <typename... KArgs, typename... Args>
void launch(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = wd_pdl_enabled ? 1 : 0;
    ++wd_launch_counter;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename T, bool kVec>
void launch_rows(const void* x, const Segs& segs, float* y, int rows, int n, int k, int ldy, bool w_static, cudaStream_t st) {
    launch(k <= 256 ? gemm_rows_kernel<T, 2, kVec> : gemm_rows_kernel<T, 3, kVec>,
           dim3((unsigned)wd_ceil_div(n, 16), (unsigned)wd_ceil_div(rows, 8)), 128, 0, st, (const T*)x, segs, y, rows, n, k, ldy, w_static ? 1 : 0);
}

template <typename T, bool kAsync>
void launch_tiles(const void* x, const Segs& segs, float* y, int rows, int n, int k, int ldy, cudaStream_t st) {
    const size_t smem = (size_t)(kAsync ? kTileStages : 2) * kTileStage * sizeof(float);
    static bool attr_done[64] = {};
    int dev = 0;
    if (kAsync && (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || !attr_done[dev])) {
        cudaFuncSetAttribute(gemm_tile_kernel<T, kAsync>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (dev >= 0 && dev < 64) attr_done[dev] = true;
    }
    launch(gemm_tile_kernel<T, kAsync>, dim3((unsigned)wd_ceil_div(n, kTileC), (unsigned)wd_ceil_div(rows, kTileR)), 256, smem, st,
           (const T*)x, segs, y, rows, n, k, ldy);
}

}  // namespace

void wd_launch_gemm_plain(int dtype, const void* x, const void* const* w, const int* n, int n_mat, float* y, int rows, int k,
                          int ldy, bool w_static, cudaStream_t st) {
    if (rows <= 0 || n_mat < 1 || n_mat > 3) return;
    Segs segs;
    int end = 0;
    bool vec = k % 4 == 0 && (uintptr_t)x % 16 == 0;
    for (int i = 0; i < 3; ++i) {
        segs.w[i] = w[i < n_mat ? i : n_mat - 1];
        if (i < n_mat) end += n[i];
        segs.end[i] = end;
        vec = vec && (uintptr_t)segs.w[i] % 16 == 0;
    }
    if (end <= 0) return;
    constexpr int kMostRows = 65535 * 8;        // of one launch (a grid holds 65535 blocks in y)
    if (rows > kMostRows) {
        const size_t size = dtype == WD_F32 ? 4 : 2;
        for (int r0 = 0; r0 < rows; r0 += kMostRows) {
            const int m = std::min(rows - r0, kMostRows);
            wd_launch_gemm_plain(dtype, (const char*)x + (size_t)r0 * k * size, w, n, n_mat, y + (size_t)r0 * ldy, m, k, ldy, w_static, st);
            if (rows - r0 <= kMostRows) return;
        }
    }
    // Tiles when the rows kernel would take longer: it works at 16 TFLOP/s in fp32 (8 where rows are not aligned) and at 15 (10)
    // in bf16, 20 (14.5) from k = 257 on, three loads in flight instead of two; a tile takes 0.85 us (1.05 through registers) of
    // its SM per 16 of K, and a lone one 0.4 more.  Measured, rows / tiles / the [32 x 64]-tile kernel before either, in us: fp32
    // 130 x 8000 k = 688 84 / 77 / 138; 520 x 2048, k = 256 33 / 29 / 51; k = 255 1024 x 2048 131 / 38 / 65, 130 x 8000 68 / 36 / 53,
    // 34 x 8000 18 / 22 / 28; bf16 2048 x 2048, k = 256 130 / 72 / 120, k = 255 201 / 72 / 120, 300 x 2048, k = 687 60 / 69 / 100.
    // In a step the rows kernel also has its weights before the previous kernel ends, about 5 us of a launch (528 rows, gate/up
    // of 2 x 688, k = 256, alike alone: normal step of the fp32 model 319 us, with tiles 332).
    const bool f32 = dtype == WD_F32;
    const double rate = f32 ? (vec ? 16.0 : 8.0) : k <= 256 ? (vec ? 15.0 : 10.0) : (vec ? 20.0 : 14.5);
    const long long n_tiles = (long long)wd_ceil_div(end, kTileC) * wd_ceil_div(rows, kTileR);
    const double us_rows = 2e-6 * rows * end * k / rate;
    const double us_tiles = wd_ceil_div(k, kTileK) * (0.4 + (f32 && vec ? 0.85 : 1.05) * (double)((n_tiles + 147) / 148));
    const bool tiles = us_tiles + (w_static ? 5.0 : 0.0) < us_rows;
    if (dtype == WD_F32) {
        if (tiles && vec) launch_tiles<float, true>(x, segs, y, rows, end, k, ldy, st);
        else if (tiles) launch_tiles<float, false>(x, segs, y, rows, end, k, ldy, st);
        else if (vec) launch_rows<float, true>(x, segs, y, rows, end, k, ldy, w_static, st);
        else launch_rows<float, false>(x, segs, y, rows, end, k, ldy, w_static, st);
    } else {
        if (tiles) launch_tiles<__nv_bfloat16, false>(x, segs, y, rows, end, k, ldy, st);
        else if (vec) launch_rows<__nv_bfloat16, true>(x, segs, y, rows, end, k, ldy, w_static, st);
        else launch_rows<__nv_bfloat16, false>(x, segs, y, rows, end, k, ldy, w_static, st);
    }
}
