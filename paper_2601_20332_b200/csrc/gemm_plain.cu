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
//
// kEpi and kNorm (WdPlainFuse) take the kernels on either side of a projection in, each of which is another link of 2-3 us in the
// step's chain however little it does:
//   kNorm    RMSNorm of the rows: their gains are multiplied into the weights before the dependency wait, the sum of squares of a
//            row is reduced like the products (the lane that ends up with a row's result has that row's sum too), and 1 / rms is
//            applied to the finished sums
//   kEpiQkv  a warp's four columns are two rotation pairs of a q or k head (or four dims of a v head): rotated and written to q and
//            the cache.  kEpiSwiglu: two gate and the two up columns that belong to them.  kEpiAdd: added to y.
// Measured, normal step of the fp32 model (two blocks of 256 / 688, 9 rows): 24 launches and 75 us with separate kernels, 15 and 52 us
// with these; a projection with its neighbours in it takes 2.1-2.9 us where the three kernels took 5.5 together.
enum { kEpiNone = 0, kEpiQkv = 1, kEpiSwiglu = 2, kEpiAdd = 3 };
template <int kEpi, bool kNorm> struct RowsArgs { WdPlainFuse f; };
template <> struct RowsArgs<kEpiNone, false> {};

// output column (of the concatenated matrices) that a warp of column group g computes as its c-th
template <int kEpi>
__device__ __forceinline__ int group_col(const WdPlainFuse& f, int g, int c) {
    if (kEpi == kEpiSwiglu) return 2 * g + (c & 1) + (c >> 1) * f.F;
    if (kEpi == kEpiQkv) {
        const int half = f.dh >> 1, rotated = (f.Hq + f.Hkv) * (half >> 1);     // groups of rotation pairs
        if (g < rotated) {
            const int h = g / (half >> 1);
            return h * f.dh + 2 * (g - h * (half >> 1)) + (c & 1) + (c >> 1) * half;
        }
        return (f.Hq + f.Hkv) * f.dh + 4 * (g - rotated) + c;
    }
    return 4 * g + c;
}

template <typename T, int kR, int NC, bool kVec, int kEpi = kEpiNone, bool kNorm = false>
__global__ void __launch_bounds__(128)
gemm_rows_kernel(const T* __restrict__ x, const Segs segs, float* __restrict__ y, int rows, int n, int k, int ldy, int w_static,
                 const RowsArgs<kEpi, kNorm> ra) {
    constexpr int kC = 4, kV = kR * kC, kDup = 32 / kV;      // sums of a warp, lanes that end up with the same one
    constexpr bool kFused = kEpi != kEpiNone || kNorm;
    WdPlainFuse f;
    if constexpr (kFused) f = ra.f;
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, group = (int)(blockIdx.x * 4 + (threadIdx.x >> 5)), row0 = (int)blockIdx.y * kR;
    if (group * kC >= n) return;
    const T* wp[kC];
#pragma unroll
    for (int c = 0; c < kC; ++c) wp[c] = weight_row<T>(segs, min(group_col<kEpi>(f, group, c), n - 1), k);
    float4 w[NC][kC];
    auto load_w = [&](int kb) {
#pragma unroll
        for (int i = 0; i < NC; ++i)
#pragma unroll
            for (int c = 0; c < kC; ++c) w[i][c] = ld_row4<T, kVec>(wp[c], kb + 128 * i + 4 * lane, k);
        if (kNorm) {
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                const float4 g = ld_row4<float, true>(f.gain, kb + 128 * i + 4 * lane, k);
#pragma unroll
                for (int c = 0; c < kC; ++c) w[i][c] = make_float4(w[i][c].x * g.x, w[i][c].y * g.y, w[i][c].z * g.z, w[i][c].w * g.w);
            }
        }
    };
    if (!w_static) pdl_wait();
    load_w(0);
    if (w_static) pdl_wait();
    // this lane's result, and what its epilogue needs beside the product
    const int own = lane / kDup, r = row0 + (own >> 2), c = group_col<kEpi>(f, group, own & 3);
    const bool mine = r < rows && c < n && lane % kDup == 0;
    float2 cs = make_float2(1.f, 0.f);
    float old = 0.f;
    int pos = 0, seq = 0;
    if (kEpi == kEpiQkv && mine) {
        pos = f.row_pos[r];
        seq = f.row_seq[r];
        if (c < (f.Hq + f.Hkv) * f.dh) cs = f.rope_tab[(size_t)r * (f.dh >> 1) + c % (f.dh >> 1)];
    }
    if (kEpi == kEpiAdd) old = Raw<float>::value(Raw<float>::load(y + (size_t)r * ldy + c, mine));
    const T* xp[kR];
#pragma unroll
    for (int i = 0; i < kR; ++i) {
        const int row = min(row0 + i, rows - 1);
        xp[i] = x + (size_t)(kNorm && f.row_idx ? f.row_idx[row] : row) * k;
    }
    float acc[kR * kC], ss[kR];
#pragma unroll
    for (int i = 0; i < kR * kC; ++i) acc[i] = 0.f;
#pragma unroll
    for (int i = 0; i < kR; ++i) ss[i] = 0.f;
    for (int kb = 0; kb < k; kb += 128 * NC) {
        if (kb > 0) load_w(kb);
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const int kk = kb + 128 * i + 4 * lane;
            float4 xv[kR];
#pragma unroll
            for (int rr = 0; rr < kR; ++rr) xv[rr] = ld_row4<T, kVec>(xp[rr], kk, k);
#pragma unroll
            for (int rr = 0; rr < kR; ++rr) {
                if (kNorm) ss[rr] = fmaf(xv[rr].x, xv[rr].x, fmaf(xv[rr].y, xv[rr].y, fmaf(xv[rr].z, xv[rr].z, fmaf(xv[rr].w, xv[rr].w, ss[rr]))));
#pragma unroll
                for (int cc = 0; cc < kC; ++cc) {
                    float& a = acc[rr * kC + cc];
                    a = fmaf(xv[rr].x, w[i][cc].x, a);
                    a = fmaf(xv[rr].y, w[i][cc].y, a);
                    a = fmaf(xv[rr].z, w[i][cc].z, a);
                    a = fmaf(xv[rr].w, w[i][cc].w, a);
                }
            }
        }
    }
    // after the step over lane bit b a lane keeps the values whose index has that bit equal to its own, while there is more than one
#pragma unroll
    for (int step = 0; step < 5; ++step) {
        const int o = 16 >> step, nv = kV >> (step + 1), ns = kR >> (step + 1);
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < kV / 2; ++i) {
            if (i >= nv) break;
            const float send = up ? acc[i] : acc[i + nv], keep = up ? acc[i + nv] : acc[i];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        if (nv == 0) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
        if (kNorm) {
#pragma unroll
            for (int i = 0; i < kR / 2; ++i) {
                if (i >= ns) break;
                const float send = up ? ss[i] : ss[i + ns], keep = up ? ss[i + ns] : ss[i];
                ss[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
            if (ns == 0) ss[0] += __shfl_xor_sync(0xffffffffu, ss[0], o);
        }
    }
    float v = acc[0];
    if (kNorm) v *= rsqrtf(ss[0] / (float)k + f.eps);
    if constexpr (kEpi == kEpiQkv) {
        const float other = __shfl_xor_sync(0xffffffffu, v, 2 * kDup);         // the partner of a rotation pair
        if (!mine) return;
        const int h = c / f.dh, j = c - h * f.dh;
        if (h < f.Hq + f.Hkv) v = v * cs.x + ((own & 2) ? other : -other) * cs.y;
        if (h < f.Hq) {
            f.q[(size_t)r * f.Hq * f.dh + c] = v;
            return;
        }
        // index check: a cache row outside the state is recorded and not written
        if ((unsigned)pos >= (unsigned)f.S || (unsigned)seq >= (unsigned)f.batch) {
            atomicCAS(f.status, 0, WD_ERR_BOUNDS);
            return;
        }
        const int kh = h < f.Hq + f.Hkv ? h - f.Hq : h - f.Hq - f.Hkv;
        if (h < f.Hq + f.Hkv) f.kcache[(((size_t)seq * f.Hkv + kh) * f.S + pos) * f.dh + j] = v;
        else f.vcache[(((size_t)seq * f.Hkv + kh) * f.dh + j) * f.Sp + pos] = v;
    } else if constexpr (kEpi == kEpiSwiglu) {
        const float up = __shfl_xor_sync(0xffffffffu, v, 2 * kDup);
        if (mine && !(own & 2)) y[(size_t)r * ldy + c] = v / (1.f + __expf(-v)) * up;
    } else {
        if (mine) y[(size_t)r * ldy + c] = kEpi == kEpiAdd ? old + v : v;
    }
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

constexpr int kFusedBlocks = 9 * 148;       // nine to an SM of a B200, see wd_launch_gemm_plain_fused

template <typename T, bool kVec, int kEpi = kEpiNone, bool kNorm = false>
void launch_rows(const void* x, const Segs& segs, float* y, int rows, int n, int k, int ldy, bool w_static, cudaStream_t st,
                 const RowsArgs<kEpi, kNorm>& ra = {}) {
    auto kernel = k <= 256 ? gemm_rows_kernel<T, 8, 2, kVec, kEpi, kNorm> : gemm_rows_kernel<T, 8, 3, kVec, kEpi, kNorm>;
    int r = 8;
    if constexpr (kEpi != kEpiNone || kNorm) {
        // Four rows to a warp while the grid stays small (nine rows waste less, and each warp has half the loads and sums in its
        // chain); then also the whole of k up to 768 in one go, one round trip instead of two.  Step of the fp32 model, two blocks of
        // 256 / 688: 9 rows 63 -> 52 us, 40 81 -> 72, 72 98 -> 89; with 13 blocks to an SM instead of nine 96.  (The add after a
        // short k is the exception: eight rows 2.1-2.4 us, four 3.7-3.8, in either block of the step, with a graph and without, and the
        // step 47.5 -> 50.9 us.  The cause was not found.)
        if (!(kEpi == kEpiAdd && k <= 256) && (long long)wd_ceil_div(n, 16) * wd_ceil_div(rows, 4) <= kFusedBlocks) {
            r = 4;
            kernel = k <= 256 ? gemm_rows_kernel<T, 4, 2, kVec, kEpi, kNorm>
                              : k <= 768 ? gemm_rows_kernel<T, 4, 6, kVec, kEpi, kNorm> : gemm_rows_kernel<T, 4, 3, kVec, kEpi, kNorm>;
        }
    }
    launch(kernel, dim3((unsigned)wd_ceil_div(n, 16), (unsigned)wd_ceil_div(rows, r)), 128, 0, st, (const T*)x, segs, y, rows, n, k, ldy,
           w_static ? 1 : 0, ra);
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

// Tiles when the rows kernel would take longer: it works at 16 TFLOP/s in fp32 (8 where rows are not aligned) and at 15 (10)
// in bf16, 20 (14.5) from k = 257 on, three loads in flight instead of two; a tile takes 0.85 us (1.05 through registers) of
// its SM per 16 of K, and a lone one 0.4 more.  Measured, rows / tiles / the [32 x 64]-tile kernel before either, in us: fp32
// 130 x 8000 k = 688 84 / 77 / 138; 520 x 2048, k = 256 33 / 29 / 51; k = 255 1024 x 2048 131 / 38 / 65, 130 x 8000 68 / 36 / 53,
// 34 x 8000 18 / 22 / 28; bf16 2048 x 2048, k = 256 130 / 72 / 120, k = 255 201 / 72 / 120, 300 x 2048, k = 687 60 / 69 / 100.
// In a step the rows kernel also has its weights before the previous kernel ends, about 5 us of a launch (528 rows, gate/up
// of 2 x 688, k = 256, alike alone: normal step of the fp32 model 319 us, with tiles 332).
bool tiles_pay(bool f32, bool vec, int rows, int n, int k, bool w_static) {
    const double rate = f32 ? (vec ? 16.0 : 8.0) : k <= 256 ? (vec ? 15.0 : 10.0) : (vec ? 20.0 : 14.5);
    const long long n_tiles = (long long)wd_ceil_div(n, kTileC) * wd_ceil_div(rows, kTileR);
    const double us_rows = 2e-6 * rows * n * k / rate;
    const double us_tiles = wd_ceil_div(k, kTileK) * (0.4 + (f32 && vec ? 0.85 : 1.05) * (double)((n_tiles + 147) / 148));
    return us_tiles + (w_static ? 5.0 : 0.0) < us_rows;
}

// the matrices side by side; false unless rows of k elements can be read four at a time
bool make_segs(const void* x, const void* const* w, const int* n, int n_mat, int k, Segs* segs, int* n_all) {
    int end = 0;
    bool vec = k % 4 == 0 && (uintptr_t)x % 16 == 0;
    for (int i = 0; i < 3; ++i) {
        segs->w[i] = w[i < n_mat ? i : n_mat - 1];
        if (i < n_mat) end += n[i];
        segs->end[i] = end;
        vec = vec && (uintptr_t)segs->w[i] % 16 == 0;
    }
    *n_all = end;
    return vec;
}

}  // namespace

void wd_launch_gemm_plain(int dtype, const void* x, const void* const* w, const int* n, int n_mat, float* y, int rows, int k,
                          int ldy, bool w_static, cudaStream_t st) {
    if (rows <= 0 || n_mat < 1 || n_mat > 3) return;
    Segs segs;
    int end = 0;
    const bool vec = make_segs(x, w, n, n_mat, k, &segs, &end);
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
    const bool f32 = dtype == WD_F32, tiles = tiles_pay(f32, vec, rows, end, k, w_static);
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

bool wd_launch_gemm_plain_fused(const WdPlainFuse& f, const void* const* w, const int* n, int n_mat, int rows, int k, cudaStream_t st) {
    if (!f.x || rows < 1 || n_mat < 1 || n_mat > 3) return false;
    Segs segs;
    int end = 0;
    const bool vec = make_segs(f.x, w, n, n_mat, k, &segs, &end) && (uintptr_t)f.gain % 16 == 0;
    // While the step is a chain of latencies: up to nine blocks of the eight-row form to an SM.  Beyond, the sums of squares taken
    // again by every group of columns cost more than the launches saved (step of the fp32 model: 300 rows 187 us with separate
    // kernels, 201 without this limit; 120 rows 101 and 99; 56 rows 75 and 64; 9 rows 74 and 52).
    if (!vec || end < 4 || end % 4 || (long long)wd_ceil_div(end, 16) * wd_ceil_div(rows, 8) > kFusedBlocks ||
        tiles_pay(true, true, rows, end, k, true))
        return false;
    switch (f.epi) {
        case WD_PLAIN_STORE:
            if (f.gain) launch_rows<float, true, kEpiNone, true>(f.x, segs, f.y, rows, end, k, f.ldy, true, st, {f});
            return f.gain != nullptr;
        case WD_PLAIN_QKV:
            if (!f.gain || f.dh % 4) return false;
            launch_rows<float, true, kEpiQkv, true>(f.x, segs, nullptr, rows, end, k, 0, true, st, {f});
            return true;
        case WD_PLAIN_SWIGLU:
            if (!f.gain || f.F % 2 || end != 2 * f.F) return false;
            launch_rows<float, true, kEpiSwiglu, true>(f.x, segs, f.y, rows, end, k, f.ldy, true, st, {f});
            return true;
        case WD_PLAIN_ADD:
            if (f.gain) return false;
            launch_rows<float, true, kEpiAdd, false>(f.x, segs, f.y, rows, end, k, f.ldy, true, st, {f});
            return true;
    }
    return false;
}
