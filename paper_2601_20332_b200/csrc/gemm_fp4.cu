// NVFP4 weight-streaming GEMM on the block-scaled tensor-core path (sm_100a), an option outside the paper
// (which calls quantisation orthogonal to its method).
//
//   y[tok, n] = gx[tok] * gw[n] * sum_blocks (sx[tok, b] * sw[n, b]) * sum_{i in block b} qx[tok, i] * qw[n, i]
//
// Operands: 4-bit e2m1 codes packed two per byte (element 2j in the low nibble), one unsigned e4m3 scale
// per block of 16 elements along K, one float scale per row.  tcgen05.mma kind::mxf4nvf4 multiplies the
// codes and applies the block scales in hardware (fp32 accumulation in tensor memory); the row scales are
// applied in the epilogue.
//
// A stage of the ring holds one K block of 256 elements: [128 weight rows x 128 bytes] and [BN tokens x 128
// bytes] of codes in the 128-byte swizzled layout, plus their block scales [rows x 16 bytes].  The hardware
// reads block scales from tensor memory: for row r of an operand the four scales of one K = 64 instruction
// sit in lane r mod 32 (of every 32-lane quarter), 32-bit column r / 32, one scale per byte.  Four warps
// copy each stage's scales from shared memory into that layout (tcgen05.st, every warp its own quarter)
// before the MMA thread issues the stage's four instructions; two scale slots alternate.
//   warp 0      TMA producer (weights, which never depend on earlier kernels, before the dependency wait)
//   warp 1      MMA issuer
//   warps 2-5   epilogue: tcgen05.ld, row scales, coalesced fp32 stores of this K slice's partial sums
//   warps 6-9   block scales: shared memory -> tensor memory
// Persistent, one CTA per SM: the K blocks of all (weight tile, token tile) units form one line that is cut into
// equal shares (stream-K, see choose_split), or whole units per CTA when that is cheaper.  The partial sums of a unit that several
// CTAs share are written side by side ([slice][tok][n]) and added by the consumer, as in the bf16 kernel.
// Measured at 34 rows, quantised input to summed result, 12288 x 4096 / 24576 x 4096 / 4096 x 12288: 11.0 / 16.4 / 12.2 us
// against 4.7 / 9.3 / 4.6 us for the bytes alone; what remains is start-up (2-3 us to the first complete stage, 2 us from the
// last MMA to the stores) around 0.28-0.39 us a stage.  (Bringing the weights into the L2 ahead of the dependency wait made it
// slower: 24.4 instead of 23.8 us for the middle shape, 107 instead of 90 us at 600 rows.)
// Every wait is bounded; on expiry the CTA records WD_ERR_DEVICE_TIMEOUT and leaves.
#include <algorithm>
#include <climits>
#include <cstring>

#include <cuda_fp8.h>

#include "gemm_tc.h"
#include "device_utils.cuh"

namespace {

using namespace wdk;

constexpr int kBM = 128;              // weight rows per tile
constexpr int kKB = 256;              // K elements per stage = 128 bytes of codes = one swizzle row
constexpr int kStageW = kBM * 128;    // 16 KB of weight codes
constexpr int kSfW = kBM * 16;        // 2 KB of weight block scales
constexpr int kThreads = 320;

struct Fp4Params {
    int rows, n_out, bn, kb_total, tok_tiles, n_slices, n_units, n_stages, buf_cols;
    int aligned;                      // whole units per CTA (one slice) instead of equal pieces of the K-block line
    int w_static;                     // the weights were written before the previous kernel started
    float* y;
    size_t split_stride;
    const float* gw;                  // [n_out] row scales of the weights
    const float* gx;                  // [rows] row scales of the activations
    int32_t* status;
    uint32_t idesc;
};

__device__ __forceinline__ void umma_fp4(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t sfa,
                                         uint32_t sfb, uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::mxf4nvf4.block_scale.block16 [%0], %1, %2, %3, [%5], [%6], p;\n}\n"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb) : "memory");
}

__global__ void __launch_bounds__(kThreads, 1)
gemm_fp4_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                const __grid_constant__ CUtensorMap map_sx, const __grid_constant__ CUtensorMap map_sw, const Fp4Params p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int NS = p.n_stages;
    const int x_bytes = p.bn * 128, sfx_bytes = p.bn * 16;
    // stage: weight codes | token codes | weight scales | token scales (rounded up to a multiple of 1024 bytes)
    const int stage_bytes = (kStageW + x_bytes + kSfW + sfx_bytes + 1023) & ~1023;
    uint64_t* bars = (uint64_t*)(smem + (size_t)NS * stage_bytes);
    // bars: [0, NS) full | [NS, 2NS) empty | 2NS.. accumulator full [2] | accumulator empty [2] | scales in tensor memory [2] |
    //       scale slot free [2]
    uint64_t* acc_full = bars + 2 * NS;
    uint64_t* acc_empty = acc_full + 2;
    uint64_t* sf_full = acc_empty + 2;
    uint64_t* sf_free = sf_full + 2;
    uint32_t* tmem_slot = (uint32_t*)(sf_free + 2);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    float* gx_s = (float*)(tmem_slot + 4);           // [128] row scales of the epilogue's token tile

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // This CTA's share [g_begin, g_end) of the line of K blocks of all units, unit = weight tile * tok_tiles + token tile
    // (neighbouring units share a weight tile): equal shares, so every SM streams the same bytes, or whole units.
    const int G = gridDim.x, c = blockIdx.x, KB = p.kb_total, W = p.n_units * KB;
    // (32-bit: the host sees to it that the products fit)
    const int g_begin = p.aligned ? c * p.n_units / G * KB : c * W / G;
    const int g_end = p.aligned ? (c + 1) * p.n_units / G * KB : (c + 1) * W / G;
    const int n_total = g_end - g_begin;
    // the piece that starts at K block g of the line: its unit's rows and tokens, first K block and length
    auto piece_at = [&](int g, int& unit, int& n0, int& tok0, int& kb0, int& len) {
        unit = g / KB;
        kb0 = g - unit * KB;
        len = min(KB - kb0, g_end - g);
        const int tile = unit / p.tok_tiles;
        n0 = tile * kBM;
        tok0 = (unit - tile * p.tok_tiles) * p.bn;
    };
    const uint32_t tmem_cols = 2u * (uint32_t)p.buf_cols + 64u <= 128u ? 128u : (2u * (uint32_t)p.buf_cols + 64u <= 256u ? 256u : 512u);

    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&bars[s]), 1);
            mbar_init(smem_u32(&bars[NS + s]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&acc_full[i]), 1);
            mbar_init(smem_u32(&acc_empty[i]), 128);
            mbar_init(smem_u32(&sf_full[i]), 128);
            mbar_init(smem_u32(&sf_free[i]), 1);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (const CUtensorMap* m : {&map_w, &map_sw, &map_x, &map_sx}) asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(tmem_slot), tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t tmem_sf = tmem_base + 2u * (uint32_t)p.buf_cols;      // two slots of 32 columns: 16 for A, 16 for B

    if (warp == 0) {
        if (n_total > 0) {
            // ------------------------------------------------ TMA producer (the whole warp, see elect_one)
            const bool leader = elect_one();
            uint64_t pol_stream;
            asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_stream));
            struct Walk { int g, left, kb, n0, tok0; };
            auto enter = [&](Walk& w) {
                int unit;
                piece_at(w.g, unit, w.n0, w.tok0, w.kb, w.left);
            };
            auto advance = [&](Walk& w) {
                ++w.kb;
                ++w.g;
                if (--w.left == 0 && w.g < g_end) enter(w);
            };
            auto load_w = [&](const Walk& w, int s) {
                if (!leader) return;
                const uint32_t sa = smem_u32(smem) + (uint32_t)(s * stage_bytes), full = smem_u32(&bars[s]);
                mbar_expect_tx(full, (uint32_t)(kStageW + x_bytes + kSfW + sfx_bytes));
                tma_load_2d_hint(sa, &map_w, full, w.kb * 128, w.n0, pol_stream);
                tma_load_2d(sa + kStageW + x_bytes, &map_sw, full, w.kb * 16, w.n0);
            };
            auto load_x = [&](const Walk& w, int s) {
                if (!leader) return;
                const uint32_t sa = smem_u32(smem) + (uint32_t)(s * stage_bytes), full = smem_u32(&bars[s]);
                tma_load_2d(sa + kStageW, &map_x, full, w.kb * 128, w.tok0);
                tma_load_2d(sa + kStageW + x_bytes + kSfW, &map_sx, full, w.kb * 16, w.tok0);
            };
            Walk w, wx;
            w.g = g_begin;
            enter(w);
            wx = w;
            const int n_pre = n_total < NS ? n_total : NS;
            if (p.w_static) {        // weights first: they depend on nothing
                for (int i = 0; i < n_pre; ++i, advance(w)) load_w(w, i);
                pdl_wait();
                for (int i = 0; i < n_pre; ++i, advance(wx)) load_x(wx, i);
            } else {                 // stage by stage, so that the first is complete as early as possible
                pdl_wait();
                for (int i = 0; i < n_pre; ++i, advance(w)) { load_w(w, i); load_x(w, i); }
            }
            int s = n_pre % NS;
            uint32_t ph = (uint32_t)(n_pre / NS) & 1u;
            for (int i = n_pre; i < n_total; ++i, advance(w)) {
                if (!mbar_wait_warp(smem_u32(&bars[NS + s]), ph ^ 1u, abort_flag)) {
                    *abort_flag = 1;
                    atomicCAS(p.status, 0, WD_ERR_DEVICE_TIMEOUT);
                    break;
                }
                load_w(w, s);
                load_x(w, s);
                if (++s == NS) { s = 0; ph ^= 1u; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        {
            // ------------------------------------------------ MMA issuer (the whole warp)
            const bool leader = elect_one();
            bool ok = true;
            int s = 0, i = 0;
            uint32_t ph = 0;
            for (int g = g_begin, u = 0; g < g_end && ok; ++u) {
                int unit, n0, tok0, kb0, kbn;
                piece_at(g, unit, n0, tok0, kb0, kbn);
                g += kbn;
                const int buf = u & 1;
                const uint32_t par = (uint32_t)(u >> 1) & 1u;
                if (!(ok = mbar_wait_warp(smem_u32(&acc_empty[buf]), par ^ 1u, abort_flag))) break;
                tc_fence_after();
                const uint32_t acc = tmem_base + (uint32_t)(buf * p.buf_cols);
                for (int j = 0; j < kbn; ++j, ++i) {
                    const int slot = i & 1;
                    if (!(ok = mbar_wait_warp(smem_u32(&bars[s]), ph, abort_flag))) break;                       // codes landed
                    if (!(ok = mbar_wait_warp(smem_u32(&sf_full[slot]), (uint32_t)(i >> 1) & 1u, abort_flag))) break;   // scales in tensor memory
                    tc_fence_after();
                    const uint32_t sa = smem_u32(smem) + (uint32_t)(s * stage_bytes);
                    const uint64_t adesc = make_sdesc(sa), bdesc = make_sdesc(sa + kStageW);
                    const uint32_t sf = tmem_sf + (uint32_t)(slot * 32);
                    if (leader) {
#pragma unroll
                        for (int kq = 0; kq < 4; ++kq)       // 64 elements = 32 bytes further along K: +2 in 16-byte units
                            umma_fp4(acc, adesc + (uint64_t)(2 * kq), bdesc + (uint64_t)(2 * kq), p.idesc, sf + (uint32_t)(4 * kq),
                                     sf + 16u + (uint32_t)(4 * kq), (j > 0 || kq > 0) ? 1u : 0u);
                        umma_commit(smem_u32(&bars[NS + s]));      // stage free once these MMAs have read it
                        umma_commit(smem_u32(&sf_free[slot]));     // ... and the scale slot
                    }
                    if (++s == NS) { s = 0; ph ^= 1u; }
                }
                if (ok && leader) umma_commit(smem_u32(&acc_full[buf]));
            }
            if (!ok) {
                *abort_flag = 1;
                atomicCAS(p.status, 0, WD_ERR_DEVICE_TIMEOUT);
            }
        }
        __syncwarp();
    } else if (warp < 6) {
        // ---------------------------------------------------- epilogue (warps 2..5)
        const int quarter = warp & 3;
        const int n_local = quarter * 32 + lane;
        pdl_wait();
        bool ok = true;
        for (int g = g_begin, u = 0; g < g_end; ++u) {
            int unit, n0, tok0, kb0, kbn;
            piece_at(g, unit, n0, tok0, kb0, kbn);
            g += kbn;
            // slice: this CTA's place among those that share the unit
            const int sl = p.aligned || kb0 == 0 ? 0 : c - ((unit * KB + 1) * G - 1) / W;
            const int buf = u & 1;
            const uint32_t par = (uint32_t)(u >> 1) & 1u;
            const int n = n0 + n_local;
            const bool n_ok = n < p.n_out;
            // the row scales while the MMAs still run: the tokens' through shared memory, the weight row's in a register
            asm volatile("bar.sync 1, 128;" ::: "memory");          // the previous piece's readers are done
            const int e = (int)threadIdx.x - 64;
            if (e < p.bn) gx_s[e] = tok0 + e < p.rows ? __ldg(p.gx + tok0 + e) : 0.f;
            const float gwn = n_ok ? p.gw[n] : 0.f;
            asm volatile("bar.sync 1, 128;" ::: "memory");
            ok = ok && mbar_wait(smem_u32(&acc_full[buf]), par, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) {               // (stays in the loop: every warp reaches the same barriers)
                *abort_flag = 1;
                continue;
            }
            tc_fence_after();
            float* ys = p.y + (size_t)sl * p.split_stride + n;
            const uint32_t t_acc = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * p.buf_cols);
            for (int cc = 0; cc < p.bn; cc += 16) {
                if (tok0 + cc >= p.rows) break;
                uint32_t v[16];
                tmem_ld16(t_acc + (uint32_t)cc, v);
                if (n_ok) {
#pragma unroll
                    for (int t = 0; t < 16; ++t) {
                        const int tok = tok0 + cc + t;
                        if (tok < p.rows) ys[(size_t)tok * p.n_out] = __uint_as_float(v[t]) * gwn * gx_s[cc + t];
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(smem_u32(&acc_empty[buf]));
            if (kb0 + kbn == KB && n_ok) {
                // this CTA finished the unit: slices that nobody wrote must read as zero
                for (int z = sl + 1; z < p.n_slices; ++z) {
                    float* yz = p.y + (size_t)z * p.split_stride + n;
                    for (int tok = tok0; tok < tok0 + p.bn && tok < p.rows; ++tok) yz[(size_t)tok * p.n_out] = 0.f;
                }
            }
        }
        if (!ok && lane == 0) {
            *abort_flag = 1;
            atomicCAS(p.status, 0, WD_ERR_DEVICE_TIMEOUT);
        }
        tc_fence_before();
    } else {
        // ---------------------------------------------------- block scales: shared memory -> tensor memory (warps 6..9)
        const int quarter = warp & 3;
        bool ok = true;
        int s = 0;
        uint32_t ph = 0;
        for (int i = 0; i < n_total; ++i) {
            const int slot = i & 1;
            ok = ok && mbar_wait(smem_u32(&bars[s]), ph, abort_flag);                                    // the stage's scales landed
            ok = ok && mbar_wait(smem_u32(&sf_free[slot]), ((uint32_t)(i >> 1) & 1u) ^ 1u, abort_flag);  // the slot's last readers are done
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint8_t* st = smem + (size_t)s * stage_bytes;
            const uint4* wsf = reinterpret_cast<const uint4*>(st + kStageW + x_bytes);                   // [128 rows] x 16 scales
            const uint4* xsf = reinterpret_cast<const uint4*>(st + kStageW + x_bytes + kSfW);            // [bn rows] x 16 scales
            uint32_t v[32];
#pragma unroll
            for (int r1 = 0; r1 < 4; ++r1) {
                // row lane + 32 r1 of either operand: its 16 scales = four instructions x four scales
                const uint4 a = wsf[lane + 32 * r1];
                const int xr = lane + 32 * r1;
                const uint4 b = xr < p.bn ? xsf[xr] : make_uint4(0u, 0u, 0u, 0u);
                v[0 + r1] = a.x; v[4 + r1] = a.y; v[8 + r1] = a.z; v[12 + r1] = a.w;          // column 4 kq + r1 of A's scales
                v[16 + r1] = b.x; v[20 + r1] = b.y; v[24 + r1] = b.z; v[28 + r1] = b.w;       // ... of B's
            }
            tmem_st32(tmem_sf + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(slot * 32), v);
            tc_fence_before();
            mbar_arrive(smem_u32(&sf_full[slot]));
            if (++s == NS) { s = 0; ph ^= 1u; }
        }
        if (!ok && lane == 0) {
            *abort_flag = 1;
            atomicCAS(p.status, 0, WD_ERR_DEVICE_TIMEOUT);
        }
        tc_fence_before();
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, tmem_cols);
    }
}

// ---------------------------------------------------------------- quantisation
// sixteen elements as bfloat16 pairs in eight words (a float input is rounded to bfloat16 first)
__device__ __forceinline__ void ld_block16(const float* p, bool vec, uint32_t (&w)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float2 v = vec ? reinterpret_cast<const float2*>(p)[i] : make_float2(p[2 * i], p[2 * i + 1]);
        const __nv_bfloat162 b = __floats2bfloat162_rn(v.x, v.y);
        w[i] = *reinterpret_cast<const uint32_t*>(&b);
    }
}
__device__ __forceinline__ void ld_block16(const __nv_bfloat16* p, bool vec, uint32_t (&w)[8]) {
    if (vec) {
        const uint4 a = reinterpret_cast<const uint4*>(p)[0], b = reinterpret_cast<const uint4*>(p)[1];
        w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
    } else {
        const uint16_t* q = reinterpret_cast<const uint16_t*>(p);
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = (uint32_t)q[2 * i] | ((uint32_t)q[2 * i + 1] << 16);
    }
}
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ float block_amax(const uint32_t (&w)[8]) {
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) m = fmaxf(m, fmaxf(fabsf(bf_lo(w[i])), fabsf(bf_hi(w[i]))));
    return m;
}

// One block per row: row scale g = max|row| / (6 * 448) (1 for a zero row); per 16-element block the scale
// s = e4m3((max|block| / 6) / g) and the codes e2m1(x / (s * g)).  The input is taken as bfloat16.  K is a multiple of 16.
// A thread owns one 16-element block, loaded once in two 16-byte pieces and kept in registers between the two passes (the
// blocks beyond kQuantThreads of a long row are read again from the L1): with few rows the kernel is one memory round trip,
// one reduction and the arithmetic.  Measured with 34 rows: K 4096 2.9 us, K 12288 4.3 us (6.2 and 15.1 us with single
// elements read in either pass).
constexpr int kQuantThreads = 1024;
template <typename T>
__global__ void __launch_bounds__(kQuantThreads)
quantize_nvfp4_kernel(const T* __restrict__ x, int K, int vec, uint8_t* __restrict__ codes, uint8_t* __restrict__ sf,
                      float* __restrict__ g_out) {
    __shared__ float red[32];
    pdl_launch_dependents();
    pdl_wait();
    const size_t row = blockIdx.x;
    const T* xr = x + row * (size_t)K;
    const int nb = K >> 4;
    uint32_t w[8];
    float bmax = 0.f, amax = 0.f;
    if ((int)threadIdx.x < nb) {
        ld_block16(xr + 16 * threadIdx.x, vec != 0, w);
        amax = bmax = block_amax(w);
    }
    for (int b = threadIdx.x + blockDim.x; b < nb; b += blockDim.x) {
        uint32_t t[8];
        ld_block16(xr + 16 * b, vec != 0, t);
        amax = fmaxf(amax, block_amax(t));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
    __syncthreads();
    amax = (threadIdx.x & 31) < (blockDim.x >> 5) ? red[threadIdx.x & 31] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    const float g = amax > 0.f ? __fdiv_rn(amax, 6.0f * 448.0f) : 1.f;
    if (threadIdx.x == 0) g_out[row] = g;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        if (b != (int)threadIdx.x) {
            ld_block16(xr + 16 * b, vec != 0, w);
            bmax = block_amax(w);
        }
        const uint32_t sc = (uint32_t)__nv_cvt_float_to_fp8(__fdiv_rn(__fdiv_rn(bmax, 6.0f), g), __NV_SATFINITE, __NV_E4M3);
        const float d = __fmul_rn(e4m3_value(sc), g);
        sf[row * (size_t)nb + b] = (uint8_t)sc;
        uint32_t lo = 0, hi = 0;
        if (d > 0.f) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                lo |= (e2m1_code(__fdiv_rn(bf_lo(w[i]), d)) | (e2m1_code(__fdiv_rn(bf_hi(w[i]), d)) << 4)) << (8 * i);
                hi |= (e2m1_code(__fdiv_rn(bf_lo(w[4 + i]), d)) | (e2m1_code(__fdiv_rn(bf_hi(w[4 + i]), d)) << 4)) << (8 * i);
            }
        }
        *reinterpret_cast<uint2*>(codes + row * (size_t)(K / 2) + 8 * b) = make_uint2(lo, hi);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {      // looked up once, by whichever thread comes first
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        return cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
                       q == cudaDriverEntryPointSuccess ? (EncodeTiledFn)p : nullptr;
    }();
    return fn;
}

// [n_rows][row_bytes] bytes, box = box_bytes x box_rows, swizzled (codes) or plain (scales); out-of-range reads give 0
wd_status encode_bytes(CUtensorMap* m, const void* ptr, int n_rows, int row_bytes, int box_bytes, int box_rows, bool swizzle) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return WD_ERR_CUDA;
    if ((uintptr_t)ptr % 16 || row_bytes % 16) return WD_ERR_MISALIGNED;
    cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)n_rows};
    cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
    cuuint32_t box[2] = {(cuuint32_t)box_bytes, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? WD_OK : WD_ERR_CUDA;
}

// How the K blocks of all units are dealt out: whole units per CTA (one slice), or the line of all K blocks cut into `grid` equal
// shares, a unit's sums then being spread over up to n_slices slices.
struct Split { int grid, n_slices, aligned; };

// Time of a split: the stages of the longest share, and for every further slice its write and re-read at HBM speed (t_slice) and 0.3
// us, for the zero fill where nobody wrote it and for its place in the chain of the kernel that adds the slices; t_sum where there is
// such a kernel only because of them (a single operation's). A stage of one CTA takes 280 ns to load and issue, what comes in at 85
// GB/s, or its part of the HBM rate beside the other CTAs: at 34 rows 390 ns with 148 CTAs, 280 with up to 106, so whole units on
// fewer CTAs lose little.  Beside all SMs the grids tried give G / n_units a denominator of at most eight: shares then start with a
// unit every few units, which costs hardly a stage and saves slices.  With fewer slices allowed than all SMs would make (a long K
// with few units, little scratch) it is a smaller grid, not whole units.
// Measured at 34 rows, quantised input to summed result: 12288 x 4096 13.2 us with 144 shares and two slices, 11.0 with 96 whole units;
// 24576 x 4096 19.4, 16.4 with 192 whole units on 96 CTAs; 4096 x 12288 keeps 144 shares, five slices.  5 rows of 300, K 16384: 12.3 us
// (48 CTAs), with whole units 34.8 (3 CTAs).
Split choose_split(int n_units, int kb, int sm_count, int max_slices, int w_bytes, int x_bytes, double t_slice, double t_sum) {
    const long long W = (long long)n_units * kb;
    auto stage = [&](int G) { return std::max({280e-9, (w_bytes + x_bytes) / 85e9, (double)w_bytes * G / 7.0e12}); };
    const int per_cta = (n_units + sm_count - 1) / sm_count, g_unit = (n_units + per_cta - 1) / per_cta;
    Split best = {std::min(sm_count, n_units), 1, 1};
    if (n_units >= 4 * sm_count) return best;               // rounds of whole units are full enough
    best.grid = g_unit;
    double t_best = (double)per_cta * kb * stage(g_unit);
    auto consider = [&](long long G) {
        if (G < 1 || G > sm_count || G > W || W * (G + 1) > INT_MAX) return;
        const int ns = wd_tc_sharers(n_units, (int)G);
        if (ns > max_slices) return;
        const double t = (double)((W + G - 1) / G) * stage((int)G) + (ns - 1) * (t_slice + 0.3e-6) + (ns > 1 ? t_sum : 0.0);
        if (t < t_best * 0.999) {
            t_best = t;
            best = {(int)G, ns, 0};
        }
    };
    for (int q = 1; q <= 8; ++q) {
        long long j = (long long)sm_count * q / n_units;
        if (q == 1) j = std::min<long long>(j, max_slices);
        if (n_units * j % q == 0) consider(n_units * j / q);
    }
    consider(sm_count);
    return best;
}

}  // namespace

size_t wd_fp4_operand_bytes(int n_rows, int K) {
    return wd_align_up((size_t)n_rows * (K / 2), 256) + wd_align_up((size_t)n_rows * (K / 16), 256) + wd_align_up((size_t)n_rows * 4, 256);
}

void wd_fp4_operand_split(void* mem, int n_rows, int K, WdFp4Operand* op) {
    char* p = (char*)mem;
    op->codes = (uint8_t*)p; p += wd_align_up((size_t)n_rows * (K / 2), 256);
    op->sf = (uint8_t*)p; p += wd_align_up((size_t)n_rows * (K / 16), 256);
    op->g = (float*)p;
    op->n_rows = n_rows;
    op->K = K;
}

void wd_launch_quantize_nvfp4(int dtype, const void* x, int n_rows, int K, const WdFp4Operand* op, cudaStream_t st) {
    if (n_rows <= 0) return;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_rows);
    cfg.blockDim = dim3((unsigned)std::min(kQuantThreads, wd_ceil_div(K / 16, 32) * 32));
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = wd_pdl_enabled ? 1 : 0;
    ++wd_launch_counter;
    for (const void* f : {(const void*)quantize_nvfp4_kernel<float>, (const void*)quantize_nvfp4_kernel<__nv_bfloat16>}) wd_prefer_max_shared(f);
    const int vec = (uintptr_t)x % 16 == 0 ? 1 : 0;
    if (dtype == WD_F32) cudaLaunchKernelEx(&cfg, quantize_nvfp4_kernel<float>, (const float*)x, K, vec, op->codes, op->sf, op->g);
    else cudaLaunchKernelEx(&cfg, quantize_nvfp4_kernel<__nv_bfloat16>, (const __nv_bfloat16*)x, K, vec, op->codes, op->sf, op->g);
}

wd_status wd_fp4_gemm(const WdFp4Operand* x, const WdFp4Operand* w, float* y, size_t y_floats, int sm_count, int32_t* status,
                      cudaStream_t stream, int* n_split_out, bool force_single_split, bool w_static, float* y_sum) {
    if (!x || !w || !y || !status) return WD_ERR_NULL;
    const int rows = x->n_rows, n_out = w->n_rows, K = x->K;
    if (rows < 1 || n_out < 1 || K < kKB || K % kKB || w->K != K) return WD_ERR_BAD_PARAM;
    Fp4Params p;
    memset(&p, 0, sizeof(p));
    p.rows = rows;
    p.n_out = n_out;
    p.tok_tiles = (rows + 127) / 128;
    p.bn = ((rows + p.tok_tiles - 1) / p.tok_tiles + 15) / 16 * 16;        // balanced token tiles, <= 128
    p.kb_total = K / kKB;
    const int n_tiles = (n_out + kBM - 1) / kBM;
    if ((long long)n_tiles * p.tok_tiles * std::max(p.kb_total, sm_count + 1) > INT_MAX) return WD_ERR_CAPACITY;
    p.n_units = n_tiles * p.tok_tiles;
    const size_t slice = (size_t)rows * n_out;
    if (slice > y_floats) return WD_ERR_CAPACITY;
    const int max_slices = (int)std::min<size_t>(WD_TC_MAX_SPLIT, y_floats / slice);
    const Split sp = choose_split(p.n_units, p.kb_total, sm_count, force_single_split ? 1 : max_slices, kStageW + kSfW, p.bn * 144,
                                  (double)slice * 8.0 / 6.5e12, y_sum ? 4e-6 : 0.0);
    if (y_sum && sp.n_slices == 1) y = y_sum;
    p.aligned = sp.aligned;
    p.n_slices = sp.n_slices;
    const int grid = sp.grid;
    int cols = 32;
    while (cols < p.bn) cols <<= 1;
    p.buf_cols = cols;
    const int stage = (kStageW + p.bn * 128 + kSfW + p.bn * 16 + 1023) & ~1023;
    p.n_stages = (200 * 1024) / stage;
    if (p.n_stages > 10) p.n_stages = 10;
    const size_t smem = (size_t)p.n_stages * stage + (2 * p.n_stages + 8) * 8 + 64 + 512 + 1024;
    p.y = y;
    p.split_stride = slice;
    p.gw = w->g;
    p.gx = x->g;
    p.status = status;
    p.w_static = w_static ? 1 : 0;
    // instruction descriptor of the block-scaled form: A and B e2m1 (format 1) K-major, unsigned e4m3 scales,
    // N in bits 17-22 (units of 8), M in bits 24-28 (units of 16), dense, K = 64
    p.idesc = (1u << 7) | (1u << 10) | ((uint32_t)(p.bn >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);

    CUtensorMap mx, mw, msx, msw;
    wd_status s;
    if ((s = encode_bytes(&mx, x->codes, rows, K / 2, 128, p.bn, true)) != WD_OK) return s;
    if ((s = encode_bytes(&mw, w->codes, n_out, K / 2, 128, kBM, true)) != WD_OK) return s;
    if ((s = encode_bytes(&msx, x->sf, rows, K / 16, 16, p.bn, false)) != WD_OK) return s;
    if ((s = encode_bytes(&msw, w->sf, n_out, K / 16, 16, kBM, false)) != WD_OK) return s;
    static bool attr_done[64] = {};
    int dev = 0;
    WD_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return WD_ERR_CUDA;
    if (!attr_done[dev]) {
        WD_CUDA_TRY(cudaFuncSetAttribute(gemm_fp4_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024));
        attr_done[dev] = true;
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)grid);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = wd_pdl_enabled ? 1 : 0;
    ++wd_launch_counter;
    WD_CUDA_TRY(cudaLaunchKernelEx(&lc, gemm_fp4_kernel, mx, mw, msx, msw, p));
    if (n_split_out) *n_split_out = p.n_slices;
    return WD_OK;
}
