// Windowed bidirectional attention on the tensor cores (sm_100a), head_dim 128, bf16.
//
//   out[r, h, :] = softmax_j( q[r,h,:] . K[kvh, j, :] / sqrt(dh) ) V[kvh, j, :],   j in [0, n_vis)
//
// for the rows computed this step.  With a decoded prompt prefix the visible set of a sequence
// is always a range [0, n_vis) (decoded prefix | external window), so K and V tiles are plain
// TMA boxes of the cache; arbitrary index lists go through the CUDA-core kernel instead.
//
// One CTA per (128-row query tile of one sequence, query head):
//   warp 0    TMA: the Q tile once, then [128 keys x 128] K boxes and [128 x 128 keys] boxes of
//             the transposed V cache into a two-stage ring
//   warp 1    tcgen05.mma: S = Q K^T into TMEM, then O_tile = P V into TMEM; software-pipelined:
//             S and O_tile are double-buffered, Q K^T of the next key tile is issued before P V
//             of the current one, so the tensor core works while the softmax threads are busy
//   warps 2-9 two threads per query row (each takes 64 of the tile's 128 columns): tcgen05.ld of
//             its half of the S row, online softmax in fp32 (exp2 with the scale folded in; the
//             two halves exchange their row maxima through shared memory), P as bf16 into shared
//             memory in the 128-byte swizzled operand layout, then tcgen05.ld of its half of the
//             O_tile row accumulated in registers with the running rescale; final O / l as bf16
// Query rows beyond the tile's valid rows are computed on whatever the box holds and discarded
// (rows are independent).  Keys at or beyond n_vis are masked by selection, and their V
// columns are zeroed in shared memory, so stale or poisoned cache rows cannot leak in.
// When there are few (tile, head) pairs, as in a normal step, the keys are also split across
// the CTAs of a thread-block cluster (grid.z = cluster size <= 8) so that the machine is filled:
// each CTA leaves its running maximum, sum and unnormalised output in its own shared memory, and
// after a cluster barrier every CTA merges a share of the rows, reading the other parts through
// distributed shared memory in a fixed order (no global round trip, no atomics).
// Every wait is bounded; on expiry the CTA records WD_ERR_DEVICE_TIMEOUT and leaves.
#include <cstring>

#include <cstdlib>

#include "attention_tc.h"
#include "device_utils.cuh"

namespace {

using namespace wdk;

constexpr int kTile = 128;                 // query rows per CTA = keys per step = head_dim
constexpr int kAtom = kTile * 64 * 2;      // one [128 x 64] bf16 swizzle-atom column: 16 KB
constexpr int kOperand = 2 * kAtom;        // a [128 x 128] bf16 operand: 32 KB
constexpr int kThreads = 320;            // TMA warp, MMA warp, 8 softmax warps
constexpr int kTmemCols = 512;             // S0, S1: columns 0..255; O_tile0, O_tile1: columns 256..511
constexpr int kBars = 21;
constexpr int kMaxCluster = 8;             // portable cluster size

struct AttnParams {
    const int32_t* qtile_seq;    // [n_tiles] sequence of the tile
    const int32_t* qtile_row0;   // [n_tiles] first row (index into the step's row list)
    const int32_t* qtile_n;      // [n_tiles] valid rows
    const int32_t* seq_nvis;     // [batch] visible positions [0, n_vis)
    const int32_t* seq_qt_off;   // [batch + 1] first tile of each sequence (two-tile kernel)
    __nv_bfloat16* out;          // [rows][Hq*dh]
    float* tap;                  // optional fp32 copy
    int Hq, Hkv, layer;
    float scale_log2e;           // log2(e) / sqrt(dh)
    int32_t* status;
    uint32_t idesc;
    // split over the keys: CTA z of (tile, head) takes key tiles [z * tiles_per_split, ...); the
    // max_parts CTAs of a (tile, head) pair form one cluster
    int tiles_per_split, max_parts;
    // head packing (grouped-query attention with few rows): a 128-row query tile holds `pack` slots of `slot`
    // rows, one query head of the same KV head each (slot >= the tile's valid rows); grid.y = Hkv * tiles_per_kv
    int pack, slot, slot_shift, tiles_per_kv;      // slot = 128 / pack = 1 << slot_shift
};

__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t dsmem_addr(uint32_t local, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 dsmem_ld4(uint32_t a) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ float2 dsmem_ld2(uint32_t a) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    return v;
}

// 2^x by the special-function unit alone (x <= 0 here: results in [0, 1], denormals flushed)
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&v);
}

// barrier indices
constexpr int kQFull = 0, kKFull = 1, kKEmpty = 4, kVFull = 7, kVEmpty = 10, kSFull = 13, kPFull = 15, kOFull = 17,
              kOEmpty = 19;
constexpr int kStages = 3;                 // K stages and V stages

// kSingle: every CTA has at most one key tile (few keys, or keys split finely over the cluster): one K and one
// V stage, one S and one O buffer (256 tensor-memory columns), no running rescale — 97 KB of shared memory
// instead of 225 KB and fewer registers, so that the CTAs of the next kernel (the output projection, with a
// ring cut to fit) can be resident beside it and fetch their weights while the attention runs.
#ifdef WD_GEMM_TRACE
__device__ unsigned long long g_attn_end[64];       // latest CTA exit per layer
__device__ unsigned long long g_attn_trace[160][8]; // per CTA (last launch): entry, wait returned, S ready, P written, O ready, part written, merged, exit
#define A_STAMP(k) do { const unsigned int b_ = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z); g_attn_trace[b_ < 160 ? b_ : 159][k] = global_ns(); } while (0)
#else
#define A_STAMP(k) do { } while (0)
#endif

template <bool kSingle>
__device__ __forceinline__ void attention_tc_body(const CUtensorMap& map_q, const CUtensorMap& map_k, const CUtensorMap& map_vt,
                                                  const AttnParams& p) {
    constexpr int NS = kSingle ? 1 : kStages;
    constexpr uint32_t kCols = kSingle ? 256u : (uint32_t)kTmemCols;
    constexpr uint32_t kOBase = kSingle ? (uint32_t)kTile : (uint32_t)(2 * kTile);     // first column of the O buffers
    extern __shared__ uint8_t smem_raw[];
    // the same offset in every CTA of the cluster (the dynamic window starts at the same address)
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sQ = smem;                          // 32 KB
    uint8_t* sK = smem + kOperand;               // 3 stages x 32 KB
    uint8_t* sV = sK + NS * kOperand;       // 3 stages x 32 KB (transposed V tiles)
    uint64_t* bars = (uint64_t*)(sV + NS * kOperand);
    // q_full | k_full[3] | k_empty[3] | v_full[3] | v_empty[3] | s_full[2] | p_full[2] | o_full[2] | o_empty[2].
    // p_full and o_empty count the 256 softmax threads.  p_full is one barrier per S buffer, not one for all
    // tiles: the softmax threads can finish P(i+1) before the MMA thread has looked at P(i)'s barrier (it waits
    // for V(i) first), and a single barrier would then have gone through two phases unseen; P(i+2) on the
    // other hand needs S(i+2), which is issued only after the MMA thread has seen P(i).  P never touches shared memory: the softmax
    // threads write it as bf16 over the S buffer they have just read (tcgen05.st) and P V takes its A
    // operand from tensor memory.  No "S empty" / "P empty" barriers are needed: the tensor core runs the
    // MMAs in issue order (Q K^T(i+1), P V(i), Q K^T(i+2), ...), so S buffer i & 1 is rewritten by
    // Q K^T(i+2) only after P V(i) has read P(i) from it, and P V(i) was issued after P(i) was complete.
    // K and V stages are released separately: a K stage as soon as Q K^T has read it, a V stage after P V.
    uint32_t* tmem_slot = (uint32_t*)(bars + kBars + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    // after the last P V the K/V ring is free: this CTA's part of a split lives there
    float* part_o = (float*)sK;                            // [128 rows][128], 16-byte chunks XOR-swizzled by row
    // [128 rows][2] running maximum, sum: behind the part's 64 KB; with one stage each that is the end of the
    // ring, so it goes where Q was (every Q K^T has completed by then)
    float* part_ml = kSingle ? (float*)sQ : (float*)(sK + 2 * kOperand);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = blockIdx.x;
    const int b = p.qtile_seq[tile], row0 = p.qtile_row0[tile], n_valid = p.qtile_n[tile];
    const int group = p.Hq / p.Hkv;
    const int kvh = (int)blockIdx.y / p.tiles_per_kv, hg = (int)blockIdx.y % p.tiles_per_kv;
    const int h = kvh * group + hg * p.pack;              // query head of slot 0; slot j holds head h + j
    const int n_slots = min(p.pack, group - hg * p.pack);  // slots of this tile that hold a head

    pdl_launch_dependents();
    // The index lists are complete before this kernel can start: a host-planned step copies them in
    // front of its first kernel, and a device-planned step's embedding kernel (the planner kernel's
    // successor) triggers its dependents only after its own wait, i.e. after the planner has finished.
    const int n_vis = p.seq_nvis[b];
    const int n_kt_all = (n_vis + kTile - 1) / kTile;
    const int n_parts = (n_kt_all + p.tiles_per_split - 1) / p.tiles_per_split;
    const int kt_begin = (int)blockIdx.z * p.tiles_per_split;
    // a CTA without key tiles still takes part in the cluster barriers below
    const bool has_work = kt_begin < n_kt_all;
    const int n_kt = has_work ? min(p.tiles_per_split, n_kt_all - kt_begin) : 0;
    uint32_t tmem_base = 0;
    if (has_work) {
        if (threadIdx.x == 0) {
            for (int i = 0; i < kBars; ++i)
                mbar_init(smem_u32(&bars[i]), (i == kPFull || i == kPFull + 1 || i == kOEmpty || i == kOEmpty + 1) ? 256u : 1u);
            *abort_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        if (warp == 1) tmem_alloc(smem_u32(tmem_slot), kCols);
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        tmem_base = *tmem_slot;
    }
    if (threadIdx.x == 64) A_STAMP(0);
    pdl_wait();                                   // q and the cache rows come from the previous kernel
    if (threadIdx.x == 64) A_STAMP(1);

    if (!has_work) {
        // nothing to compute
    } else if (warp == 0) {
        {
            // ---------------------------------------------------- TMA producer (the whole warp, see elect_one)
            const bool leader = elect_one();
            const uint32_t qf = smem_u32(&bars[kQFull]);
            // slot j: rows [row0, row0 + slot) of head h + j at tile rows [j * slot, ...); slots without a head
            // stay unwritten (their rows of S and O are never read)
            if (leader) mbar_expect_tx(qf, (uint32_t)(n_slots * p.slot * 256));
            for (int j = 0; j < n_slots; ++j) {
                const uint32_t dst = smem_u32(sQ) + (uint32_t)(j * p.slot * 128);
                if (!leader) continue;
                tma_load_2d(dst, &map_q, qf, (h + j) * kTile, row0);
                tma_load_2d(dst + kAtom, &map_q, qf, (h + j) * kTile + 64, row0);
            }
            const int bh = b * p.Hkv + kvh;
            auto load_k = [&](int j) -> bool {
                const int ks = j % NS;
                const uint32_t ph = (uint32_t)(j / NS) & 1u;
                const uint32_t kfull = smem_u32(&bars[kKFull + ks]);
                if (!mbar_wait_warp(smem_u32(&bars[kKEmpty + ks]), ph ^ 1u, abort_flag)) return false;   // stage free
                const uint32_t sk = smem_u32(sK) + (uint32_t)(ks * kOperand);
                const int kv0 = (kt_begin + j) * kTile;
                if (leader) {
                    mbar_expect_tx(kfull, kOperand);
                    tma_load_4d(sk, &map_k, kfull, 0, kv0, bh, p.layer);            // keys kv0.., dims 0..63
                    tma_load_4d(sk + kAtom, &map_k, kfull, 64, kv0, bh, p.layer);   // dims 64..127
                }
                return true;
            };
            // order of need: K(0), K(1), V(0), K(2), V(1), ...
            bool ok = load_k(0);
            for (int i = 0; i < n_kt && ok; ++i) {
                if (i + 1 < n_kt && !(ok = load_k(i + 1))) break;
                const int vs = i % NS;
                const uint32_t ph = (uint32_t)(i / NS) & 1u;
                const uint32_t vfull = smem_u32(&bars[kVFull + vs]);
                const uint32_t sv = smem_u32(sV) + (uint32_t)(vs * kOperand);
                const int kv0 = (kt_begin + i) * kTile;
                if (!(ok = mbar_wait_warp(smem_u32(&bars[kVEmpty + vs]), ph ^ 1u, abort_flag))) break;   // stage free
                if (leader) {
                    mbar_expect_tx(vfull, kOperand);
                    tma_load_4d(sv, &map_vt, vfull, kv0, 0, bh, p.layer);           // all dims, keys kv0..kv0+63
                    tma_load_4d(sv + kAtom, &map_vt, vfull, kv0 + 64, 0, bh, p.layer);
                }
            }
            if (!ok) {
                *abort_flag = 1;
                atomicCAS(p.status, 0, WD_ERR_DEVICE_TIMEOUT);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        {
            // ---------------------------------------------------- MMA issuer (the whole warp)
            const bool leader = elect_one();
            // tile i uses K/V stage i % 3, S buffer i & 1, O_tile buffer i & 1
            bool ok = mbar_wait_warp(smem_u32(&bars[kQFull]), 0, abort_flag);
            const uint64_t qd0 = make_sdesc(smem_u32(sQ)), qd1 = make_sdesc(smem_u32(sQ) + kAtom);
            auto issue_qk = [&](int j) -> bool {           // S[j&1] = Q K(j)^T
                const int s = j & 1, ks = j % NS;
                if (!mbar_wait_warp(smem_u32(&bars[kKFull + ks]), (uint32_t)(j / NS) & 1u, abort_flag)) return false;   // K(j) landed
                tc_fence_after();
                const uint32_t sk = smem_u32(sK) + (uint32_t)(ks * kOperand);
                const uint64_t kd0 = make_sdesc(sk), kd1 = make_sdesc(sk + kAtom);
                const uint32_t acc = tmem_base + (uint32_t)(s * kTile);
                if (leader) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) umma_bf16(acc, qd0 + 2 * kk, kd0 + 2 * kk, p.idesc, kk > 0);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) umma_bf16(acc, qd1 + 2 * kk, kd1 + 2 * kk, p.idesc, 1u);
                    umma_commit(smem_u32(&bars[kKEmpty + ks]));    // K stage free once these MMAs have read it
                    umma_commit(smem_u32(&bars[kSFull + s]));
                }
                return true;
            };
            ok = ok && issue_qk(0);
            for (int i = 0; i < n_kt && ok; ++i) {
                const int s = i & 1, vs = i % NS;
                const uint32_t ph = (uint32_t)(i >> 1) & 1u;
                if (i + 1 < n_kt && !(ok = issue_qk(i + 1))) break;                           // runs ahead of the softmax
                if (!(ok = mbar_wait_warp(smem_u32(&bars[kVFull + vs]), (uint32_t)(i / NS) & 1u, abort_flag))) break;   // V(i) landed
                if (!(ok = mbar_wait_warp(smem_u32(&bars[kPFull + s]), ph, abort_flag))) break;              // P(i) written
                if (!(ok = mbar_wait_warp(smem_u32(&bars[kOEmpty + s]), ph ^ 1u, abort_flag))) break;        // O_tile(i-2) folded
                tc_fence_after();
                const uint32_t sv = smem_u32(sV) + (uint32_t)(vs * kOperand);
                const uint64_t vd0 = make_sdesc(sv), vd1 = make_sdesc(sv + kAtom);
                const uint32_t acc = tmem_base + kOBase + (uint32_t)(s * kTile);
                const uint32_t pa = tmem_base + (uint32_t)(s * kTile);       // P(i): 64 columns over S(i)
                // O_tile = P V: reduction over the 128 keys of the tile, 16 keys = 8 columns of P per MMA
                if (leader) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) umma_bf16_ta(acc, pa + 8 * kk, vd0 + 2 * kk, p.idesc, kk > 0);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) umma_bf16_ta(acc, pa + 32 + 8 * kk, vd1 + 2 * kk, p.idesc, 1u);
                    umma_commit(smem_u32(&bars[kVEmpty + vs]));    // V stage free
                    umma_commit(smem_u32(&bars[kOFull + s]));      // O_tile(i) ready
                }
            }
            if (!ok) {
                *abort_flag = 1;
                atomicCAS(p.status, 0, WD_ERR_DEVICE_TIMEOUT);
            }
        }
        __syncwarp();
    } else {
        // -------------------------------------------------------- softmax + accumulate (two threads per row)
        const int quarter = warp & 3;                      // TMEM lanes 32*quarter .. +31
        const int hf = (warp - 2) >> 2;                    // which 64 columns of a 128-wide tile
        const int r = quarter * 32 + lane;                 // query row of the tile = TMEM lane
        // warps whose 32 rows are all beyond the valid ones only keep the barrier counts right.
        // The test is per warp, not per row: tcgen05.ld is warp-collective and must not diverge.
        const int sj = r >> p.slot_shift, rr_ = r & (p.slot - 1);       // slot (head h + sj) and row within the slot
        const bool live = ((quarter * 32) >> p.slot_shift) < n_slots && ((quarter * 32) & (p.slot - 1)) < n_valid;
        const bool valid = sj < n_slots && rr_ < n_valid;
        const int c_off = 64 * hf;
        const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16);
        float* xch = (float*)(tmem_slot + 4);              // [2][128] exchange between the two halves (row sums)
        uint16_t* xm = (uint16_t*)xch;                     // the same 1 KB as [2 parities][2][128] bf16 row maxima
        float o[64];
#pragma unroll
        for (int c = 0; c < 64; ++c) o[c] = 0.f;
        float m = -INFINITY, l = 0.f, alpha_prev = 0.f;
        bool ok = true;
        // o += O_tile(j) with tile j's rescale factor; done one tile late so that P V(j) has had
        // time to finish while this thread was busy with the next tile's softmax
        auto fold = [&](int j, float alpha) {
            const int s = j & 1;
            mbar_wait_stay(smem_u32(&bars[kOFull + s]), (uint32_t)(j >> 1) & 1u, abort_flag, ok);
            tc_fence_after();
            if (live) {
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += 32) {
                    uint32_t v[32];
                    tmem_ld32(t_row + kOBase + (uint32_t)(s * kTile + c_off + c0), v);
#pragma unroll
                    for (int c = 0; c < 32; ++c) o[c0 + c] = kSingle ? __uint_as_float(v[c]) : o[c0 + c] * alpha + __uint_as_float(v[c]);
                }
            }
            tc_fence_before();
            mbar_arrive(smem_u32(&bars[kOEmpty + s]));     // O_tile buffer may be overwritten
        };
        for (int i = 0; i < n_kt; ++i) {
            const int s = i & 1;
            // A failed wait must not leave the loop: the other warps would wait at the named barrier below for ever.  It
            // raises the CTA's abort flag, and every thread goes through the remaining tiles, whose waits give up at once.
            mbar_wait_stay(smem_u32(&bars[kSFull + s]), (uint32_t)(i >> 1) & 1u, abort_flag, ok);
            tc_fence_after();
            if (threadIdx.x == 64 && i == 0) A_STAMP(2);
            const int n_keys = min(kTile, n_vis - (kt_begin + i) * kTile);   // valid keys in this tile
            // keys past n_vis may hold anything: zero their V columns so that 0 * garbage stays 0.
            // Thread (r, hf) owns row r (a head dim) of atom hf (keys 64*hf..) of the transposed V tile.
            if (n_keys < c_off + 64) {
                mbar_wait_stay(smem_u32(&bars[kVFull + i % NS]), (uint32_t)(i / NS) & 1u, abort_flag, ok);   // V landed
                uint8_t* vt = sV + (size_t)(i % NS) * kOperand + hf * kAtom + r * 128;
                for (int kv = max(n_keys - c_off, 0); kv < 64; ++kv)
                    *reinterpret_cast<uint16_t*>(vt + (((kv >> 3) ^ (r & 7)) << 4) + (kv & 7) * 2) = 0;
            }
            // This thread's 64 raw scores stay in registers for both passes.  The softmax warps are
            // bound by instruction issue, so the passes are kept to one FMNMX, then one FFMA + one MUFU
            // + one FADD (+ half a pack) per score: the scale is folded into the exponent's FFMA
            // (exp2(s * c - m * c)), and only the last, ragged key tile pays for the masking.
            float sc[64];
            float mx = -INFINITY;
            if (live) {
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += 32) {
                    uint32_t v[32];
                    tmem_ld32(t_row + (uint32_t)(s * kTile + c_off + c0), v);
                    if (n_keys >= kTile) {
#pragma unroll
                        for (int c = 0; c < 32; ++c) {
                            sc[c0 + c] = __uint_as_float(v[c]);
                            mx = fmaxf(mx, sc[c0 + c]);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 32; ++c) {
                            sc[c0 + c] = (c_off + c0 + c < n_keys) ? __uint_as_float(v[c]) : -INFINITY;
                            mx = fmaxf(mx, sc[c0 + c]);
                        }
                    }
                }
                mx *= p.scale_log2e;                       // the scale is positive; -inf stays -inf
            }
            // The two halves of a row must use the same reference value, and any upper bound of the scores
            // serves (softmax does not depend on it): each half rounds its maximum up to bf16 and both take
            // the larger.  Sixteen bits per value leave room for one buffer per tile parity, so a thread
            // that is already a tile ahead cannot overwrite what its partner has yet to read.
            {
                uint32_t mb = __float_as_uint(mx);
                mb = (mb & 0x80000000u) ? (mb & 0xffff0000u) : ((mb + 0xffffu) & 0xffff0000u);
                mx = __uint_as_float(mb);
                xm[((i & 1) * 2 + hf) * kTile + r] = (uint16_t)(mb >> 16);
            }
            asm volatile("bar.sync 1, 256;" ::: "memory");
            float alpha = 0.f;
            if (live) {
                mx = fmaxf(fmaxf(mx, __uint_as_float((uint32_t)xm[((i & 1) * 2 + (hf ^ 1)) * kTile + r] << 16)), m);
                alpha = ex2_approx(m - mx);                // m = -inf on the first tile gives 0
                m = mx;
                l *= alpha;
            }
            // P(i) as bf16 pairs over the S buffer: both threads of the row hold their scores in registers
            // (the barrier above), and the tensor core is done with whatever these columns held before
            if (live) {
                uint32_t pw[32];
                const float neg_mx = -mx;
                float l0 = 0.f, l1 = 0.f;
#pragma unroll
                for (int g = 0; g < 32; ++g) {
                    // masked keys: fma(-inf, c, -m) = -inf, exp2(-inf) = 0
                    const float p0 = ex2_approx(fmaf(sc[2 * g], p.scale_log2e, neg_mx));
                    const float p1 = ex2_approx(fmaf(sc[2 * g + 1], p.scale_log2e, neg_mx));
                    l0 += p0;
                    l1 += p1;
                    pw[g] = pack_bf16(p0, p1);
                }
                l += l0 + l1;
                tmem_st32(t_row + (uint32_t)(s * kTile + 32 * hf), pw);
            }
            fence_proxy_async_smem();                      // the zeroed V columns -> visible to the MMA
            tc_fence_before();
            mbar_arrive(smem_u32(&bars[kPFull + s]));
            if (threadIdx.x == 64 && i == n_kt - 1) A_STAMP(3);
            if (!kSingle && i > 0) fold(i - 1, alpha_prev);
            alpha_prev = alpha;
        }
        if (n_kt > 0) fold(n_kt - 1, alpha_prev);
        if (threadIdx.x == 64) A_STAMP(4);
        // row sum = sum of the two halves (same running maximum on both sides)
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (*abort_flag) {
            ok = false;
            if (threadIdx.x == 64) atomicCAS(p.status, 0, WD_ERR_DEVICE_TIMEOUT);
        }
        xch[hf * kTile + r] = l;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        l += xch[(hf ^ 1) * kTile + r];
        if (n_parts == 1) {
            if (ok && valid) {
                const float inv = 1.f / l;
                const size_t base = ((size_t)(row0 + rr_) * p.Hq + h + sj) * kTile + c_off;
                uint4* dst = reinterpret_cast<uint4*>(p.out + base);
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    uint4 u;
                    u.x = pack_bf16(o[8 * g + 0] * inv, o[8 * g + 1] * inv);
                    u.y = pack_bf16(o[8 * g + 2] * inv, o[8 * g + 3] * inv);
                    u.z = pack_bf16(o[8 * g + 4] * inv, o[8 * g + 5] * inv);
                    u.w = pack_bf16(o[8 * g + 6] * inv, o[8 * g + 7] * inv);
                    dst[g] = u;
                }
                if (p.tap) {
#pragma unroll
                    for (int c = 0; c < 64; ++c) p.tap[base + c] = o[c] * inv;
                }
            }
        } else if (valid) {
            // this CTA's part: every tensor-core read of the K/V ring has completed (the last fold
            // waited for the last P V), so the ring is reused.  Chunk c of row r sits at c ^ (r & 31).
            float4* dst = reinterpret_cast<float4*>(part_o + (size_t)r * kTile);
#pragma unroll
            for (int g = 0; g < 16; ++g)
                dst[(hf * 16 + g) ^ (r & 31)] = make_float4(o[4 * g], o[4 * g + 1], o[4 * g + 2], o[4 * g + 3]);
            if (hf == 0) *reinterpret_cast<float2*>(part_ml + r * 2) = make_float2(m, l);
        }
    }
    if (p.max_parts > 1) {
        // ------------------------------------------------------------ merge across the cluster
        if (threadIdx.x == 64) A_STAMP(5);
        cluster_sync_all();                                // every part is in place and visible
        if (has_work && n_parts > 1 && warp >= 2) {
            // CTA z merges rows [z * per, (z + 1) * per).  An item = (row, group of 4 columns); a
            // thread takes items t, t + 256, ... and keeps kItems x kParts remote loads in flight.
            constexpr int kItems = 2, kParts = 4;
            // (rows are counted over the valid rows of all slots: index q = slot * n_valid + row within the slot)
            const int n_tot = n_slots * n_valid;
            const int per = (n_tot + n_parts - 1) / n_parts;
            const int r_lo = min((int)blockIdx.z * per, n_tot), r_hi = min(r_lo + per, n_tot);
            const int t = (int)threadIdx.x - 64, n_items = (r_hi - r_lo) * 32;
            const uint32_t lo = smem_u32(part_o), lml = smem_u32(part_ml);
            for (int it0 = t; it0 < n_items; it0 += 256 * kItems) {
                float mxx[kItems], lsum[kItems];
                float4 acc[kItems];
#pragma unroll
                for (int u = 0; u < kItems; ++u) {
                    mxx[u] = -INFINITY;
                    lsum[u] = 0.f;
                    acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                for (int z0 = 0; z0 < n_parts; z0 += kParts) {       // parts in order of z
                    float2 ml[kItems][kParts];
                    float4 v[kItems][kParts];
#pragma unroll
                    for (int u = 0; u < kItems; ++u) {
                        const int item = it0 + u * 256, qq = r_lo + (item >> 5), cg = item & 31;
                        const int rr = (qq / n_valid) * p.slot + qq % n_valid;         // tile row
#pragma unroll
                        for (int zz = 0; zz < kParts; ++zz) {
                            ml[u][zz] = make_float2(-INFINITY, 0.f);
                            v[u][zz] = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (item < n_items && z0 + zz < n_parts) {
                                ml[u][zz] = dsmem_ld2(dsmem_addr(lml + (uint32_t)rr * 8u, (uint32_t)(z0 + zz)));
                                v[u][zz] = dsmem_ld4(dsmem_addr(lo + (uint32_t)rr * 512u + (uint32_t)((cg ^ (rr & 31)) << 4),
                                                                (uint32_t)(z0 + zz)));
                            }
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kItems; ++u) {
                        if (it0 + u * 256 >= n_items) continue;
                        float mnew = mxx[u];
#pragma unroll
                        for (int zz = 0; zz < kParts; ++zz) mnew = fmaxf(mnew, ml[u][zz].x);
                        const float keep = exp2f(mxx[u] - mnew);       // -inf on the first chunk gives 0
                        mxx[u] = mnew;
                        lsum[u] *= keep;
                        acc[u].x *= keep; acc[u].y *= keep; acc[u].z *= keep; acc[u].w *= keep;
#pragma unroll
                        for (int zz = 0; zz < kParts; ++zz) {
                            const float wgt = exp2f(ml[u][zz].x - mnew);   // absent parts: exp2(-inf) = 0
                            lsum[u] += ml[u][zz].y * wgt;
                            acc[u].x += v[u][zz].x * wgt; acc[u].y += v[u][zz].y * wgt;
                            acc[u].z += v[u][zz].z * wgt; acc[u].w += v[u][zz].w * wgt;
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < kItems; ++u) {
                    const int item = it0 + u * 256, qq = r_lo + (item >> 5), cg = item & 31;
                    if (item >= n_items) continue;
                    const float inv = 1.f / lsum[u];
                    const size_t base = ((size_t)(row0 + qq % n_valid) * p.Hq + h + qq / n_valid) * kTile + 4 * cg;
                    uint2 w2;
                    w2.x = pack_bf16(acc[u].x * inv, acc[u].y * inv);
                    w2.y = pack_bf16(acc[u].z * inv, acc[u].w * inv);
                    *reinterpret_cast<uint2*>(p.out + base) = w2;
                    if (p.tap)
                        *reinterpret_cast<float4*>(p.tap + base) =
                            make_float4(acc[u].x * inv, acc[u].y * inv, acc[u].z * inv, acc[u].w * inv);
                }
            }
        }
        if (threadIdx.x == 64) A_STAMP(6);
        cluster_sync_all();                                // no CTA leaves while its part may still be read
    }
    if (has_work) {
        tc_fence_before();
        __syncthreads();
        if (warp == 1) {
            tc_fence_after();
            tmem_dealloc(tmem_base, kCols);
        }
    }
#ifdef WD_GEMM_TRACE
    if (threadIdx.x == 0) atomicMax(&g_attn_end[p.layer & 63], global_ns());
    if (threadIdx.x == 64) A_STAMP(7);
#endif
}

__global__ void __launch_bounds__(kThreads, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                    const __grid_constant__ CUtensorMap map_vt, const AttnParams p) {
    attention_tc_body<false>(map_q, map_k, map_vt, p);
}

// (128 registers: 320 threads of this kernel and the 192 of a GEMM CTA fit the register file together)
__global__ void __maxnreg__(128)
attention_tc_single_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                           const __grid_constant__ CUtensorMap map_vt, const AttnParams p) {
    attention_tc_body<true>(map_q, map_k, map_vt, p);
}

// ------------------------------------------------------------------------------------------
// Two query tiles per CTA (the rule stands in wd_attn_tc_launch)
// ------------------------------------------------------------------------------------------
// A single-tile CTA is bound by its softmax warps: 2800 cycles per key tile, one phase after another (scores, maxima, a barrier
// between the two halves of a row, exponentials, P, the rescale of O in registers), against 1024 of the tensor core.  Here a CTA
// works on two query tiles over the same keys: consecutive (row tile, query head) items of one sequence and KV head.
//   warps 0, 1         TMA, MMA (2 and 3 are there to make a warpgroup, which hands its registers to the others)
//   warps 4-7 / 8-11   softmax of tile 0 / tile 1, one thread per query row: no exchange between threads, a row's 128 scores in
//                      registers, and while one tile's scores are exponentiated the tensor core works on the other's
//   O                  stays in tensor memory: P V accumulates over the key tiles, and a warp rescales its rows only when a row's
//                      maximum has grown by more than 2^8 since the reference value in use (any reference cancels in O / l)
// (Two tiles in turn and the rescale left out while the maximum grows little are the steps that FlashAttention-4 made known;
// written here from their description.)
// Tensor memory: S (and P over it) 2 x 128 columns, O 2 x 128.  Shared memory: two Q tiles, two K and two V stages, 192 KB.
// The tensor core runs Q K^T and P V in issue order, so S(i + 1) complete means P V(i) has read P(i) and has been added to O;
// one barrier each for S and P of a tile suffices (P(i + 1) needs S(i + 1), which is issued only after P(i) has been seen).
// What bounds it: the softmax, 3100 cycles per key tile and pair of query tiles without the MMAs, of which 2048 are the exponentials' (16 a
// cycle); K/V loads and MMAs hide behind it, now that their issue loops are run by converged warps (one lane alone took 3280 cycles for
// the MMAs of a key tile, and the launch of 1792 rows, 128 heads 255 us instead of 225; 640 rows, 40 heads, 2048 keys 43.5 / 38.1).
// Beside the loop a CTA spends 3 us until its first scores, 1.1
// us after the last exponentials and the write of O, so a few key tiles are dominated by both ends: one row of O per thread took
// 2.1-4.6 us (a warp's store touched 32 lines), staged through shared memory 0.5-1; loading tile 0 and its keys before tile 1, and
// zeroing V columns by 16 bytes while the scores are still being computed, the rest of 113 -> 98 us for eight sequences of
// 672 rows, 28 query and 4 KV heads, and 257 -> 249 us for 1792 rows, 128 heads.
// Measured per launch against the single-tile kernel: see wd_attn_tc_launch.
constexpr int kDThreads = 384;
// Registers per thread after the hand-over: 56 for the first warpgroup, 224 for the other two.  The launch has 168 for each of
// the 384 threads (the most that fit the register file), and 128 * 56 + 256 * 224 = 384 * 168.
constexpr int kDBars = 16;
constexpr int kDQ = 0, kDKFull = 2, kDKEmpty = 4, kDVFull = 6, kDVEmpty = 8, kDSFull = 10, kDPFull = 12, kDODone = 14;
constexpr size_t kDualSmem = 6 * (size_t)kOperand + (kDBars + 2) * 8 + 1024;

__device__ __forceinline__ uint64_t f32x2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f32x2_get(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t f32x2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t f32x2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__global__ void __launch_bounds__(kDThreads, 1)
attention_tc_dual_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                         const __grid_constant__ CUtensorMap map_vt, const AttnParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sQ = smem;                              // two tiles
    uint8_t* sK = smem + 2 * kOperand;               // two stages
    uint8_t* sV = sK + 2 * kOperand;                 // two stages (transposed V tiles)
    uint64_t* bars = (uint64_t*)(sV + 2 * kOperand);
    uint32_t* tmem_slot = (uint32_t*)(bars + kDBars);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    pdl_launch_dependents();
    // (the index lists are complete before this kernel can start: see attention_tc_body)
    const int b = blockIdx.z, kvh = blockIdx.y, item0 = 2 * (int)blockIdx.x;
    const int tile0 = p.seq_qt_off[b], n_items = (p.seq_qt_off[b + 1] - tile0) * p.tiles_per_kv;
    if (item0 >= n_items) return;                    // a shorter sequence of the batch
    const int n_q = min(2, n_items - item0);         // query tiles of this CTA
    const int n_vis = p.seq_nvis[b], n_kt = (n_vis + kTile - 1) / kTile;
    const int group = p.Hq / p.Hkv;
    struct Item { int row0, n_valid, h, n_slots; };
    auto item = [&](int t) {
        const int e = item0 + t, hg = e % p.tiles_per_kv;
        const int tile = tile0 + e / p.tiles_per_kv;
        Item r;
        r.row0 = p.qtile_row0[tile];
        r.n_valid = p.qtile_n[tile];
        r.h = kvh * group + hg * p.pack;             // query head of slot 0
        r.n_slots = min(p.pack, group - hg * p.pack);
        return r;
    };

    if (threadIdx.x == 0) {
        for (int i = 0; i < kDBars; ++i) mbar_init(smem_u32(&bars[i]), (i == kDPFull || i == kDPFull + 1) ? 128u : 1u);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (const CUtensorMap* m : {&map_q, &map_k, &map_vt}) asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(tmem_slot), (uint32_t)kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();                                      // q and the cache rows come from the previous kernel
    // (the hand-over stands inside the branches: the compiler gives each the registers it has after it)
    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp == 0) {
            {
                // ---------------------------------------------------- TMA producer (the whole warp)
                const bool leader = elect_one();
                const int bh = b * p.Hkv + kvh;
                auto load_q = [&](int t) {
                    const Item q = item(t);
                    const uint32_t qf = smem_u32(&bars[kDQ + t]);
                    if (leader) mbar_expect_tx(qf, (uint32_t)(q.n_slots * p.slot * 256));
                    for (int j = 0; j < q.n_slots; ++j) {
                        if (!leader) continue;
                        const uint32_t dst = smem_u32(sQ) + (uint32_t)(t * kOperand + j * p.slot * 128);
                        tma_load_2d(dst, &map_q, qf, (q.h + j) * kTile, q.row0);
                        tma_load_2d(dst + kAtom, &map_q, qf, (q.h + j) * kTile + 64, q.row0);
                    }
                };
                load_q(0);                                             // the first tile and its keys come first: S(0) of tile 0 starts on them
                bool ok = true;
                for (int i = 0; i < n_kt && ok; ++i) {
                    const int s = i & 1, kv0 = i * kTile;
                    const uint32_t ph = ((uint32_t)(i >> 1) & 1u) ^ 1u;
                    const uint32_t kf = smem_u32(&bars[kDKFull + s]), vf = smem_u32(&bars[kDVFull + s]);
                    const uint32_t sk = smem_u32(sK) + (uint32_t)(s * kOperand), sv = smem_u32(sV) + (uint32_t)(s * kOperand);
                    if (!(ok = mbar_wait_warp(smem_u32(&bars[kDKEmpty + s]), ph, abort_flag))) break;
                    if (leader) {
                        mbar_expect_tx(kf, kOperand);
                        tma_load_4d(sk, &map_k, kf, 0, kv0, bh, p.layer);             // keys kv0.., dims 0..63
                        tma_load_4d(sk + kAtom, &map_k, kf, 64, kv0, bh, p.layer);    // dims 64..127
                    }
                    if (i == 0 && n_q == 2) load_q(1);
                    if (!(ok = mbar_wait_warp(smem_u32(&bars[kDVEmpty + s]), ph, abort_flag))) break;
                    if (leader) {
                        mbar_expect_tx(vf, kOperand);
                        tma_load_4d(sv, &map_vt, vf, kv0, 0, bh, p.layer);            // all dims, keys kv0..kv0+63
                        tma_load_4d(sv + kAtom, &map_vt, vf, kv0 + 64, 0, bh, p.layer);
                    }
                }
                if (!ok) {
                    *abort_flag = 1;
                    atomicCAS(p.status, 0, WD_ERR_DEVICE_TIMEOUT);
                }
            }
            __syncwarp();
        } else if (warp == 1) {
            {
                // ---------------------------------------------------- MMA issuer (the whole warp)
                const bool leader = elect_one();
                auto issue_qk = [&](int t, int i) {                   // S_t = Q_t K(i)^T
                    if (!leader) return;
                    const uint64_t qd = make_sdesc(smem_u32(sQ) + (uint32_t)(t * kOperand));
                    const uint64_t kd = make_sdesc(smem_u32(sK) + (uint32_t)((i & 1) * kOperand));
                    const uint32_t acc = tmem_base + (uint32_t)(t * kTile);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {
                        const uint64_t o = (uint64_t)((kk >> 2) * (kAtom >> 4) + 2 * (kk & 3));
                        umma_bf16(acc, qd + o, kd + o, p.idesc, kk > 0);
                    }
                    umma_commit(smem_u32(&bars[kDSFull + t]));
                    if (t == n_q - 1) umma_commit(smem_u32(&bars[kDKEmpty + (i & 1)]));     // K stage free
                };
                bool ok = mbar_wait_warp(smem_u32(&bars[kDKFull]), 0, abort_flag);
                for (int t = 0; t < n_q && ok; ++t) {
                    if (!(ok = mbar_wait_warp(smem_u32(&bars[kDQ + t]), 0, abort_flag))) break;
                    tc_fence_after();
                    issue_qk(t, 0);
                }
                for (int i = 0; i < n_kt && ok; ++i) {
                    const uint32_t ph = (uint32_t)(i >> 1) & 1u;
                    if (!(ok = mbar_wait_warp(smem_u32(&bars[kDVFull + (i & 1)]), ph, abort_flag))) break;          // V(i) landed
                    for (int t = 0; t < n_q; ++t) {
                        if (!(ok = mbar_wait_warp(smem_u32(&bars[kDPFull + t]), (uint32_t)i & 1u, abort_flag))) break;   // P_t(i) written, O_t rescaled
                        tc_fence_after();
                        const uint64_t vd = make_sdesc(smem_u32(sV) + (uint32_t)((i & 1) * kOperand));
                        const uint32_t acc = tmem_base + (uint32_t)(2 * kTile + t * kTile), pa = tmem_base + (uint32_t)(t * kTile);
                        if (leader) {
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk)                // 16 keys = 8 columns of P per MMA
                                umma_bf16_ta(acc, pa + 8 * kk, vd + (uint64_t)((kk >> 2) * (kAtom >> 4) + 2 * (kk & 3)), p.idesc, (i > 0 || kk > 0) ? 1u : 0u);
                            if (t == n_q - 1) umma_commit(smem_u32(&bars[kDVEmpty + (i & 1)]));     // V stage free
                            if (i == n_kt - 1) umma_commit(smem_u32(&bars[kDODone + t]));
                        }
                        if (i + 1 < n_kt) {
                            if (t == 0 && !(ok = mbar_wait_warp(smem_u32(&bars[kDKFull + ((i + 1) & 1)]), (uint32_t)((i + 1) >> 1) & 1u, abort_flag))) break;
                            tc_fence_after();
                            issue_qk(t, i + 1);
                        }
                    }
                }
                if (!ok) {
                    *abort_flag = 1;
                    atomicCAS(p.status, 0, WD_ERR_DEVICE_TIMEOUT);
                }
            }
            __syncwarp();
        }
        __syncwarp();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        // -------------------------------------------------------- softmax, one thread per query row
        const int t = (warp - 4) >> 2, quarter = warp & 3;        // query tile; TMEM lanes 32*quarter .. +31
        const int r = quarter * 32 + lane;
        bool ok = true;
        if (t < n_q) {
            const Item q = item(t);
            // warps whose rows are all beyond the valid ones only keep the barrier counts right (the test is per warp:
            // tcgen05.ld and .st are warp-collective)
            const int sj = r >> p.slot_shift, rr = r & (p.slot - 1);          // slot (head q.h + sj) and row within it
            const bool live = ((quarter * 32) >> p.slot_shift) < q.n_slots && ((quarter * 32) & (p.slot - 1)) < q.n_valid;
            const uint32_t t_s = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(t * kTile);
            const uint32_t t_o = t_s + (uint32_t)(2 * kTile);
            const uint64_t c2 = f32x2(p.scale_log2e, p.scale_log2e);
            float m = 0.f, l = 0.f;
            for (int i = 0; i < n_kt; ++i) {
                const int n_keys = min(kTile, n_vis - i * kTile);             // valid keys of this tile
                // keys past n_vis may hold anything: zero their V columns so that 0 * garbage stays 0 (tile 0's threads, row r
                // of the transposed V tile = head dim r; P V of either tile is issued after tile 0's P has been seen)
                if (n_keys < kTile && t == 0) {
                    mbar_wait_stay(smem_u32(&bars[kDVFull + (i & 1)]), (uint32_t)(i >> 1) & 1u, abort_flag, ok);
                    uint8_t* vt = sV + (size_t)(i & 1) * kOperand + r * 128;
                    auto at = [&](int kv) { return vt + (kv >> 6) * kAtom + ((((kv & 63) >> 3) ^ (r & 7)) << 4) + (kv & 7) * 2; };
                    int kv = n_keys;
                    for (; kv & 7; ++kv) *reinterpret_cast<uint16_t*>(at(kv)) = 0;
                    for (; kv < kTile; kv += 8) *reinterpret_cast<uint4*>(at(kv)) = make_uint4(0, 0, 0, 0);
                    fence_proxy_async_smem();
                }
                mbar_wait_stay(smem_u32(&bars[kDSFull + t]), (uint32_t)i & 1u, abort_flag, ok);      // (a failed wait goes on: its output is not written)
                tc_fence_after();
                if (live) {
                    uint32_t sc[4][32];
                    float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        tmem_ld32(t_s + (uint32_t)(32 * c), sc[c]);
                        if (n_keys < kTile) {
#pragma unroll
                            for (int k = 0; k < 32; ++k)
                                if (32 * c + k >= n_keys) sc[c][k] = __float_as_uint(-INFINITY);
                        }
#pragma unroll
                        for (int k = 0; k < 32; k += 2) {
                            mx0 = fmaxf(mx0, __uint_as_float(sc[c][k]));
                            mx1 = fmaxf(mx1, __uint_as_float(sc[c][k + 1]));
                        }
                    }
                    const float mx = fmaxf(mx0, mx1) * p.scale_log2e;          // the scale is positive
                    if (i == 0) {
                        m = mx;
                    } else if (__any_sync(0xffffffffu, mx > m + 8.f)) {
                        // (P V(i - 1) is complete: S(i) was issued behind it)
                        const float mn = fmaxf(m, mx), alpha = ex2_approx(m - mn);
                        m = mn;
                        l *= alpha;
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            uint32_t v[32];
                            tmem_ld32(t_o + (uint32_t)(32 * c), v);
#pragma unroll
                            for (int k = 0; k < 32; ++k) v[k] = __float_as_uint(__uint_as_float(v[k]) * alpha);
                            tmem_st32(t_o + (uint32_t)(32 * c), v);
                        }
                    }
                    const uint64_t nm2 = f32x2(-m, -m);
                    uint64_t l2[2] = {0ull, 0ull};
#pragma unroll
                    for (int hc = 0; hc < 2; ++hc) {
                        uint32_t pw[32];
#pragma unroll
                        for (int g = 0; g < 32; ++g) {
                            // masked keys: fma(-inf, c, -m) = -inf, exp2(-inf) = 0
                            const uint32_t* q2 = &sc[2 * hc + (g >> 4)][2 * (g & 15)];
                            float a, c;
                            f32x2_get(f32x2_fma(f32x2(__uint_as_float(q2[0]), __uint_as_float(q2[1])), c2, nm2), a, c);
                            a = ex2_approx(a);
                            c = ex2_approx(c);
                            l2[g & 1] = f32x2_add(l2[g & 1], f32x2(a, c));
                            pw[g] = pack_bf16(a, c);
                        }
                        tmem_st32(t_s + (uint32_t)(32 * hc), pw);             // P over the S columns: all scores are in registers
                    }
                    float a, c;
                    f32x2_get(f32x2_add(l2[0], l2[1]), a, c);
                    l += a + c;
                }
                tc_fence_before();
                mbar_arrive(smem_u32(&bars[kDPFull + t]));
            }
            mbar_wait_stay(smem_u32(&bars[kDODone + t]), 0, abort_flag, ok);
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after();
            if (ok && live) {
                // through shared memory (the warp's rows of the Q tile, which no MMA reads any more), so that a store instruction
                // writes two whole rows of 256 bytes: with a thread to a row it touched 32 lines
                const float inv = 1.f / l;
                const int rr0 = (quarter * 32) & (p.slot - 1), n_out = min(32, q.n_valid - rr0);     // the warp's valid rows
                uint8_t* st = sQ + (size_t)t * kOperand + quarter * 8192;
                __nv_bfloat16* out = p.out + ((size_t)(q.row0 + rr0) * p.Hq + q.h + sj) * kTile;
                const size_t pitch = (size_t)p.Hq * kTile;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t v[32];
                    tmem_ld32(t_o + (uint32_t)(32 * c), v);
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        uint4 u;
                        u.x = pack_bf16(__uint_as_float(v[8 * g]) * inv, __uint_as_float(v[8 * g + 1]) * inv);
                        u.y = pack_bf16(__uint_as_float(v[8 * g + 2]) * inv, __uint_as_float(v[8 * g + 3]) * inv);
                        u.z = pack_bf16(__uint_as_float(v[8 * g + 4]) * inv, __uint_as_float(v[8 * g + 5]) * inv);
                        u.w = pack_bf16(__uint_as_float(v[8 * g + 6]) * inv, __uint_as_float(v[8 * g + 7]) * inv);
                        *reinterpret_cast<uint4*>(st + lane * 256 + (((4 * c + g) ^ (lane & 7)) << 4)) = u;
                    }
                    if (p.tap && lane < n_out) {
#pragma unroll
                        for (int k = 0; k < 32; ++k)
                            p.tap[((size_t)(q.row0 + rr) * p.Hq + q.h + sj) * kTile + 32 * c + k] = __uint_as_float(v[k]) * inv;
                    }
                }
                __syncwarp();
                for (int r0 = lane >> 4; r0 < n_out; r0 += 8) {
                    uint4 u[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        u[k] = *reinterpret_cast<const uint4*>(st + (r0 + 2 * k) * 256 + (((lane & 15) ^ ((r0 + 2 * k) & 7)) << 4));
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (r0 + 2 * k < n_out) *reinterpret_cast<uint4*>(out + (r0 + 2 * k) * pitch + 8 * (lane & 15)) = u[k];
                }
            }
            if (!ok) {
                *abort_flag = 1;
                if (lane == 0) atomicCAS(p.status, 0, WD_ERR_DEVICE_TIMEOUT);
            }
        }
        tc_fence_before();
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)kTmemCols);
    }
}

#ifdef WD_GEMM_TRACE
extern "C" __attribute__((visibility("default"))) int wd_debug_attn_stamps(unsigned long long* host /*[160][8]*/) {
    cudaDeviceSynchronize();
    return (int)cudaMemcpyFromSymbol(host, g_attn_trace, sizeof(unsigned long long) * 160 * 8);
}
extern "C" __attribute__((visibility("default"))) int wd_debug_attn_trace(unsigned long long* host /*[64]*/) {
    cudaDeviceSynchronize();
    return (int)cudaMemcpyFromSymbol(host, g_attn_end, sizeof(unsigned long long) * 64);
}
#endif

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

}  // namespace

// K cache [L][BH][S][dh] -> dims (dh, S, BH, L), box (64, 128, 1, 1);
// transposed V cache [L][BH][dh][Sp] -> dims (Sp, dh, BH, L), box (64, 128, 1, 1)
wd_status wd_attn_tc_encode_cache(CUtensorMap* map_k, CUtensorMap* map_vt, const void* kcache, const void* vcache,
                                  int L, int BH, int S, int Sp, int dh) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return WD_ERR_CUDA;
    if (dh != kTile) return WD_ERR_BAD_PARAM;
    {
        cuuint64_t dims[4] = {(cuuint64_t)dh, (cuuint64_t)S, (cuuint64_t)BH, (cuuint64_t)L};
        cuuint64_t strides[3] = {(cuuint64_t)dh * 2, (cuuint64_t)S * dh * 2, (cuuint64_t)BH * S * dh * 2};
        cuuint32_t box[4] = {64, 128, 1, 1}, estr[4] = {1, 1, 1, 1};
        if (enc(map_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(kcache), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return WD_ERR_CUDA;
    }
    {
        cuuint64_t dims[4] = {(cuuint64_t)Sp, (cuuint64_t)dh, (cuuint64_t)BH, (cuuint64_t)L};
        cuuint64_t strides[3] = {(cuuint64_t)Sp * 2, (cuuint64_t)dh * Sp * 2, (cuuint64_t)BH * dh * Sp * 2};
        cuuint32_t box[4] = {64, 128, 1, 1}, estr[4] = {1, 1, 1, 1};
        if (enc(map_vt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(vcache), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return WD_ERR_CUDA;
    }
    return WD_OK;
}

wd_status wd_attn_tc_launch(const void* q, int n_rows, int n_tiles, const int32_t* qtile_seq, const int32_t* qtile_row0,
                            const int32_t* qtile_n, const int32_t* seq_nvis, const CUtensorMap* map_k,
                            const CUtensorMap* map_vt, void* out, float* tap, int Hq, int Hkv, int dh, int layer,
                            int max_vis, int sm_count, int32_t* status, cudaStream_t stream, int max_tile_rows,
                            size_t* smem_used, const int32_t* seq_qt_off, int batch, int max_seq_tiles, WdAttnQ* q_maps) {
    if (dh != kTile) return WD_ERR_BAD_PARAM;
    if (n_tiles <= 0) return WD_OK;
    EncodeTiledFn enc = get_encode();
    if (!enc) return WD_ERR_CUDA;
    int dev = 0;
    WD_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return WD_ERR_CUDA;
    // Grouped-query attention with few rows per tile: 2 or 4 query heads of one KV head share a 128-row tile
    // (slots of 64 or 32 rows), so their K/V tiles are loaded once and the grid shrinks by that factor
    const int group = Hq / Hkv;
    static const int pack_max = getenv("WD_ATTN_PACK") ? atoi(getenv("WD_ATTN_PACK")) : 4;     // 1 switches packing off
    int pack = 1;
    if (max_tile_rows > 0 && group > 1) {
        if (max_tile_rows <= 32 && group >= 4) pack = 4;
        else if (max_tile_rows <= 64) pack = 2;
        if (pack > pack_max) pack = pack_max >= 2 ? 2 : 1;
        if (pack == 2 && max_tile_rows > 64) pack = 1;
    }
    const int slot = kTile / pack;
    CUtensorMap mq;
    const WdAttnQ::Entry* known = nullptr;
    for (int i = 0; q_maps && i < 2; ++i) {
        const WdAttnQ::Entry& e = q_maps->entries[i];
        if (e.q == q && e.rows == n_rows && e.heads == Hq && e.slot == slot) known = &e;
    }
    if (known) {
        mq = known->map;
    } else {
        cuuint64_t dims[2] = {(cuuint64_t)Hq * dh, (cuuint64_t)n_rows};
        cuuint64_t strides[1] = {(cuuint64_t)Hq * dh * 2};
        cuuint32_t box[2] = {64, (cuuint32_t)slot}, estr[2] = {1, 1};
        if (enc(&mq, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(q), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return WD_ERR_CUDA;
        if (q_maps) {
            q_maps->entries[q_maps->next] = {q, n_rows, Hq, slot, mq};
            q_maps->next ^= 1;
        }
    }
    AttnParams p;
    memset(&p, 0, sizeof(p));
    p.qtile_seq = qtile_seq; p.qtile_row0 = qtile_row0; p.qtile_n = qtile_n; p.seq_nvis = seq_nvis;
    p.out = (__nv_bfloat16*)out; p.tap = tap;
    p.Hq = Hq; p.Hkv = Hkv; p.layer = layer;
    p.scale_log2e = 1.4426950408889634f / sqrtf((float)dh);
    p.status = status;
    p.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTile >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
    // split the keys across the CTAs of a cluster while (tile, head) pairs alone would leave SMs idle
    const int max_kt = (max_vis + kTile - 1) / kTile;
    p.pack = pack;
    p.slot = slot;
    p.slot_shift = pack == 1 ? 7 : (pack == 2 ? 6 : 5);
    p.tiles_per_kv = (group + pack - 1) / pack;
    const int grid_y = Hkv * p.tiles_per_kv;
    static bool attr_done[64] = {};     // the attribute is per device
    // Two tiles per CTA when that takes fewer rounds over the SMs: a CTA with two tiles takes 1.05-1.4 times a CTA with one, so
    // halving the rounds pays and the same number of rounds does not (pairs are formed inside one sequence and KV head: with one
    // tile for each there are none).  Measured, single / two tiles, in us; rounds 2 and 1: 583 rows, 32 heads 33 / 23.4; 128 keys
    // 700 rows, 28 query and 4 KV heads 14.8 / 10.0; 2048 keys, 640 rows, 40 heads 63 / 42.5.  3 and 2: 290 rows, 100 heads, 512
    // keys 32.5 / 28.2.  2 and 2: 34 rows, 160 heads, 512 keys 21.7 / 24.2; 290 rows, 80 heads, 2048 keys 65 / 75; 640 rows, 50
    // heads, 1024 keys 37.6 / 42.7.  With the same rounds it still wins where a CTA is mostly start and end, one key tile and
    // more than 64 rows in a tile (128 rows, 160 heads 14.3 / 13.2; 64 rows 12.7 / 13.1) or two and more than 96 (256 keys: 97
    // rows 17.5 / 17.1, 128 rows 17.8 / 17.0, 80 rows 16.6 / 16.9; at 512 keys 128 rows 23.8 / 24.2).
    static const int dual_on = getenv("WD_ATTN_DUAL") ? atoi(getenv("WD_ATTN_DUAL")) : 1;
    const int ctas_one = n_tiles * grid_y;
    const int ctas_two = Hkv * ((n_tiles * p.tiles_per_kv + (p.tiles_per_kv & 1 ? batch : 0)) / 2);   // (each sequence may end in half a pair)
    const int rounds_one = (ctas_one + sm_count - 1) / sm_count, rounds_two = (ctas_two + sm_count - 1) / sm_count;
    const int tile_rows = max_tile_rows > 0 ? max_tile_rows : kTile;
    const bool short_ctas = rounds_one > 1 && ((max_kt == 1 && tile_rows > 64) || (max_kt == 2 && tile_rows > 96));
    if (dual_on && seq_qt_off && (rounds_two < rounds_one || (rounds_two == rounds_one && short_ctas))) {
        static bool dual_done[64] = {};
        if (!dual_done[dev]) {
            WD_CUDA_TRY(cudaFuncSetAttribute(attention_tc_dual_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDualSmem));
            dual_done[dev] = true;
        }
        p.seq_qt_off = seq_qt_off;
        if (smem_used) *smem_used = kDualSmem;
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3((unsigned)((max_seq_tiles * p.tiles_per_kv + 1) / 2), (unsigned)Hkv, (unsigned)batch);
        lc.blockDim = dim3(kDThreads);
        lc.dynamicSmemBytes = kDualSmem;
        lc.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        lc.attrs = attr;
        lc.numAttrs = wd_pdl_enabled ? 1 : 0;
        ++wd_launch_counter;
        WD_CUDA_TRY(cudaLaunchKernelEx(&lc, attention_tc_dual_kernel, mq, *map_k, *map_vt, p));
        return WD_OK;
    }
    int want = sm_count / (n_tiles * grid_y);
    if (want < 1) want = 1;
    if (want > kMaxCluster) want = kMaxCluster;
    if (want > max_kt) want = max_kt;
    p.tiles_per_split = (max_kt + want - 1) / want;
    p.max_parts = (max_kt + p.tiles_per_split - 1) / p.tiles_per_split;
    static const int single_on = getenv("WD_ATTN_SINGLE") ? atoi(getenv("WD_ATTN_SINGLE")) : 1;
    const bool single = single_on && p.tiles_per_split == 1;
    const size_t smem_of[2] = {(1 + 2 * kStages) * (size_t)kOperand + (kBars + 1) * 8 + 16 + 2 * kTile * 4 + 1024,
                               (1 + 2) * (size_t)kOperand + (kBars + 1) * 8 + 16 + 2 * kTile * 4 + 1024};
    const size_t smem = smem_of[single ? 1 : 0];
    if (smem_used) *smem_used = smem;
    if (!attr_done[dev]) {
        WD_CUDA_TRY(cudaFuncSetAttribute(attention_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of[0]));
        WD_CUDA_TRY(cudaFuncSetAttribute(attention_tc_single_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of[1]));
        // the whole SM's shared memory although the kernel takes less than half: the output projection's CTAs are
        // to be resident beside it, and an SM keeps its carve-out while blocks are resident
        if (!(getenv("WD_NO_CARVEOUT") && atoi(getenv("WD_NO_CARVEOUT"))))
            WD_CUDA_TRY(cudaFuncSetAttribute(attention_tc_single_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                             cudaSharedmemCarveoutMaxShared));
        attr_done[dev] = true;
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(n_tiles, grid_y, p.max_parts);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    cudaLaunchAttribute attr[2];
    int n_attr = 0;
    if (p.max_parts > 1) {
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = 1;
        attr[n_attr].val.clusterDim.y = 1;
        attr[n_attr].val.clusterDim.z = (unsigned)p.max_parts;
        ++n_attr;
    }
    if (wd_pdl_enabled) {
        attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
        ++n_attr;
    }
    lc.attrs = attr;
    lc.numAttrs = n_attr;
    ++wd_launch_counter;
    if (single) WD_CUDA_TRY(cudaLaunchKernelEx(&lc, attention_tc_single_kernel, mq, *map_k, *map_vt, p));
    else WD_CUDA_TRY(cudaLaunchKernelEx(&lc, attention_tc_kernel, mq, *map_k, *map_vt, p));
    return WD_OK;
}
