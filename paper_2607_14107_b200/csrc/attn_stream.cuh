// Bidirectional attention rows with drift (Eq. 3, Eq. 4) as a STREAM over the key tiles: one CTA per
// (128 query rows, head) walks all keys twice, with the tensor core, the loads and the sixteen statistics warps
// overlapped through rings of operand tiles and two score accumulators in tensor memory.  bf16, head_dim 128,
// any number of keys.  For a single key tile, and in forwards over up to 512 keys for steps with many rows (block entries,
// batches), where the kernel of attn_tc.cuh -- one tile per CTA, key ranges combined across a cluster -- spends its time in
// start-up and exchange; beyond that the one-pass kernel of attn_flash.cuh takes over.
//
//   pass 1   S_t = Q K_t^T for every key tile t (tcgen05.mma into accumulator t & 1); the statistics warps read
//            each S_t from tensor memory (lane = row, four threads per row) and keep a running maximum and sum:
//            the row's log-sum-exp
//   pass 2   S_t again (K comes back through the ring, from L2); p = 2^(t - lse), normalised BEFORE it is rounded
//            to bf16 (the rounding point of a plain implementation), the drift sum A = sum p (s - s_old) against the
//            stored row, the new stored row s, and P into tensor memory as the A operand of O += P V_t (V as an
//            MN-major operand, accumulated in tensor memory over the tiles); S_{t+1} is computed while the
//            warps work on S_t
//   rows     the stored rows move as tensor boxes (or 512-byte bulk copies per row) between global memory and two staging
//            tiles in shared memory: the statistics warps never wait on global memory.  Q and P are tensor-memory operands
//            to make room for the second staging tile
//   end      O from tensor memory to the output rows, KL = A - (lse - lse_old)
//
// Computing S twice costs tensor time (which this kernel has to spare) and saves the rescaling of a running
// output, the second rounding point it brings, and any exchange between CTAs.  Stored rows are scaled scores plus
// one log-sum-exp per row, as in attn_tc.cuh.  Every mbarrier wait is bounded.
#pragma once
#include "attn_tc.cuh"

namespace ps {
namespace ast {

using namespace atc;

constexpr int THREADS = 576;              // warp 0: TMA, warp 1: MMA + tensor memory, warps 2..17: statistics / epilogue
constexpr int NS = 2;                     // slots of the operand ring (K and V tiles in the order the tensor core uses them)
constexpr uint32_t XPITCH = 512 + 16;     // bytes per row of the stored-row staging tile (the pad spreads the rows over the banks)
constexpr uint32_t XQ_BYTES = 17 * 1024;  // a lane quarter's share of a staging tile: 32 rows of XPITCH bytes, or four swizzled [32 rows][32 keys] boxes
constexpr uint32_t XBOX_BYTES = 32 * 128;
constexpr uint32_t X_BYTES = 4 * XQ_BYTES;
static_assert(32 * XPITCH <= XQ_BYTES && 4 * XBOX_BYTES <= XQ_BYTES, "staging tile");
constexpr uint32_t TILE_BYTES = 2 * BOX_BYTES;       // [128][128] bf16 as two [128][64] boxes
// Tensor memory: S0, S1, O (128 fp32 columns each), P and Q (two bf16 per column).  Both A operands live there, which
// leaves shared memory for two staging tiles.
constexpr uint32_t TMEM_COLS = 512, COL_O = 2 * KEYS, COL_P = COL_O + DH, COL_Q = COL_P + KEYS / 2;
static_assert(COL_Q + DH / 2 <= TMEM_COLS, "tensor memory");

__host__ __device__ constexpr size_t smem_bytes() { return (size_t)NS * TILE_BYTES + 2 * X_BYTES + 1024; }     // ring, X0, X1

// A from tensor memory (lane = row, K-major, two bf16 per column), B from shared memory
__device__ __forceinline__ void umma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
        ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// 16 columns of this thread's lane, complete on return (the whole warp calls)
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void bar_sync_stat() { asm volatile("bar.sync 1, 512;" ::: "memory"); }
// one row segment global -> shared (bytes counted on the mbarrier) and shared -> global (bulk group); 16-byte aligned
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}

// [32 rows][32 keys] boxes of the stored rows (128-byte swizzle in shared memory)
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int x, int y, int z) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"(map), "r"(src), "r"(x), "r"(y), "r"(z) : "memory");
}

// "Tile j of a quarter is written": one barrier per staging tile, so each serves every second key tile.  With one barrier
// for both, a warp that is a tile ahead (the old rows of tile j + 1 were requested before tile j was worked on) would arrive
// in place of a slower one, and tile j would be stored without the slower warp's columns.
__host__ __device__ constexpr int written_bar(int j) { return j & 1; }
__host__ __device__ constexpr uint32_t written_parity(int j) { return (j >> 1) & 1; }

struct Args {
    AttnArgs a;
    int maps;               // bit 0: map_p describes a.pprev, bit 1: map_r describes a.aprev (else null rows or unaligned: plain path)
    int rows_per_seq;       // forward rows per sequence (stand-alone: n_rows)
    int tiles_per_seq;      // 128-row tiles per sequence
    int* status;            // set to 1 when a bounded wait gave up (null: nowhere to report)
};

__global__ void __launch_bounds__(THREADS, 1)
attention_stream_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                        const __grid_constant__ CUtensorMap map_p, const __grid_constant__ CUtensorMap map_r, Args g) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bars[4 + 2 * NS + 4 + 8 + 8];
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_sh;
    __shared__ float* prev_sh[ROWS];
    __shared__ float* lsep_sh[ROWS];
    __shared__ int valid_sh[ROWS];
    __shared__ int box_row_sh[4], box_map_sh[4];   // lane quarters whose 32 stored rows are consecutive: first row, which map (-1: not so)
    __shared__ float2 part_ml[4][ROWS];            // (maximum, sum) of each column quarter
    __shared__ float part_A[3][ROWS];              // drift sums of the upper three column quarters

    const AttnArgs& a = g.a;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int seq = blockIdx.x / g.tiles_per_seq, tile = blockIdx.x - seq * g.tiles_per_seq;
    const int h = blockIdx.y;
    const int g_kv = (h * a.n_kv) / a.n_heads;
    const int dq = a.n_heads * DH;
    const int row0 = seq * g.rows_per_seq + tile * ROWS;
    const int n_in_tile = min(ROWS, g.rows_per_seq - tile * ROWS);
    const int kv_seq = a.rows ? seq : 0;
    const int n = (a.N + KEYS - 1) / KEYS;                 // key tiles

    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t smem_base = smem_u32(smem);
    auto ring_s = [&](int s) { return smem_base + (uint32_t)s * TILE_BYTES; };
    const uint32_t bar_q = smem_u32(&bars[0]), bar_o = smem_u32(&bars[1]), bar_pfull = smem_u32(&bars[2]), bar_pfree = smem_u32(&bars[3]);
    auto bar_full = [&](int s) { return smem_u32(&bars[4 + s]); };
    auto bar_free = [&](int s) { return smem_u32(&bars[4 + NS + s]); };
    auto bar_sfull = [&](int s) { return smem_u32(&bars[4 + 2 * NS + s]); };
    auto bar_sfree = [&](int s) { return smem_u32(&bars[6 + 2 * NS + s]); };
    // staging tiles, per lane quarter (32 rows, the four warps that share them): "X_b may be worked on", "the warps are done with it"
    auto bar_x = [&](int b, int q) { return smem_u32(&bars[8 + 2 * NS + 4 * b + q]); };
    auto bar_w = [&](int j, int q) { return smem_u32(&bars[16 + 2 * NS + 4 * written_bar(j) + q]); };
    auto x_s = [&](int b) { return smem_base + (uint32_t)NS * TILE_BYTES + (uint32_t)b * X_BYTES; };

    if (threadIdx.x == 0) {
        mbar_init(bar_q, 16); mbar_init(bar_o, 1); mbar_init(bar_pfull, 16); mbar_init(bar_pfree, 1);
        for (int s = 0; s < NS; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_free(s), 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(bar_sfull(s), 1); mbar_init(bar_sfree(s), 16); }
        for (int q = 0; q < 4; ++q) { mbar_init(bar_x(0, q), 32); mbar_init(bar_x(1, q), 32); mbar_init(bar_w(0, q), 4); mbar_init(bar_w(1, q), 4); }
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_sh), TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();
    const uint32_t tmem_base = tmem_base_sh;
    volatile int* abort_flag = &abort_sh;
    // Operand units, in the order the tensor core consumes them (3 n in all, unit u in ring slot u % NS):
    //   K_0 .. K_{n-1}                          pass 1
    //   K_0, (K_1, V_0), (K_2, V_1), ..., V_{n-1}   pass 2: S of tile j + 1 is issued before P V of tile j
    // Score unit t (t < n: pass 1, else pass 2, tile t mod n) uses accumulator t & 1.  The k-th use of a ring slot or
    // accumulator completes phase k & 1 of its barriers.
    auto unit_tile = [&](int u, bool& is_v) {
        is_v = false;
        if (u < n) return u;
        if (u == n) return 0;
        const int w = u - n - 1;
        if (w == 2 * (n - 1)) { is_v = true; return n - 1; }
        if (w & 1) { is_v = true; return (w - 1) >> 1; }
        return (w >> 1) + 1;
    };

    if (warp == 0) {
        if (elect_one()) {
            auto clean = [&](int kt) {          // tile last written by an earlier forward: loadable before the dependency wait
                const int lo = kt * KEYS, hi = lo + KEYS;
                return hi <= a.dirty_lo || lo >= a.dirty_hi;
            };
            auto load = [&](int u) {
                bool is_v;
                const int kt = unit_tile(u, is_v), sl = u % NS;
                mbar_expect_tx(bar_full(sl), TILE_BYTES);
                for (int kb = 0; kb < 2; ++kb)
                    tma_load_3d(ring_s(sl) + kb * BOX_BYTES, is_v ? &map_v : &map_k, bar_full(sl), g_kv * DH + kb * 64, kt * KEYS, kv_seq);
            };
            int u = 0;
            bool ok = true;
            // the first ring slots need no wait; tiles that no kernel of this step writes are requested right away
            for (; u < min(NS, 3 * n); ++u) {
                bool is_v;
                if (!clean(unit_tile(u, is_v))) break;
                load(u);
            }
            pdl_wait();      // the K / V rows written this step come from the projection that ran just before
            trace_stamp(7);
            for (; u < 3 * n && ok; ++u) {
                if (u >= NS) ok = mbar_wait(bar_free(u % NS), (uint32_t)(u / NS - 1) & 1u, abort_flag);
                if (ok) load(u);
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc_s = instr_desc_bf16(ROWS, KEYS);
            const uint32_t idesc_o = instr_desc_bf16(ROWS, DH) | (1u << 16);       // B (= V) is MN-major
            bool ok = mbar_wait(bar_q, 0, abort_flag);          // q is in tensor memory
            int u = 0;                   // operand units consumed so far
            auto take = [&]() {          // next unit of the ring: its slot, once the tile has landed
                const int sl = u % NS;
                ok = ok && mbar_wait(bar_full(sl), (uint32_t)(u / NS) & 1u, abort_flag);
                ++u;
                return sl;
            };
            auto mma_s = [&](int t) {
                const int sl = take(), b = t & 1;
                if (t >= 2) ok = ok && mbar_wait(bar_sfree(b), (uint32_t)((t >> 1) - 1) & 1u, abort_flag);
                if (!ok) return;
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < DH / UMMA_K; ++k) {
                    const uint64_t db = smem_desc_sw128(ring_s(sl) + (k >> 2) * BOX_BYTES) + (uint64_t)((k & 3) * 2);
                    umma_bf16_ta(tmem_base + (uint32_t)(b * KEYS), tmem_base + COL_Q + (uint32_t)(k * (UMMA_K / 2)), db, idesc_s, k > 0 ? 1u : 0u);
                }
                umma_commit(bar_free(sl));
                umma_commit(bar_sfull(b));
            };
            for (int t = 0; t < n && ok; ++t) mma_s(t);
            if (ok) mma_s(n);
            for (int j = 0; j < n && ok; ++j) {
                if (j + 1 < n) mma_s(n + j + 1);
                const int sl = take();
                ok = ok && mbar_wait(bar_pfull, (uint32_t)j & 1u, abort_flag);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < KEYS / UMMA_K; ++k) {
                    // B = V_j: 16 keys = two 8-row groups further down
                    const uint64_t db = smem_desc_mn_sw128(ring_s(sl) + (uint32_t)k * 2048u, BOX_BYTES);
                    umma_bf16_ta(tmem_base + COL_O, tmem_base + COL_P + (uint32_t)(k * (UMMA_K / 2)), db, idesc_o, (j > 0 || k > 0) ? 1u : 0u);
                }
                umma_commit(bar_free(sl));
                umma_commit(bar_pfree);
            }
            umma_commit(bar_o);          // (also on failure: the statistics warps then see the abort flag)
        }
    } else {
        // ---- statistics / epilogue warps: TMEM lane = row; the four warps of a lane quarter split the columns ----
        const int ew = warp - 2;
        const int quarter = warp & 3;             // tensor-memory lanes 32 * quarter .. + 31
        const int cq = ew >> 2;                   // columns 32 * cq .. + 31 of every tile
        const int row = quarter * 32 + lane;
        const uint32_t taddr0 = tmem_base + ((uint32_t)(quarter * 32) << 16);
        pdl_wait();            // the row table, q and the stored rows all come from earlier kernels of the stream
        if (cq == 0) {
            float* prev = nullptr; float* lsep = nullptr;
            int valid = 0, stored = -1, arr = -1;              // index of the stored row, 0: pprev, 1: aprev
            if (row < n_in_tile) {
                const int r = row0 + row;
                if (a.rows) {
                    const int4 rw = __ldg(reinterpret_cast<const int4*>(a.rows) + r);      // {seq, pos, widx, aidx}
                    if (rw.y >= 0) {
                        valid = 1;
                        if (a.cluster_K > 0 ? (row_is_proxy(rw.z) && a.pprev != nullptr) : (rw.z >= 0 && a.pprev != nullptr)) {
                            // recorded drift rows: the window rows, or (centroid proxies) the clusters' proxy rows
                            const size_t i = a.cluster_K > 0 ? ((size_t)rw.x * a.cluster_K + row_cluster(rw.z)) * a.n_heads + h
                                                             : ((size_t)rw.x * a.W_max + rw.z) * a.n_heads + h;
                            prev = a.pprev + i * a.N; lsep = a.pprev_lse + i; stored = (int)(i / a.n_heads); arr = 0;
                        } else if (rw.w >= 0 && a.aprev) {
                            const size_t i = ((size_t)rw.x * a.B + rw.w) * a.n_heads + h;
                            prev = a.aprev + i * a.N; lsep = a.aprev_lse + i; stored = (int)(i / a.n_heads); arr = 1;
                        }
                    }
                } else {
                    valid = 1;
                    if (a.pprev) { const size_t i = (size_t)r * a.n_heads + h; prev = a.pprev + i * a.N; lsep = a.pprev_lse + i; stored = r; arr = 0; }
                }
            }
            prev_sh[row] = prev; lsep_sh[row] = lsep; valid_sh[row] = valid;
            // (rows behind the last one of a stand-alone call lie outside its map: loads fill, stores leave them out)
            const int s0 = __shfl_sync(0xffffffffu, stored, 0), arr0 = __shfl_sync(0xffffffffu, arr, 0);
            const bool run = __all_sync(0xffffffffu, (stored == s0 + lane && arr == arr0) || (!a.rows && s0 >= 0 && s0 + lane >= a.n_rows)) != 0;
            if (lane == 0) { box_row_sh[quarter] = s0; box_map_sh[quarter] = (run && s0 >= 0 && ((g.maps >> arr0) & 1)) ? arr0 : -1; }
        }
        {
            // this thread's 32 channels of its row of q, straight into tensor memory
            uint32_t qw[16];
            if (row < n_in_tile) {
                const uint4* src = reinterpret_cast<const uint4*>((const __nv_bfloat16*)a.q + (size_t)(row0 + row) * dq + h * DH + cq * 32);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 v = __ldcg(src + i);
                    qw[4 * i] = v.x; qw[4 * i + 1] = v.y; qw[4 * i + 2] = v.z; qw[4 * i + 3] = v.w;
                }
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) qw[i] = 0u;
            }
            __syncwarp();
            tmem_st16(taddr0 + COL_Q + (uint32_t)(cq * 16), qw);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_q);
        }
        bar_sync_stat();
        float* const prev = prev_sh[row];
        const bool valid = valid_sh[row] != 0;
        // tensor-memory loads are warp-wide (.sync.aligned): whether a warp reads at all is decided per warp
        const bool warp_valid = __any_sync(0xffffffffu, valid) != 0;
        const bool use_old = prev != nullptr && a.record_kl != 0;
        const bool vec = (a.N & 3) == 0 && (((uintptr_t)a.pprev | (uintptr_t)a.aprev) & 15) == 0;
        // stored rows are handled a warp at a time: nothing of it runs in a warp none of whose rows is recorded
        const bool warp_prev = __any_sync(0xffffffffu, prev != nullptr) != 0;
        float lse_old = 0.f;
        if (cq == 0 && lsep_sh[row] && a.record_kl) lse_old = __ldcg(lsep_sh[row]);
        const float scale2 = a.scale * LOG2E_F;
        bool ok = true;

        // Stored rows travel through two staging tiles X_0 / X_1 in shared memory, a lane quarter (32 rows, four warps) at a
        // time: the statistics warps never touch global memory, and DRAM sees whole row segments.  A quarter whose 32 stored
        // rows are consecutive moves them as swizzled [32 rows][32 keys] tensor boxes (four copies per tile), any other as
        // one 512-byte bulk copy per row, issued by the row's first thread.  "X_b may be worked on for tile j" is phase
        // j / 2 of bar_x(b, quarter): the quarter's 32 first threads arrive on it once the store of tile j - 2 has read X_b,
        // together with the bytes of the old rows of tile j when there are any: tile j + 1 is on its way while tile j is
        // worked on.  2048 rows x 2048 keys x 32 heads, rows read and written: one staging tile and row copies 434 us, two
        // 381, boxes 293, now 281 (without any stored rows: 157); 256 x 2048: 102 / 94 / 74.  Rows that no bulk copy takes
        // (length or base no multiple of 16 bytes) go through the same tiles, a warp at a time (patch_load below).
        const bool use_x = vec && warp_prev;                     // (the same in the four warps of a quarter, like everything here)
        const bool patch = !vec && warp_prev;
        const bool boxes = use_x && box_map_sh[quarter] >= 0;
        const CUtensorMap* const map_x = box_map_sh[quarter] == 1 ? &map_r : &map_p;
        auto x_quarter = [&](int b) { return x_s(b) + (uint32_t)quarter * XQ_BYTES; };
        auto x_ready = [&](int j) {         // first threads: X may take tile j; request the old rows if there are any
            const int b = j & 1, keys = min(KEYS, a.N - j * KEYS);
            if (boxes) {
                if (lane == 0 && a.record_kl) {
                    const int nb = (keys + 31) >> 5;
                    mbar_expect_tx(bar_x(b, quarter), (uint32_t)nb * XBOX_BYTES);
                    for (int c = 0; c < nb; ++c)
                        tma_load_3d(x_quarter(b) + (uint32_t)c * XBOX_BYTES, map_x, bar_x(b, quarter), j * KEYS + 32 * c, h, box_row_sh[quarter]);
                } else {
                    mbar_arrive(bar_x(b, quarter));
                }
            } else if (use_old) {
                mbar_expect_tx(bar_x(b, quarter), (uint32_t)keys * 4u);
                bulk_load(x_quarter(b) + (uint32_t)lane * XPITCH, prev + j * KEYS, (uint32_t)keys * 4u, bar_x(b, quarter));
            } else {
                mbar_arrive(bar_x(b, quarter));
            }
        };
        if (use_x && cq == 0) { x_ready(0); if (n > 1) x_ready(1); }
        // Each warp keeps its own [32 rows][32 keys] patch of the staging tiles, filled two tiles ahead by four-byte asynchronous
        // copies and written back a row of the warp's 32 keys at a time: whole sectors, no waiting for other warps.  Every thread
        // reading and writing its own row touched 32 lines per instruction (403 keys, 200 rows x 32 heads: 137 us, now 35; 2047 keys,
        // 256 rows x 8 heads: 616, 114), and its 32 registers of old scores made the other forms spill.
        auto patch_s = [&](int j, int r) { return x_quarter(j & 1) + (uint32_t)r * XPITCH + (uint32_t)cq * 128u + (uint32_t)lane * 4u; };
        auto patch_load = [&](int j) {
            const int k = j * KEYS + cq * 32 + lane;
            if (a.record_kl && k < a.N)
                for (int r = 0; r < 32; ++r) {
                    const float* src = prev_sh[quarter * 32 + r];
                    if (src) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(patch_s(j, r)), "l"(src + k) : "memory");
                }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        if (patch) { patch_load(0); if (n > 1) patch_load(1); }

        // ---- pass 1: running (maximum, sum) of this thread's columns (four independent chains each: two or four warps
        // per scheduler cannot hide one long dependent chain) ----
        float mx = -INFINITY, l = 0.f;
        for (int t = 0; t < n; ++t) {
            const int b = t & 1;
            ok = mbar_wait(bar_sfull(b), (uint32_t)(t >> 1) & 1u, abort_flag) && ok && !*abort_flag;
            ok = __all_sync(0xffffffffu, ok) != 0;
            if (!ok) break;
            tc_fence_after();
            const int kb = t * KEYS + cq * 32;
            if (warp_valid) {
                uint32_t r[2][16];
#pragma unroll
                for (int u = 0; u < 2; ++u) tmem_ld16_issue(taddr0 + (uint32_t)(b * KEYS + cq * 32 + 16 * u), r[u]);
                tmem_ld_wait();
                if (kb + 32 > a.N) {         // the tile's columns beyond the last key do not take part
#pragma unroll
                    for (int u = 0; u < 2; ++u)
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (kb + 16 * u + i >= a.N) r[u][i] = 0xff800000u;      // -inf
                }
                float tm4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int i = 0; i < 16; ++i) tm4[i & 3] = fmaxf(tm4[i & 3], __uint_as_float(r[u][i]));
                const float tm = fmaxf(fmaxf(tm4[0], tm4[1]), fmaxf(tm4[2], tm4[3])) * scale2;      // scale2 > 0: the maximum commutes with it
                const float nm = fmaxf(mx, tm);
                if (nm > -INFINITY) {
                    float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int u = 0; u < 2; ++u)
#pragma unroll
                        for (int i = 0; i < 16; ++i) s4[i & 3] += ex2(fmaf(__uint_as_float(r[u][i]), scale2, -nm));     // (2^-inf = 0)
                    l = l * ex2(mx - nm) + ((s4[0] + s4[1]) + (s4[2] + s4[3]));       // (mx = -inf: l is 0 and 2^(-inf) = 0)
                }
                mx = nm;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_sfree(b));
        }
        part_ml[cq][row] = make_float2(mx, l);
        bar_sync_stat();
        float lse2;
        {
            float M = -INFINITY;
#pragma unroll
            for (int c = 0; c < 4; ++c) M = fmaxf(M, part_ml[c][row].x);
            float L = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 ml = part_ml[c][row];
                if (ml.y > 0.f) L = fmaf(ml.y, ex2(ml.x - M), L);
            }
            lse2 = M + log2f(L);
        }
        float dlse = 0.f;
        if (cq == 0) {
            // the row's log-sum-exp is kept in natural-log units, like the stored rows
            float* lsep = lsep_sh[row];
            const float lse = lse2 * LN2_F;
            dlse = lse - lse_old;
            if (lsep && valid && ok) *lsep = lse;
        }

        // ---- pass 2: probabilities (normalised before they are rounded to bf16), P, then drift sum and the new stored row ----
        float A4[4] = {0.f, 0.f, 0.f, 0.f};
        const float neg_lse2 = -lse2;
        // this thread's 128 bytes of its row: sixteen-byte chunk c at x_seg + ((c ^ x_swz) << 4)
        const uint32_t x_seg = boxes ? (uint32_t)cq * XBOX_BYTES + (uint32_t)lane * 128u : (uint32_t)lane * XPITCH + (uint32_t)cq * 128u;
        const uint32_t x_swz = boxes ? (uint32_t)(lane & 7) : 0u;
        for (int j = 0; j < n && ok; ++j) {
            const int t = n + j, b = t & 1;
            const int kb = j * KEYS + cq * 32;
            const bool edge = kb + 32 > a.N;
            ok = mbar_wait(bar_sfull(b), (uint32_t)(t >> 1) & 1u, abort_flag) && ok && !*abort_flag;
            ok = __all_sync(0xffffffffu, ok) != 0;
            if (!ok) break;
            tc_fence_after();
            uint32_t pw[16];             // P of this thread's 32 columns, two bf16 per word
            uint32_t r[2][16];
            float pr[32];
            if (warp_valid) {
#pragma unroll
                for (int u = 0; u < 2; ++u) tmem_ld16_issue(taddr0 + (uint32_t)(b * KEYS + cq * 32 + 16 * u), r[u]);
                tmem_ld_wait();
                if (edge || !valid) {        // columns beyond the last key, rows that are not valid: probability zero
#pragma unroll
                    for (int u = 0; u < 2; ++u)
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (!valid || kb + 16 * u + i >= a.N) r[u][i] = 0xff800000u;      // -inf
                }
#pragma unroll
                for (int i = 0; i < 32; ++i) pr[i] = ex2(fmaf(__uint_as_float(r[i >> 4][i & 15]), scale2, neg_lse2));      // (masked entries are -inf: p = 0)
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    __nv_bfloat162 bb = __floats2bfloat162_rn(pr[2 * i], pr[2 * i + 1]);
                    pw[i] = *reinterpret_cast<uint32_t*>(&bb);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) pw[i] = 0u;
            }
            // the scores are in registers: the accumulator may take the tile after next
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_sfree(b));
            // P of the previous tile must have been consumed by its P V before the buffer is rewritten
            if (j > 0) {
                ok = mbar_wait(bar_pfree, (uint32_t)(j - 1) & 1u, abort_flag) && ok && !*abort_flag;
                ok = __all_sync(0xffffffffu, ok) != 0;
                if (!ok) break;
            }
            // P as the A operand of P V
            tc_fence_after();
            __syncwarp();
            tmem_st16(taddr0 + COL_P + (uint32_t)(cq * 16), pw);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_pfull);
            // ---- the tensor core has what it needs; now the stored row of this tile
            // old scores out of the staging tile, drift sum, new scores into their place
            auto new_rows = [&](uint32_t x) {
                if (!warp_valid) return;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    float o0, o1, o2, o3;
                    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(o0), "=f"(o1), "=f"(o2), "=f"(o3) : "r"(x + (((uint32_t)c ^ x_swz) << 4)) : "memory");
                    float sn[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i)       // (rounded products, never fused into the subtraction below: an unchanged row gives exactly zero)
                        sn[i] = __fmul_rn(__fmul_rn(__uint_as_float(r[c >> 2][4 * (c & 3) + i]), scale2), LN2_F);
                    if (use_old) {
                        const float od[4] = {o0, o1, o2, o3};
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (pr[4 * c + i] > 0.f) A4[i] = fmaf(pr[4 * c + i], sn[i] - od[i], A4[i]);      // (p = 0: also the masked entries)
                    }
                    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(x + (((uint32_t)c ^ x_swz) << 4)), "f"(sn[0]), "f"(sn[1]), "f"(sn[2]), "f"(sn[3]) : "memory");
                }
            };
            if (use_x) {
                const int xb = j & 1;
                if (cq == 0 && j > 0) {
                    // the bulk store of the previous tile has read its staging tile by now: the tile after this one may come
                    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                    __syncwarp();
                    if (j + 1 < n) x_ready(j + 1);
                }
                ok = mbar_wait(bar_x(xb, quarter), (uint32_t)(j >> 1) & 1u, abort_flag) && ok && !*abort_flag;
                ok = __all_sync(0xffffffffu, ok) != 0;
                if (!ok) break;
                new_rows(x_quarter(xb) + x_seg);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the bulk store reads what was just written
                // the quarter's rows are complete once its four warps have passed here (an mbarrier, not a named barrier:
                // its wait is bounded like every other)
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_w(j, quarter));
                if (cq == 0) {
                    ok = mbar_wait(bar_w(j, quarter), written_parity(j), abort_flag) && ok && !*abort_flag;
                    ok = __all_sync(0xffffffffu, ok) != 0;
                    if (!ok) break;
                    const int keys = min(KEYS, a.N - j * KEYS);
                    if (boxes) {
                        if (lane == 0) {
                            for (int c = 0; c < (keys + 31) >> 5; ++c)
                                tma_store_3d(map_x, x_quarter(xb) + (uint32_t)c * XBOX_BYTES, j * KEYS + 32 * c, h, box_row_sh[quarter]);
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        }
                    } else if (prev) {
                        bulk_store(prev + j * KEYS, x_quarter(xb) + (uint32_t)lane * XPITCH, (uint32_t)keys * 4u);
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
            } else if (patch) {
                if (j + 1 < n) asm volatile("cp.async.wait_group 1;" ::: "memory");
                else asm volatile("cp.async.wait_group 0;" ::: "memory");
                __syncwarp();                    // the patch has landed for every lane
                new_rows(x_quarter(j & 1) + x_seg);
                __syncwarp();                    // ... and holds the new rows: out, a row of the warp's keys at a time
                const int k = kb + lane;
                if (k < a.N)
                    for (int rr = 0; rr < 32; ++rr) {
                        float* dst = prev_sh[quarter * 32 + rr];
                        float v;
                        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(patch_s(j, rr)) : "memory");
                        if (dst) __stcg(dst + k, v);
                    }
                __syncwarp();
                if (j + 2 < n) patch_load(j + 2);
            }
        }
        if (use_x && cq == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");      // the last stores have left
        if (patch) asm volatile("cp.async.wait_all;" ::: "memory");         // (a wait that gave up left copies in flight)

        // ---- output rows and drift ----
        const float A = (A4[0] + A4[1]) + (A4[2] + A4[3]);
        if (cq > 0) part_A[cq - 1][row] = A;
        ok = mbar_wait(bar_o, 0, abort_flag) && ok && !*abort_flag;
        ok = __all_sync(0xffffffffu, ok) != 0;
        tc_fence_after();
        bar_sync_stat();
        if (ok && warp_valid) {
            uint32_t r[2][16];
#pragma unroll
            for (int u = 0; u < 2; ++u) tmem_ld16_issue(taddr0 + COL_O + (uint32_t)(cq * 32 + 16 * u), r[u]);
            tmem_ld_wait();
            if (valid && a.out) {
                __nv_bfloat16* dst = (__nv_bfloat16*)a.out + (size_t)(row0 + row) * dq + h * DH + cq * 32;
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t w[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            __nv_bfloat162 bb = __floats2bfloat162_rn(__uint_as_float(r[u][8 * c + 2 * i]), __uint_as_float(r[u][8 * c + 2 * i + 1]));
                            w[i] = *reinterpret_cast<uint32_t*>(&bb);
                        }
                        *reinterpret_cast<uint4*>(dst + 16 * u + 8 * c) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
            }
        }
        if (ok && cq == 0 && valid && a.kl)
            a.kl[(size_t)(row0 + row) * a.n_heads + h] =
                (lsep_sh[row] && a.record_kl) ? ((A + part_A[0][row]) + (part_A[1][row] + part_A[2][row])) - dlse : 0.f;
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, TMEM_COLS);
    trace_stamp(312, 64);
    if (threadIdx.x == 0 && abort_sh && g.status) atomicExch(g.status, 1);
}

}  // namespace ast
}  // namespace ps
