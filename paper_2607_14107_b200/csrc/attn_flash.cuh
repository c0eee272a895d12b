// Bidirectional attention rows with drift (Eq. 3, Eq. 4) in ONE pass over the key tiles, two streams of (128 rows x key tiles)
// per CTA: while the warps of one stream work on its scores, the tensor core computes the other's.  bf16, head_dim 128, any
// number of keys, rows and heads per K/V head.
//
//   rows     the query rows of all heads that share a K/V head form one list (head-major: virtual row = head in the group *
//            rows + row), cut into tiles of 128, so grouped heads fill the tiles even when a step has few rows
//   streams  ROW SPLIT: two row tiles, every key tile serves both.  KEY SPLIT (fewer row tiles than would fill the GPU): one
//            row tile, the streams take the even and the odd key tiles, and their partial rows are put together at the end
//   scores   S = Q K^T into the stream's accumulator in tensor memory; four warps, one thread per row, read the row's 128
//            scores, keep a running maximum m and sum, and write p = 2^(s - m), rounded to bf16, over the scores, where it is the A
//            operand of O += P V.  Output rows are divided by the sum at the end.  m follows the true maximum only when that has
//            grown by more than 2^8 (the row's O, sum and drift sum are then rescaled): the scale of p does not matter to its
//            rounding, and after the first tile it hardly ever moves.  In forwards m is a whole number (AttnArgs::p_pow2): the rounding of
//            p is then that of e^score on its own, whatever the order of the tiles, and the oracle's
//   drift    A = sum p (s - s_old) is accumulated and rescaled like the sum; KL = A / sum - (lse - lse_old), exactly zero for an
//            unchanged row (s - s_old and lse - lse_old are: same bits in, same bits out)
//   stored   the stored rows (scaled scores plus one log-sum-exp, as in attn_tc.cuh) pass through two staging patches of [32
//            rows][64 keys] per warp, the next one loaded while one is worked on and stored from where it was replaced: as swizzled
//            tensor boxes where the warp's 32 stored rows are consecutive, else in coalesced pieces.  Rows that are never
//            recorded (most of a block entry's) are the work of other CTAs of the same launch (FlashPart)
//
// Without stored rows a tile costs a stream ~2200 cycles of softmax and ~1600 of waiting for its two products (512 tensor cycles each
// and the hand-over); the streams hide one another's waits, and packed arithmetic (two fp32 per instruction) keeps issue
// slots free.  us, against two passes with normalised probabilities on one row tile (attn_stream.cuh), 32 heads: 2048 x 2048
// 161 -> 82 (839 TFLOP/s), 900 x 1024 47 -> 25, 512 x 512 17.0 -> 11.5.  With stored rows HBM and the chain of a patch (wait, old scores
// out of shared memory, new ones in, store) share the time: 2048 x 2048 284 -> 230 (4.7 TB/s), 192 x 2048 69 -> 53, 512 x 512 27.6 ->
// 21.7; rows of no whole 16 bytes, 1000 x 1501, 192 -> 165.  Measured and dropped: sixteen softmax warps with two threads per row
// (302 us: a third of the registers, so spills), three 32-key patches per warp (237), the tile's 128 columns unrolled (246: the
// loop no longer fits the instruction cache; without stored rows the unrolled form is the faster one, 82 / 91).
//
// The method is published: a running maximum and sum in one pass (Milakov and Gimelshein, 2018) over key tiles (FlashAttention: Dao
// et al., 2022), two row tiles whose softmax and products alternate (FlashAttention-3: Shah et al., 2024), a reference that moves only
// when the maximum has outgrown it (FlashAttention-4: Dao et al., 2025).  Drift, stored rows, the key split and the code are this library's.
//
// Every mbarrier wait is bounded.
#pragma once
#include <type_traits>

#include "attn_stream.cuh"

namespace ps {
namespace afl {

using namespace ast;

constexpr int FL_THREADS = 320;           // warp 0: TMA, warp 1: MMA + tensor memory, warps 2..9: four per stream
constexpr int FL_MAX_SLOTS = 6;
constexpr int FL_PLAIN_SLOTS = 4;         // K / V ring of the form without stored rows
constexpr int FL_REC_SLOTS = 2;           // ... and of a CTA with recorded rows; one without uses the patches' room for four more
constexpr uint32_t PBOX_BYTES = 32 * 128, PATCH_BYTES = 2 * PBOX_BYTES;      // a box is [32 rows][32 keys] fp32
static_assert(8 * 2 * PATCH_BYTES == (FL_MAX_SLOTS - FL_REC_SLOTS) * TILE_BYTES, "the patches take the room of four slots");
constexpr float FL_SLACK = 8.f;           // log2 of how far the running maximum may lag behind
__host__ __device__ constexpr size_t flash_smem_bytes(bool rec) { return (size_t)(rec ? 1 + FL_MAX_SLOTS : 2 + FL_PLAIN_SLOTS) * TILE_BYTES + 1024; }

__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t* r) {
    tmem_ld16_issue(taddr, r);
    tmem_ld16_issue(taddr + 16, r + 16);
}
__device__ __forceinline__ void tmem_st16_issue(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
// two fp32 values per instruction (rounded as the single operations are)
__device__ __forceinline__ uint64_t f2_pack(float x, float y) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y)); return r; }
__device__ __forceinline__ uint64_t f2_pack(uint32_t x, uint32_t y) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(x), "r"(y)); return r; }
__device__ __forceinline__ void f2_unpack(uint64_t v, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) { uint64_t r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) { uint64_t r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) { uint64_t r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ float f2_sum(uint64_t v) { float x, y; f2_unpack(v, x, y); return x + y; }
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void bar_sync_streams() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// A part of the forward's rows, the same of every sequence: `rows` of them, row r of the part being forward row r of the sequence,
// or r + skip from `skip_at` on
struct FlashPart {
    int rows, skip_at, skip;
    int vrows;              // virtual rows per sequence and K/V head: rows x heads per K/V head
    int key_split;          // the streams split the keys of one row tile instead of taking a row tile each
    int tiles;              // CTAs per sequence and K/V head
};
struct FlashArgs {
    AttnArgs a;
    int maps;               // bit 0: map_p describes a.pprev, bit 1: map_r describes a.aprev
    int stride;             // forward rows per sequence
    int rec_ctas;           // the first rec_ctas of a grid row work on part 0, which may have recorded rows and is split by keys; the
                            // others on part 1, which has none
    FlashPart part[2];
    int* status;            // set to 1 when a bounded wait gave up (null: nowhere to report)
};

template <bool REC>
__global__ void __launch_bounds__(FL_THREADS, 1)
attention_flash_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                       const __grid_constant__ CUtensorMap map_p, const __grid_constant__ CUtensorMap map_r, const __grid_constant__ FlashArgs f) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bars[1 + 2 * FL_MAX_SLOTS + 6 + 16];
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_sh;

    const AttnArgs& a = f.a;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool rec_cta = REC && (int)blockIdx.x < f.rec_ctas;
    const FlashPart& part = f.part[rec_cta ? 0 : 1];
    const int bx = (int)blockIdx.x - (rec_cta ? 0 : f.rec_ctas);
    const int seq = bx / part.tiles, tile = bx - seq * part.tiles;
    const int g_kv = blockIdx.y, hpg = a.n_heads / a.n_kv;
    const int dq = a.n_heads * DH;
    const int kv_seq = a.rows ? seq : 0;
    const int n = (a.N + KEYS - 1) / KEYS;               // key tiles
    const bool ksplit = part.key_split != 0;
    const int vr0 = tile * (ksplit ? ROWS : 2 * ROWS);   // first virtual row of the CTA
    const int cnt0 = ksplit ? (n + 1) >> 1 : n;          // key tiles of stream 0 ...
    const int cnt1 = ksplit ? n >> 1 : (vr0 + ROWS < part.vrows ? n : 0);       // ... and of stream 1

    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t smem_base = smem_u32(smem);
    auto q_s = [&](int g) { return smem_base + (uint32_t)g * TILE_BYTES; };
    const int q_tiles = rec_cta ? 1 : 2;                 // (a CTA with recorded rows: the second one's room belongs to the patches)
    auto ring_s = [&](int s) { return smem_base + (uint32_t)(q_tiles + s) * TILE_BYTES; };
    const uint32_t bar0 = smem_u32(&bars[0]);
    const uint32_t bar_q = bar0;
    auto bar_full = [&](int s) { return bar0 + 8u * (uint32_t)(1 + s); };
    auto bar_free = [&](int s) { return bar0 + 8u * (uint32_t)(1 + FL_MAX_SLOTS + s); };
    auto bar_s = [&](int g) { return bar0 + 8u * (uint32_t)(1 + 2 * FL_MAX_SLOTS + g); };          // scores of the stream's next tile are in its accumulator
    auto bar_p = [&](int g) { return bar0 + 8u * (uint32_t)(3 + 2 * FL_MAX_SLOTS + g); };          // ... and replaced by its probabilities
    auto bar_o = [&](int g) { return bar0 + 8u * (uint32_t)(5 + 2 * FL_MAX_SLOTS + g); };          // the stream's last P V has completed
    auto bar_x = [&](int w, int b) { return bar0 + 8u * (uint32_t)(7 + 2 * FL_MAX_SLOTS + 2 * w + b); };

    if (threadIdx.x == 0) {
        mbar_init(bar_q, 8);
        for (int s = 0; s < FL_MAX_SLOTS; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_free(s), 1); }
        for (int g = 0; g < 2; ++g) { mbar_init(bar_s(g), 1); mbar_init(bar_p(g), 4); mbar_init(bar_o(g), 1); }
        for (int w = 0; w < 8; ++w) for (int b = 0; b < 2; ++b) mbar_init(bar_x(w, b), 1);
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_sh), 512);       // S / P of stream 0 and 1, O of stream 0 and 1: 128 columns each
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();
    const uint32_t tmem_base = tmem_base_sh;
    volatile int* abort_flag = &abort_sh;
    const int slots = rec_cta ? FL_REC_SLOTS : (REC ? FL_MAX_SLOTS - 1 : FL_PLAIN_SLOTS);

    // Operand tiles in the order the tensor core takes them: row split K_0, V_0, K_1, V_1, ...; key split K_0, K_1, V_0, K_2, V_1,
    // K_3, ..., V_{n-2}, V_{n-1}.
    if (warp == 0) {
        if (elect_one()) {
            auto unit_tile = [&](int u, bool& is_v) {
                if (!ksplit || n == 1) { is_v = (u & 1) != 0; return u >> 1; }
                if (u < 2) { is_v = false; return u; }
                const int w = u - 2;
                if (w < 2 * (n - 2)) { is_v = (w & 1) == 0; return is_v ? w >> 1 : (w >> 1) + 2; }
                is_v = true;
                return n - 2 + (w - 2 * (n - 2));
            };
            auto load = [&](int u, int sl) {
                bool is_v;
                const int kt = unit_tile(u, is_v);
                mbar_expect_tx(bar_full(sl), TILE_BYTES);
                for (int kb = 0; kb < 2; ++kb)
                    tma_load_3d(ring_s(sl) + kb * BOX_BYTES, is_v ? &map_v : &map_k, bar_full(sl), g_kv * DH + kb * 64, kt * KEYS, kv_seq);
            };
            int u = 0;
            // the first two slots need no wait; tiles that no kernel of this step writes are requested right away
            for (; u < 2; ++u) {
                bool is_v;
                const int lo = unit_tile(u, is_v) * KEYS;
                if (!(lo + KEYS <= a.dirty_lo || lo >= a.dirty_hi)) break;
                load(u, u);
            }
            pdl_wait();      // the K / V rows written this step come from the projection that ran just before
            trace_stamp(7);
            for (; u < 2; ++u) load(u, u);
            bool ok = true;
            Ring r(2, slots);
            for (; u < 2 * n && ok; ++u, r.next(slots)) {
                if (u >= slots) ok = mbar_wait(bar_free(r.slot), r.phase ^ 1u, abort_flag);
                if (ok) load(u, r.slot);
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc_s = instr_desc_bf16(ROWS, KEYS);
            const uint32_t idesc_o = instr_desc_bf16(ROWS, DH) | (1u << 16);       // B (= V) is MN-major
            bool ok = mbar_wait(bar_q, 0, abort_flag);          // q is in shared memory
            Ring r(0, slots);
            auto take = [&]() {          // next tile of the ring: its slot, once it has landed
                const int sl = r.slot;
                ok = ok && mbar_wait(bar_full(sl), r.phase, abort_flag);
                r.next(slots);
                tc_fence_after();
                return sl;
            };
            auto mma_s = [&](int g, int sl) {
                if (!ok) return;
                const uint32_t q = q_s(ksplit ? 0 : g);
#pragma unroll
                for (int k = 0; k < DH / UMMA_K; ++k)
                    umma_bf16(tmem_base + (uint32_t)(g * KEYS), smem_desc_sw128(q + (k >> 2) * BOX_BYTES) + (uint64_t)((k & 3) * 2),
                              smem_desc_sw128(ring_s(sl) + (k >> 2) * BOX_BYTES) + (uint64_t)((k & 3) * 2), idesc_s, k > 0 ? 1u : 0u);
                umma_commit(bar_s(g));
            };
            auto mma_o = [&](int g, int k0, int sl) {
                ok = ok && mbar_wait(bar_p(g), (uint32_t)k0 & 1u, abort_flag);
                if (!ok) return;
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < KEYS / UMMA_K; ++k)         // B = V: 16 keys = two 8-row groups further down
                    umma_bf16_ta(tmem_base + (uint32_t)(2 * KEYS + g * DH), tmem_base + (uint32_t)(g * KEYS + k * (UMMA_K / 2)),
                                 smem_desc_mn_sw128(ring_s(sl) + (uint32_t)k * 2048u, BOX_BYTES), idesc_o, (k0 > 0 || k > 0) ? 1u : 0u);
            };
            auto release = [&](int sl) { if (ok) umma_commit(bar_free(sl)); };
            // The scores of tile k + 1 overwrite the probabilities of tile k: issued behind the P V that reads them, products
            // complete in order.
            if (!ksplit) {
                int ks = take();
                mma_s(0, ks);
                if (cnt1 > 0) mma_s(1, ks);
                release(ks);
                for (int k = 0; k < n && ok; ++k) {
                    const int vs = take();
                    mma_o(0, k, vs);
                    if (k + 1 < n) { ks = take(); mma_s(0, ks); }
                    if (cnt1 > 0) {
                        mma_o(1, k, vs);
                        release(vs);
                        if (k + 1 < n) mma_s(1, ks);
                    } else {
                        release(vs);
                    }
                    if (k + 1 < n) release(ks);
                }
            } else {
                for (int g = 0; g < min(n, 2); ++g) { const int ks = take(); mma_s(g, ks); release(ks); }
                for (int t = 0; t < n && ok; ++t) {
                    const int vs = take();
                    mma_o(t & 1, t >> 1, vs);
                    release(vs);
                    if (t + 2 < n) { const int ks = take(); mma_s(t & 1, ks); release(ks); }
                }
            }
            umma_commit(bar_o(0));       // (also on failure: the other warps then see the abort flag)
            umma_commit(bar_o(1));
        }
    } else {
        // ---- softmax warps: tensor-memory lane = row ---------------------------------------------------------------
        const int sw = warp - 2, g = sw >> 2, quarter = warp & 3;
        const int row = quarter * 32 + lane;                       // of the stream's row tile
        const int cnt = g ? cnt1 : cnt0;
        const uint32_t tS = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(g * KEYS);
        const uint32_t tO = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(2 * KEYS + g * DH);
        const int vr = vr0 + ((g && !ksplit) ? ROWS : 0) + row;
        auto head_row = [&](int v, int& hd) {                      // virtual row -> head, forward row
            const int hv = hpg == 1 ? 0 : v / part.rows, r = v - hv * part.rows;
            hd = g_kv * hpg + hv;
            return seq * f.stride + r + (r >= part.skip_at ? part.skip : 0);
        };
        int h;
        const int rr = head_row(vr, h);
        pdl_wait();            // the row table, q and the stored rows all come from earlier kernels of the stream
        float* prev = nullptr; float* lsep = nullptr;
        bool valid = false;
        int rec = 0, box_row = -1, box_arr = 0;                    // 0: the warp records nothing, 1: as boxes, 2: row by row
        {
            int stored = -1, arr = -1;                             // index of the stored row, 0: pprev, 1: aprev
            if (vr < part.vrows) {
                if (a.rows) {
                    const int4 rw = __ldg(reinterpret_cast<const int4*>(a.rows) + rr);      // {seq, pos, widx, aidx}
                    if (rw.y >= 0) {
                        valid = true;
                        if (REC && (a.cluster_K > 0 ? (row_is_proxy(rw.z) && a.pprev != nullptr) : (rw.z >= 0 && a.pprev != nullptr))) {
                            // recorded drift rows: the window rows, or (centroid proxies) the clusters' proxy rows
                            stored = a.cluster_K > 0 ? rw.x * a.cluster_K + row_cluster(rw.z) : rw.x * a.W_max + rw.z;
                            arr = 0;
                        } else if (REC && rw.w >= 0 && a.aprev) {
                            stored = rw.x * a.B + rw.w;
                            arr = 1;
                        }
                    }
                } else {
                    valid = true;
                    if (REC && a.pprev) { stored = rr; arr = 0; }
                }
            }
            if (rec_cta && stored >= 0) {
                const size_t i = (size_t)stored * a.n_heads + h;
                prev = (arr ? a.aprev : a.pprev) + i * a.N;
                lsep = (arr ? a.aprev_lse : a.pprev_lse) + i;
            }
            if (rec_cta && __any_sync(0xffffffffu, stored >= 0)) {
                // (rows behind the last one of a stand-alone call lie outside its map: loads fill, stores leave them out)
                const int s0 = __shfl_sync(0xffffffffu, stored, 0), h0 = __shfl_sync(0xffffffffu, h, 0);
                box_arr = __shfl_sync(0xffffffffu, arr, 0);
                const bool run = __all_sync(0xffffffffu, (stored == s0 + lane && arr == box_arr && h == h0) ||
                                                             (!a.rows && vr >= part.vrows && s0 + lane >= a.n_rows)) != 0;
                rec = (run && s0 >= 0 && ((f.maps >> box_arr) & 1)) ? 1 : 2;
                box_row = s0;
                if (cnt == 0) rec = 0;
            }
        }
        // q rows into shared memory in the operand layout, half a warp per row (the streams of a key split take 16 rows each)
        if (cnt > 0 || ksplit) {
            const int first = quarter * 32 + (ksplit ? 16 * g : 0), pairs = ksplit ? 8 : 16, ch = lane & 15;
            const int vq0 = vr0 + ((g && !ksplit) ? ROWS : 0) + first + (lane >> 4);
            const uint32_t dst = q_s(ksplit ? 0 : g) + (uint32_t)(ch >> 3) * BOX_BYTES;
            for (int i0 = 0; i0 < pairs; i0 += 8) {
                uint4 v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int vq = vq0 + 2 * (i0 + i);
                    v[i] = make_uint4(0u, 0u, 0u, 0u);
                    if (vq < part.vrows) {
                        int qh;
                        const int qr = head_row(vq, qh);
                        v[i] = __ldcg(reinterpret_cast<const uint4*>((const __nv_bfloat16*)a.q + (size_t)qr * dq + qh * DH) + ch);
                    }
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int lr = first + (lane >> 4) + 2 * (i0 + i);
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (uint32_t)lr * 128u + ((uint32_t)((ch ^ lr) & 7) << 4)),
                                 "r"(v[i].x), "r"(v[i].y), "r"(v[i].z), "r"(v[i].w) : "memory");
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_q);

        const float scale2 = a.scale * LOG2E_F;
        const bool use_old = REC && prev != nullptr && a.record_kl != 0;
        float lse_old = 0.f;
        if (REC && lsep && a.record_kl && (g == 0 || !ksplit)) lse_old = __ldcg(lsep);

        // ---- stored rows: patch i of this warp's sequence of [32 rows][64 keys] patches lies in buffer i & 1 as two boxes,
        // sixteen-byte piece c of a box's row r at r * 128 + ((c ^ (r & 7)) << 4)
        const uint32_t x0 = ring_s(FL_REC_SLOTS) + (uint32_t)sw * (2 * PATCH_BYTES);
        const bool vec = (a.N & 3) == 0 && (((uintptr_t)a.pprev | (uintptr_t)a.aprev) & 15) == 0;
        auto tile_of = [&](int k) { return ksplit ? 2 * k + g : k; };
        auto patch_key = [&](int i) { return tile_of(i >> 1) * KEYS + (i & 1) * 64; };
        const int patches = (REC && rec) ? 2 * (cnt - 1) + (a.N - tile_of(cnt - 1) * KEYS > 64 ? 2 : 1) : 0;
        auto patch_load = [&](int i) {
            const int k0 = patch_key(i);
            const uint32_t x = x0 + (uint32_t)(i & 1) * PATCH_BYTES;
            if (__builtin_expect(rec == 1, 1)) {
                if (lane == 0 && a.record_kl) {
                    const int nb = a.N - k0 > 32 ? 2 : 1;
                    mbar_expect_tx(bar_x(sw, i & 1), (uint32_t)nb * PBOX_BYTES);
                    for (int b = 0; b < nb; ++b)
                        tma_load_3d(x + (uint32_t)b * PBOX_BYTES, box_arr ? &map_r : &map_p, bar_x(sw, i & 1), k0 + 32 * b, h, box_row);
                }
            } else {
                if (a.record_kl) {
                    if (vec) {
#pragma unroll 4
                        for (int it = 0; it < 16; ++it) {
                            const int r = 2 * it + (lane >> 4), c = lane & 15;
                            const float* src = (const float*)__shfl_sync(0xffffffffu, (unsigned long long)prev, r);
                            if (src && k0 + 4 * c < a.N)
                                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(x + (uint32_t)(c >> 3) * PBOX_BYTES + (uint32_t)r * 128u + ((uint32_t)((c ^ r) & 7) << 4)), "l"(src + k0 + 4 * c) : "memory");
                        }
                    } else {
#pragma unroll 4
                        for (int r = 0; r < 32; ++r) {
                            const float* src = (const float*)__shfl_sync(0xffffffffu, (unsigned long long)prev, r);
                            for (int b = 0; b < 2; ++b)
                                if (src && k0 + 32 * b + lane < a.N)
                                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(x + (uint32_t)b * PBOX_BYTES + (uint32_t)r * 128u + ((uint32_t)(((lane >> 2) ^ r) & 7) << 4) + 4u * (lane & 3)),
                                                 "l"(src + k0 + 32 * b + lane) : "memory");
                        }
                    }
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
        };
        if (REC && rec) {
            for (int i = 0; i < min(patches, 2); ++i) patch_load(i);
        }

        float m = -INFINITY, l = 0.f;
        uint64_t A2[2] = {0ull, 0ull};
        bool ok = true;
        int ip = 0;                                        // next patch
        // (two copies of the loop: a warp without recorded rows takes the shorter one)
        auto stream_loop = [&](auto with_rows) {
        constexpr bool RW = decltype(with_rows)::value;
        for (int k = 0; k < cnt; ++k) {
            ok = mbar_wait(bar_s(g), (uint32_t)k & 1u, abort_flag) && ok && !*abort_flag;
            ok = __all_sync(0xffffffffu, ok) != 0;
            if (!ok) break;
            tc_fence_after();
            const int kb = tile_of(k) * KEYS;
            // All 128 scores are read for the maximum, the first 64 stay in registers and the others are read again.
            const bool edge = kb + KEYS > a.N;               // columns beyond the last key do not take part
            auto mask = [&](uint32_t* r, int c0) {
#pragma unroll
                for (int i = 0; i < 32; ++i) if (kb + c0 + i >= a.N) r[i] = 0xff800000u;      // -inf
            };
            uint32_t ra[32], rb[32];
            float tm4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
            auto top = [&](const uint32_t* x, const uint32_t* y, int j) {
#pragma unroll
                for (int i = 0; i < 32; ++i) tm4[j + (i & 1)] = fmaxf(tm4[j + (i & 1)], fmaxf(__uint_as_float(x[i]), __uint_as_float(y[i])));
            };
            if constexpr (RW) {              // (half at a time: the other form's registers are taken by the stored rows)
                tmem_ld32_issue(tS + 64u, ra);
                tmem_ld32_issue(tS + 96u, rb);
                tmem_ld_wait16(ra); tmem_ld_wait16(ra + 16); tmem_ld_wait16(rb); tmem_ld_wait16(rb + 16);
                if (__builtin_expect(edge, 0)) { mask(ra, 64); mask(rb, 96); }
                top(ra, rb, 0);
                tmem_ld32_issue(tS, ra);
                tmem_ld32_issue(tS + 32u, rb);
                tmem_ld_wait16(ra); tmem_ld_wait16(ra + 16); tmem_ld_wait16(rb); tmem_ld_wait16(rb + 16);
                if (__builtin_expect(edge, 0)) { mask(ra, 0); mask(rb, 32); }
                top(ra, rb, 2);
            } else {
                uint32_t rc[32], rd[32];
                tmem_ld32_issue(tS, ra);
                tmem_ld32_issue(tS + 32u, rb);
                tmem_ld32_issue(tS + 64u, rc);
                tmem_ld32_issue(tS + 96u, rd);
                tmem_ld_wait16(ra); tmem_ld_wait16(ra + 16); tmem_ld_wait16(rb); tmem_ld_wait16(rb + 16);
                tmem_ld_wait16(rc); tmem_ld_wait16(rc + 16); tmem_ld_wait16(rd); tmem_ld_wait16(rd + 16);
                if (__builtin_expect(edge, 0)) { mask(ra, 0); mask(rb, 32); mask(rc, 64); mask(rd, 96); }
                top(ra, rb, 0);
                top(rc, rd, 2);
            }
            float tm = fmaxf(fmaxf(tm4[0], tm4[1]), fmaxf(tm4[2], tm4[3])) * scale2;      // scale2 > 0: the maximum commutes with it
            if (a.p_pow2) tm = ceilf(tm);
            if (k == 0) {
                m = tm;
            } else if (__builtin_expect(__any_sync(0xffffffffu, tm > m + FL_SLACK), 0)) {
                // (the P V of the previous tile has completed: it was issued in front of the scores just read)
                // Decided row by row: a row's bits must not hang on the rows that share its warp, or one that has not changed would
                // drift when it is measured in other company (a block entry's rows, then a refresh step's).
                const bool up = tm > m + FL_SLACK;
                const float nm = up ? tm : m, al = up ? ex2(m - nm) : 1.f;
                l *= al;
                A2[0] = f2_mul(A2[0], f2_pack(al, al)); A2[1] = f2_mul(A2[1], f2_pack(al, al));
                m = nm;
#pragma unroll 1
                for (int c = 0; c < DH; c += 16) {
                    uint32_t o[16];
                    tmem_ld16_issue(tO + (uint32_t)c, o);
                    tmem_ld_wait16(o);
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * al);
                    tmem_st16_issue(tO + (uint32_t)c, o);
                }
                tmem_st_wait();
            }
            const float neg_m = m == -INFINITY ? 0.f : -m;       // (only -inf so far: p = 0)
            const uint64_t sc2 = f2_pack(scale2, scale2), nm2 = f2_pack(neg_m, neg_m);
            uint64_t l2[2] = {0ull, 0ull};
            // 64 columns (a patch) at a time; with stored rows in a rolled loop: straight-line code for all 128 misses the instruction cache
#pragma unroll (RW ? 1 : 2)
            for (int h2 = 0; h2 < 2; ++h2) {
                if (h2) {
                    tmem_ld_wait16(ra); tmem_ld_wait16(ra + 16); tmem_ld_wait16(rb); tmem_ld_wait16(rb + 16);
                    if (__builtin_expect(edge, 0)) { mask(ra, 64); mask(rb, 96); }
                }
                const int k0 = kb + 64 * h2;
                const bool patch = RW && k0 < a.N;
                const uint32_t x = x0 + (uint32_t)(ip & 1) * PATCH_BYTES;
                if (patch) {
                    if (__builtin_expect(rec == 1, 1)) {
                        if (ip >= 1) {
                            // the store of the patch before has read its buffer: the next patch may come there
                            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                            if (ip + 1 < patches) patch_load(ip + 1);
                            __syncwarp();
                        }
                        if (a.record_kl) ok = mbar_wait(bar_x(sw, ip & 1), (uint32_t)(ip >> 1) & 1u, abort_flag) && ok;
                    } else {
                        if (ip + 1 < patches) asm volatile("cp.async.wait_group 1;" ::: "memory");
                        else asm volatile("cp.async.wait_group 0;" ::: "memory");
                        __syncwarp();
                    }
                }
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                uint32_t* const r = c ? rb : ra;
                const uint32_t xr = x + (uint32_t)c * PBOX_BYTES + (uint32_t)lane * 128u;
                // sixteen columns at a time: the old scores are on their way while the exponentials are taken
                uint32_t pw[16];
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    float od[16], p[16];
                    if (patch) {
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(od[4 * q]), "=f"(od[4 * q + 1]), "=f"(od[4 * q + 2]), "=f"(od[4 * q + 3])
                                         : "r"(xr + ((uint32_t)(((4 * hf + q) ^ lane) & 7) << 4)));
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        float y0, y1;
                        f2_unpack(f2_fma(f2_pack(r[16 * hf + 2 * i], r[16 * hf + 2 * i + 1]), sc2, nm2), y0, y1);
                        p[2 * i] = ex2(y0); p[2 * i + 1] = ex2(y1);
                        l2[i & 1] = f2_add(l2[i & 1], f2_pack(p[2 * i], p[2 * i + 1]));
                        __nv_bfloat162 bb = __floats2bfloat162_rn(p[2 * i], p[2 * i + 1]);
                        pw[8 * hf + i] = *reinterpret_cast<uint32_t*>(&bb);
                    }
                    if (patch) {
                        // drift sum (entries without probability do not take part, whatever their difference: masked columns
                        // are -inf), new scores into the old ones' place
                        uint64_t sn[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {         // (rounded products: an unchanged row gives exactly zero)
                            sn[i] = f2_mul(f2_mul(f2_pack(r[16 * hf + 2 * i], r[16 * hf + 2 * i + 1]), sc2), f2_pack(LN2_F, LN2_F));
                            float d0, d1;
                            f2_unpack(f2_fma(f2_pack(od[2 * i], od[2 * i + 1]), f2_pack(-1.f, -1.f), sn[i]), d0, d1);
                            d0 = p[2 * i] > 0.f ? d0 : 0.f; d1 = p[2 * i + 1] > 0.f ? d1 : 0.f;
                            A2[i & 1] = f2_fma(f2_pack(p[2 * i], p[2 * i + 1]), f2_pack(d0, d1), A2[i & 1]);
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            float w[4];
                            f2_unpack(sn[2 * q], w[0], w[1]); f2_unpack(sn[2 * q + 1], w[2], w[3]);
                            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(xr + ((uint32_t)(((4 * hf + q) ^ lane) & 7) << 4)), "f"(w[0]), "f"(w[1]), "f"(w[2]), "f"(w[3]));
                        }
                    }
                }
                tmem_st16_issue(tS + (uint32_t)(32 * h2 + 16 * c), pw);
                if (h2 == 0) tmem_ld32_issue(tS + 64u + 32u * (uint32_t)c, r);
                }
                if (patch) {                                 // the patch is complete
                    if (__builtin_expect(rec == 1, 1)) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the store reads what was just written
                        __syncwarp();
                        if (lane == 0) {
                            for (int b = 0; b < (a.N - k0 > 32 ? 2 : 1); ++b) tma_store_3d(box_arr ? &map_r : &map_p, x + (uint32_t)b * PBOX_BYTES, k0 + 32 * b, h, box_row);
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        }
                    } else {
                        __syncwarp();
                        if (vec) {
#pragma unroll 4
                            for (int it = 0; it < 16; ++it) {
                                const int r2 = 2 * it + (lane >> 4), c2 = lane & 15;
                                float* dst = (float*)__shfl_sync(0xffffffffu, (unsigned long long)prev, r2);
                                float4 v;
                                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                                             : "r"(x + (uint32_t)(c2 >> 3) * PBOX_BYTES + (uint32_t)r2 * 128u + ((uint32_t)((c2 ^ r2) & 7) << 4)) : "memory");
                                if (dst && k0 + 4 * c2 < a.N) __stcg(reinterpret_cast<float4*>(dst + k0) + c2, v);
                            }
                        } else {
#pragma unroll 4
                            for (int r2 = 0; r2 < 32; ++r2) {
                                float* dst = (float*)__shfl_sync(0xffffffffu, (unsigned long long)prev, r2);
                                for (int b = 0; b < 2; ++b) {
                                    float v;
                                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(x + (uint32_t)b * PBOX_BYTES + (uint32_t)r2 * 128u + ((uint32_t)(((lane >> 2) ^ r2) & 7) << 4) + 4u * (lane & 3)) : "memory");
                                    if (dst && k0 + 32 * b + lane < a.N) __stcg(dst + k0 + 32 * b + lane, v);
                                }
                            }
                        }
                        __syncwarp();
                        if (ip + 2 < patches) patch_load(ip + 2);
                    }
                    ++ip;
                }
            }
            l += f2_sum(f2_add(l2[0], l2[1]));
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_p(g));
        }
        };
        if constexpr (REC) { if (rec) stream_loop(std::true_type{}); else stream_loop(std::false_type{}); }
        else stream_loop(std::false_type{});
        if (REC && rec == 1) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");       // the last stores have left
        if (REC && rec == 2) asm volatile("cp.async.wait_all;" ::: "memory");                // (a wait that gave up left copies in flight)

        // ---- output rows and drift ----
        float A = f2_sum(f2_add(A2[0], A2[1]));
        ok = mbar_wait(bar_o(0), 0, abort_flag) && mbar_wait(bar_o(1), 0, abort_flag) && ok && !*abort_flag;
        ok = __all_sync(0xffffffffu, ok) != 0;
        tc_fence_after();
        float w0 = 1.f / l, w1 = 0.f;                      // weights of the streams' O
        if (ksplit) {
            // the streams' parts of the row (m, l, A) meet in the first ring slot's place: every product has completed
            float* ex = reinterpret_cast<float*>(smem + q_tiles * TILE_BYTES);
            ex[(3 * g) * ROWS + row] = m; ex[(3 * g + 1) * ROWS + row] = l; ex[(3 * g + 2) * ROWS + row] = A;
            bar_sync_streams();
            const float m0 = ex[row], m1 = ex[3 * ROWS + row];
            m = fmaxf(m0, m1);
            const float a0 = ex2(m0 - m), a1 = ex2(m1 - m);           // (a stream without tiles: m1 = -inf, a1 = 0)
            l = ex[ROWS + row] * a0 + ex[4 * ROWS + row] * a1;
            A = ex[2 * ROWS + row] * a0 + ex[5 * ROWS + row] * a1;
            w0 = a0 / l; w1 = a1 / l;
        }
        if (ok && (cnt > 0 || ksplit)) {
            const float lse = (m + log2f(l)) * LN2_F;             // natural-log units, like the stored rows
            if (g == 0 || !ksplit) {
                if (REC && lsep && valid) *lsep = lse;
                if (valid && a.kl) a.kl[(size_t)rr * a.n_heads + h] = use_old ? A / l - (lse - lse_old) : 0.f;
            }
            const int c_lo = ksplit ? 64 * g : 0, c_hi = ksplit ? c_lo + 64 : DH;
            const uint32_t t0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(2 * KEYS);
            __nv_bfloat16* dst = (__nv_bfloat16*)a.out + (size_t)rr * dq + h * DH;
            for (int c = c_lo; c < c_hi; c += 32) {
                uint32_t o[32], o1[32];
                tmem_ld32_issue((ksplit ? t0 : tO) + (uint32_t)c, o);
                if (ksplit && cnt1 > 0) tmem_ld32_issue(t0 + (uint32_t)(DH + c), o1);
                tmem_ld_wait16(o); tmem_ld_wait16(o + 16);
                if (ksplit && cnt1 > 0) {
                    tmem_ld_wait16(o1); tmem_ld_wait16(o1 + 16);
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * w0 + __uint_as_float(o1[i]) * w1);
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * w0);
                }
                if (valid && a.out) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t w[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            __nv_bfloat162 bb = __floats2bfloat162_rn(__uint_as_float(o[8 * q + 2 * i]), __uint_as_float(o[8 * q + 2 * i + 1]));
                            w[i] = *reinterpret_cast<uint32_t*>(&bb);
                        }
                        *reinterpret_cast<uint4*>(dst + c + 8 * q) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, 512);
    if (threadIdx.x == 0 && abort_sh && f.status) atomicExch(f.status, 1);
}

}  // namespace afl
}  // namespace ps
