// CUDA-core kernels of the Polestar step: row table, embedding, RMSNorm staging, a plain
// tiled GEMM (fp32 models and debugging), attention with drift (fp32 models), select /
// compaction, confidence and commit.
#pragma once
#include "common.cuh"

namespace ps {

// ---------------------------------------------------------------------------------------
// Row table of one forward (Algorithm 1: E_b at block entry, J_b plus Omega_b within a block)
// ---------------------------------------------------------------------------------------
__global__ void build_rows_kernel(StepDesc sd, Row* rows) {
    KERNEL_PROLOGUE(1);   // build_rows_kernel
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int total = sd.batch * sd.rows_per_seq;
    if (i >= total) return;
    const int s = i / sd.rows_per_seq, j = i - s * sd.rows_per_seq;
    Row r;
    r.seq = s; r.pos = -1; r.widx = -1; r.aidx = -1;
    const int n_plain = sd.rows_per_seq - sd.K;      // the proxy rows of the clusters come last
    if (j >= n_plain) {
        // proxy row: position and emptiness are per layer (cluster tables); unused on steps without refresh
        if (sd.kind != 2 || sd.refresh.v[s]) { r.pos = 0; r.widx = -2 - (j - n_plain); }
    } else if (sd.kind == 2) {
        if (j < sd.B) {
            r.pos = sd.act_start + j; r.aidx = j;
        } else {
            const int w = j - sd.B;
            if (w < sd.W && sd.refresh.v[s]) { r.pos = window_pos(sd, w); r.widx = w; }
        }
    } else {
        const int pos = sd.e0 + j;
        if (pos < sd.N) {
            r.pos = pos;
            if (pos >= sd.act_start && pos < sd.act_start + sd.B) r.aidx = pos - sd.act_start;
            else r.widx = window_index(sd, pos);
        }
    }
    rows[i] = r;
}

// ---------------------------------------------------------------------------------------
// Layer-0 inputs: embeddings of forwarded rows; on refresh steps the layer-0 packet holds the
// embeddings of window positions whose token changed since their cached row was written
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void embed_rows_kernel(StepDesc sd, const Row* rows, const int* y, const T* emb, int d,
                                  float* x, float* packet, unsigned char* patch0, int* tok_at_h0,
                                  int* stats) {
    KERNEL_PROLOGUE(2);   // embed_rows_kernel
    const int r = blockIdx.x;
    const Row rw = rows[r];
    if (rw.pos < 0 || row_is_proxy(rw.widx)) return;
    const int tok = y[rw.seq * sd.N + rw.pos];
    const T* e = emb + (size_t)tok * d;
    if (sd.within && rw.widx >= 0) {
        const int o = rw.seq * sd.W_max + rw.widx;
        const bool changed = tok_at_h0[o] != tok;
        if (changed) {
            float* dst = packet + (size_t)o * d;
            for (int c = threadIdx.x; c < d; c += blockDim.x) dst[c] = to_f<T>(e[c]);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            patch0[o] = changed ? 1 : 0;
            tok_at_h0[o] = tok;
            if (changed) atomicAdd(stats, 1);
        }
    } else {
        float* dst = x + (size_t)r * d;
        for (int c = threadIdx.x; c < d; c += blockDim.x) dst[c] = to_f<T>(e[c]);
        if (!sd.within && rw.widx >= 0 && threadIdx.x == 0) tok_at_h0[rw.seq * sd.W_max + rw.widx] = tok;
    }
}

// ---------------------------------------------------------------------------------------
// One row of RMSNorm + staging, held in registers: every thread owns up to NORM_VPT float4 chunks,
// so the row is read once (all loads in flight together), reduced, scaled and stored.
// Requires d % 4 == 0 and d <= 4 * NORM_VPT * blockDim.x.
// ---------------------------------------------------------------------------------------
constexpr int NORM_THREADS = 512;
constexpr int NORM_VPT = 8;
template <typename T>
__device__ __forceinline__ void store4(T* p, float a, float b, float c, float d4);
template <>
__device__ __forceinline__ void store4<float>(float* p, float a, float b, float c, float d4) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d4);
}
template <>
__device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* p, float a, float b, float c, float d4) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d4);
    uint2 u;
    u.x = *reinterpret_cast<uint32_t*>(&lo);
    u.y = *reinterpret_cast<uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(p) = u;
}
// src row -> a_out row (normed, times gain); optional copies of the raw row to up to two fp32 destinations
template <typename T>
__device__ __forceinline__ void norm_row(const float* __restrict__ src, const float* __restrict__ gain, float eps, int d,
                                         T* a_out, float* copy0, float* copy1, float* red) {
    const int n4 = d >> 2;
    float4 v[NORM_VPT];
    float ss = 0.f;
#pragma unroll
    for (int u = 0; u < NORM_VPT; ++u) {
        const int c4 = threadIdx.x + u * blockDim.x;
        v[u] = c4 < n4 ? __ldcg(reinterpret_cast<const float4*>(src) + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
        // the gains are needed only after the reduction: have them in L1 by then
        if (c4 < n4) asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const float4*>(gain) + c4));
    }
#pragma unroll
    for (int u = 0; u < NORM_VPT; ++u) ss += v[u].x * v[u].x + v[u].y * v[u].y + v[u].z * v[u].z + v[u].w * v[u].w;
    ss = block_sum(ss, red);
    const float inv = rsqrtf(ss / (float)d + eps);
#pragma unroll
    for (int u = 0; u < NORM_VPT; ++u) {
        const int c4 = threadIdx.x + u * blockDim.x;
        if (c4 < n4) {
            const float4 g = __ldg(reinterpret_cast<const float4*>(gain) + c4);
            store4<T>(a_out + 4 * c4, v[u].x * inv * g.x, v[u].y * inv * g.y, v[u].z * inv * g.z, v[u].w * inv * g.w);
            if (copy0) reinterpret_cast<float4*>(copy0)[c4] = v[u];
            if (copy1) reinterpret_cast<float4*>(copy1)[c4] = v[u];
        }
    }
}
template <typename T>
__device__ __forceinline__ void zero_row(T* a, int d) {
    for (int c = threadIdx.x; c < d; c += blockDim.x) a[c] = from_f<T>(0.f);
}

// ---------------------------------------------------------------------------------------
// Patch + RMSNorm + staging of the QKV projection's input rows (Algorithm 1 "Patch")
//   window rows of a within-block step read the hidden cache (after taking the packet row if
//   the previous layer selected them); every other row reads the residual stream x.
// ---------------------------------------------------------------------------------------
// TABS false: a step without cluster tables (no proxy rows, no quantised cache), whose rows need half of the registers
template <typename T, bool TABS = true>
__device__ __forceinline__ void prep_qkv_row(const StepDesc& sd, int r, const Row* rows, float* x, float* hc, const float* packet,
                                             const unsigned char* patch, const float* gain, float eps, int d,
                                             T* a_out, unsigned char* kvflag, float* red, const ClusterTabs& ct) {
    const Row rw = rows[r];
    T* a = a_out + (size_t)r * d;
    if (rw.pos < 0) {
        zero_row<T>(a, d);
        if (threadIdx.x == 0) kvflag[r] = 0;
        return;
    }
    if (TABS && row_is_proxy(rw.widx)) {
        // Proxy of a cluster = mean of its members' current hidden rows (Sec. 4.1: the centroid follows its refreshed
        // members; rebuilding the mean from the cache is that incremental update without its rounding drift).
        // Members are added in ascending window order by every thread for its own columns: deterministic.
        const int c = row_cluster(rw.widx);
        const int n = ct.zcnt[rw.seq * ct.K + c];
        if (threadIdx.x == 0) kvflag[r] = 0;
        if (n <= 0) { zero_row<T>(a, d); return; }
        const int* mem = ct.members + (size_t)rw.seq * sd.W_max + ct.moff[rw.seq * (ct.K + 1) + c];
        float* z = ct.zbuf + ((size_t)rw.seq * ct.K + c) * d;
        const float inv_n = 1.f / (float)n;
        const int n4 = d >> 2;
        // the members' row tables go through shared memory in groups, so that the loads of the rows themselves do not
        // wait on a chain of dependent index loads
        constexpr int GROUP = 64;
        __shared__ const float* s_src[GROUP];
        __shared__ int s_o[GROUP];                               // row of the cache; bit 30: the row enters the cache now
        float4 acc[NORM_VPT], rf[NORM_VPT];
#pragma unroll
        for (int u = 0; u < NORM_VPT; ++u) {
            const int c4 = threadIdx.x + u * blockDim.x;
            acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            rf[u] = (ct.hq && c4 < n4) ? __ldg(reinterpret_cast<const float4*>(ct.z0 + ((size_t)rw.seq * ct.K + c) * d) + c4)
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int t0 = 0; t0 < n; t0 += GROUP) {
            __syncthreads();
            if (threadIdx.x < GROUP && t0 + threadIdx.x < n) {
                const int w = mem[t0 + threadIdx.x];
                const int o = rw.seq * sd.W_max + w;
                const bool pt = sd.within && patch[o];
                s_src[threadIdx.x] = !sd.within ? x + ((size_t)rw.seq * sd.rows_per_seq + (window_pos(sd, w) - sd.e0)) * d
                                                : (pt ? packet + (size_t)o * d : hc + (size_t)o * d);
                s_o[threadIdx.x] = o | ((!sd.within || pt) ? (1 << 30) : 0);
            }
            __syncthreads();
            const int nb = min(GROUP, n - t0);
#pragma unroll
            for (int u = 0; u < NORM_VPT; ++u) {
                const int c4 = threadIdx.x + u * blockDim.x;
                const bool in = c4 < n4;
                if (u * (int)blockDim.x >= n4) continue;         // (the whole block is past the row)
                // members in ascending window order for every column (deterministic): all loads of a group are issued before
                // the first of them is used, sixteen of a plain cache's (a refresh step with eight proxies at the 8B widths: 5833 -> 5669
                // us), four of a quantised one's
                if (!ct.hq) {
                    for (int t = 0; t < nb; t += 16) {
                        float4 v[16];
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            v[k] = (t + k < nb && in) ? __ldcg(reinterpret_cast<const float4*>(s_src[t + k]) + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            if (t + k < nb) { acc[u].x += v[k].x; acc[u].y += v[k].y; acc[u].z += v[k].z; acc[u].w += v[k].w; }
                    }
                    continue;
                }
                for (int t = 0; t < nb; t += 4) {
                    float4 v[4];
                    unsigned cd[4], sb[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                        cd[k] = sb[k] = 0;
                        if (t + k < nb && in) {
                            const int so = s_o[t + k];
                            const size_t o = (size_t)(so & ~(1 << 30));
                            const bool fresh = (so >> 30) & 1;
                            if (!ct.hq || fresh) v[k] = __ldcg(reinterpret_cast<const float4*>(s_src[t + k]) + c4);
                            if (ct.hq) {
                                // the member's STORED value: the codes in the cache, or (a row that enters the cache in this
                                // step) what the codec makes of the plain row, or the codes imposed on it
                                const bool imposed = fresh && ct.fmask && ct.fmask[o];
                                const unsigned char* q = imposed ? ct.fq : ct.hq;
                                const unsigned char* sc = imposed ? ct.fs : ct.hs;
                                if (!fresh || imposed) {
                                    cd[k] = *reinterpret_cast<const unsigned short*>(q + o * (size_t)(d >> 1) + 2 * c4);
                                    sb[k] = sc[o * (size_t)(d >> 4) + (c4 >> 2)];
                                }
                            }
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (t + k < nb) {                        // (uniform: the codec's lanes act together)
                            if (ct.hq) {
                                const int so = s_o[t + k];
                                const bool fresh = (so >> 30) & 1;
                                const bool imposed = fresh && ct.fmask && ct.fmask[(size_t)(so & ~(1 << 30))];
                                if (fresh && !imposed) {
                                    unsigned c_, s_;
                                    v[k] = nvfp4_residual_chunk(v[k], rf[u], &c_, &s_);
                                } else if (in) {
                                    v[k] = nvfp4_dequant_chunk(cd[k], sb[k], rf[u]);
                                }
                            }
                            acc[u].x += v[k].x; acc[u].y += v[k].y; acc[u].z += v[k].z; acc[u].w += v[k].w;
                        }
                    }
                }
            }
        }
        // the mean row (kept for read-back) and its RMSNorm, straight from the registers
        float ss = 0.f;
#pragma unroll
        for (int u = 0; u < NORM_VPT; ++u) {
            const int c4 = threadIdx.x + u * blockDim.x;
            acc[u] = make_float4(acc[u].x * inv_n, acc[u].y * inv_n, acc[u].z * inv_n, acc[u].w * inv_n);
            if (c4 < n4) {
                reinterpret_cast<float4*>(z)[c4] = acc[u];
                ss += acc[u].x * acc[u].x + acc[u].y * acc[u].y + acc[u].z * acc[u].z + acc[u].w * acc[u].w;
            }
        }
        ss = block_sum(ss, red);
        const float inv = rsqrtf(ss / (float)d + eps);
#pragma unroll
        for (int u = 0; u < NORM_VPT; ++u) {
            const int c4 = threadIdx.x + u * blockDim.x;
            if (c4 < n4) {
                const float4 g = __ldg(reinterpret_cast<const float4*>(gain) + c4);
                store4<T>(a + 4 * c4, acc[u].x * inv * g.x, acc[u].y * inv * g.y, acc[u].z * inv * g.z, acc[u].w * inv * g.w);
            }
        }
        return;
    }
    float* xr = x + (size_t)r * d;
    bool kv = true;
    if (TABS && rw.widx >= 0 && ct.hq) {
        // ---- NVFP4 residual cache: the row's codes against its cluster's block-entry centroid
        const size_t o = (size_t)rw.seq * sd.W_max + rw.widx;
        const float* ref = ct.z0 + ((size_t)rw.seq * ct.K + ct.labels[o]) * d;
        unsigned char* cq = ct.hq + o * (size_t)(d >> 1);
        unsigned char* cs = ct.hs + o * (size_t)(d >> 4);
        const bool patched = sd.within && patch[o] != 0;
        const bool fresh = !sd.within || patched;              // block entry records the row; a packet row replaces it
        const bool imposed = fresh && ct.fmask && ct.fmask[o];
        kv = fresh;
        const float* src = !sd.within ? xr : packet + o * d;
        const int n4 = d >> 2;
        float4 v[NORM_VPT];
        float ss = 0.f;
#pragma unroll
        for (int u = 0; u < NORM_VPT; ++u) {
            const int c4 = threadIdx.x + u * blockDim.x;
            const bool in = c4 < n4;
            const float4 rf = in ? __ldg(reinterpret_cast<const float4*>(ref) + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
            v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (u * (int)blockDim.x >= n4) continue;           // (the whole block is past the row)
            if (fresh) {
                const float4 raw = in ? __ldcg(reinterpret_cast<const float4*>(src) + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
                unsigned cd, sb;
                float4 q = nvfp4_residual_chunk(raw, rf, &cd, &sb);
                if (in && imposed) {
                    cd = *reinterpret_cast<const unsigned short*>(ct.fq + o * (size_t)(d >> 1) + 2 * c4);
                    sb = ct.fs[o * (size_t)(d >> 4) + (c4 >> 2)];
                    q = nvfp4_dequant_chunk(cd, sb, rf);
                }
                if (in) {
                    *reinterpret_cast<unsigned short*>(cq + 2 * c4) = (unsigned short)cd;
                    if ((c4 & 3) == 0) cs[c4 >> 2] = (unsigned char)sb;
                    // a block-entry forward goes on with the plain row (only later steps read the cache); a refreshed
                    // row is what the cache now holds
                    v[u] = sd.within ? q : raw;
                }
            } else if (in) {
                v[u] = nvfp4_dequant_chunk(*reinterpret_cast<const unsigned short*>(cq + 2 * c4), cs[c4 >> 2], rf);
            }
            ss += v[u].x * v[u].x + v[u].y * v[u].y + v[u].z * v[u].z + v[u].w * v[u].w;
        }
        ss = block_sum(ss, red);
        const float inv = rsqrtf(ss / (float)d + eps);
#pragma unroll
        for (int u = 0; u < NORM_VPT; ++u) {
            const int c4 = threadIdx.x + u * blockDim.x;
            if (c4 < n4) {
                const float4 g = __ldg(reinterpret_cast<const float4*>(gain) + c4);
                store4<T>(a + 4 * c4, v[u].x * inv * g.x, v[u].y * inv * g.y, v[u].z * inv * g.z, v[u].w * inv * g.w);
                if (sd.within) reinterpret_cast<float4*>(xr)[c4] = v[u];
            }
        }
    } else if (rw.widx >= 0) {
        const size_t o = (size_t)rw.seq * sd.W_max + rw.widx;
        float* h = hc + o * d;
        if (sd.within) {
            // window row of a within-block step: the packet row if the previous layer selected it
            // (then it also replaces the cached hidden row), else the cached hidden row
            const bool patched = patch[o] != 0;
            kv = patched;
            norm_row<T>(patched ? packet + o * d : h, gain, eps, d, a, xr, patched ? h : nullptr, red);
        } else {
            norm_row<T>(xr, gain, eps, d, a, h, nullptr, red);      // block entry: record the hidden row
        }
    } else {
        norm_row<T>(xr, gain, eps, d, a, nullptr, nullptr, red);
    }
    if (threadIdx.x == 0) kvflag[r] = kv ? 1 : 0;
}
// Imposed NVFP4 codes written straight into the cache: one block per window row of one layer.
__global__ void impose_codes_kernel(const unsigned char* fmask, const unsigned char* fq, const unsigned char* fs, unsigned char* hq,
                                    unsigned char* hs, int d) {
    const size_t o = blockIdx.x;
    if (!fmask[o]) return;
    for (int i = threadIdx.x; i < (d >> 1); i += blockDim.x) hq[o * (size_t)(d >> 1) + i] = fq[o * (size_t)(d >> 1) + i];
    for (int i = threadIdx.x; i < (d >> 4); i += blockDim.x) hs[o * (size_t)(d >> 4) + i] = fs[o * (size_t)(d >> 4) + i];
}

template <typename T, bool TABS>
__global__ void prep_qkv_kernel(StepDesc sd, const Row* rows, float* x, float* hc, const float* packet,
                                const unsigned char* patch, const float* gain, float eps, int d,
                                T* a_out, unsigned char* kvflag, ClusterTabs ct) {
    KERNEL_PROLOGUE(3);   // prep_qkv_kernel
    __shared__ float red[33];
    prep_qkv_row<T, TABS>(sd, blockIdx.x, rows, x, hc, packet, patch, gain, eps, d, a_out, kvflag, red, ct);
}

// RMSNorm of a compacted list of rows (FFN input, LM-head input).
//   src row = list ? list[i] : i;  packet_rows: rows flagged as window rows read the packet
//   packet != null (steps whose down projection adds onto its output rows): the residual row of a selected window row is
//   also copied to its packet row, where that projection's parts then land
template <typename T>
__device__ __forceinline__ void prep_rows_row(int i, const float* x, const int* list, const int* m_count, const float* gain,
                                              float eps, int d, T* a_out, float* red, const Row* rows = nullptr,
                                              float* packet = nullptr, int W_max = 0) {
    T* a = a_out + (size_t)i * d;
    if (m_count && i >= *m_count) {
        for (int c = threadIdx.x; c < d; c += blockDim.x) a[c] = from_f<T>(0.f);
        return;
    }
    const int r = list ? list[i] : i;
    float* copy = nullptr;
    if (packet && rows) {
        const Row rw = rows[r];
        if (rw.pos >= 0 && rw.widx >= 0) copy = packet + ((size_t)rw.seq * W_max + rw.widx) * d;
    }
    norm_row<T>(x + (size_t)r * d, gain, eps, d, a, copy, nullptr, red);
}
template <typename T>
__global__ void prep_rows_kernel(const float* x, const int* list, const int* m_count, const float* gain,
                                 float eps, int d, T* a_out, const Row* rows, float* packet, int W_max) {
    KERNEL_PROLOGUE(4);   // prep_rows_kernel
    __shared__ float red[33];
    prep_rows_row<T>(blockIdx.x, x, list, m_count, gain, eps, d, a_out, red, rows, packet, W_max);
}

// Rows of a compacted list, gathered: dst row i <- src row list[i] (`bytes` a multiple of 16, rows 16-byte aligned).  Bound by
// the copy; four 16-byte loads in flight per thread.
__global__ void __launch_bounds__(128) gather_rows_kernel(const char* src, const int* list, const int* m_count, int bytes, char* dst) {
    KERNEL_PROLOGUE(6);   // gather_rows_kernel
    const int i = blockIdx.x;
    if (i >= __ldcg(m_count)) return;
    const uint4* s = reinterpret_cast<const uint4*>(src + (size_t)__ldcg(list + i) * bytes);
    uint4* d = reinterpret_cast<uint4*>(dst + (size_t)i * bytes);
    const int n = bytes >> 4;
    for (int c = threadIdx.x; c < n; c += 4 * 128) {
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) if (c + 128 * k < n) v[k] = __ldcg(s + c + 128 * k);
#pragma unroll
        for (int k = 0; k < 4; ++k) if (c + 128 * k < n) d[c + 128 * k] = v[k];
    }
}

// LM-head input rows: entry i < n_act reads x[act_rows...]; later entries read packet rows.
struct HeadSrc { int kind; int index; };  // kind 0: x row `index`; 1: packet row `index` (= seq*W_max+w)
template <typename T>
__global__ void prep_head_kernel(const float* x, const float* packet, const HeadSrc* src_list,
                                 const int* m_count, const float* gain, float eps, int d, T* a_out) {
    KERNEL_PROLOGUE(5);   // prep_head_kernel
    __shared__ float red[33];
    const int i = blockIdx.x;
    T* a = a_out + (size_t)i * d;
    if (i >= *m_count) {
        for (int c = threadIdx.x; c < d; c += blockDim.x) a[c] = from_f<T>(0.f);
        return;
    }
    const HeadSrc hs = src_list[i];
    norm_row<T>((hs.kind ? packet : x) + (size_t)hs.index * d, gain, eps, d, a, nullptr, nullptr, red);
}

// Gather + RMSNorm for the stand-alone refresh kernel: row (s, i) <- h[s][idx[s][i]], `TPR` threads per row.
// The same launch also prepares what the projection behind it needs: the rotary table rope_tab[pos][half] (the first
// `rope_blocks` blocks: the entries of the selected positions, or of all P with `rope_all`) and, in its first row block, zeroed
// split-tile counters and status word of the caller's scratch.
//
// Few rows are bound by latency (read, reduce, store), many by the copy.  Rows whose layout allows it (`vec`: d a multiple of
// eight, 16-byte aligned rows and gains) are read once, in 16-byte loads that are all in flight together, and stay in
// registers: a block per row, or from REFRESH_WARP_ROWS rows on a warp per row, which has no block barriers (a barrier per 8 KB
// row leaves the memory system idle).  The rotary entries (a pow and a sincos in double precision: several microseconds in a row) are the
// work of blocks of their own, beside the rows instead of in front of each.
// Gather and projection, K = 4096, 12288 features, against element loads in two passes with the rotary entries in the row blocks,
// us: 41 rows 32.8 -> 26.8, 205 48.5 -> 42.1, 1024 114 -> 98, 600 of 600 92 -> 70, 8192 697 -> 653 (power limited).
constexpr int REFRESH_THREADS = 256;
constexpr int REFRESH_VPT = 16;              // 16-byte chunks a thread can hold
constexpr int REFRESH_WARP_ROWS = 1024;      // a warp per row from here on: all SMs then have a block of eight rows
template <int TPR>
__global__ void __launch_bounds__(REFRESH_THREADS)
prep_refresh_kernel(const __nv_bfloat16* h, const int* idx, const int* counts, int batch, int max_rows, int P, const float* gain, float eps, int d,
                    int vec, __nv_bfloat16* a_out, float2* rope_tab, int rope_blocks, int rope_all, int half, double theta, int* counters,
                    int n_counters, int* status) {
    // The projection behind this launch requests weights before its own dependency wait, so it may start only when whatever
    // ran before this launch (the caller's kernel that wrote those weights, for one) is complete: wait, then trigger.  What
    // that costs: the weight stream no longer starts under the selection in front of the refresh.
    pdl_wait();
    pdl_trigger();
    trace_stamp(6);   // prep_refresh_kernel
    __shared__ float red[33];
    const int t = threadIdx.x;
    if ((int)blockIdx.x < rope_blocks) {
        // a thread keeps its column: one pow, then a sincos per position
        const int cols = min(half, REFRESH_THREADS), side = REFRESH_THREADS / cols, r = t / cols;
        if (r >= side) return;
        const int n = rope_all ? P : batch * max_rows;
        for (int k = t - r * cols; k < half; k += cols) {
            const double inv = pow(theta, -(double)k / (double)half);
            for (int m = (int)blockIdx.x * side + r; m < n; m += rope_blocks * side) {
                int pos = m;
                if (!rope_all) {
                    const int s = m / max_rows;
                    if (m - s * max_rows >= counts[s]) continue;
                    pos = idx[m];
                }
                const double ang = (double)pos * inv;
                rope_tab[(size_t)pos * half + k] = make_float2((float)cos(ang), (float)sin(ang));
            }
        }
        return;
    }
    const int blk = (int)blockIdx.x - rope_blocks;
    if (blk == 0 && counters) {
        for (int c = t; c < n_counters; c += REFRESH_THREADS) counters[c] = 0;
        if (t == 0 && status) *status = 0;
    }
    constexpr int ROWS = REFRESH_THREADS / TPR;
    const int m = blk * ROWS + t / TPR, tr = t % TPR;
    if (m >= batch * max_rows) return;                   // (TPR < REFRESH_THREADS: whole warps; no block barrier below)
    const int s = m / max_rows;
    __nv_bfloat16* a = a_out + (size_t)m * d;
    const bool live = m - s * max_rows < counts[s];
    if (!vec) {
        if (!live) { for (int c = tr; c < d; c += TPR) a[c] = from_f<__nv_bfloat16>(0.f); return; }
        const __nv_bfloat16* src = h + ((size_t)s * P + idx[m]) * d;
        float ss = 0.f;
        for (int c = tr; c < d; c += TPR) { const float v = to_f<__nv_bfloat16>(src[c]); ss += v * v; }
        ss = TPR == 32 ? warp_sum(ss) : block_sum(ss, red);
        const float inv = rsqrtf(ss / (float)d + eps);
        for (int c = tr; c < d; c += TPR) a[c] = from_f<__nv_bfloat16>(to_f<__nv_bfloat16>(src[c]) * inv * gain[c]);
        return;
    }
    const int n16 = d >> 3;
    uint4* dst = reinterpret_cast<uint4*>(a);
    if (!live) { for (int c = tr; c < n16; c += TPR) dst[c] = make_uint4(0u, 0u, 0u, 0u); return; }
    const uint4* src = reinterpret_cast<const uint4*>(h + ((size_t)s * P + idx[m]) * d);
    uint4 v[REFRESH_VPT];
    float ss = 0.f;
#pragma unroll
    for (int u = 0; u < REFRESH_VPT; ++u) {
        const int c = tr + u * TPR;
        v[u] = c < n16 ? __ldcg(src + c) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int u = 0; u < REFRESH_VPT; ++u) {
        const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float lo = __uint_as_float(w[i] << 16), hi = __uint_as_float(w[i] & 0xFFFF0000u);
            ss += lo * lo + hi * hi;
        }
    }
    ss = TPR == 32 ? warp_sum(ss) : block_sum(ss, red);
    const float inv = rsqrtf(ss / (float)d + eps);
#pragma unroll
    for (int u = 0; u < REFRESH_VPT; ++u) {
        const int c = tr + u * TPR;
        if (c >= n16) break;
        const float4 g0 = __ldg(reinterpret_cast<const float4*>(gain) + 2 * c), g1 = __ldg(reinterpret_cast<const float4*>(gain) + 2 * c + 1);
        const float g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
        const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float lo = __uint_as_float(w[i] << 16), hi = __uint_as_float(w[i] & 0xFFFF0000u);
            __nv_bfloat162 b2 = __floats2bfloat162_rn(lo * inv * g[2 * i], hi * inv * g[2 * i + 1]);
            o[i] = *reinterpret_cast<uint32_t*>(&b2);
        }
        dst[c] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// ---------------------------------------------------------------------------------------
// Spherical K-means of the window's hidden rows at block entry (Sec. 4.1 "Cluster and Quantize Hidden States";
// Algorithm 1 "SphericalKMeans"), one CTA per sequence, and the cluster tables that follow from the labels.
// Deterministic reading: centre j starts at the unit vector of window row floor((j + 1/2) W / K); `iters` Lloyd
// iterations (assign to the largest cosine, lowest cluster on ties; centre = normalised sum of the members' unit
// vectors, an empty cluster keeps its centre); no more rows than clusters: every row its own cluster.
// All sums run in a fixed order.  K <= KM_MAX_K, W <= KM_MAX_W (what a configuration with proxies admits).
// A chain of dependent phases on L2-resident rows: each keeps eight or sixteen loads per thread in flight (rows in flat member
// order, across cluster boundaries, in the centre update) and groups the rows by ballots.  96 rows x 4096, 8 clusters, in the pipeline,
// with single floats, centres in shared memory, a chain per cluster and loops over the labels 130 us, now 88 (83 of them without the
// comparisons in 64 bits).
// ---------------------------------------------------------------------------------------
constexpr int KM_MAX_K = 16, KM_MAX_W = 256, KM_THREADS = 512, KM_CL = 8, KM_SMEM_BYTES = 160 * 1024;
// A row's fp32 cosines are compared where they differ by more than their sums' rounding can: two chains of at most 40 additions for
// the product and the centre's norm, 80 x 2^-24.  Centres within that of the best are compared again by products and norms in 64 bits (rows of the
// lower layers, masked positions above all, are nearly parallel: the cosines of a decision are then within 1e-7 of one another).
constexpr float KM_NEAR = 5e-6f;
// What is left is the rounding of the centres, fp32 sums of up to KM_MAX_W unit vectors.  Rows that agree give centres along the same line, each of
// whose columns is off by at most n 2^-24 of itself, so their cosines are at least 1 - (n 2^-24)^2 / 2: closer than that is a tie.
constexpr double KM_TIE = 0.5 * (KM_MAX_W / 16777216.0) * (KM_MAX_W / 16777216.0);
struct KmeansArgs {
    const float* x;            // entry forward: residual-stream rows of this layer [rows][d]
    int d, K, iters;
    float* invn;               // scratch [batch][W_max]: the rows' 1 / norm
    int* labels; int* zpos; int* zcnt; int* members; int* moff;      // this layer's tables (see ClusterTabs)
    const int* forced_labels;  // [batch][W_max], first entry < 0: not forced (parity replay of another clustering)
    float* z0;                 // NVFP4 residual cache: [batch][K][d] member means of the plain rows (null: not kept)
};
// A cluster of KM_CL CTAs per sequence.  The columns are split over the CTAs: each keeps its columns of the centres in shared
// memory, works out its part of every (row, centre) product with four centres at a time in registers (a row's values against centres in
// shared memory were bound by its bandwidth), and adds up its columns of the members.  The rows are split over the CTAs for the decision: a row's
// owner receives the parts in its shared memory, adds them in rank order and sends the label to all.
__host__ __device__ inline int km_columns(int d) { return (((d + KM_CL - 1) / KM_CL) + 3) & ~3; }                     // per CTA
__host__ __device__ inline size_t km_smem(int d, int K, int W) { return ((size_t)K * km_columns(d) + (size_t)2 * KM_CL * ((W + KM_CL - 1) / KM_CL) * K) * sizeof(float); }
__device__ __forceinline__ void km_cluster_sync() {
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// a value into the same place of CTA `cta`'s shared memory
__device__ __forceinline__ void km_push(float* p, float v, int cta) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dsmem_addr((uint32_t)__cvta_generic_to_shared(p), cta)), "f"(v) : "memory");
}
__device__ __forceinline__ void km_push(int* p, int v, int cta) {
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(dsmem_addr((uint32_t)__cvta_generic_to_shared(p), cta)), "r"(v) : "memory");
}
__device__ __forceinline__ void km_push(double* p, double v, int cta) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dsmem_addr((uint32_t)__cvta_generic_to_shared(p), cta)), "d"(v) : "memory");
}
// sum of n products (n a multiple of four, 16-byte aligned) in 64 bits, by a warp
__device__ __forceinline__ double km_dot(const float* x, const float* y, int n, int lane) {
    double acc = 0.;
    for (int c = 4 * lane; c < n; c += 128) {
        const float4 u = *reinterpret_cast<const float4*>(x + c), v = *reinterpret_cast<const float4*>(y + c);
        acc = fma((double)u.x, (double)v.x, acc); acc = fma((double)u.y, (double)v.y, acc);
        acc = fma((double)u.z, (double)v.z, acc); acc = fma((double)u.w, (double)v.w, acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}
__global__ void __cluster_dims__(KM_CL, 1, 1) __launch_bounds__(KM_THREADS) kmeans_kernel(StepDesc sd, KmeansArgs a) {
    KERNEL_PROLOGUE(18);   // kmeans_kernel
    extern __shared__ __align__(16) float Cs[];             // [K][columns of this CTA]: the centres (member sums, not normalised)
    __shared__ float invn[KM_MAX_W];
    __shared__ int lab[KM_MAX_W];
    __shared__ float inv_c[KM_MAX_K];
    __shared__ int cnt[KM_MAX_K + 1], off[KM_MAX_K + 1];
    __shared__ unsigned short ord[KM_MAX_W];                 // window rows grouped by cluster, ascending inside a cluster
    // ... their rows of x, 1 / norm, and (last of a cluster) the cluster + 1
    __shared__ int ord_row[KM_MAX_W];
    __shared__ float ord_inv[KM_MAX_W];
    __shared__ unsigned char ord_last[KM_MAX_W];
    __shared__ int wcnt[KM_MAX_W / 32][KM_MAX_K];
    __shared__ float c2[KM_CL][KM_MAX_K];                    // every CTA's part of |centre|^2
    __shared__ double c2_64[KM_CL][KM_MAX_K];
    const int s = blockIdx.y, rk = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = KM_THREADS / 32;
    const int W = sd.W, K = a.K, d = a.d;
    auto row_index = [&](int w) { return s * sd.rows_per_seq + (window_pos(sd, w) - sd.e0); };
    auto row = [&](int w) { return a.x + (size_t)row_index(w) * d; };
    // lab[] -> cnt[], off[], ord[], ord_row[] (the whole block calls): ballots of the rows' labels, a warp per 32 rows
    auto group_rows = [&]() {
        __syncthreads();
        const int mine = t < W ? lab[t] : -1;
        int before = 0;                                      // rows of the own cluster in front of this one in its warp
        if (warp < KM_MAX_W / 32)
            for (int j = 0; j < K; ++j) {
                const unsigned b = __ballot_sync(0xffffffffu, mine == j);
                if (lane == 0) wcnt[warp][j] = __popc(b);
                if (mine == j) before = __popc(b & ((1u << lane) - 1u));
            }
        __syncthreads();
        if (t < 32) {
            int n = 0;
            if (t < K) for (int q = 0; q < KM_MAX_W / 32; ++q) { const int c = wcnt[q][t]; wcnt[q][t] = n; n += c; }
            int inc = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int up = __shfl_up_sync(0xffffffffu, inc, o); if (t >= o) inc += up; }
            if (t < K) { cnt[t] = n; off[t] = inc - n; }
            if (t == K - 1) off[K] = inc;
        }
        __syncthreads();
        if (mine >= 0) {
            const int o = off[mine] + wcnt[warp][mine] + before;
            ord[o] = (unsigned short)t;
            ord_row[o] = row_index(t);
            ord_inv[o] = invn[t];
            ord_last[o] = o + 1 == off[mine] + cnt[mine] ? mine + 1 : 0;
        }
        __syncthreads();
    };
    // sums over the members of every cluster for one column, rows in flat member order: done(cluster, sum), empty clusters left out
    auto member_sums = [&](int c, auto term, auto done) {
        float acc = 0.f;
        for (int i0 = 0; i0 < W; i0 += 16) {
            float v[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = i0 + k < W ? __ldg(a.x + (size_t)ord_row[i0 + k] * d + c) : 0.f;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                if (i0 + k >= W) break;
                acc = term(acc, v[k], i0 + k);
                const int last = ord_last[i0 + k];
                if (last) { done(last - 1, acc); acc = 0.f; }
            }
        }
    };
    float* invn_g = a.invn + (size_t)s * sd.W_max;
    int* labels = a.labels + (size_t)s * sd.W_max;
    const int per = (W + KM_CL - 1) / KM_CL, w_lo = min(W, rk * per), w_hi = min(W, w_lo + per);     // this CTA's rows
    const int dper = km_columns(d), c_lo = min(d, rk * dper), c_hi = min(d, c_lo + dper), cols = c_hi - c_lo;        // ... and columns
    const int n_rk = (d + dper - 1) / dper;                  // CTAs with columns (few of them leave the last CTAs none): only these have parts
    float* const part = Cs + (size_t)K * dper;               // [W][K] this CTA's part of the products
    float* const recv = part + (size_t)KM_CL * per * K;      // [CTA][per][K] the parts of this CTA's rows
    double* const recv_64 = reinterpret_cast<double*>(part); // [CTA][per][K] the same in 64 bits, in the place of both
    const int* forced = a.forced_labels ? a.forced_labels + (size_t)s * sd.W_max : nullptr;
    if (forced && forced[0] >= 0) {
        for (int w = w_lo + t; w < w_hi; w += KM_THREADS) labels[w] = min(max(forced[w], 0), K - 1);
    } else if (W <= K) {
        for (int w = w_lo + t; w < w_hi; w += KM_THREADS) labels[w] = w;
    } else {
        for (int w = w_lo + warp; w < w_hi; w += nw) {
            float ss = 0.f;
            const float4* h4 = reinterpret_cast<const float4*>(row(w));
            for (int q0 = lane; q0 < (d >> 2); q0 += 8 * 32) {
                float4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = q0 + 32 * u < (d >> 2) ? __ldg(h4 + q0 + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int u = 0; u < 8; ++u) ss = fmaf(v[u].x, v[u].x, fmaf(v[u].y, v[u].y, fmaf(v[u].z, v[u].z, fmaf(v[u].w, v[u].w, ss))));
            }
            ss = warp_sum(ss);
            if (lane == 0) invn_g[w] = ss > 0.f ? rsqrtf(ss) : 0.f;
        }
        // starting centres: rows floor((j + 1/2) W / K) of the window
        for (int e = t; e < K * cols; e += KM_THREADS) {
            const int j = e / cols, c = e - j * cols;
            Cs[(size_t)j * dper + c] = row((int)(((2 * j + 1) * (long long)W) / (2 * K)))[c_lo + c];
        }
        km_cluster_sync();
        for (int w = t; w < W; w += KM_THREADS) invn[w] = __ldcg(invn_g + w);
        const int groups = (K + 3) / 4, team = nw / groups;      // warps per group of four centres
        const int grp = warp / team, wt = warp - grp * team;
        for (int it = 0; it < a.iters; ++it) {
            // ---- this CTA's part of every product
            __syncthreads();
            if (grp < groups) {
                for (int q_lo = 0; q_lo < cols; q_lo += 512) {
                    float4 cv[4][4];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int c = q_lo + 4 * (lane + 32 * u);
                            cv[j][u] = (4 * grp + j < K && c < cols) ? *reinterpret_cast<const float4*>(Cs + (size_t)(4 * grp + j) * dper + c) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                    float4 hv[2][4];                              // this row and the next one, on its way
                    auto fetch = [&](int w, float4 (&v)[4]) {
                        const float* h = row(min(w, W - 1)) + c_lo;
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int c = q_lo + 4 * (lane + 32 * u);
                            v[u] = c < cols ? __ldg(reinterpret_cast<const float4*>(h + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                    };
                    auto products = [&](int w, const float4 (&hv)[4]) {
                        float dot[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            dot[j] = 0.f;
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                dot[j] = fmaf(hv[u].x, cv[j][u].x, fmaf(hv[u].y, cv[j][u].y, fmaf(hv[u].z, cv[j][u].z, fmaf(hv[u].w, cv[j][u].w, dot[j]))));
                        }
                        // four sums over the warp: after two exchange steps a lane carries one of them
                        const float x0 = __shfl_xor_sync(0xffffffffu, (lane & 1) ? dot[0] : dot[1], 1), x1 = __shfl_xor_sync(0xffffffffu, (lane & 1) ? dot[2] : dot[3], 1);
                        const float y0 = ((lane & 1) ? dot[1] : dot[0]) + x0, y1 = ((lane & 1) ? dot[3] : dot[2]) + x1;
                        float z = ((lane & 2) ? y1 : y0) + __shfl_xor_sync(0xffffffffu, (lane & 2) ? y0 : y1, 2);
                        z += __shfl_xor_sync(0xffffffffu, z, 4);
                        z += __shfl_xor_sync(0xffffffffu, z, 8);
                        z += __shfl_xor_sync(0xffffffffu, z, 16);
                        const int j = 4 * grp + (lane & 3);                  // (lane 0: 0, 1: 1, 2: 2, 3: 3)
                        if (lane < 4 && j < K) {
                            float* dst = part + w * K + j;
                            *dst = q_lo ? *dst + z : z;
                        }
                    };
                    fetch(wt, hv[0]);
                    for (int w = wt; w < W; w += 2 * team) {
                        fetch(w + team, hv[1]);
                        products(w, hv[0]);
                        if (w + team >= W) break;
                        fetch(w + 2 * team, hv[0]);
                        products(w + team, hv[1]);
                    }
                }
            }
            if (rk < n_rk && warp < K) {
                float n2 = 0.f;
                for (int c = 4 * lane; c < cols; c += 128) {
                    const float4 v = *reinterpret_cast<const float4*>(Cs + (size_t)warp * dper + c);
                    n2 = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, n2))));
                }
                n2 = warp_sum(n2);
                if (lane < KM_CL) km_push(&c2[rk][warp], n2, lane);
            }
            __syncthreads();
            if (rk < n_rk) for (int e = t; e < W * K; e += KM_THREADS) {
                const int w = e / K, o = w / per;
                km_push(recv + ((size_t)rk * per + (w - o * per)) * K + (e - w * K), part[e], o);
            }
            km_cluster_sync();
            // ---- labels of this CTA's rows, to every CTA
            if (t < K) {
                float n2 = 0.f;
#pragma unroll
                for (int r = 0; r < KM_CL; ++r) n2 += r < n_rk ? c2[r][t] : 0.f;
                inv_c[t] = n2 > 0.f ? rsqrtf(n2) : 0.f;
            }
            __syncthreads();
            // a half warp per row, a lane per centre
            for (int w0 = w_lo; w0 < w_hi; w0 += KM_THREADS / 16) {
                const int w = w0 + (t >> 4), j = t & 15;
                float cs = -INFINITY;
                if (w < w_hi && j < K) {
                    float dot = 0.f;
#pragma unroll
                    for (int r = 0; r < KM_CL; ++r) dot += r < n_rk ? recv[((size_t)r * per + (w - w_lo)) * K + j] : 0.f;
                    cs = dot * inv_c[j] * invn[w];
                }
                float best = cs;
#pragma unroll
                for (int o = 1; o < 16; o <<= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
                // the centre with the largest cosine (the lowest cluster for a row of NaN), or (upper half) all those that may have it
                const unsigned near = (__ballot_sync(0xffffffffu, j < K && cs >= best - KM_NEAR) >> (t & 16)) & 0xffffu;
                const int bj = max(__ffs(near) - 1, 0);
                if (w < w_hi) {
                    if (j == 0) labels[w] = bj;
                    if (j < KM_CL) km_push(lab + w, __popc(near) > 1 ? (int)(near << 16) : bj, j);
                }
            }
            km_cluster_sync();
            // ---- rows with several such centres (the same ones in every CTA): their products in 64 bits
            const bool any_near = __syncthreads_or(t < W && (lab[min(t, W - 1)] & 0xffff0000) != 0) != 0;
            if (any_near) {
                if (rk < n_rk) {
                    for (int w = warp; w < W; w += nw) {
                        const int o = w / per;
                        for (unsigned m = (unsigned)lab[w] >> 16; m; m &= m - 1) {
                            const int j = __ffs(m) - 1;
                            const double dot = km_dot(row(w) + c_lo, Cs + (size_t)j * dper, cols, lane);
                            if (lane == 0) km_push(recv_64 + ((size_t)rk * per + (w - o * per)) * K + j, dot, o);
                        }
                    }
                    if (warp < K) {
                        const double n2 = km_dot(Cs + (size_t)warp * dper, Cs + (size_t)warp * dper, cols, lane);
                        if (lane < KM_CL) km_push(&c2_64[rk][warp], n2, lane);
                    }
                }
                km_cluster_sync();
                for (int w0 = w_lo; w0 < w_hi; w0 += KM_THREADS / 16) {
                    const int w = w0 + (t >> 4), j = t & 15;
                    const unsigned near = w < w_hi ? (unsigned)lab[w] >> 16 : 0u;
                    double cs = -INFINITY;
                    if ((near >> j) & 1) {
                        double dot = 0., n2 = 0.;
                        for (int r = 0; r < n_rk; ++r) { dot += recv_64[((size_t)r * per + (w - w_lo)) * K + j]; n2 += c2_64[r][j]; }
                        cs = n2 > 0. ? dot / sqrt(n2) * invn[w] : 0.;
                    }
                    double best = cs;
#pragma unroll
                    for (int o = 1; o < 16; o <<= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
                    // (lowest cluster on ties)
                    const unsigned tie = (__ballot_sync(0xffffffffu, ((near >> j) & 1) && cs >= best - KM_TIE) >> (t & 16)) & 0xffffu;
                    const int bj = max(__ffs(tie) - 1, 0);
                    if (near) {
                        if (j == 0) labels[w] = bj;
                        if (j < KM_CL) km_push(lab + w, bj, j);
                    }
                }
                km_cluster_sync();
            }
            if (it + 1 == a.iters) break;          // the centres of the last update are never used
            // ---- update of this CTA's columns: members added in ascending row order; an empty cluster keeps its centre
            group_rows();
            for (int c = c_lo + t; c < c_hi; c += KM_THREADS)
                member_sums(c, [&](float acc, float v, int i) { return acc + v * ord_inv[i]; }, [&](int j, float sum) { Cs[(size_t)j * dper + c - c_lo] = sum; });
        }
    }
    km_cluster_sync();
    // ---- tables: member counts, groups of members, rotary position of every proxy (first CTA); labels of the unused rows
    for (int w = t; w < W; w += KM_THREADS) lab[w] = __ldcg(labels + w);
    group_rows();
    if (rk == 0) {
        for (int w = W + t; w < sd.W_max; w += KM_THREADS) labels[w] = -1;
        if (t < K) {
            const int n = cnt[t];
            long long sp = 0;
            for (int i = off[t]; i < off[t + 1]; ++i) sp += window_pos(sd, ord[i]);
            a.zcnt[s * K + t] = n;
            a.zpos[s * K + t] = n > 0 ? (int)((2 * sp + n) / (2 * n)) : -1;       // floor(mean + 1/2)
        }
        if (t <= K) a.moff[s * (K + 1) + t] = off[t];
        for (int i = t; i < W; i += KM_THREADS) a.members[(size_t)s * sd.W_max + i] = ord[i];
    }
    if (a.z0) {
        // reference rows of the residual codec: the clusters' centroids as this block entry sees them (this CTA's columns)
        for (int c = c_lo + t; c < c_hi; c += KM_THREADS) {
            for (int j = 0; j < K; ++j) if (cnt[j] == 0) a.z0[((size_t)s * K + j) * d + c] = 0.f;
            member_sums(c, [&](float acc, float v, int) { return acc + v; },
                        [&](int j, float sum) { a.z0[((size_t)s * K + j) * d + c] = sum * (1.f / (float)cnt[j]); });
        }
    }
}

// The codec on its own: codes, scales and stored values of rows x against reference rows ref (one CTA per row).
__global__ void nvfp4_residual_kernel(const float* x, const float* ref, int d, unsigned char* codes, unsigned char* scales, float* deq) {
    KERNEL_PROLOGUE(19);   // nvfp4_residual_kernel
    const size_t r = blockIdx.x;
    const int n4 = d >> 2;
    for (int c0 = 0; c0 < n4; c0 += blockDim.x) {
        const int c4 = c0 + threadIdx.x;
        const bool in = c4 < n4;
        const float4 v = in ? reinterpret_cast<const float4*>(x + r * d)[c4] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 rf = in ? reinterpret_cast<const float4*>(ref + r * d)[c4] : make_float4(0.f, 0.f, 0.f, 0.f);
        unsigned cd, sb;
        const float4 q = nvfp4_residual_chunk(v, rf, &cd, &sb);
        if (in) {
            *reinterpret_cast<unsigned short*>(codes + r * (size_t)(d >> 1) + 2 * c4) = (unsigned short)cd;
            if ((c4 & 3) == 0) scales[r * (size_t)(d >> 4) + (c4 >> 2)] = (unsigned char)sb;
            reinterpret_cast<float4*>(deq + r * d)[c4] = q;
        }
    }
}

// ---------------------------------------------------------------------------------------
// Plain tiled GEMM on CUDA cores: out[m][n] = sum_k A[m][k] W[n][k], fp32 accumulate.
// 64x64 tile, 16-wide K slices, 256 threads, 4x4 outputs per thread.
// ---------------------------------------------------------------------------------------
template <typename T, int EPI>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const T* __restrict__ A, const T* __restrict__ Wt,
                                                        int M, int Nout, int K, int w_tiled, EpiArgs e) {
    KERNEL_PROLOGUE(7);   // __launch_bounds__
    __shared__ float As[16][64 + 4];
    __shared__ float Ws[16][64 + 4];
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    const int Mv = e.m_count ? min(M, *e.m_count) : M;
    if (m0 >= Mv) return;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int k0 = 0; k0 < K; k0 += 16) {
        for (int t = threadIdx.x; t < 64 * 16; t += 256) {
            const int rr = t >> 4, kk = t & 15;
            const int m = m0 + rr, n = n0 + rr, k = k0 + kk;
            As[kk][rr] = (m < M && k < K) ? to_f<T>(A[(size_t)m * K + k]) : 0.f;
            // tile-major weights: block (n / 256, k / 64) is a contiguous [256][64] chunk
            const size_t wi = w_tiled ? ((size_t)((n >> 8) * (K >> 6) + (k >> 6)) << 14) + ((n & 255) << 6) + (k & 63)
                                      : (size_t)n * K + k;
            Ws[kk][rr] = (n < Nout && k < K) ? to_f<T>(Wt[wi]) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Ws[kk][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
        if (m >= Mv) continue;
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
            const int n = n0 + tx * 4 + j;
            if (n + 1 < Nout) epilogue_pair<T, EPI>(e, m, n, acc[i][j], acc[i][j + 1]);
        }
    }
}

// ---------------------------------------------------------------------------------------
// The same product for fp32 models: 16 x 32 outputs per CTA, the K dimension split over the CTA's eight warps.
// These models are small (tens of rows, K of a few hundred), so a launch is a latency chain, not a throughput problem:
// 64 x 64 tiles leave most SMs idle and every 16-wide K slice is a round trip to L2.  Here the operands of three
// 64-wide K slices are in flight at once (cp.async ring; the weights' share of it before the dependency wait), each
// warp multiplies eight k of a slice, and the eight partial tiles are added in warp order through shared memory.
// Where the output tiles leave most SMs idle and K is long, the slices are split over a cluster of up to eight CTAs (gridDim.z), which
// push their tiles into the first one's shared memory; it adds them in rank order.
// Rows / columns beyond the matrix and k beyond K arrive as zeros.  Needs K % 4 == 0 and 16-byte aligned operands.
// Measured against 64 x 64 tiles (rows x columns x K): 32 x 768 x 256 5.6 / 29 us, 32 x 256 x 1024 11 / 109 us,
// 128 x 2048 x 256 11 / 31 us, 512 x 2048 x 256 29 / 37 us, 4096 x 4096 x 1024 1160 / 1522 us: faster at every size, so the
// 64 x 64 tiles above are left with bf16 operands and unaligned ones.
// ---------------------------------------------------------------------------------------
constexpr int LAT_TM = 16, LAT_TN = 32, LAT_KC = 64, LAT_STAGES = 4, LAT_LD = LAT_KC + 4;
constexpr int LAT_SMEM = LAT_STAGES * (LAT_TM + LAT_TN) * LAT_LD * 4;
__device__ __forceinline__ void cp_async16_zfill(float* dst, const float* src, bool ok) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    const int n = ok ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
template <int EPI>
__global__ void __launch_bounds__(256) gemm_f32_kernel(const float* __restrict__ A, const float* __restrict__ Wt,
                                                       int M, int Nout, int K, EpiArgs e) {
    constexpr int STAGE = (LAT_TM + LAT_TN) * LAT_LD;
    static_assert(8 * LAT_TM * LAT_TN <= LAT_STAGES * STAGE, "the partial tiles reuse the operand ring");
    extern __shared__ __align__(16) float lat_sm[];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int m0 = blockIdx.y * LAT_TM, n0 = blockIdx.x * LAT_TN;
    // this CTA's slices of K
    const int slices_all = (K + LAT_KC - 1) / LAT_KC, cl = gridDim.z, rank = blockIdx.z;
    const int s_begin = slices_all * rank / cl, slices = slices_all * (rank + 1) / cl - s_begin;
    // thread t copies 16 bytes of A (row t / 16, k chunk t % 16) and twice 16 bytes of W (rows t / 16 and t / 16 + 16)
    const int cr = t >> 4, ck = (t & 15) * 4;
    auto load_w = [&](int s) {
        const int k = (s_begin + s) * LAT_KC + ck;
        float* st = lat_sm + (s % LAT_STAGES) * STAGE + LAT_TM * LAT_LD;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int n = n0 + cr + 16 * i;
            const bool ok = n < Nout && k < K;
            cp_async16_zfill(st + (cr + 16 * i) * LAT_LD + ck, ok ? Wt + (size_t)n * K + k : Wt, ok);
        }
    };
    auto load_a = [&](int s) {
        const int k = (s_begin + s) * LAT_KC + ck;
        const bool ok = m0 + cr < M && k < K;
        cp_async16_zfill(lat_sm + (s % LAT_STAGES) * STAGE + cr * LAT_LD + ck, ok ? A + (size_t)(m0 + cr) * K + k : A, ok);
    };
    pdl_trigger();
    for (int s = 0; s < min(LAT_STAGES - 1, slices); ++s) load_w(s);       // no kernel of a forward writes weights
    pdl_wait();
    trace_stamp(7);
    const int Mv = e.m_count ? min(M, *e.m_count) : M;
    if (m0 >= Mv) {                             // (the whole cluster)
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
    }
    for (int s = 0; s < LAT_STAGES - 1; ++s) {
        if (s < slices) load_a(s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const int mi = lane >> 3, ni = lane & 7;    // outputs: rows mi + 4 i, columns ni + 8 j
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int s = 0; s < slices; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(LAT_STAGES - 2) : "memory");
        __syncthreads();                        // slice s has landed for every thread; the slot of slice s - 1 is free
        if (s + LAT_STAGES - 1 < slices) { load_w(s + LAT_STAGES - 1); load_a(s + LAT_STAGES - 1); }
        asm volatile("cp.async.commit_group;" ::: "memory");
        const float* as = lat_sm + (s % LAT_STAGES) * STAGE + warp * 8;
        const float* ws = as + LAT_TM * LAT_LD;
#pragma unroll
        for (int kk = 0; kk < 8; kk += 4) {
            float4 a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(as + (mi + 4 * i) * LAT_LD + kk);
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(ws + (ni + 8 * j) * LAT_LD + kk);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
                    acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
                    acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
                    acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
                }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (cl > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");     // this CTA's ring is free
    float* red = lat_sm + warp * (LAT_TM * LAT_TN);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) red[(mi + 4 * i) * LAT_TN + ni + 8 * j] = acc[i][j];
    __syncthreads();
    const int m = m0 + (t >> 4), n = n0 + (t & 15) * 2;
    float2 sum = make_float2(0.f, 0.f);
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const float2 v = *reinterpret_cast<const float2*>(lat_sm + w * (LAT_TM * LAT_TN) + t * 2);
        sum.x += v.x; sum.y += v.y;
    }
    if (cl > 1) {
        // the other CTAs' tiles, behind the partial tiles in the first CTA's ring
        static_assert((8 + 7) * LAT_TM * LAT_TN <= LAT_STAGES * STAGE, "and so do the cluster's tiles");
        float2* const peer = reinterpret_cast<float2*>(lat_sm + 8 * LAT_TM * LAT_TN) + t;
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (rank > 0) {
            const uint32_t dst = dsmem_addr((uint32_t)__cvta_generic_to_shared(peer + (rank - 1) * 256), 0);
            asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(sum.x), "f"(sum.y) : "memory");
        }
        cluster_sync_all();
        if (rank > 0) return;
        for (int c = 1; c < cl; ++c) { const float2 v = peer[(c - 1) * 256]; sum.x += v.x; sum.y += v.y; }
    }
    if (m < Mv && n + 1 < Nout) epilogue_pair<float, EPI>(e, m, n, sum.x, sum.y);
}

// ---------------------------------------------------------------------------------------
// Attention rows with drift, CUDA-core version: one warp per (row, head).
//   logp_j = s_j - logsumexp(s), s_j = q.k_j / sqrt(dh) over all N cache rows (Eq. 3, no mask);
//   out = sum_j p_j v_j;  recorded rows: kl = sum_j p_j (logp_j - prev_j), prev <- logp (Eq. 4).
// Dynamic shared memory: warps_per_block * N floats.
// ---------------------------------------------------------------------------------------
struct AttnArgs {
    const Row* rows; int n_rows;
    const void* q; const void* kc; const void* vc; void* out;
    // Stored attention rows: a row and one float per row such that log-probability = row - lse.  The tensor-core
    // kernel keeps scaled scores and their log-sum-exp; the other kernels keep log-probabilities and leave lse at 0.
    float* pprev;    // window rows: [batch][W_max][n_heads][N]   (null: none recorded)
    float* aprev;    // active rows: [batch][B][n_heads][N]       (null: none recorded)
    float* pprev_lse;   // [batch][W_max][n_heads]
    float* aprev_lse;   // [batch][B][n_heads]
    float* kl;       // [n_rows][n_heads]
    int N, n_heads, n_kv, head_dim, W_max, B, record_kl;
    int rows_per_seq, batch;   // layout of the forward's rows (stand-alone: n_rows, 1)
    float scale;
    int p_pow2;                // round exp(score) to bf16 times a power of two (any: it does not matter to the rounding) instead of the normalised
                               // probability, and normalise in fp32 behind P V: what a kernel that sees every key once can do
    int cluster_K;             // > 0: centroid proxies: pprev / pprev_lse hold [batch][cluster_K] proxy rows per head and
                               // window rows are not recorded
    int rec_lo, rec_hi;        // rows [lo, hi) of every sequence hold all the recorded ones (hi 0: any row may be recorded)
    int dirty_lo, dirty_hi;    // key positions [lo, hi) of every sequence that the kernel running just before may have
                               // written; all other K/V rows were complete before this forward was launched
    // stand-alone form: rows == null, row r belongs to sequence 0 and records into pprev[r]
};
// Whether every stored row can be read and written in pieces of `floats` (a power of two) floats.
static inline bool stored_rows_in_pieces(const AttnArgs& a, int floats) {
    return a.N % floats == 0 && (((uintptr_t)a.pprev | (uintptr_t)a.aprev) & (uintptr_t)(4 * floats - 1)) == 0;
}

// One CTA of four warps per (row, head): a chain of dependent loads at the sizes of these models, so the keys are split over the
// warps and everything a thread needs of K (16-byte pieces of its keys, sixteen in flight) and V (its columns of 32 keys) is
// requested at once.  Parts are put together in warp order.  fp32, 4 heads of 64, 128 keys, in the pipeline, us,
// against a warp per (row, head): 32 rows 14.4 -> 7.5, 128 rows with stored rows 19.6 - 33 -> 12.
constexpr int SIMT_WARPS = 4;
__host__ __device__ constexpr size_t simt_attn_smem(int N, int dh) { return ((size_t)N + SIMT_WARPS * dh + 2 * SIMT_WARPS) * sizeof(float); }
template <typename T>
__global__ void __launch_bounds__(SIMT_WARPS * 32) attention_simt_kernel(AttnArgs a) {
    KERNEL_PROLOGUE(8);   // attention_simt_kernel
    extern __shared__ float sm[];
    const int t = threadIdx.x, wid = t >> 5, lane = t & 31;
    const int r = blockIdx.x, h = blockIdx.y;
    int seq = 0;
    float* prev = nullptr;
    if (a.rows) {
        const Row rw = a.rows[r];
        if (rw.pos < 0) return;
        seq = rw.seq;
        if (a.cluster_K > 0) {
            if (row_is_proxy(rw.widx) && a.pprev) prev = a.pprev + (((size_t)seq * a.cluster_K + row_cluster(rw.widx)) * a.n_heads + h) * a.N;
            else if (rw.aidx >= 0 && a.aprev) prev = a.aprev + (((size_t)seq * a.B + rw.aidx) * a.n_heads + h) * a.N;
        }
        else if (rw.widx >= 0 && a.pprev) prev = a.pprev + (((size_t)seq * a.W_max + rw.widx) * a.n_heads + h) * a.N;
        else if (rw.aidx >= 0 && a.aprev) prev = a.aprev + (((size_t)seq * a.B + rw.aidx) * a.n_heads + h) * a.N;
    } else if (a.pprev) {
        prev = a.pprev + ((size_t)r * a.n_heads + h) * a.N;
    }
    const int dh = a.head_dim, g = (h * a.n_kv) / a.n_heads;
    float* const sc = sm;                              // scores, then probabilities
    float* const part = sm + a.N;                      // [warp][dh] partial output rows
    float* const red = part + SIMT_WARPS * dh;         // [2][warp]
    const int dq = a.n_heads * dh, dkv = a.n_kv * dh;
    const T* q = (const T*)a.q + (size_t)r * dq + h * dh;
    const T* K = (const T*)a.kc + (size_t)seq * a.N * dkv + g * dh;
    const T* V = (const T*)a.vc + (size_t)seq * a.N * dkv + g * dh;
    // one value of every warp, combined in warp order
    auto combine = [&](float v, int slot, auto op) {
        if (lane == 0) red[slot * SIMT_WARPS + wid] = v;
        __syncthreads();
        float x = red[slot * SIMT_WARPS];
#pragma unroll
        for (int w = 1; w < SIMT_WARPS; ++w) x = op(x, red[slot * SIMT_WARPS + w]);
        return x;
    };
    // scores
    float mx = -INFINITY;
    const bool vec = sizeof(T) == 4 && (dh & 31) == 0 && (dq & 3) == 0 && (dkv & 3) == 0 && (((uintptr_t)a.q | (uintptr_t)a.kc) & 15) == 0;
    for (int j = t; j < a.N; j += SIMT_WARPS * 32) {
        const T* kj = K + (size_t)j * dkv;
        float s = 0.f;
        if (vec) {
            const float4* k4 = reinterpret_cast<const float4*>(kj);
            const float4* q4 = reinterpret_cast<const float4*>(q);
            for (int c = 0; c < (dh >> 2); c += 16) {
                float4 kv[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) if (c + i < (dh >> 2)) kv[i] = k4[c + i];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    if (c + i >= (dh >> 2)) break;
                    const float4 qv = q4[c + i];
                    s = fmaf(qv.x, kv[i].x, s); s = fmaf(qv.y, kv[i].y, s);
                    s = fmaf(qv.z, kv[i].z, s); s = fmaf(qv.w, kv[i].w, s);
                }
            }
        } else {
            for (int c = 0; c < dh; ++c) s = fmaf(to_f<T>(q[c]), to_f<T>(kj[c]), s);
        }
        s *= a.scale;
        sc[j] = s;
        mx = fmaxf(mx, s);
    }
    mx = combine(warp_max(mx), 0, [](float x, float y) { return fmaxf(x, y); });
    float sum = 0.f;
    for (int j = t; j < a.N; j += SIMT_WARPS * 32) sum += expf(sc[j] - mx);
    sum = combine(warp_sum(sum), 1, [](float x, float y) { return x + y; });
    const float lse = mx + logf(sum);
    float kl = 0.f;
    for (int j = t; j < a.N; j += SIMT_WARPS * 32) {
        const float lp = sc[j] - lse;
        const float p = expf(lp);
        if (prev) {
            if (a.record_kl) kl += p * (lp - prev[j]);
            prev[j] = lp;
        }
        sc[j] = round_to<T>(p);
    }
    kl = combine(warp_sum(kl), 0, [](float x, float y) { return x + y; });        // (also: the probabilities are complete)
    if (a.kl && t == 0) a.kl[(size_t)r * a.n_heads + h] = (prev && a.record_kl) ? kl : 0.f;
    if (a.out) {
        // a warp takes every fourth group of 32 keys, a lane one column or two adjacent ones
        const bool two = sizeof(T) == 4 && (dh & 63) == 0 && (dkv & 1) == 0 && (((uintptr_t)a.vc) & 7) == 0;
        for (int c = two ? 2 * lane : lane; c < dh; c += two ? 64 : 32) {
            float a0 = 0.f, a1 = 0.f;
            for (int j0 = 32 * wid; j0 < a.N; j0 += 32 * SIMT_WARPS) {
                const T* vj = V + (size_t)j0 * dkv + c;
                if (j0 + 32 <= a.N) {
                    if (two) {
                        float2 v[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = *reinterpret_cast<const float2*>(vj + (size_t)i * dkv);
#pragma unroll
                        for (int i = 0; i < 32; ++i) { const float p = sc[j0 + i]; a0 = fmaf(p, v[i].x, a0); a1 = fmaf(p, v[i].y, a1); }
                    } else {
                        T v[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = vj[(size_t)i * dkv];
#pragma unroll
                        for (int i = 0; i < 32; ++i) a0 = fmaf(sc[j0 + i], to_f<T>(v[i]), a0);
                    }
                } else {
                    for (int i = 0; j0 + i < a.N; ++i) {
                        const float p = sc[j0 + i];
                        a0 = fmaf(p, to_f<T>(vj[(size_t)i * dkv]), a0);
                        if (two) a1 = fmaf(p, to_f<T>(vj[(size_t)i * dkv + 1]), a1);
                    }
                }
            }
            part[wid * dh + c] = a0;
            if (two) part[wid * dh + c + 1] = a1;
        }
        __syncthreads();
        T* o = (T*)a.out + (size_t)r * dq + h * dh;
        for (int c = t; c < dh; c += SIMT_WARPS * 32) {
            float x = part[c];
#pragma unroll
            for (int w = 1; w < SIMT_WARPS; ++w) x += part[w * dh + c];
            o[c] = from_f<T>(x);
        }
    }
}

// ---------------------------------------------------------------------------------------
// Squared hidden-state change per row (Appendix B, Cor. 1): one warp per row, 128-bit loads.
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void hidden_delta_kernel(const T* __restrict__ a, const T* __restrict__ b, float* out, int rows, int d) {
    KERNEL_PROLOGUE(9);   // hidden_delta_kernel
    const int wpb = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int per = 16 / (int)sizeof(T);
    for (int r = blockIdx.x * wpb + wid; r < rows; r += gridDim.x * wpb) {
        const uint4* pa = reinterpret_cast<const uint4*>(a + (size_t)r * d);
        const uint4* pb = reinterpret_cast<const uint4*>(b + (size_t)r * d);
        float acc = 0.f;
        const int nv = d / per;
        for (int i = lane; i < nv; i += 32) {
            const uint4 ua = __ldg(pa + i), ub = __ldg(pb + i);
            const T* ea = reinterpret_cast<const T*>(&ua);
            const T* eb = reinterpret_cast<const T*>(&ub);
#pragma unroll
            for (int t = 0; t < per; ++t) { const float dd = to_f<T>(ea[t]) - to_f<T>(eb[t]); acc = fmaf(dd, dd, acc); }
        }
        for (int c = nv * per + lane; c < d; c += 32) {
            const float dd = to_f<T>(a[(size_t)r * d + c]) - to_f<T>(b[(size_t)r * d + c]);
            acc = fmaf(dd, dd, acc);
        }
        acc = warp_sum(acc);
        if (lane == 0) out[r] = acc;
    }
}

// ---------------------------------------------------------------------------------------
// Stale-row selection + compaction for one sequence (Sec. 4.1; Algorithm 1 "TopK").
// Block-wide radix select of the k-th largest drift, ties to the lower index, then a
// prefix-sum compaction to an ascending index list.  W <= SEL_MAX_W.
// ---------------------------------------------------------------------------------------
constexpr int SEL_THREADS = 1024;
constexpr int SEL_ITEMS = 4;
constexpr int SEL_MAX_W = SEL_THREADS * SEL_ITEMS;

struct SelSmem {
    int hist[2][256];
    int scan[33];
    unsigned prefix; int kleft; int ncand;
};

__device__ __forceinline__ unsigned float_key(float v) {   // order-preserving map to unsigned
    const unsigned u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// D[i] valid for i < W.  Writes idx_out[0..count) ascending and (optional) flag_out[i] in {0,1}.
// Returns count (same value in every thread).  Must be called by all SEL_THREADS threads.
// A chain of barriers: two per radix pass (the other pass's histogram is cleared meanwhile), the candidate count under the first
// pass's.  Only the leading byte, which drift values share, is counted with one addition per distinct bucket of a warp.  us, against
// four barriers a pass and scans: 4096 values, one sequence 6.8 -> 5.8, eight 8.8 -> 6.0.
__device__ int select_one(const float* D, int W, int mode, int k, float thresh, float floor_,
                          int* idx_out, unsigned char* flag_out, SelSmem& s) {
    const int t = threadIdx.x;
    unsigned key[SEL_ITEMS];
    float val[SEL_ITEMS];
    bool cand[SEL_ITEMS], sel[SEL_ITEMS];
    // items are blocked: thread t owns indices t*ITEMS .. t*ITEMS+ITEMS-1 (keeps index order in scans)
    if (t < 256) s.hist[0][t] = 0;
    if (t == 0) { s.ncand = 0; s.prefix = 0u; s.kleft = k; }
    if (t * SEL_ITEMS + SEL_ITEMS <= W && ((uintptr_t)D & 15) == 0) {
        const float4 v = *reinterpret_cast<const float4*>(D + t * SEL_ITEMS);
        val[0] = v.x; val[1] = v.y; val[2] = v.z; val[3] = v.w;
    } else {
#pragma unroll
        for (int u = 0; u < SEL_ITEMS; ++u) val[u] = t * SEL_ITEMS + u < W ? D[t * SEL_ITEMS + u] : 0.f;
    }
    int ncand_local = 0;
#pragma unroll
    for (int u = 0; u < SEL_ITEMS; ++u) {
        cand[u] = (t * SEL_ITEMS + u < W) && (val[u] > floor_);          // NaN compares false: never a candidate
        key[u] = float_key(val[u]);
        sel[u] = false;
        ncand_local += cand[u];
    }
    ncand_local = __reduce_add_sync(0xffffffffu, ncand_local);
    __syncthreads();
    if ((t & 31) == 0 && ncand_local) atomicAdd(&s.ncand, ncand_local);
    if (mode < 2) {
#pragma unroll
        for (int u = 0; u < SEL_ITEMS; ++u) {
            const unsigned bkt = cand[u] ? key[u] >> 24 : 256u;
            const unsigned same = __match_any_sync(0xffffffffu, bkt);
            if (cand[u] && (t & 31) == __ffs(same) - 1) atomicAdd(&s.hist[0][bkt], __popc(same));
        }
    }
    __syncthreads();
    const int ncand = s.ncand;
    if (mode == 3) {                                  // ALL: every row
#pragma unroll
        for (int u = 0; u < SEL_ITEMS; ++u) sel[u] = (t * SEL_ITEMS + u) < W;
    } else if (mode == 2) {                           // THRESHOLD
#pragma unroll
        for (int u = 0; u < SEL_ITEMS; ++u) sel[u] = cand[u] && (val[u] > thresh);
    } else if (mode == 4 || k <= 0) {                 // NONE
    } else if (k >= ncand) {
#pragma unroll
        for (int u = 0; u < SEL_ITEMS; ++u) sel[u] = cand[u];
    } else {
        // radix select, most significant byte first
        for (int pass = 0; pass < 4; ++pass) {
            const int shift = 24 - 8 * pass;
            int* const hist = s.hist[pass & 1];
            const unsigned prefix = s.prefix;
            if (pass > 0) {
                const unsigned himask = 0xFFFFFFFFu << (shift + 8);
#pragma unroll
                for (int u = 0; u < SEL_ITEMS; ++u)
                    if (cand[u] && (key[u] & himask) == prefix) atomicAdd(&hist[(key[u] >> shift) & 255u], 1);
                __syncthreads();
            }
            if (t < 32) {
                // the bucket that holds the k-th candidate, from the top: lane t owns buckets 255 - 8 t ... 248 - 8 t
                int c[8], sum = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) { c[j] = hist[255 - 8 * t - j]; sum += c[j]; }
                int inc = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int up = __shfl_up_sync(0xffffffffu, inc, o);
                    if (t >= o) inc += up;
                }
                int left = s.kleft;
                __syncwarp();
                if (inc - sum < left && inc >= left) {        // (one lane: the counts add up to at least k)
                    left -= inc - sum;
                    int j = 0;
#pragma unroll
                    for (int i = 0; i < 7; ++i) if (j == i && c[i] < left) { left -= c[i]; ++j; }
                    s.kleft = left;
                    s.prefix = prefix | ((unsigned)(255 - 8 * t - j) << shift);
                }
            } else if (t < 288) {
                s.hist[(pass & 1) ^ 1][t - 32] = 0;
            }
            __syncthreads();
        }
        const unsigned kth = s.prefix;     // key of the k-th largest candidate
        const int need_eq = s.kleft;       // how many rows equal to it are taken (lowest indices)
        int eq_local = 0;
#pragma unroll
        for (int u = 0; u < SEL_ITEMS; ++u) eq_local += (cand[u] && key[u] == kth);
        int eq_total;
        int eq_before = block_excl_scan(eq_local, s.scan, &eq_total);
#pragma unroll
        for (int u = 0; u < SEL_ITEMS; ++u) {
            if (!cand[u]) continue;
            if (key[u] > kth) sel[u] = true;
            else if (key[u] == kth) { sel[u] = eq_before < need_eq; ++eq_before; }
        }
    }
    int nsel_local = 0;
#pragma unroll
    for (int u = 0; u < SEL_ITEMS; ++u) nsel_local += sel[u];
    int count;
    int off = block_excl_scan(nsel_local, s.scan, &count);
#pragma unroll
    for (int u = 0; u < SEL_ITEMS; ++u) {
        const int i = t * SEL_ITEMS + u;
        if (i < W && flag_out) flag_out[i] = sel[u] ? 1 : 0;
        if (sel[u]) idx_out[off++] = i;
    }
    __syncthreads();
    return count;
}

// Small windows (W <= SEL_SMALL_W, the in-step case: W = 3B): rank counting, two barriers.
// Thread i owns row i; rank = number of candidates ahead of it in (drift descending, index ascending) order.
constexpr int SEL_SMALL_W = 256;
// `i` = index of the calling thread among the participating threads (at least W of them); bar < 0: they are the
// whole block (__syncthreads), else they synchronise on named barrier `bar` with `nthr` threads.
__device__ __forceinline__ void sel_sync(int bar, int nthr) {
    if (bar < 0) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(nthr) : "memory");
}
// Place of a chosen index among the chosen ones (ascending) and their number, by the warps' ballots.  All participating threads
// (whole warps, chosen indices below SEL_SMALL_W) call; wcnt: eight ints of shared memory.
__device__ __forceinline__ int chosen_place(bool sel, int i, int* total, int* wcnt, int bar, int nthr) {
    const unsigned b = __ballot_sync(0xffffffffu, sel);
    const int w = i >> 5, lane = i & 31;
    if (w < SEL_SMALL_W / 32 && lane == 0) wcnt[w] = __popc(b);
    sel_sync(bar, nthr);
    int pos = __popc(b & ((1u << lane) - 1u)), sum = 0;
#pragma unroll
    for (int q = 0; q < SEL_SMALL_W / 32; ++q) {
        const int c = wcnt[q];
        pos += q < w ? c : 0;
        sum += c;
    }
    *total = sum;
    return pos;
}
// Rank counting from shared memory, four values a load, and ballots for the compaction; us, against loops over single values and
// flags: 96 values 6.8 -> 2.3, eight times 192 12.4 -> 3.6.  At least SEL_SMALL_W threads.  D: shared memory, 16-byte aligned, with room for W rounded up to four
__device__ int select_small(float* D, int W, int mode, int k, float thresh, float floor_,
                            int* idx_out, unsigned char* flag_out, int* wcnt /* [8] */, int i, int bar, int nthr) {
    const float v = i < W ? D[i] : 0.f;
    const bool cand = i < W && v > floor_;
    bool sel = false;
    if (mode == 3) sel = i < W;
    else if (mode == 2) sel = cand && v > thresh;
    else if (mode != 4 && k > 0) {
        if (i >= W && i < ((W + 3) & ~3)) D[i] = -INFINITY;
        sel_sync(bar, nthr);
        if (cand) {
            // (whatever is as large as a candidate is one)
            int rank = 0;
            for (int j = 0; j < W; j += 4) {
                const float4 d = *reinterpret_cast<const float4*>(D + j);
                rank += (d.x > v || (d.x == v && j < i)) + (d.y > v || (d.y == v && j + 1 < i)) + (d.z > v || (d.z == v && j + 2 < i)) +
                        (d.w > v || (d.w == v && j + 3 < i));
            }
            sel = rank < k;
        }
    }
    int total;
    const int pos = chosen_place(sel, i, &total, wcnt, bar, nthr);
    if (i < W) {
        if (flag_out) flag_out[i] = sel ? 1 : 0;
        if (sel) idx_out[pos] = i;
    }
    sel_sync(bar, nthr);
    return total;
}

__global__ void __launch_bounds__(SEL_THREADS) select_kernel(const float* drift, int W, int mode, int k,
                                                             float thresh, float floor_, int* idx, int* count) {
    KERNEL_PROLOGUE(7);   // __launch_bounds__
    __shared__ SelSmem s;
    const int b = blockIdx.x;
    __shared__ __align__(16) float dsh[SEL_SMALL_W];
    if (W <= SEL_SMALL_W) {
        if ((int)threadIdx.x < W) dsh[threadIdx.x] = drift[(size_t)b * W + threadIdx.x];
        __syncthreads();
    }
    const int c = W <= SEL_SMALL_W ? select_small(dsh, W, mode, k, thresh, floor_, idx + (size_t)b * W, nullptr, s.scan, threadIdx.x, -1, SEL_THREADS)
                                   : select_one(drift + (size_t)b * W, W, mode, k, thresh, floor_, idx + (size_t)b * W, nullptr, s);
    if (threadIdx.x == 0) count[b] = c;
}

// In-step selection for every refreshing sequence, plus the compacted row list of the sparse
// forward: all valid non-window rows followed by the selected window rows.
struct StepSelArgs {
    const float* kl;            // [rows][n_heads] per-head drift of the forward's rows
    float* drift;               // [batch][W_max] (output, this layer)
    int* sel_idx; int* sel_cnt; // this layer: [batch][W_max], [batch]
    unsigned char* flag_next;   // patch flags of the next layer [batch][W_max]
    const int* forced_idx; const int* forced_cnt;   // this layer (cnt < 0: not forced)
    int* list; int* list_count; // compacted rows of the sparse forward
    int* stats;                 // [0] += refreshed rows
    int n_heads, mode, k, W_max;
    float thresh, floor_;
    ClusterTabs ct;             // centroid proxies (ct.K > 0): drift per cluster, the top cluster_k clusters' members
    int cluster_k;
};

// The same work for a batch of one sequence with a window of at most SEL_SMALL_W rows, done by `nthr` >= W threads
// (t = 0 .. nthr-1) of a kernel that is busy otherwise: they synchronise on named barrier `bar` only.  Used by
// the O projection, whose idle warps select the stale rows while the weights stream.
__device__ __forceinline__ void step_select_inline(const StepDesc& sd, const StepSelArgs& a, int t, int nthr, int bar,
                                                   float* dsh /* [SEL_SMALL_W], 16-byte aligned */, int* wcnt /* [8] */) {
    int cnt = 0;
    int* idx = a.sel_idx;
    if (sd.refresh.v[0]) {
        for (int w0 = 0; w0 < sd.W; w0 += nthr / 8) {
            const int w = w0 + (t >> 3), part = t & 7;
            float acc = 0.f;
            if (w < sd.W) {
                const float* kr = a.kl + (size_t)(sd.B + w) * a.n_heads;
                for (int h = part; h < a.n_heads; h += 8) acc += __ldcg(kr + h);
            }
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            acc += __shfl_xor_sync(0xffffffffu, acc, 4);
            if (w < sd.W && part == 0) {
                const float dv = acc / (float)a.n_heads;
                dsh[w] = dv;
                a.drift[w] = dv;
            }
        }
        sel_sync(bar, nthr);
        unsigned char* fl = a.flag_next;
        const int fc = a.forced_cnt ? a.forced_cnt[0] : -1;
        if (fc >= 0) {
            for (int w = t; w < sd.W; w += nthr) fl[w] = 0;
            sel_sync(bar, nthr);
            for (int i = t; i < fc; i += nthr) { const int w = a.forced_idx[i]; idx[i] = w; fl[w] = 1; }
            cnt = fc;
            sel_sync(bar, nthr);
        } else {
            cnt = select_small(dsh, sd.W, a.mode, a.k, a.thresh, a.floor_, idx, fl, wcnt, t, bar, nthr);
        }
    }
    // compacted row list of the sparse forward: the active rows, then the selected window rows
    for (int i = t; i < sd.B; i += nthr) a.list[i] = i;
    for (int i = t; i < cnt; i += nthr) a.list[sd.B + i] = sd.B + idx[i];
    if (t == 0) {
        a.sel_cnt[0] = cnt;
        *a.list_count = sd.B + cnt;
        atomicAdd(a.stats, cnt);
    }
}

// One CTA per sequence; the CTA that finishes last (arrival counter a.stats[3], left at zero again) builds the
// compacted row list from all sequences' selections.
__global__ void __launch_bounds__(SEL_THREADS) step_select_kernel(StepDesc sd, StepSelArgs a) {
    KERNEL_PROLOGUE(7);   // __launch_bounds__
    __shared__ SelSmem s;
    __shared__ __align__(16) float dsh[SEL_MAX_W > 1024 ? 1024 : SEL_MAX_W];
    __shared__ int offs[65];
    __shared__ int last_sh;
    const int t = threadIdx.x;
    const int sq = blockIdx.x;
    int cnt = 0;
    if (sd.refresh.v[sq] && a.ct.K > 0) {
        // ---- centroid proxies (Sec. 4.1; Algorithm 1 "KL", "TopK", M[K]): drift of the K proxy rows, the
        // cluster_k clusters with the largest drift, then their member rows in ascending order
        __shared__ int ctmp[KM_MAX_K];
        __shared__ unsigned char csel[KM_MAX_K];
        const int K = a.ct.K;
        const int label = t < sd.W ? a.ct.labels[(size_t)sq * a.W_max + t] : 0;
        if (t < 8 * KM_MAX_K) {                              // eight lanes per proxy row, as for the window rows below
            const int c = t >> 3, part = t & 7;
            float acc = 0.f;
            if (c < K) {
                const float* kr = a.kl + (size_t)(sq * sd.rows_per_seq + sd.B + sd.W + c) * a.n_heads;
                for (int h = part; h < a.n_heads; h += 8) acc += __ldg(kr + h);
            }
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            acc += __shfl_xor_sync(0xffffffffu, acc, 4);
            if (c < K && part == 0) {
                const float dv = a.ct.zcnt[sq * K + c] > 0 ? acc / (float)a.n_heads : 0.f;       // an empty cluster never drifts
                dsh[c] = dv;
                a.drift[sq * a.W_max + c] = dv;
            }
        }
        __syncthreads();
        int* idx = a.sel_idx + sq * a.W_max;
        unsigned char* fl = a.flag_next + sq * a.W_max;
        const int fc = a.forced_cnt ? a.forced_cnt[sq] : -1;
        if (fc >= 0) {
            for (int w = t; w < sd.W; w += blockDim.x) fl[w] = 0;
            __syncthreads();
            for (int i = t; i < fc; i += blockDim.x) { const int w = a.forced_idx[sq * a.W_max + i]; idx[i] = w; fl[w] = 1; }
            cnt = fc;
        } else {
            select_small(dsh, K, 1 /* top-k count */, a.cluster_k, a.thresh, a.floor_, ctmp, csel, s.scan, t, -1, SEL_THREADS);
            const bool sel = t < sd.W && csel[label] != 0;
            int total;
            const int pos = chosen_place(sel, t, &total, s.scan, -1, SEL_THREADS);
            if (t < sd.W) { fl[t] = sel ? 1 : 0; if (sel) idx[pos] = t; }
            cnt = total;
        }
    } else if (sd.refresh.v[sq]) {
        // head mean of the per-head drift (Eq. 4): eight lanes per row, all loads of a row in flight at once;
        // the partial sums are combined in a fixed order
        for (int w0 = 0; w0 < sd.W; w0 += blockDim.x / 8) {
            const int w = w0 + (t >> 3), part = t & 7;
            float acc = 0.f;
            if (w < sd.W) {
                const float* kr = a.kl + (size_t)(sq * sd.rows_per_seq + sd.B + w) * a.n_heads;
                for (int h = part; h < a.n_heads; h += 8) acc += __ldg(kr + h);
            }
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            acc += __shfl_xor_sync(0xffffffffu, acc, 4);
            if (w < sd.W && part == 0) {
                const float dv = acc / (float)a.n_heads;
                dsh[w] = dv;
                a.drift[sq * a.W_max + w] = dv;
            }
        }
        __syncthreads();
        int* idx = a.sel_idx + sq * a.W_max;
        unsigned char* fl = a.flag_next + sq * a.W_max;
        const int fc = a.forced_cnt ? a.forced_cnt[sq] : -1;
        if (fc >= 0) {
            for (int w = t; w < sd.W; w += blockDim.x) fl[w] = 0;
            __syncthreads();
            for (int i = t; i < fc; i += blockDim.x) { const int w = a.forced_idx[sq * a.W_max + i]; idx[i] = w; fl[w] = 1; }
            cnt = fc;
        } else {
            cnt = sd.W <= SEL_SMALL_W ? select_small(dsh, sd.W, a.mode, a.k, a.thresh, a.floor_, idx, fl, s.scan, t, -1, SEL_THREADS)
                                      : select_one(dsh, sd.W, a.mode, a.k, a.thresh, a.floor_, idx, fl, s);
        }
    }
    __syncthreads();
    if (t == 0) {
        a.sel_cnt[sq] = cnt;
        int last = 1;
        if (sd.batch > 1) {
            __threadfence();
            last = atomicAdd(a.stats + 3, 1) == sd.batch - 1;
            __threadfence();
        }
        last_sh = last;
    }
    __syncthreads();
    if (!last_sh) return;
    // compacted row list of the sparse forward: all active rows (row id = s*rows_per_seq + j), then the selected
    // window rows sequence by sequence
    const int nb = sd.batch * sd.B;
    if (t == 0) {
        int base = nb;
        for (int q = 0; q < sd.batch; ++q) { offs[q] = base; base += __ldcg(a.sel_cnt + q); }
        offs[sd.batch] = base;
        *a.list_count = base;
        atomicAdd(a.stats, base - nb);
        a.stats[3] = 0;
    }
    for (int i = t; i < nb; i += blockDim.x) a.list[i] = (i / sd.B) * sd.rows_per_seq + (i % sd.B);
    __syncthreads();
    for (int q = 0; q < sd.batch; ++q) {
        const int b0 = offs[q], n = offs[q + 1] - b0;
        for (int i = t; i < n; i += blockDim.x) a.list[b0 + i] = q * sd.rows_per_seq + sd.B + __ldcg(a.sel_idx + q * a.W_max + i);
    }
}

// ---------------------------------------------------------------------------------------
// LM-head row list: every active row, then (refresh steps with suffix commit) the rows the last
// layer selected that lie in the suffix window and are still masked (Sec. 4.2 "Suffix Block Commit")
// ---------------------------------------------------------------------------------------
__global__ void build_head_list_kernel(StepDesc sd, const int* y, int mask_id, const int* sel_idx,
                                       const int* sel_cnt, int use_suffix, int act_row0_stride,
                                       HeadSrc* list, int* count, int* suf_seq, int* suf_w) {
    KERNEL_PROLOGUE(10);   // build_head_list_kernel
    // act_row0_stride: forward row of active j in sequence s = s*rows_per_seq + (act offset) + j
    const int t = threadIdx.x;
    const int nb = sd.batch * sd.B;
    const int act_off = sd.kind == 2 ? 0 : (sd.act_start - sd.e0);
    for (int i = t; i < nb; i += blockDim.x) {
        HeadSrc h; h.kind = 0; h.index = (i / sd.B) * sd.rows_per_seq + act_off + (i % sd.B);
        list[i] = h;
    }
    // the block compacts a sequence's selected rows in order (one thread walking them all: 48 us for a batch of eight)
    __shared__ int sc[33];
    int n = nb;
    if (use_suffix) {
        for (int s = 0; s < sd.batch; ++s) {
            if (!sd.refresh.v[s]) continue;
            const int c = sel_cnt[s];
            for (int i0 = 0; i0 < c; i0 += blockDim.x) {
                const int w = i0 + t < c ? sel_idx[s * sd.W_max + i0 + t] : -1;
                const bool take = w >= sd.n_pre && y[s * sd.N + window_pos(sd, w)] == mask_id;
                int total;
                const int o = n + block_excl_scan(take ? 1 : 0, sc, &total);
                if (take) {
                    HeadSrc h; h.kind = 1; h.index = s * sd.W_max + w;
                    list[o] = h; suf_seq[o - nb] = s; suf_w[o - nb] = w;
                }
                n += total;
            }
        }
    }
    if (t == 0) *count = n;
    (void)act_row0_stride;
}

// ---------------------------------------------------------------------------------------
// Confidence of logits rows (Eq. 1 and the confidence of Sec. 2).  One launch: a cluster of up to eight CTAs per row, every warp
// pushes its (maximum, sum, best) into the first CTA's shared memory, whose first warp combines them in a fixed order; no
// scratch in global memory.
//
// Few rows are a latency chain (loads, running maximum, combination), many are bound by the read.  Every thread has CONF_U
// 16-byte loads in flight and takes one rescaling and independent exponentials (expf: with __expf, 7 - 8 % faster, a term's error grows with
// its distance from the maximum) per batch; the vocabulary need not be a multiple
// of four.  us, against 32 chunks of a row in blocks of their own, a rescaling per 16 bytes (single floats in the second) and
// a second launch that combined them: 32 rows x 126464 8.9 -> 7.6, 64 x 50258 13.9 -> 7.5, 512 x 126464 78 -> 55 (4.7 TB/s),
// 512 x 2000 35 -> 4.5.
// ---------------------------------------------------------------------------------------
struct ConfPart { float mx_all; float sum; float mx_ex; int arg_ex; };
constexpr int CONF_CL = 8, CONF_MAX_THREADS = 512, CONF_U = 4;

struct ConfRun {
    float mx = -INFINITY, sum = 0.f, mxe = -INFINITY;       // maximum, sum of exp relative to it, best non-[MASK] value
    int arg = 0x7fffffff;
    __device__ __forceinline__ void best(float x, int v, int mask_id) {
        if (v != mask_id && (x > mxe || (x == mxe && v < arg))) { mxe = x; arg = v; }
    }
    __device__ __forceinline__ void one(float x, int v, int mask_id) {
        const float nm = fmaxf(mx, x), ref = nm == -INFINITY ? 0.f : nm;        // (only -inf so far: every term is exp(-inf))
        sum = sum * expf(mx - ref) + expf(x - ref);
        mx = nm;
        best(x, v, mask_id);
    }
    // CONF_U 16-byte pieces, piece u from element v + u * step on (ascending, so the lowest index of equal values comes first);
    // one rescaling and independent exponentials for all of them.  Missing pieces are -inf.
    __device__ __forceinline__ void batch(const float4 (&x)[CONF_U], int v, int step, int mask_id) {
        float m = -INFINITY;
#pragma unroll
        for (int u = 0; u < CONF_U; ++u) m = fmaxf(m, fmaxf(fmaxf(x[u].x, x[u].y), fmaxf(x[u].z, x[u].w)));
        const float nm = fmaxf(mx, m), ref = nm == -INFINITY ? 0.f : nm;
        float s = 0.f;
#pragma unroll
        for (int u = 0; u < CONF_U; ++u) s += (expf(x[u].x - ref) + expf(x[u].y - ref)) + (expf(x[u].z - ref) + expf(x[u].w - ref));
        sum = sum * expf(mx - ref) + s;
        mx = nm;
#pragma unroll
        for (int u = 0; u < CONF_U; ++u) {
            float e[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
            const int vu = v + u * step;
            if ((unsigned)(mask_id - vu) < 4u) {
#pragma unroll
                for (int i = 0; i < 4; ++i) if (vu + i == mask_id) e[i] = -INFINITY;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) if (e[i] > mxe) { mxe = e[i]; arg = vu + i; }
        }
    }
    // the warp's lanes combined: every lane ends with the same values
    __device__ __forceinline__ void warp_combine() {
        const float all = warp_max(mx);
        sum = warp_sum(sum > 0.f ? sum * expf(mx - all) : 0.f);
        mx = all;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, mxe, o);
            const int oi = __shfl_xor_sync(0xffffffffu, arg, o);
            if (ov > mxe || (ov == mxe && oi < arg)) { mxe = ov; arg = oi; }
        }
    }
};
__global__ void __launch_bounds__(CONF_MAX_THREADS) confidence_kernel(const float* logits, const int* m_count, int V, int mask_id, int cl, int* yhat, float* conf) {
    KERNEL_PROLOGUE(11);   // confidence_kernel
    __shared__ ConfPart parts[CONF_CL * (CONF_MAX_THREADS / 32)];
    const int r = (int)blockIdx.x / cl, ch = (int)blockIdx.x - r * cl;
    if (m_count && r >= *m_count) return;                    // (the whole cluster)
    // (the first CTA must run before anything is pushed into its shared memory: the barrier passes under the loads)
    if (cl > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, wid = t >> 5, nw = nt >> 5;
    // The row from its first 16-byte boundary on in 16-byte pieces, whatever the vocabulary; up to three elements in
    // front of that and three behind are the last CTA's.
    const float* l = logits + (size_t)r * V;
    const int lead = min(V, (int)((4 - (((uintptr_t)l >> 2) & 3)) & 3)), n4 = (V - lead) >> 2, tail = V - lead - 4 * n4;
    const int per = (n4 + cl - 1) / cl, c0 = ch * per, c1 = min(n4, c0 + per);
    const float4* l4 = reinterpret_cast<const float4*>(l + lead);
    ConfRun a;
    if (c0 + t < c1) { a.arg = lead + 4 * (c0 + t); a.arg += a.arg == mask_id; }      // (a row of -inf predicts its lowest token)
    for (int i = c0 + t; i < c1; i += CONF_U * nt) {
        float4 x[CONF_U];
#pragma unroll
        for (int u = 0; u < CONF_U; ++u) x[u] = i + u * nt < c1 ? __ldg(l4 + i + u * nt) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        a.batch(x, lead + 4 * i, 4 * nt, mask_id);
    }
    if (ch == cl - 1 && t < lead + tail) {
        const int v = t < lead ? t : V - tail + (t - lead);
        a.one(__ldg(l + v), v, mask_id);
    }
    a.warp_combine();
    if (cl > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (lane == 0) {
        const uint32_t dst = dsmem_addr((uint32_t)__cvta_generic_to_shared(parts + ch * nw + wid), 0);
        asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(__float_as_uint(a.mx)), "r"(__float_as_uint(a.sum)),
                     "r"(__float_as_uint(a.mxe)), "r"(a.arg) : "memory");
    }
    if (cl > 1) cluster_sync_all(); else __syncthreads();
    if (ch != 0 || wid != 0) return;
    ConfRun f;
    for (int c = lane; c < cl * nw; c += 32) {
        const ConfPart q = parts[c];
        const float nm = fmaxf(f.mx, q.mx_all);
        if (f.sum > 0.f) f.sum *= expf(f.mx - nm);
        if (q.sum > 0.f) f.sum += q.sum * expf(q.mx_all - nm);
        f.mx = nm;
        if (q.mx_ex > f.mxe || (q.mx_ex == f.mxe && q.arg_ex < f.arg)) { f.mxe = q.mx_ex; f.arg = q.arg_ex; }
    }
    f.warp_combine();
    if (lane == 0) { yhat[r] = f.arg; conf[r] = expf(f.mxe - f.mx) / f.sum; }
}

// ---------------------------------------------------------------------------------------
// Commit rule (Sec. 4.2; Algorithm 1 after the layer loop; Eq. 2): one block per sequence.
// ---------------------------------------------------------------------------------------
struct CommitArgs {
    int* y;                      // [batch][N]
    const float* conf; const int* yhat;   // LM rows: active rows first ([batch*B]), then suffix rows
    const float* kl;             // per-head drift of the forward's rows (last layer) [rows][n_heads]
    float* delta_out;            // [batch][B]
    float* Delta_out; float* taud_out;
    float* theta; int* theta_cnt;   // [batch][hist][B] ring, [batch] number pushed so far
    int* commit_flags;           // [batch][B]
    int* own_flags;              // [batch][B]: the rule's own decision, before a forced decision replaces it
    int* suffix_flags;           // [batch][W_max]
    const int* head_count; const int* suf_seq; const int* suf_w;
    const int* forced_pos; int forced_n;      // [batch][forced_n] absolute positions, -1 unused (null: free-running)
    const int* forced_tok;                    // optional tokens written at the forced positions (null: own prediction)
    int* seq_info;               // [batch][8]: committed, by_conf, by_drift, by_quota, suffix, eos, masked_left, nonfinite;
                                 // then 8 more words: the step's counters (stats[0..3]) and the GEMM status word
    const int* stats; const int* status; int batch;
    int n_heads, hist, mask_id, eos_id, act_row_off, steps_used, steps_per_block, use_drift, use_suffix, ge;
    float tau_s, alpha, tau_suffix;
};

__global__ void commit_kernel(StepDesc sd, CommitArgs a) {
    KERNEL_PROLOGUE(13);   // commit_kernel
    __shared__ float s_conf[256];
    __shared__ unsigned char s_masked[256], s_flag[256];
    __shared__ int cnt[8];
    const int s = blockIdx.x, j = threadIdx.x, B = sd.B;
    if (j < 8) cnt[j] = 0;
    __syncthreads();
    const bool within = sd.record_kl != 0;
    float c = 0.f, dl = 0.f, Dl = 0.f, td = 0.f;
    int tok = 0, yh = 0;
    bool masked = false;
    int flag = 0;
    if (j < B) {
        tok = a.y[s * sd.N + sd.act_start + j];
        masked = tok == a.mask_id;
        c = a.conf[s * B + j];
        yh = a.yhat[s * B + j];
        if (within) {
            dl = a.delta_out[s * B + j];      // written by delta_kernel at the end of the forward
            const int pushed = a.theta_cnt[s];
            const int nh = min(pushed, a.hist);
            float mean = 0.f;
            if (nh > 0) {
                // oldest to newest, like a running list
                for (int u = 0; u < nh; ++u) mean += a.theta[((size_t)s * a.hist + ((pushed - nh + u) % a.hist)) * B + j];
                mean /= (float)nh;
            }
            Dl = dl - mean;
            if (a.hist > 0) a.theta[((size_t)s * a.hist + (pushed % a.hist)) * B + j] = dl;
        }
        td = a.alpha * (a.tau_s - c) * (a.tau_s - c);
        if (masked) {
            if (!(c == c)) atomicAdd(&cnt[7], 1);
            const bool c_ok = a.ge ? (c >= a.tau_s) : (c > a.tau_s);
            const bool d_ok = within && a.use_drift && (a.ge ? (Dl >= td) : (Dl > td));
            if (c_ok) flag = 1 | 2;
            else if (d_ok) flag = 1 | 4;
        }
        a.delta_out[s * B + j] = dl;
        a.Delta_out[s * B + j] = Dl;
        a.taud_out[s * B + j] = td;
        s_conf[j] = c; s_masked[j] = masked; s_flag[j] = (unsigned char)flag;
        if (masked) atomicAdd(&cnt[6], 1);
        if (flag) atomicAdd(&cnt[0], 1);
    }
    __syncthreads();
    if (j == 0 && within && a.hist > 0) a.theta_cnt[s] = a.theta_cnt[s] + 1;
    const int n_masked = cnt[6];
    {
        // quota top-up: the most confident masked rows not yet committed (ties: lowest position)
        const int denom = max(1, a.steps_per_block - a.steps_used);
        const int quota = n_masked > 0 ? (n_masked + denom - 1) / denom : 0;
        const int need = quota - cnt[0];
        if (need > 0 && j < B && masked && !flag) {
            int rank = 0;
            for (int u = 0; u < B; ++u)
                if (s_masked[u] && !s_flag[u] && (s_conf[u] > c || (s_conf[u] == c && u < j))) ++rank;
            if (rank < need) flag = 1 | 8;
        }
    }
    if (j < B) a.own_flags[s * B + j] = flag;
    if (a.forced_pos) {
        // a forced decision replaces the rule's own (kept in own_flags); the label of a row the rule also chose stays
        if (j < B) {
            const int own = flag;
            flag = 0;
            const int pos = sd.act_start + j;
            for (int u = 0; u < a.forced_n; ++u)
                if (a.forced_pos[s * a.forced_n + u] == pos) {
                    flag = own ? own : (1 | 8);
                    if (a.forced_tok) yh = a.forced_tok[s * a.forced_n + u];
                }
            if (!masked) flag = 0;
        }
    }
    __syncthreads();
    if (j < 6) cnt[j] = 0;
    __syncthreads();
    if (j < B) {
        a.commit_flags[s * B + j] = flag;
        if (flag & 1) {
            a.y[s * sd.N + sd.act_start + j] = yh;
            atomicAdd(&cnt[0], 1);
            if (flag & 2) atomicAdd(&cnt[1], 1);
            if (flag & 4) atomicAdd(&cnt[2], 1);
            if (flag & 8) atomicAdd(&cnt[3], 1);
            if (yh == a.eos_id) atomicAdd(&cnt[5], 1);
        }
    }
    // suffix rows of the final packet: confidence alone decides
    for (int w = j; w < sd.W_max; w += blockDim.x) a.suffix_flags[s * sd.W_max + w] = 0;
    __syncthreads();
    if (a.use_suffix && within) {
        const int n_suf = *a.head_count - sd.batch * B;
        for (int i = j; i < n_suf; i += blockDim.x) {
            if (a.suf_seq[i] != s) continue;
            const int w = a.suf_w[i];
            const int pos = window_pos(sd, w);
            const float sc = a.conf[sd.batch * B + i];
            bool ok = a.ge ? (sc >= a.tau_suffix) : (sc > a.tau_suffix);
            int t2 = a.yhat[sd.batch * B + i];
            int f = 1 | (ok ? 4 : 0);          // bit 2: the rule's own decision for this eligible row
            if (a.forced_pos) {
                ok = false;
                for (int u = 0; u < a.forced_n; ++u)
                    if (a.forced_pos[s * a.forced_n + u] == pos) { ok = true; if (a.forced_tok) t2 = a.forced_tok[s * a.forced_n + u]; }
            }
            if (ok && a.y[s * sd.N + pos] == a.mask_id) {
                a.y[s * sd.N + pos] = t2;
                f |= 2;
                atomicAdd(&cnt[0], 1); atomicAdd(&cnt[4], 1);
                if (t2 == a.eos_id) atomicAdd(&cnt[5], 1);
            }
            a.suffix_flags[s * sd.W_max + w] = f;
        }
    }
    __syncthreads();
    if (j == 0) {
        int* o = a.seq_info + s * 8;
        o[0] = cnt[0]; o[1] = cnt[1]; o[2] = cnt[2]; o[3] = cnt[3]; o[4] = cnt[4]; o[5] = cnt[5];
        o[6] = n_masked - (cnt[0] - cnt[4]);
        o[7] = cnt[7];
        if (s == 0) {        // one record for the host: a single copy brings everything the controller reads
            int* t = a.seq_info + a.batch * 8;
            t[0] = a.stats[0]; t[1] = a.stats[1]; t[2] = a.stats[2]; t[3] = a.stats[3];
            t[4] = *a.status;
        }
    }
}

// Last-layer drift of the active rows (Algorithm 1, delta): mean over heads of the per-head KL.
__global__ void delta_kernel(StepDesc sd, const float* kl, int act_row_off, int n_heads, float* delta) {
    KERNEL_PROLOGUE(14);   // delta_kernel
    const int s = blockIdx.x, j = threadIdx.x;
    if (j >= sd.B) return;
    float dl = 0.f;
    if (sd.record_kl) {
        const float* kr = kl + (size_t)(s * sd.rows_per_seq + act_row_off + j) * n_heads;
        float acc = 0.f;
        for (int h = 0; h < n_heads; ++h) acc += kr[h];
        dl = acc / (float)n_heads;
    }
    delta[s * sd.B + j] = dl;
}

// gather rows of x into a keep buffer: dst[s][j][:] = x[row(s, j)][:]
__global__ void keep_hidden_kernel(StepDesc sd, const float* x, int act_row_off, int d, float* dst) {
    KERNEL_PROLOGUE(15);   // keep_hidden_kernel
    const int i = blockIdx.x;
    const int s = i / sd.B, j = i - s * sd.B;
    const float* src = x + (size_t)(s * sd.rows_per_seq + act_row_off + j) * d;
    float* o = dst + (size_t)i * d;
    for (int c = threadIdx.x; c < d; c += blockDim.x) o[c] = src[c];
}

// y = [prompt ; MASK ...] from a prompt that already lives on the device (ids clamped to the vocabulary)
__global__ void init_tokens_kernel(int* y, const int* prompt, int batch, int prompt_len, int N, int mask_id, int vocab) {
    KERNEL_PROLOGUE(16);   // init_tokens_kernel
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= batch * N) return;
    const int s = i / N, pos = i - s * N;
    int t = mask_id;
    if (pos < prompt_len) {
        t = prompt[s * prompt_len + pos];
        t = t < 0 ? 0 : (t >= vocab ? vocab - 1 : t);
        if (t == mask_id) t = (mask_id + 1) % vocab;
    }
    y[i] = t;
}

// rotary table: tab[pos][i] = (cos, sin)(pos * theta^(-2i/dh)), computed in double precision
__global__ void rope_table_kernel(float2* tab, int N, int half, double theta) {
    KERNEL_PROLOGUE(17);   // rope_table_kernel
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * half) return;
    const int pos = i / half, k = i - pos * half;
    const double inv = pow(theta, -(double)k / (double)half);
    const double ang = (double)pos * inv;
    tab[i] = make_float2((float)cos(ang), (float)sin(ang));
}

}  // namespace ps
