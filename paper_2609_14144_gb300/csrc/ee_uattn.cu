// Causal attention of a batch of positions on the fifth-generation tensor
// cores (sm_103a): the multi-position layer pass's attention for batches of at
// least kUaMinRows rows (ee_rows.cu has the warp-level one for fewer).
//
// CTA (head h, key split s, row tile t): the 128 rows of tile t of the batch
// for query head h against keys [s KC, (s + 1) KC) of the layer's cache (no
// further than its own rows look), in blocks of 64 keys:
//   S = Q K^T with the scaled query split into three bf16 parts (high + middle
//     + low = q exactly), one tcgen05.mma of M = 128 x N = 64 per part and 16
//     dimensions; the high parts' products and the middle and low parts' in
//     separate accumulators, as in the projections;
//   softmax in registers: tensor-memory lane = row, a row's 64 scores shared by
//     four threads (warps w, w + 4, w + 8 and w + 12); keys past a row's position
//     are masked;
//   O = P V with the probabilities split into three parts the same way and
//     written to shared memory as the A operand; V is the B operand as it lies
//     in the cache (dimensions contiguous).  The products of up to kUaChain
//     blocks add up in tensor memory and are then added to the row's running
//     sum in registers, in fp32 with rounding to nearest.
// A row's probabilities are taken relative to a reference that follows its
// maximum only when it is outgrown by e^8, which ends the chain (the splits'
// merge needs a common reference, not the exact maximum).
// The scores of block j + 1 are issued before the softmax of block j, and the
// product of block j runs under the softmax of block j + 1.  Keys and values
// come with cp.async into two buffers each, as [16-byte chunk of the head
// dimension][64 keys][16 bytes]: the canonical no-swizzle layout of K as a
// K-major operand and of V as an N-major one.
//
// What bounds it: the registers' side (two loads, an exponential, a split into
// three parts and three stores per score, and the read-back of the products)
// has four warps a scheduler and issues on 40% of the cycles, between the two
// barriers of a block; the tensor pipe is active on 16%.  A 256-row batch of 16
// heads of 128 over 2200 keys on average takes 40.9 us a layer, 92.6 us with
// the warp-level kernel (four warps per SM, its shared memory's worth; twelve
// warps with the same products took 67 us: close to the mma.sync rate).  A
// 4099-position prompt of six such layers went from 20.8 to 16.8 ms.
//
// Each split writes its unnormalised output, maximum and sum per (row, head) as
// the warp-level kernel does; k_rows_amerge combines them.  Every wait is
// bounded; after one runs out the kernel flags kErrStall, does not wait for
// further ones, lets its products in flight end (bounded), frees its tensor
// memory and returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "ee_internal.h"
#include "ee_split3.cuh"
#include "ee_umma.cuh"

namespace ee {
namespace {

constexpr int kUaSplit = 4;                    // threads that share a row
constexpr int kUaRows = 128;                   // query rows per CTA
constexpr int kUaThreads = kUaSplit * kUaRows;
constexpr int kUaKeys = 64;                    // keys per block
constexpr int kUaChain = 8;                    // blocks whose products meet in tensor memory (at most)
constexpr int kUaPages = 1024;                 // page-table entries kept in shared memory

// Shared memory: the queries' parts, two key and two value buffers, the
// probabilities' parts, row statistics exchanged between the two halves.
template <int D>
struct UaSmem {
    static constexpr int CH = D / 8;  // 16-byte chunks of a row
    // From one chunk to the next: the rows, and 16 bytes so that the lanes that
    // write neighbouring chunks of a row fall in different banks.
    static constexpr int q_step = kUaRows * 16 + 16, kv_step = kUaKeys * 16 + 16;
    static constexpr int q_part = CH * q_step;  // one part of the queries
    static constexpr int kv = CH * kv_step;     // one block of keys or values
    static constexpr int p_part = kUaKeys / 8 * kUaRows * 16;
    static constexpr int at_k = 3 * q_part, at_v = at_k + 2 * kv, at_p = at_v + 2 * kv, at_x = at_p + 3 * p_part;
    static constexpr int at_bar = at_x + kUaSplit * kUaRows * 4;
    static constexpr int bytes = at_bar + 64 + 1024;  // barriers, then alignment slack
};

// Eight floats as three 16-byte pieces of bf16 parts.
__device__ __forceinline__ void ua_split8(const float (&x)[8], uint4 (&p)[3]) {
    uint32_t w[4][3];
#pragma unroll
    for (int e = 0; e < 4; ++e) split3(x[2 * e], x[2 * e + 1], w[e]);
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k] = make_uint4(w[0][k], w[1][k], w[2][k], w[3][k]);
}
__device__ __forceinline__ void ua_cp16(uint32_t dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void ua_commit_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void ua_wait_group() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ua_proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

template <int D>
__global__ void __launch_bounds__(kUaThreads, 1)
    k_rows_uattn(DevModel m, int j, const float* __restrict__ Q, const int32_t* __restrict__ pos, int Mj, int KC, int t_max,
                 float* __restrict__ part) {
    using L = UaSmem<D>;
    constexpr int CH = L::CH, HC = D / kUaSplit, SC = kUaKeys / kUaSplit;  // output columns and scores of a thread
    extern __shared__ __align__(1024) uint8_t ua_smem_raw[];
    __shared__ uint32_t tmem_slot;
    __shared__ int p_last[kUaThreads / 32];
    __shared__ int s_page[kUaPages];
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(ua_smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sb = u_saddr(sm);
    float* xch = reinterpret_cast<float*>(sm + L::at_x);  // [kUaSplit][rows]
    uint64_t* s_full = reinterpret_cast<uint64_t*>(sm + L::at_bar);  // [2] scores of a block are there
    uint64_t* pv_done = s_full + 2;                                  // a block's product is there
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int qt = w >> 2, row = (w & 3) * 32 + lane;  // this thread's share of the columns, and its row of the tile
    if (tid == 0) {
        u_mb_init(&s_full[0], 1);
        u_mb_init(&s_full[1], 1);
        u_mb_init(pv_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (w == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(u_saddr(&tmem_slot)), "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int h = blockIdx.x, s = blockIdx.y, r0 = blockIdx.z * kUaRows, G = m.A / m.KH, g = h / G;
    const int my_pos = r0 + row < Mj ? pos[r0 + row] : -1;
    int pw = my_pos;
#pragma unroll
    for (int o = 16; o; o >>= 1) pw = max(pw, __shfl_xor_sync(0xffffffffu, pw, o));
    if (lane == 0) p_last[w] = pw;
    u_fence_before();
    __syncthreads();
    u_fence_after();
    const uint32_t tmem = tmem_slot;
    const int k0 = s * KC;
    int kend = 0;
#pragma unroll
    for (int i = 0; i < kUaThreads / 32; ++i) kend = max(kend, p_last[i] + 1);
    kend = min(kend, min(k0 + KC, t_max));
    const int nb = kend > k0 ? (kend - k0 + kUaKeys - 1) / kUaKeys : 0;
    volatile int* everr = &m.ctl->err;

    if (nb > 0) {
        // The pages of the split's keys (page lengths are powers of two).
        const int ps = 31 - __clz(m.page_size), pg0 = k0 >> ps, npg = ((kend - 1) >> ps) - pg0 + 1;
        if (npg <= kUaPages) {
            for (int i = tid; i < npg; i += kUaThreads) s_page[i] = m.page_table[pg0 + i];
            __syncthreads();
        }
        const int64_t page_elems = (int64_t)m.KH * m.page_size * D;
        const int64_t layer_off = (int64_t)j * m.kv_layer_stride + (int64_t)g * m.page_size * D + (tid % CH) * 8;
        // 64 keys (or values) from key kb on into buffer `at`; past kend zeros
        auto load = [&](const uint16_t* pool, int b, int at) {
            if (b < nb) {
#pragma unroll
                for (int u = 0; u < kUaKeys * CH / kUaThreads; ++u) {
                    const int r = tid / CH + u * (kUaThreads / CH), t = k0 + b * kUaKeys + r;
                    const bool ok = t < kend;
                    const int pi = (t >> ps) - pg0;
                    const int page = !ok ? 0 : npg <= kUaPages ? s_page[pi] : m.page_table[pg0 + pi];
                    const int64_t off = ok ? layer_off + page * page_elems + (t & (m.page_size - 1)) * D : 0;
                    ua_cp16(sb + at + (tid % CH) * L::kv_step + r * 16, pool + off, ok ? 16 : 0);
                }
            }
            ua_commit_group();
        };
        load(m.kpool, 0, L::at_k);
        load(m.kpool, 1, L::at_k + L::kv);
        load(m.vpool, 0, L::at_v);
        // the tile's queries, scaled, as three parts: [part][chunk][row][16 bytes]
        const float scale = 1.0f / sqrtf((float)D);
#pragma unroll 4
        for (int e = tid; e < kUaRows * CH; e += kUaThreads) {
            const int r = e / CH, c = e % CH, i = r0 + r;
            float x[8];
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (i < Mj) {
                const float4* q = reinterpret_cast<const float4*>(Q + (int64_t)i * m.A * D + (int64_t)h * D + c * 8);
                a = q[0], b = q[1];
            }
            x[0] = a.x * scale, x[1] = a.y * scale, x[2] = a.z * scale, x[3] = a.w * scale;
            x[4] = b.x * scale, x[5] = b.y * scale, x[6] = b.z * scale, x[7] = b.w * scale;
            uint4 p[3];
            ua_split8(x, p);
#pragma unroll
            for (int k = 0; k < 3; ++k) *reinterpret_cast<uint4*>(sm + k * L::q_part + c * L::q_step + r * 16) = p[k];
        }
        constexpr uint32_t kOHi = 256, kOLo = 256 + D;  // tensor-memory columns; scores: 128 per buffer from 0 on
        const uint32_t id_s = u_idesc(kUaKeys), id_o = u_idesc(D, true);
        auto issue_scores = [&](int b) {  // one thread
            const uint32_t kd = sb + L::at_k + (b & 1) * L::kv, d = tmem + (b & 1) * 128;
#pragma unroll
            for (int c = 0; c < D / 16; ++c)
#pragma unroll
                for (int p = 0; p < 3; ++p)
                    u_mma(d + (p ? 64 : 0), u_desc(sb + p * L::q_part + 2 * c * L::q_step, L::q_step, 128),
                          u_desc(kd + 2 * c * L::kv_step, L::kv_step, 128), id_s, (c > 0 || p == 2) ? 1u : 0u);
            u_commit(&s_full[b & 1]);
        };
        auto issue_product = [&](int b, bool more) {  // one thread; more: onto the products there
            const uint32_t vd = sb + L::at_v + (b & 1) * L::kv;
#pragma unroll
            for (int c = 0; c < kUaKeys / 16; ++c)
#pragma unroll
                for (int p = 0; p < 3; ++p)
                    u_mma(tmem + (p ? kOLo : kOHi), u_desc(sb + L::at_p + p * L::p_part + 2 * c * (kUaRows * 16), kUaRows * 16, 128),
                          u_desc(vd + c * 256, 128, L::kv_step), id_o, (more || c > 0 || p == 2) ? 1u : 0u);
            u_commit(pv_done);
        };
        const uint32_t lane_t = tmem + ((uint32_t)((w & 3) * 32) << 16);
        float o[HC], mx = -INFINITY, l = 0.f;
#pragma unroll
        for (int i = 0; i < HC; ++i) o[i] = 0.f;
        // a wait of every thread of the CTA
        auto wait = [&](uint64_t* bar, int parity) {
            if (!u_mb_wait(bar, parity, everr)) atomicOr(&m.ctl->err, kErrStall);
            u_fence_after();
            __syncwarp();  // the tensor-memory loads that follow are warp-wide
        };
        // o += the products since the last read-back
        auto add_products = [&]() {
#pragma unroll
            for (int i = 0; i < HC; i += 16) {
                uint32_t hi[16], lo[16];
                u_ld16(lane_t + kOHi + qt * HC + i, hi);
                u_ld16(lane_t + kOLo + qt * HC + i, lo);
                u_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) o[i + e] += __uint_as_float(hi[e]) + __uint_as_float(lo[e]);
            }
        };
        ua_wait_group<2>();  // the first keys
        ua_proxy_fence();
        __syncthreads();  // (and the queries)
        if (tid == 0) issue_scores(0);
        int since = 0;  // products in tensor memory not yet added to o
        for (int b = 0; b < nb; ++b) {
            wait(&s_full[b & 1], (b >> 1) & 1);
            load(m.kpool, b + 2, L::at_k + (b & 1) * L::kv);  // the scores of b have read its keys
            float sc[SC];
            {
                uint32_t hi[SC], lo[SC];
                u_ld16(lane_t + (b & 1) * 128 + qt * SC, hi);
                u_ld16(lane_t + (b & 1) * 128 + 64 + qt * SC, lo);
                u_wait_ld();
#pragma unroll
                for (int e = 0; e < SC; ++e) sc[e] = __uint_as_float(hi[e]) + __uint_as_float(lo[e]);
                const int last = my_pos - (k0 + b * kUaKeys + qt * SC);  // keys up to here are looked at
                if (!__all_sync(0xffffffffu, last >= SC - 1))
#pragma unroll
                    for (int e = 0; e < SC; ++e) sc[e] = e <= last ? sc[e] : -INFINITY;
            }
            float bm = sc[0];
#pragma unroll
            for (int e = 1; e < SC; ++e) bm = fmaxf(bm, sc[e]);
            xch[qt * kUaRows + row] = bm;
            // keys b + 1 have landed (in flight at most: values b, keys b + 2)
            ua_wait_group<2>();
            ua_proxy_fence();
            u_fence_before();
            // a row whose scores outgrow its reference by more than e^8
            const bool grow = __syncthreads_or(bm > mx + 8.f);
            if (tid == 0 && b + 1 < nb) {
                u_fence_after();
                issue_scores(b + 1);
            }
            if (b > 0) wait(pv_done, (b - 1) & 1);
            if (since > 0 && (grow || since == kUaChain)) {
                add_products();
                since = 0;
            }
            if (grow) {
                float mn = bm;
#pragma unroll
                for (int e = 0; e < kUaSplit; ++e) mn = fmaxf(mn, xch[e * kUaRows + row]);
                if (mn > mx + 8.f) {
                    const float c = expf(mx - mn);  // 0 for a row's first key
                    mx = mn;
                    l *= c;
#pragma unroll
                    for (int i = 0; i < HC; ++i) o[i] *= c;
                }
            }
            // a row with no key yet keeps reference -inf, probabilities 0
            const bool any = mx != -INFINITY;
#pragma unroll
            for (int e = 0; e < SC; ++e) {
                sc[e] = any ? expf(sc[e] - mx) : 0.f;
                l += sc[e];
            }
            load(m.vpool, b + 1, L::at_v + ((b + 1) & 1) * L::kv);  // the product of b - 1 has read its values
#pragma unroll
            for (int q = 0; q < SC / 8; ++q) {
                float x[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = sc[8 * q + e];
                uint4 p[3];
                ua_split8(x, p);
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    *reinterpret_cast<uint4*>(sm + L::at_p + k * L::p_part + ((qt * (SC / 8) + q) * kUaRows + row) * 16) = p[k];
            }
            ua_wait_group<2>();  // values b (in flight at most: keys b + 2, values b + 1)
            ua_proxy_fence();
            u_fence_before();
            __syncthreads();
            if (tid == 0) {
                u_fence_after();
                issue_product(b, since > 0);
            }
            ++since;
        }
        wait(pv_done, (nb - 1) & 1);
        if (*everr & kErrStall) u_mb_wait(pv_done, (nb - 1) & 1, nullptr);  // products in flight end
        add_products();
        ua_wait_group<0>();
        // the split's unnormalised output, maximum and sum: part[((s Mj + row) A + h)][kAttnLd(D)]
        __syncthreads();
        xch[qt * kUaRows + row] = l;
        __syncthreads();
        if (my_pos >= k0) {
            float* out = part + ((int64_t)(s * Mj + r0 + row) * m.A + h) * kAttnLd(D);
#pragma unroll
            for (int i = 0; i < HC; i += 4)
                *reinterpret_cast<float4*>(out + qt * HC + i) = make_float4(o[i], o[i + 1], o[i + 2], o[i + 3]);
            float lt = 0.f;
#pragma unroll
            for (int e = 0; e < kUaSplit; ++e) lt += xch[e * kUaRows + row];
            if (qt == 0) *reinterpret_cast<float2*>(out + D) = make_float2(mx, lt);
        }
    }
    u_fence_before();
    __syncthreads();
    if (w == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

}  // namespace

// Keys per split: a multiple of the block, the split count that needs the
// least time by a simple count: the waves of CTAs (one resident per SM) times
// a CTA's blocks and its set-up and write-out (about two blocks' time; four
// more for a split beyond the first, which the merge reads back).
int uattn_keys_per_split(int t_max, int A, int M, int n_sm, int max_splits) {
    const int units = A * ((M + kUaRows - 1) / kUaRows), blocks = (t_max + kUaKeys - 1) / kUaKeys;
    int best = blocks;
    int64_t least = INT64_MAX;
    for (int S = 1; S <= std::min(max_splits, blocks); ++S) {
        const int per = (blocks + S - 1) / S, n = (blocks + per - 1) / per;
        const int64_t waves = ((int64_t)units * n + n_sm - 1) / n_sm;
        const int64_t t = 2 * waves * (per + 2) + n;
        if (t < least) {
            least = t;
            best = per;
        }
    }
    return best * kUaKeys;
}

cudaError_t configure_uattn() {
    cudaError_t e = cudaFuncSetAttribute(k_rows_uattn<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, UaSmem<128>::bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_rows_uattn<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, UaSmem<64>::bytes);
    return e;
}

cudaError_t launch_uattn(const DevModel& m, int j, const float* Q, const int32_t* d_pos, int Mj, int KC, int t_max, float* part,
                         cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(m.A, (t_max + KC - 1) / KC, (Mj + kUaRows - 1) / kUaRows);
    cfg.blockDim = dim3(kUaThreads);
    cfg.dynamicSmemBytes = m.D == 128 ? UaSmem<128>::bytes : UaSmem<64>::bytes;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (m.D == 128) return cudaLaunchKernelEx(&cfg, k_rows_uattn<128>, m, j, Q, d_pos, Mj, KC, t_max, part);
    return cudaLaunchKernelEx(&cfg, k_rows_uattn<64>, m, j, Q, d_pos, Mj, KC, t_max, part);
}

}  // namespace ee
