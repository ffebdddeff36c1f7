// Fifth-generation tensor-core projections of the multi-position layer pass
// (the prompt and the full-depth re-pass, ee_rows.cu) on sm_103a: tcgen05.mma
// with operands staged in shared memory by TMA and the fp32 accumulator in
// tensor memory.
//
// One projection of a batch of positions: Y[row][n] = sum_k W[n][k]
// x[row][k] for the n_rows x K tile-packed bf16 weights W.  Each activation
// is carried as three bf16 parts (x = high + middle + low, ee_rows.cu), each
// part of a block of at most 256 of the batch's rows stored as N operand rows;
// every K = 16 step issues three MMAs of shape M = 128 (weight rows) x N (the
// block's rows rounded up to 16), one per part, into two fp32 accumulators whose column is the batch
// row: the high parts' products into the first, the middle and low parts'
// (2^-8 of the size and less) into the second, so that their small terms are
// not added into the large sum step by step; the epilogue adds the two.  The
// bf16 products are exact.
//
// CTA (x, s, z): weight rows [128 x, 128 x + 128) (four 32-row tiles) over the
// K range of split s for row block z, 32 columns per pipeline stage, four
// stages in flight (eight for a small batch, whose stages are 20 KB):
//   - the producer warp's lane 0 loads a stage: the 128 x 32 weight block with one TMA
//     tensor copy (a three-dimensional view of the tile-packed layout whose
//     box lands in shared memory in the UMMA canonical K-major layout with
//     no swizzle: 8-row x 16-byte core matrices, 128 bytes apart along the
//     rows, 2048 along K) and the batch's activations with bulk copies (the
//     activation buffer is stored chunk-major with a row stride of N, so a
//     stage is one contiguous range in the same canonical layout: a part's N
//     rows N x 16 bytes long, the three parts of a chunk side by side, chunks
//     3 N x 16 bytes apart along K; 48 KB for a full batch);
//   - the MMA warp's lane 0 issues six MMAs per stage into the tensor-memory
//     accumulators and commits each stage back to its producer barrier;
//   - the epilogue warps read the accumulators (warps w and w + 4 hold
//     tensor-memory lanes 32 w .. 32 w + 31, the weight rows of tile w, half of
//     the columns each): the high parts' after every chain of stages, added to
//     running sums in registers, both after the last stage, when they write the
//     split's partial sums part[s][row][n], which the consumer adds in split
//     order as with the warp-level path.  (A small batch's chains have an
//     accumulator each, all read after the last stage.)
// The tensor core adds with truncation, so the error of a sum grows with the
// number of steps it is carried through: with a whole K range in one chain a
// 4099-position prompt was 2.0e-4 from 64 bits in its final state, with chains
// of 4 stages 2.5e-5.  Reading a chain back costs little tensor time: the next
// stages' middle and low parts' products are issued first and run under it
// (gate/up of an 820-row batch at 3B: 162 us, 145 us in one chain).  A chain is
// never longer than a split of a 256-row batch (umma_chain): where K is short
// and the splits are many there, fewer splits must not mean longer chains.
// Every wait is bounded; after a wait runs out the kernel flags kErrStall in
// the device error word, waits (bounded, whatever the word says) for its
// copies in flight and for the MMAs it issued, frees its tensor memory and
// returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "ee_internal.h"
#include "ee_umma.cuh"

namespace ee {
namespace {

constexpr int kUMRows = 128;                        // weight rows per CTA (UMMA M)
constexpr int kUKStage = 32;                        // K columns per stage
constexpr int kUABytes = kUMRows * kUKStage * 2;    // 8 KB

// A launch's shape.  EW epilogue warps read the accumulators (warp w:
// tensor-memory lanes 32 (w mod 4), columns from HC (w / 4) on), then come the
// producer warp and the MMA warp; NA accumulators of the high parts' products,
// CH stages to a chain (0: as many as the launch says).
template <int EW_, int HC_, int NA_, int CH_, int ST_>
struct UShape {
    static constexpr int EW = EW_, HC = HC_, NA = NA_, CH = CH_, ST = ST_;
    static constexpr int threads = 32 * (EW + 2);
    static constexpr int rows = EW / 4 * HC;  // a block's rows, at most
    // a stage: the weight block and the activations of a full block (8 + 48, 8 + 12 KB)
    static constexpr int stage_bytes = kUABytes + kUKStage / 8 * 3 * rows * 16;
    static constexpr int lo = NA * rows;      // the middle and low parts' accumulator
    static constexpr int tmem_cols = 512;     // accumulators of one fp32 column per position (a CTA has the SM to itself)
    static constexpr size_t smem = (size_t)ST * stage_bytes + 256 + 1024;
    static_assert(lo + rows <= tmem_cols, "the accumulators fit tensor memory");
};
using ULarge = UShape<8, kRowsBlock / 2, 1, 4, 4>;
using UShort = UShape<8, kRowsBlock / 2, 1, 0, 4>;  // short K ranges: shorter chains
// A small batch: fewer threads and registers, so that the launches before and
// after find room beside it (programmatic launch).  Its products are too short
// to run under a read-back, but its accumulators are narrow: each chain has one
// of its own, all read after the last stage.  Eight of its small stages,
// so that most splits have their whole range in flight at once, the weights
// since before the programmatic wait (33 positions at 0.5B: 1254 us with four
// stages as long as a full block's, 1267 with four short ones, 1244 with eight).
using USmall = UShape<4, 64, 4, 0, 8>;

// ---------------------------------------------------------------- copies
__device__ __forceinline__ void u_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(u_saddr(bar)), "r"(bytes) : "memory");
}
// The 128 x 32 weight block at (tile t0, 16-byte column chunk c0) of the
// three-dimensional view {256 elements (one chunk of a 32-row tile), tiles,
// chunks}.
__device__ __forceinline__ void u_tma_w(void* dst, const CUtensorMap* map, int t0, int c0, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(u_saddr(dst)),
        "l"(map), "r"(0), "r"(t0), "r"(c0), "r"(u_saddr(bar))
        : "memory");
}
__device__ __forceinline__ void u_bulk(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     u_saddr(dst)),
                 "l"(src), "r"(bytes), "r"(u_saddr(bar))
                 : "memory");
}

template <class U>
__global__ void __launch_bounds__(U::threads, 1)
    k_rows_umma(const __grid_constant__ CUtensorMap wmap, const uint16_t* __restrict__ x3, int ldx, int n_tiles, int K,
                int M_all, int S, int chain, float* __restrict__ part, int Np, int* err) {
    const int ch = U::CH ? U::CH : chain;
    extern __shared__ __align__(1024) uint8_t u_smem_raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(u_smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(sm + U::ST * U::stage_bytes);
    uint64_t* empty = full + U::ST;
    uint64_t* done = empty + U::ST;
    uint64_t* sum_full = done + 1;    // a chain of the high parts' products is complete
    uint64_t* sum_empty = done + 2;   // it has been read
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 3);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile0 = blockIdx.x * 4, s = blockIdx.y;
    const int nk = (K + kUKStage - 1) / kUKStage;
    const int k0 = (int)((int64_t)nk * s / S), k1 = (int)((int64_t)nk * (s + 1) / S), ks = k1 - k0;
    // operand rows of the batch's blocks (UMMA N); the rows of the last one past
    // M_all give accumulator columns that are never read
    // (the activation parts are stored with this row stride, x3_rows(M_all))
    const int N = x3_rows(M_all), row0 = blockIdx.z * N;
    const int M = M_all - row0 < N ? M_all - row0 : N;  // this block's rows
    x3 += (int64_t)blockIdx.z * (ldx / 8) * 3 * N * 8;
    const int part_bytes = N * 16;  // one part of one 16-byte chunk
    const uint32_t act_bytes = (uint32_t)(kUKStage / 8 * 3 * part_bytes);
    const uint32_t stage_tx = (uint32_t)kUABytes + act_bytes;
    volatile int* everr = err;

    if (threadIdx.x == 0) {
        for (int i = 0; i < U::ST; ++i) {
            u_mb_init(&full[i], 1);
            u_mb_init(&empty[i], 1);
        }
        u_mb_init(done, 1);
        u_mb_init(sum_full, 1);
        u_mb_init(sum_empty, U::EW);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (w == U::EW) {  // tensor memory for the accumulators
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(u_saddr(tmem_slot)),
                     "r"(U::tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    u_fence_before();
    __syncthreads();
    u_fence_after();
    const uint32_t tmem = *tmem_slot;
    // The weights do not depend on the previous kernel: the first stages'
    // weight blocks are requested before the programmatic wait, so that
    // their HBM latency overlaps the previous kernel's tail.
    const int pre = ks < U::ST ? ks : U::ST;
    if (w == U::EW && lane == 0)
        for (int i = 0; i < pre; ++i) {
            u_expect_tx(&full[i], stage_tx);
            u_tma_w(sm + i * U::stage_bytes, &wmap, tile0, (k0 + i) * (kUKStage / 8), &full[i]);
        }
    // the set-up above overlaps the previous kernel (programmatic launch)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (w == U::EW && lane == 0) {
        // producer: stage i of this split, the ring reused once its MMAs are done
        int issued = 0;
        bool ok = true;
        for (int i = 0; i < ks && ok; ++i) {
            const int st = i % U::ST;
            if (i >= U::ST && !u_mb_wait(&empty[st], ((i / U::ST) - 1) & 1, everr)) {
                atomicOr(err, kErrStall);
                ok = false;
                break;
            }
            uint8_t* a = sm + st * U::stage_bytes;
            const int kc = (k0 + i) * (kUKStage / 8);  // first 16-byte chunk of the stage
            if (i >= pre) {  // (the first stages' weights are in flight already)
                u_expect_tx(&full[st], stage_tx);
                u_tma_w(a, &wmap, tile0, kc, &full[st]);
            }
            // the stage's activations: one contiguous range
            u_bulk(a + kUABytes, x3 + (int64_t)kc * 3 * N * 8, act_bytes, &full[st]);
            ++issued;
        }
        // every issued copy lands before the CTA may leave
        for (int i = issued > U::ST ? issued - U::ST : 0; i < issued; ++i)
            u_mb_wait(&full[i % U::ST], (i / U::ST) & 1, nullptr);
    } else if (w == U::EW + 1 && lane == 0) {
        // MMA issuer
        const uint32_t idesc = u_idesc(N);
        // each K = 16 step: the weights times the high parts of the block into
        // the first accumulator, times the middle and the low parts into the
        // second
        // (a descriptor's start address is in units of 16 bytes in its low bits)
        const uint32_t a0 = u_saddr(sm);
        const uint64_t da0 = u_desc(a0, 2048, 128), db0 = u_desc(a0 + kUABytes, 3 * part_bytes, 128);
        const uint32_t part16 = part_bytes >> 4;
        auto mma = [&](int st, int kk, int pp, int acc, bool fresh) {
            const uint32_t at = st * (U::stage_bytes >> 4);
            u_mma(tmem + (pp ? U::lo : acc * U::rows), da0 + (at + kk * 256), db0 + (at + (kk * 6 + pp) * part16), idesc, fresh ? 0u : 1u);
        };
        auto landed = [&](int i) {
            const bool ok = u_mb_wait(&full[i % U::ST], (i / U::ST) & 1, everr);
            if (!ok) atomicOr(err, kErrStall);
            u_fence_after();
            return ok;
        };
        bool ok = true;
        int since = 0, q = 0;  // stages of the chain so far; the chain
        for (int i = 0; i < ks && ok;) {
            if (since == ch) {
                since = 0;
                ++q;
                if constexpr (U::NA == 1) {
                    // The high parts start a new chain in the one accumulator:
                    // two stages' middle and low parts' products first, which
                    // run while the epilogue warps read the old chain.
                    u_commit(sum_full);
                    const int n = min(ks - i, min(ch, 2));
                    for (int k = 0; k < n && ok; ++k) {
                        ok = landed(i + k);
#pragma unroll
                        for (int kk = 0; kk < kUKStage / 16 && ok; ++kk) {
                            mma((i + k) % U::ST, kk, 1, 0, false);
                            mma((i + k) % U::ST, kk, 2, 0, false);
                        }
                    }
                    if (ok && !u_mb_wait(sum_empty, (q - 1) & 1, everr)) {
                        atomicOr(err, kErrStall);
                        ok = false;
                    }
                    if (!ok) break;
                    u_fence_after();
                    for (int k = 0; k < n; ++k) {
#pragma unroll
                        for (int kk = 0; kk < kUKStage / 16; ++kk) mma((i + k) % U::ST, kk, 0, 0, k == 0 && kk == 0);
                        u_commit(&empty[(i + k) % U::ST]);
                    }
                    i += n;
                    since = n;
                    continue;
                }
            }
            ok = landed(i);
            if (!ok) break;
#pragma unroll
            for (int kk = 0; kk < kUKStage / 16; ++kk)
#pragma unroll
                for (int pp = 0; pp < 3; ++pp)
                    mma(i % U::ST, kk, pp, U::NA == 1 ? 0 : q, kk == 0 && (pp ? i == 0 && pp == 1 : since == 0));
            u_commit(&empty[i % U::ST]);
            ++i;
            ++since;
        }
        u_commit(done);  // after every MMA this thread issued
    }
    __syncwarp();
    if (w < U::EW) {
        // epilogue: a thread is one weight row (tensor-memory lane) and half of
        // the block's rows (accumulator columns)
        constexpr int HC = U::HC;
        const int col0 = (w >> 2) * HC, tile = tile0 + (w & 3);
        const uint32_t lane_addr = tmem + ((uint32_t)(32 * (w & 3)) << 16) + col0;
        float sum[U::NA == 1 ? HC : 1];
        if constexpr (U::NA == 1) {
#pragma unroll
            for (int i = 0; i < HC; ++i) sum[i] = 0.f;
            for (int f = 0; f < (ks - 1) / ch; ++f) {
                if (!u_mb_wait(sum_full, f & 1, everr)) {
                    atomicOr(err, kErrStall);
                    break;
                }
                u_fence_after();
                __syncwarp();
#pragma unroll
                for (int c = 0; c < HC; c += 32)
                    if (col0 + c < M) {
                        uint32_t v0[16], v1[16];
                        u_ld16(lane_addr + c, v0);
                        u_ld16(lane_addr + c + 16, v1);
                        u_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            sum[c + i] += __uint_as_float(v0[i]);
                            sum[c + 16 + i] += __uint_as_float(v1[i]);
                        }
                    }
                u_fence_before();
                __syncwarp();
                if (lane == 0) u_mb_arrive(sum_empty);
            }
        }
        bool have = u_mb_wait(done, 0, nullptr);  // the MMA thread commits done after every wait of its own
        if (!have) have = u_mb_wait(done, 0, nullptr);
        u_fence_after();
        // the tensor-memory loads are warp-wide: the whole warp reads or none of it
        if (__all_sync(0xffffffffu, have && ks > 0 && !(*everr & kErrStall))) {
            const int n = tile * 32 + lane;  // output row of the projection
            float* ps = part + ((int64_t)s * M_all + row0 + col0) * Np;
#pragma unroll
            for (int c = 0; c < HC; c += 16)
                if (col0 + c < M) {
                    float t[16];
                    if constexpr (U::NA == 1) {
                        uint32_t hi[16], lo[16];
                        u_ld16(lane_addr + c, hi);
                        u_wait_ld();
                        u_ld16(lane_addr + U::lo + c, lo);
                        u_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) t[i] = sum[c + i] + (__uint_as_float(hi[i]) + __uint_as_float(lo[i]));
                    } else {  // the chains that there are, then the middle and low parts
                        uint32_t v[U::NA + 1][16];
#pragma unroll
                        for (int k = 0; k < U::NA; ++k)
                            if (k * ch < ks) u_ld16(lane_addr + k * U::rows + c, v[k]);
                        u_ld16(lane_addr + U::lo + c, v[U::NA]);
                        u_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) t[i] = __uint_as_float(v[U::NA][i]);
#pragma unroll
                        for (int k = 0; k < U::NA; ++k)
                            if (k * ch < ks)
#pragma unroll
                                for (int i = 0; i < 16; ++i) t[i] += __uint_as_float(v[k][i]);
                    }
                    if (tile < n_tiles)
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (col0 + c + i < M) ps[(int64_t)(c + i) * Np + n] = t[i];
                }
        }
    }
    u_fence_before();
    __syncthreads();
    if (w == U::EW) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(U::tmem_cols) : "memory");
}

// ---------------------------------------------------------------- host side
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

bool encode_fn() {
    std::call_once(g_encode_once, [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
        cudaGetLastError();
    });
    return g_encode != nullptr;
}

// The tile-packed weights as {256 elements, tiles, 16-byte chunks} with byte
// strides {-, 64 K, 512}: the 32 rows of one tile's chunk are 512 contiguous
// bytes.  A box of {256, 4, kUKStage / 8} lands as row * 16 + chunk * 2048
// bytes (row = 32 tile + row within the tile), the canonical layout, in 512-byte
// rows of the copy.
bool weight_map(CUtensorMap* map, const uint16_t* W, int64_t n_tiles, int K) {
    if (!encode_fn() || K % 8 || ((uintptr_t)W & 15)) return false;
    const cuuint64_t dim[3] = {256, (cuuint64_t)n_tiles, (cuuint64_t)(K / 8)};
    const cuuint64_t stride[2] = {(cuuint64_t)K * 64, 512};
    const cuuint32_t box[3] = {256, 4, kUKStage / 8};
    const cuuint32_t estr[3] = {1, 1, 1};
    return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<uint16_t*>(W), dim, stride, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool small_batch(int M) { return x3_rows(M) <= USmall::rows; }

}  // namespace

bool configure_umma() {
    int dev = 0, major = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    CUtensorMap probe;
    static const uint16_t dummy[64 * 8] __attribute__((aligned(16))) = {};
    auto smem = [](auto kern, size_t bytes) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
    };
    const bool ok = major == 10 && encode_fn() && weight_map(&probe, dummy, 4, 64) &&
                    smem(k_rows_umma<ULarge>, ULarge::smem) && smem(k_rows_umma<UShort>, UShort::smem) &&
                    smem(k_rows_umma<USmall>, USmall::smem) && configure_uattn() == cudaSuccess;
    cudaGetLastError();
    return ok;
}

// K splits: as many as keep the grid within one wave (one CTA per SM: the
// stages take most of the shared memory), at most one per stage.  A small batch
// (USmall) waits for latencies, not for the tensor cores: a split more shortens
// every CTA's run of stages and lengthens the sum that the next launch starts
// with, each by about the same time, so there are at most sqrt(2 stages) of
// them.  A 33-position prompt at 0.5B (21 splits of two stages or fewer became
// 7 of four, 21 of seven became 17 of nine): 1300 us before, 1254 with it
// (1244 since USmall has eight stages); 1262 with sqrt(stages) splits, 1263 with
// sqrt(4 stages).
int umma_splits(int64_t n_tiles, int K, int M, int n_sm) {
    const int64_t mt = (n_tiles + 3) / 4 * rows_blocks(M);
    const int nk = (K + kUKStage - 1) / kUKStage;
    int64_t want = std::min<int64_t>(n_sm / mt, nk);
    if (small_batch(M))
        while (want * want > 2 * nk) --want;
    return (int)std::max<int64_t>(1, want);
}

// Stages per chain.  A small batch: as many as give every chain one of its four
// accumulators (feed-forward of 33 rows against 64 bits, in chains of up to 24 and
// now: 0.5B 1.2e-6, 4.1e-7; 1.5B 2.3e-6, 9.5e-7; 33 positions at 0.5B take 1227 us
// for 1225).  A full block: 4, fewer where a split of a 256-row batch (one CTA per
// SM) would be shorter, so that short K ranges are summed no less exactly when
// larger batches leave them fewer splits (1000 rows at width 256: 3.4e-7 in
// chains of 4, 1.9e-7 now, 1.8e-7 in splits of one stage).
static int umma_chain(int64_t n_tiles, int K, int M, int S, int n_sm) {
    const int nk = (K + kUKStage - 1) / kUKStage;
    if (small_batch(M)) return ((nk + S - 1) / S + USmall::NA - 1) / USmall::NA;
    const int64_t splits = std::max<int64_t>(1, n_sm / ((n_tiles + 3) / 4));
    return (int)std::max<int64_t>(1, std::min<int64_t>(ULarge::CH, (nk + splits - 1) / splits));
}

cudaError_t launch_mm_umma(const uint16_t* W, int64_t n_rows, int K, const uint16_t* x3, int ldx, int M, int S, int n_sm,
                           float* part, int Np, int* err, cudaStream_t s) {
    const int64_t nt = tile_count(n_rows);
    CUtensorMap map;
    if (!weight_map(&map, W, nt, K)) return cudaErrorNotSupported;
    const dim3 grid((unsigned)((nt + 3) / 4), (unsigned)S, (unsigned)rows_blocks(M));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    const bool small = small_batch(M);
    const int ch = umma_chain(nt, K, M, S, n_sm);
    cfg.blockDim = dim3(small ? USmall::threads : ULarge::threads);
    cfg.dynamicSmemBytes = small ? USmall::smem : ULarge::smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (small) return cudaLaunchKernelEx(&cfg, k_rows_umma<USmall>, map, x3, ldx, (int)nt, K, M, S, ch, part, Np, err);
    if (ch < ULarge::CH) return cudaLaunchKernelEx(&cfg, k_rows_umma<UShort>, map, x3, ldx, (int)nt, K, M, S, ch, part, Np, err);
    return cudaLaunchKernelEx(&cfg, k_rows_umma<ULarge>, map, x3, ldx, (int)nt, K, M, S, ch, part, Np, err);
}

}  // namespace ee
