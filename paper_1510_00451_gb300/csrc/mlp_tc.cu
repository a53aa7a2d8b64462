// Tensor-core (tcgen05) inference of the surrogate ensemble: one CTA runs all
// four layers of one member on a 128-row tile.  Two kernels: k_mlp_tma (TMA
// ring, used when the tensor maps can be built) and k_mlp_tc (operands staged
// by the threads; the fallback).
//
//   * operands are staged in shared memory in the canonical no-swizzle
//     K-major layout: 8-row x 16-byte core matrices, consecutive along K
//     (leading-byte offset 128 B) and SBO bytes apart along M / N;
//   * one elected thread issues tcgen05.mma (kind::f16, bfloat16 A and B,
//     FP32 accumulator in tensor memory, M = 128, K = 16 per instruction),
//     tcgen05.commit signals an mbarrier the CTA waits on (bounded);
//   * the epilogue reads the accumulator rows with tcgen05.ld (thread t of
//     warp w owns row 32 w + t), adds the bias, applies the exact-erf GELU,
//     rounds to bfloat16 and writes the next layer's A operand in shared memory.
// A wait that exceeds its iteration limit latches MLSD_ETIMEOUT, skips the rest
// of the tile, frees the tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstdint>
#include <cstring>

#include "async_copy.cuh"
#include "mlsd_internal.cuh"

namespace mlsd {
namespace {

constexpr int TM = 128;                // rows per tile (MMA M)
constexpr int KC = 64;                 // K chunk staged per round
constexpr int HMAX = 256;              // hidden width supported by this kernel
constexpr unsigned TMEM_COLS = 256;
constexpr long long kWaitClocks = 1ll << 31;   // about a second of SM clocks

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// no-swizzle K-major shared-memory matrix descriptor (sm_100 family)
__device__ __forceinline__ uint64_t mat_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;              // descriptor version for tcgen05
    return d;                            // base offset 0, swizzle none
}

// instruction descriptor: D FP32, A and B bfloat16, both K-major, M x N
__host__ __device__ constexpr uint32_t inst_desc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        :: "r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 :: "r"(mbar) : "memory");
}

// bounded wait for the mbarrier phase with the given parity; false once about
// a second of SM clocks has passed without the phase completing
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity)
{
    const long long t0 = clock64();
    for (;;) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
        if (ok) return true;
        if (clock64() - t0 > kWaitClocks) return false;
    }
}

// 32 consecutive FP32 columns of this warp's 32 TMEM lanes, one wait for all
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
          "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ float gelu_tc(float z)
{
    return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f));
}

// byte offset of element (r, k) in a no-swizzle K-major tile with K columns
__device__ __forceinline__ uint32_t cm_off(int r, int k, int K)
{
    return (uint32_t)(((r >> 3) * (K >> 3) + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// stage rows [0, R) x columns [k0, k0 + KC) of a row-major bfloat16 matrix (ld elements
// per row, rows >= rows_valid read as zero) into a core-matrix tile with K = KC
__device__ __forceinline__ void stage_chunk(unsigned char *dst, const __nv_bfloat16 *src, int R,
                                            int rows_valid, long long ld, int k0)
{
    for (int t = threadIdx.x; t < R * (KC / 8); t += blockDim.x) {
        const int r = t / (KC / 8), kc = t % (KC / 8);
        uint4 v = make_uint4(0, 0, 0, 0);
        if (r < rows_valid) v = *reinterpret_cast<const uint4 *>(src + (long long)r * ld + k0 + 8 * kc);
        *reinterpret_cast<uint4 *>(dst + cm_off(r, 8 * kc, KC)) = v;
    }
}

struct TcArgs {
    const __nv_bfloat16 *X;      // [M][640]
    long long M;
    int h, members;
    const __nv_bfloat16 *const *wb;   // per member bfloat16 parameters (layout of the ABI)
    const float *const *wf;           // per member FP32 parameters (biases are read here)
    float *out;                  // [members][M][3]
    int *status;
};

__global__ void __launch_bounds__(128, 1) k_mlp_tc(TcArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *As = smem;                        // [128][64] bf16 chunk, 16 KB
    unsigned char *Bs = As + TM * KC * 2;            // [256][64] bf16 chunk, 32 KB
    unsigned char *Hs = Bs + HMAX * KC * 2;          // [128][256] bf16 activations, 64 KB
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_slot;
    __shared__ int failed;

    const int member = blockIdx.y;
    const long long row0 = (long long)blockIdx.x * TM;
    const int rows_valid = (int)min((long long)TM, a.M - row0);
    const int h = a.h;
    const __nv_bfloat16 *wb = a.wb[member];
    const float *wf = a.wf[member];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // parameter offsets (W1 b1 W2 b2 W3 b3 W4 b4)
    const long long oW1 = 0, ob1 = oW1 + (long long)h * MLSD_SUR_IN, oW2 = ob1 + h;
    const long long ob2 = oW2 + (long long)h * h, oW3 = ob2 + h, ob3 = oW3 + (long long)h * h;
    const long long oW4 = ob3 + h, ob4 = oW4 + 3LL * h;

    if (threadIdx.x == 0) {
        failed = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&mbar)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&tmem_slot)), "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const uint32_t mb = smem_u32(&mbar);
    uint32_t phase = 0;
    const uint32_t taddr_row = tmem + ((uint32_t)(warp * 32) << 16);   // this warp's 32 lanes

    // one layer: D[128][N] = A[128][K] W^T with W [N][K] row-major in global memory.
    // a_from_h: A is the activation tile in Hs (K = h), else X chunks from global.
    auto layer = [&](bool a_from_h, int K, int N, int n_rows_w, const __nv_bfloat16 *W) -> bool {
        const uint32_t idesc = inst_desc(TM, N);
        for (int k0 = 0; k0 < K; k0 += KC) {
            if (!a_from_h) stage_chunk(As, a.X + row0 * MLSD_SUR_IN, TM, rows_valid, MLSD_SUR_IN, k0);
            stage_chunk(Bs, W, N, n_rows_w, K, k0);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (threadIdx.x == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int ks = 0; ks < KC / 16; ++ks) {
                    uint64_t da, db;
                    if (a_from_h) da = mat_desc(smem_u32(Hs + ((k0 + ks * 16) >> 3) * 128), 128, (h >> 3) * 128);
                    else da = mat_desc(smem_u32(As + ks * 2 * 128), 128, (KC >> 3) * 128);
                    db = mat_desc(smem_u32(Bs + ks * 2 * 128), 128, (KC >> 3) * 128);
                    mma_bf16(tmem, da, db, idesc, (k0 > 0 || ks > 0) ? 1u : 0u);
                }
                mma_commit(mb);
            }
            const bool ok = mbar_wait(mb, phase);
            phase ^= 1u;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (!ok) { failed = 1; }
            __syncthreads();
            if (failed) return false;
        }
        return true;
    };

    // epilogue: bias + GELU -> bfloat16 activations in Hs (K = h)
    auto epilogue_hidden = [&](const float *bias) {
        const int r = warp * 32 + lane;
        for (int c0 = 0; c0 < h; c0 += 16) {
            float v[16];
            tmem_ld16(taddr_row + (uint32_t)c0, v);
            __align__(16) __nv_bfloat16 o[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = __float2bfloat16_rn(gelu_tc(v[i] + bias[c0 + i]));
            *reinterpret_cast<uint4 *>(Hs + cm_off(r, c0, h)) = *reinterpret_cast<const uint4 *>(o);
            *reinterpret_cast<uint4 *>(Hs + cm_off(r, c0 + 8, h)) = *reinterpret_cast<const uint4 *>(o + 8);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
    };

    bool ok = layer(false, MLSD_SUR_IN, h, h, wb + oW1);
    if (ok) { epilogue_hidden(wf + ob1); ok = layer(true, h, h, h, wb + oW2); }
    if (ok) { epilogue_hidden(wf + ob2); ok = layer(true, h, h, h, wb + oW3); }
    if (ok) { epilogue_hidden(wf + ob3); ok = layer(true, h, 16, 3, wb + oW4); }
    if (ok) {
        const int r = warp * 32 + lane;
        float v[16];
        tmem_ld16(taddr_row, v);
        if (r < rows_valid) {
            float *o = a.out + ((long long)member * a.M + row0 + r) * 3;
            o[0] = v[0] + wf[ob4];
            o[1] = v[1] + wf[ob4 + 1];
            o[2] = v[2] + wf[ob4 + 2];
        }
    } else if (threadIdx.x == 0) {
        atomicCAS(a.status, 0, MLSD_ETIMEOUT);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(TMEM_COLS));
    }
}

// ---------------------------------------------------------------------------
// TMA-fed variant.  Boxes of 64 elements x rows of each row-major [rows][K] bfloat16 matrix
// arrive by cp.async.bulk.tensor with the 128-byte swizzle.
// A 3-slot ring (full / empty mbarriers) prefetches 64-wide K chunks across the
// layers while one thread issues the MMAs; the epilogue writes activations as
// K-group-major slabs of 128 x 16 bytes (conflict-free 16-byte stores), the no-swizzle K-major
// core-matrix layout, for the next layer's A operand.  9216 rows x 4 members, 256 wide:
// 65 us, 90 with core-matrix boxes (rows of 16 bytes) for all operands.
constexpr int RING = 3;
// 16 warps: warp w reads TMEM lanes 32 (w % 4) .. +31 (the lane quarter a warp may
// access) and the 32-column chunks w / 4, w / 4 + 4, ... of the layer's outputs, so the
// bias + GELU epilogue between layers runs on four times the warps of the 128 rows
// and hides more of its latency
constexpr int TMA_THREADS = 512;
constexpr int A_BYTES = TM * KC * 2;           // 16 KB
constexpr int B_BYTES = HMAX * KC * 2;         // 32 KB
constexpr int SLOT = A_BYTES + B_BYTES;

struct TmaArgs {
    CUtensorMap xmap;                          // X [M][640]
    CUtensorMap wmap[4][4];                    // [member][layer]
    long long M;
    int h, members;
    const float *const *wf;
    float *out;
    int *status;
};

__device__ __forceinline__ void expect_tx(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(mbar), "r"(bytes)
                 : "memory");
}

__global__ void __launch_bounds__(TMA_THREADS, 1) k_mlp_tma(const __grid_constant__ TmaArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    // RING x (A 16 KB | B 32 KB), on swizzle atoms
    unsigned char *ring = smem + ((1024 - (smem_u32(smem) & 1023)) & 1023);
    unsigned char *Hs = ring + RING * SLOT;              // [K/8][128][16 B] activations
    __shared__ __align__(8) uint64_t full[RING], empty[RING], accb;
    __shared__ uint32_t tmem_slot;
    __shared__ int failed;
    __shared__ float sbias[3][HMAX];                    // the hidden layers' biases

    const int member = blockIdx.y;
    const long long row0 = (long long)blockIdx.x * TM;
    const int rows_valid = (int)min((long long)TM, a.M - row0);
    const int h = a.h;
    const float *wf = a.wf[member];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long ob1 = (long long)h * MLSD_SUR_IN, ob2 = ob1 + h + (long long)h * h;
    const long long ob3 = ob2 + h + (long long)h * h, ob4 = ob3 + h + 3LL * h;

    // chunk schedule over the four layers: K chunks of 64, N rows of the weight tile
    const int nk1 = MLSD_SUR_IN / KC, nkh = h / KC;
    const int total = nk1 + 3 * nkh;
    auto layer_of = [&](int q) { return q < nk1 ? 0 : 1 + (q - nk1) / nkh; };
    auto kc_of = [&](int q) { return q < nk1 ? q : (q - nk1) % nkh; };
    auto nrows = [&](int l) { return l < 3 ? h : 16; };

    for (int i = threadIdx.x; i < 3 * h; i += blockDim.x) {
        const int l = i / h, c = i % h;
        sbias[l][c] = wf[(l == 0 ? ob1 : (l == 1 ? ob2 : ob3)) + c];
    }
    if (threadIdx.x == 0) {
        failed = 0;
        for (int i = 0; i < RING; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&full[i])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&empty[i])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&accb)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&tmem_slot)), "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const int lq = warp & 3, cgrp = warp >> 2;           // lane quarter, column group
    const uint32_t taddr_row = tmem + ((uint32_t)(lq * 32) << 16);

    auto issue_load = [&](int q) {
        const int l = layer_of(q), kc = kc_of(q), slot = q % RING;
        unsigned char *sA = ring + slot * SLOT, *sB = sA + A_BYTES;
        const uint32_t fb = smem_u32(&full[slot]);
        const int nr = nrows(l);
        expect_tx(fb, (l == 0 ? A_BYTES : 0) + nr * KC * 2);
        if (l == 0) tma_load_2d(smem_u32(sA), &a.xmap, kc * KC, (int)row0, fb);
        tma_load_2d(smem_u32(sB), &a.wmap[member][l], kc * KC, 0, fb);
    };

    uint32_t acc_phase = 0;
    bool ok = true;
    int issued = 0;                          // chunks whose loads thread 0 has issued
    if (threadIdx.x == 0)
        for (; issued < RING && issued < total; ++issued) issue_load(issued);
    int q = 0;
    for (int l = 0; l < 4 && ok; ++l) {
        const int nk = l == 0 ? nk1 : nkh;
        const int N = nrows(l);
        const uint32_t idesc = inst_desc(TM, N);
        if (threadIdx.x == 0) {
            for (int kc = 0; kc < nk && ok; ++kc, ++q) {
                const int slot = q % RING;
                if (!mbar_wait(smem_u32(&full[slot]), (uint32_t)((q / RING) & 1))) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                unsigned char *sA = ring + slot * SLOT, *sB = sA + A_BYTES;
#pragma unroll
                for (int ks = 0; ks < KC / 16; ++ks) {
                    uint64_t da, db;
                    if (l == 0) da = desc_sw128(smem_u32(sA) + ks * 32);
                    else da = mat_desc(smem_u32(Hs + ((kc * KC + ks * 16) >> 3) * (TM * 16)), TM * 16, 128);
                    db = desc_sw128(smem_u32(sB) + ks * 32);
                    mma_bf16(tmem, da, db, idesc, (kc > 0 || ks > 0) ? 1u : 0u);
                }
                mma_commit(smem_u32(&empty[slot]));
                if (kc == nk - 1) mma_commit(smem_u32(&accb));
                // refill the slot of the previous chunk once its MMAs are done
                const int qn = q - 1 + RING;
                if (q >= 1 && qn < total) {
                    const int ps = (q - 1) % RING;
                    if (!mbar_wait(smem_u32(&empty[ps]), (uint32_t)(((q - 1) / RING) & 1))) { ok = false; break; }
                    issue_load(qn);
                    issued = qn + 1;
                }
            }
            if (!ok) failed = 1;
        } else {
            q += nk;
        }
        // accumulator of layer l complete
        const bool got = mbar_wait(smem_u32(&accb), acc_phase);
        acc_phase ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!got) failed = 1;
        __syncthreads();
        if (failed) { ok = false; break; }
        const int r = lq * 32 + lane;
        if (l < 3) {
            const float *bias = sbias[l];                // staged at entry: broadcast reads
            // 32-column chunks dealt round-robin to the column groups
            for (int c0 = 32 * cgrp; c0 < h; c0 += 32 * (TMA_THREADS / 128)) {
                float v[32];
                tmem_ld32(taddr_row + (uint32_t)c0, v);
                __align__(16) __nv_bfloat16 o[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] = __float2bfloat16_rn(gelu_tc(v[i] + bias[c0 + i]));
#pragma unroll
                for (int g = 0; g < 4; ++g)
                    *reinterpret_cast<uint4 *>(Hs + ((c0 >> 3) + g) * (TM * 16) + r * 16) =
                        *reinterpret_cast<const uint4 *>(o + 8 * g);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncthreads();
        } else if (cgrp == 0) {
            float v[16];
            tmem_ld16(taddr_row, v);
            if (r < rows_valid) {
                float *o = a.out + ((long long)member * a.M + row0 + r) * 3;
                o[0] = v[0] + wf[ob4];
                o[1] = v[1] + wf[ob4 + 1];
                o[2] = v[2] + wf[ob4 + 2];
            }
        }
    }
    if (!ok && threadIdx.x == 0) {
        atomicCAS(a.status, 0, MLSD_ETIMEOUT);
        // let the copies still in flight land (bounded) before the CTA leaves
        for (int k = q; k < issued; ++k) mbar_wait(smem_u32(&full[k % RING]), (uint32_t)((k / RING) & 1));
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(TMEM_COLS));
    }
}

typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encoder()
{
    static EncodeTiled fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
    }
    return fn;
}

}  // namespace

// 2-D view of a row-major bfloat16 matrix [rows][K], rows ld elements apart, box of box_rows rows
// of 64 elements, 128-byte swizzle.  K is rounded up to 8 (the caller keeps the padding zero);
// what a box reaches past it is zero-filled.
bool encode_rows_bf16(void *map, const void *base, long long rows, long long K, long long ld,
                      int box_rows)
{
    EncodeTiled enc = encoder();
    if (!enc || ld % 8 || ld < 8 * ((K + 7) / 8)) return false;
    cuuint64_t dims[2] = {(cuuint64_t)(8 * ((K + 7) / 8)), (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return enc(static_cast<CUtensorMap *>(map), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
               const_cast<void *>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D view of a row-major [height][width] FP32 array with a box of box_h rows of
// box_w elements (zero fill outside the array)
bool encode_f32_2d(void *map, const float *base, long long width, long long height, int box_w,
                   int box_h)
{
    EncodeTiled enc = encoder();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)width, (cuuint64_t)height};
    cuuint64_t strides[1] = {(cuuint64_t)width * 4};
    cuuint32_t box[2] = {(cuuint32_t)box_w, (cuuint32_t)box_h};
    cuuint32_t es[2] = {1, 1};
    return enc(static_cast<CUtensorMap *>(map), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
               const_cast<float *>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {

// Failure-path check of mbar_wait: one thread waits on a fresh mbarrier that
// receives no arrival (no copy or MMA is in flight), so the wait expires and
// the kernel latches MLSD_ETIMEOUT the way the inference kernels do.
__global__ void k_wait_check_mbar(int *status)
{
    __shared__ __align__(8) unsigned long long bar;
    const uint32_t mb = smem_u32(&bar);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(mb) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0 && !mbar_wait(mb, 0)) atomicCAS(status, 0, MLSD_ETIMEOUT);
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" :: "r"(mb) : "memory");
}

}  // namespace

// Host: tensor maps of every member's weights; false when TMA views are unavailable.
bool mlp_tma_prepare(int h, int members, void *const *wb_host, void *maps_out)
{
    if (h % KC || h > HMAX || members > 4) return false;
    CUtensorMap *mp = static_cast<CUtensorMap *>(maps_out);     // [4][4]
    std::memset(mp, 0, sizeof(CUtensorMap) * 16);
    for (int m = 0; m < members; ++m) {
        const __nv_bfloat16 *w = static_cast<const __nv_bfloat16 *>(wb_host[m]);
        const long long oW2 = (long long)h * MLSD_SUR_IN + h, oW3 = oW2 + (long long)h * h + h;
        const long long oW4 = oW3 + (long long)h * h + h;
        if (!encode_rows_bf16(&mp[m * 4 + 0], w, h, MLSD_SUR_IN, MLSD_SUR_IN, h)) return false;
        if (!encode_rows_bf16(&mp[m * 4 + 1], w + oW2, h, h, h, h)) return false;
        if (!encode_rows_bf16(&mp[m * 4 + 2], w + oW3, h, h, h, h)) return false;
        if (!encode_rows_bf16(&mp[m * 4 + 3], w + oW4, 3, h, h, 16)) return false;
    }
    return true;
}

size_t mlp_tma_maps_bytes() { return sizeof(CUtensorMap) * 16; }

cudaError_t launch_wait_check_mbar(int *status, cudaStream_t s)
{
    count_launches(1);
    k_wait_check_mbar<<<1, 32, 0, s>>>(status);
    return cudaGetLastError();
}

cudaError_t launch_mlp_tma(const void *X, long long M, int h, int members, const void *maps,
                           const float *const *wf_dev, float *out, int *status, cudaStream_t s)
{
    TmaArgs a;
    std::memset(&a, 0, sizeof(a));
    if (!encode_rows_bf16(&a.xmap, X, M, MLSD_SUR_IN, MLSD_SUR_IN, TM)) return cudaErrorNotSupported;
    std::memcpy(a.wmap, maps, sizeof(a.wmap));
    a.M = M;
    a.h = h;
    a.members = members;
    a.wf = wf_dev;
    a.out = out;
    a.status = status;
    const size_t smem = 1024 + (size_t)RING * SLOT + (size_t)TM * HMAX * 2;
    cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(&k_mlp_tma),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((M + TM - 1) / TM), (unsigned)members);
    count_launches(1);
    k_mlp_tma<<<grid, TMA_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

size_t mlp_tc_smem() { return (size_t)TM * KC * 2 + (size_t)HMAX * KC * 2 + (size_t)TM * HMAX * 2; }

bool mlp_tc_supported(int h) { return h % 64 == 0 && h <= HMAX && h >= 64; }

cudaError_t launch_mlp_tc(const void *X, long long M, int h, int members, const void *const *wb_dev,
                          const float *const *wf_dev, float *out, int *status, cudaStream_t s)
{
    TcArgs a;
    a.X = static_cast<const __nv_bfloat16 *>(X);
    a.M = M;
    a.h = h;
    a.members = members;
    a.wb = reinterpret_cast<const __nv_bfloat16 *const *>(wb_dev);
    a.wf = wf_dev;
    a.out = out;
    a.status = status;
    const size_t smem = mlp_tc_smem();
    cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(&k_mlp_tc),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((M + TM - 1) / TM), (unsigned)members);
    count_launches(1);
    k_mlp_tc<<<grid, 128, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace mlsd
