// Learned sphere proposer: a small MLP (3 hidden layers of 128, BF16 weights
// and activations, FP32 accumulation) trained and evaluated on the GPU with
// the library's own kernels.  The paper has no counterpart: it grows every
// sphere by sphere shrinking (Sec. 5.1); here the network proposes the
// radius of the sphere a pin will grow into, the shrinking starts from that
// proposal instead of from a radius above the mesh's extent, and the
// shrinking itself (and the exact RPD check after the insertion) decides.
//
// The dense layers are tile GEMMs on the 5th-generation tensor cores:
// D[128 x N] (TMEM, FP32) += A[128 x K] B[N x K]^T with both operands BF16 in
// shared memory, issued by one thread as tcgen05.mma kind::f16 (M = 128,
// K = 16 per instruction), completion signalled through an mbarrier by
// tcgen05.commit, the accumulator read back by tcgen05.ld.  Operands are in
// the canonical no-swizzle K-major layout: 8 rows x 16 bytes per core matrix,
// core matrices consecutive along K (leading byte offset 128) and rows of core
// matrices K * 2 bytes x 8 apart (stride byte offset).
//
// One kernel (k_mlp_step) takes a 128-row tile through the whole network,
// forward and backward, without leaving the SM: see its comment.
#include <cuda_runtime.h>
#include <math.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "internal.cuh"
#include "prim.cuh"

namespace {

inline unsigned nblk(long long n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr int TM = 128;                 // rows of a tile (tcgen05 M)
constexpr int STEP_THREADS = 256;       // 8 warps: two per 32 TMEM lanes, each takes half of the columns
constexpr int MAX_CTAS = 152;           // one per SM
constexpr long long MBAR_SPIN_LIMIT = 1ll << 24;

// ----------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor: no swizzle, K-major.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);            // start address, bits 0-13
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;        // leading byte offset, bits 16-29
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;        // stride byte offset, bits 32-45
    d |= (uint64_t)1 << 46;                              // descriptor version 1
    return d;                                            // base offset 0, layout SWIZZLE_NONE (0)
}

// Instruction descriptor of kind::f16: D FP32, A and B BF16, both K-major.
__device__ __forceinline__ uint32_t instr_desc(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Bounded wait for phase `phase` of the barrier; false when the bound ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase) {
    const uint32_t a = smem_u32(bar);
    for (long long it = 0; it < MBAR_SPIN_LIMIT; it++) {
        uint32_t done = 0;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(a), "r"(phase)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, int ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, int ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, int acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void fence_before_sync() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after_sync() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// 32 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 32; k++) v[k] = __uint_as_float(r[k]);
}

// Byte offset of element (row, k) in a no-swizzle K-major tile of kdim
// columns: core matrix (row / 8, k / 8) at ((row / 8) * (kdim / 8) + k / 8)
// * 128, row % 8 at 16-byte steps, k % 8 at 2-byte steps.
__device__ __forceinline__ uint32_t tile_off(int row, int k, int kdim) {
    return (uint32_t)((((row >> 3) * (kdim >> 3) + (k >> 3)) << 7) + ((row & 7) << 4) + ((k & 7) << 1));
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

constexpr int HID = 128;   // hidden width
constexpr int NIN = 32;    // padded input width
// parameter offsets in the FP32 master vector
constexpr long long OW0 = 0, OB0 = OW0 + HID * NIN, OW1 = OB0 + HID, OB1 = OW1 + HID * HID, OW2 = OB1 + HID,
                    OB2 = OW2 + HID * HID, OW3 = OB2 + HID, OB3 = OW3 + HID, NPARAM = OB3 + 1;
constexpr int PSTRIDE = 37440;   // floats of one CTA's partial gradient: NPARAM, the loss at NPARAM, padding
// BF16 copies of the weights as tile images (K-major, no swizzle): W0 [n][k],
// W1, W2 [n][k], and W1, W2 transposed [k][n] for the input gradients
constexpr int IW0 = 0, IW1 = IW0 + HID * NIN, IW2 = IW1 + HID * HID, IW1T = IW2 + HID * HID, IW2T = IW1T + HID * HID,
              NIMG = IW2T + HID * HID;

// Shared memory of one CTA (one per SM): 222 KB.
// A transposed tile has the core matrices of a column block of eight rows next
// to each other and the blocks TR_LBO bytes apart: the lanes of a warp hold
// consecutive columns, and this stride spreads their eight-column blocks over
// the banks (consecutive core matrices along K put them all on the same eight:
// four-way conflicts on every transposed store, 11k a CTA; the whole kernel has
// 870 in 14.4k wavefronts now).
constexpr uint32_t TR_LBO = 16 * 128 + 32;
constexpr int TR_ELEMS = 16 * (int)TR_LBO / 2;
struct StepSmem {
    union {
        __nv_bfloat16 x[TM * NIN];             // the tile's inputs by row, for the first GEMM only
        uint32_t mask[3][2][STEP_THREADS];     // then ReLU masks by layer, 32 columns a word
    };
    __nv_bfloat16 xt[NIN * TM];                // inputs transposed
    __nv_bfloat16 w0[HID * NIN];
    __nv_bfloat16 wa[HID * HID], wb[HID * HID];   // W1 then W2^T; W2 then W1^T
    __nv_bfloat16 row[TM * HID];                  // the A operand: H0, H1, dZ2, dZ1 by row
    __nv_bfloat16 h0t[TR_ELEMS], h1t[TR_ELEMS];   // transposed activations (weight gradients' B operand)
    __nv_bfloat16 zt[TR_ELEMS];                   // H2, then dZ2, dZ1, dZ0, transposed (their A operand)
    float bias[3][HID], w3[HID], dy[TM], red[HID], lred[4];
    uint64_t bar;
    uint32_t tmem;
};

// 16-byte chunks of a tile image into shared memory (its own commit group).
__device__ __forceinline__ void load_image(__nv_bfloat16* dst, const __nv_bfloat16* __restrict__ src, int n) {
    for (int c = threadIdx.x; c < n / 8; c += STEP_THREADS) cp_async16(dst + 8 * c, src + 8 * c);
    cp_async_commit();
}

__device__ __forceinline__ char* at(__nv_bfloat16* base, int row, int k, int kdim) {
    return reinterpret_cast<char*>(base) + tile_off(row, k, kdim);
}

__device__ __forceinline__ char* at_tr(__nv_bfloat16* base, int row, int k) {
    return reinterpret_cast<char*>(base) + (uint32_t)(k >> 3) * TR_LBO + (uint32_t)((row >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// 32 values of one tile row m, columns c0..c0+31, as BF16: by row (when row
// is not NULL) and transposed.  The transposed stores pair the lanes of two
// neighbouring rows into 32-bit words.
__device__ __forceinline__ void put_tile(__nv_bfloat16* row, __nv_bfloat16* tr, int m, int c0,
                                         const __nv_bfloat16 (&o)[32]) {
    if (row) {
#pragma unroll
        for (int q = 0; q < 4; q++)
            *reinterpret_cast<uint4*>(at(row, m, c0 + 8 * q, HID)) = reinterpret_cast<const uint4*>(o)[q];
    }
    const uint32_t* w = reinterpret_cast<const uint32_t*>(o);
    const int odd = m & 1;
#pragma unroll
    for (int q = 0; q < 16; q++) {   // columns c0 + 2q (even lane's) and c0 + 2q + 1 (odd lane's)
        const uint32_t other = __shfl_xor_sync(0xffffffffu, w[q], 1);
        const uint32_t v = odd ? __byte_perm(w[q], other, 0x3276) : __byte_perm(w[q], other, 0x5410);
        *reinterpret_cast<uint32_t*>(at_tr(tr, c0 + 2 * q + odd, m & ~1)) = v;
    }
}

// The network on 128-row tiles, one CTA of 8 warps per SM, tiles strided over
// the grid.  Forward: three GEMMs, each followed by an epilogue that adds the
// bias, applies ReLU and writes the BF16 activations back to shared memory,
// by row (the next GEMM's A operand) and, with GRAD, transposed (the weight
// gradient's B operand).  The head (w3, b3) runs on the CUDA cores.  Backward:
// dZ2 from the head's gradient and the ReLU mask; then per layer one batch of
// MMAs computes the tile's weight gradient, in an accumulator of its own, and the
// input gradient, whose epilogue masks it into the next dZ.  Every CTA adds
// its tiles' weight gradients up in its own partial gradient, which k_adam sums
// in order: no atomics.
//
// What bounds it: latency.  A training batch of 8192 rows is 64 tiles, one per
// SM: eight dependent MMA batches of about 0.1 us each and as many epilogues
// through shared memory.  The form before this one ran a kernel per layer and
// direction with global round trips in between and one FP32 atomic per weight
// and tile: 206 us per step of 8192 rows, 17 launches; now 24 us and 2.  Of the
// shared memory wavefronts of this kernel half were bank conflicts before the
// transposed tiles were padded (TR_LBO), and the partial gradients went out one
// line per lane: 25.0 us then, 20.6 us now, 100 steps of 8192 rows 3.29 -> 2.90 ms (2.43 with
// the launches overlapped, launch_step).
//
// Rows past n (the last tile's) have zero activations and dy = 0.
// x rows: row r of the pass is row (cur[0] + r) mod n_total of the data when
// cur is given, else row r.
template <bool GRAD>
__global__ void __launch_bounds__(STEP_THREADS, 1)
    k_mlp_step(const float* __restrict__ x, const float* __restrict__ t, long long n, int n_in, long long n_total,
               long long* cur, const float* p, const __nv_bfloat16* img, float* __restrict__ y, float* part, int* err) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    StepSmem& S = *reinterpret_cast<StepSmem*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int quad = warp & 3, half = warp >> 2;   // TMEM lanes 32 quad.., columns 64 half..
    const int m = 32 * quad + lane;                // this thread's row of the tile
    const uint32_t D = 0, DW2 = 128, DW1 = 256, DW0 = 384;   // TMEM columns
    const uint32_t tlane = (uint32_t)(32 * quad) << 16;
    if (warp == 0) tmem_alloc(&S.tmem, 512);
    if (tid == 0) mbar_init(&S.bar, 1);
    // In a training run the launches overlap (launch_step): the next k_adam may
    // become resident now, and this CTA waits for the last one to end before it
    // reads or writes anything.  No pointer to what either of the two kernels
    // writes (cur, p, img, part, err here; in k_adam also g, m, v and loss) may
    // carry __restrict__: it would allow loads and stores to be moved above the
    // wait.
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    const long long base = cur ? cur[0] : 0;
    load_image(S.w0, img + IW0, HID * NIN);
    for (int k = tid; k < HID; k += STEP_THREADS) {
        S.bias[0][k] = p[OB0 + k];
        S.bias[1][k] = p[OB1 + k];
        S.bias[2][k] = p[OB2 + k];
        S.w3[k] = p[OW3 + k];
    }
    const float b3 = p[OB3];
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t T0 = S.tmem;
    uint32_t phase = 0;
    bool ok = true;
    // staged operands visible to the tensor cores, then one thread issues
    auto begin_mma = [&]() {
        fence_proxy_async();
        fence_before_sync();
        __syncthreads();
        fence_after_sync();
    };
    // operands by row (consecutive core matrices along K), or transposed (tr)
    auto issue = [&](uint32_t d, __nv_bfloat16* a, bool a_tr, __nv_bfloat16* b, bool b_tr, int K, int N) {
        const uint32_t idesc = instr_desc(TM, N), a0 = smem_u32(a), b0 = smem_u32(b);
        const uint32_t al = a_tr ? TR_LBO : 128u, as = a_tr ? 128u : 16u * K;
        const uint32_t bl = b_tr ? TR_LBO : 128u, bs = b_tr ? 128u : 16u * K;
        for (int j = 0; j < K / 16; j++)
            mma_bf16(T0 + d, smem_desc(a0 + 2u * al * j, al, as), smem_desc(b0 + 2u * bl * j, bl, bs), idesc,
                     j > 0);
    };
    auto end_mma = [&]() {   // every thread waits for the committed MMAs; uniform over the CTA
        const bool done = mbar_wait(&S.bar, phase);
        phase ^= 1;
        ok = __syncthreads_and(done) && ok;
        fence_after_sync();
    };
    float gw3 = 0.0f, gb[3] = {0.0f, 0.0f, 0.0f}, gb3 = 0.0f, lsum = 0.0f;   // column sums of this thread's half rows
    // sum over 64 rows (this half's) of row `col` of zt, optionally weighted by dy
    auto col_sum = [&](bool weighted) {
        const int col = tid & 127, r0 = 64 * (tid >> 7);
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const uint4 v = *reinterpret_cast<const uint4*>(at_tr(S.zt, col, r0 + 8 * q));
            const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
            for (int z = 0; z < 4; z++) {
                const float2 f = __bfloat1622float2(h[z]);
                if (weighted) {
                    s += __fmul_rn(f.x, S.dy[r0 + 8 * q + 2 * z]);
                    s += __fmul_rn(f.y, S.dy[r0 + 8 * q + 2 * z + 1]);
                } else {
                    s += f.x + f.y;
                }
            }
        }
        return s;
    };
    // The tile's weight gradients into this CTA's partial gradient, which the
    // first tile sets.  FP32 additions, not more MMAs into the same accumulators:
    // those round towards zero, and over the 103 tiles of a CTA at 2 M rows left
    // W0's gradient 2.2e-5 off in norm (1.8e-6 so, 2.7e-6 with FP32 atomics; 1.33 ->
    // 2.21 ms a step there, nothing where a CTA has one tile).  Through shared
    // memory: a lane holds a row, so stores straight from the accumulators would
    // touch 32 lines each.
    auto add_weights = [&](bool set) {
        constexpr int LD = HID + 4;
        float* stage = reinterpret_cast<float*>(S.wa);   // wa, wb and row are free now
        static_assert(TM * LD * sizeof(float) <= 3 * sizeof(S.wa), "stage");
        float* g = part + (long long)blockIdx.x * PSTRIDE;
#pragma unroll 1
        for (int layer = 0; layer < 3; layer++) {
            const int K = layer == 0 ? NIN : HID;
            const uint32_t d = layer == 0 ? DW0 : (layer == 1 ? DW1 : DW2);
            float4* gw = reinterpret_cast<float4*>(g + (layer == 0 ? OW0 : (layer == 1 ? OW1 : OW2)));
#pragma unroll 1
            for (int c = 0; c < 2; c++) {
                const int c0 = K == HID ? 64 * half + 32 * c : 0;
                if (K == NIN && (half || c)) continue;   // warp-uniform
                float v[32];
                tmem_ld32(T0 + d + tlane + (uint32_t)c0, v);
#pragma unroll
                for (int q = 0; q < 8; q++)
                    *reinterpret_cast<float4*>(stage + m * LD + c0 + 4 * q) =
                        make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
            __syncthreads();
            const int per = K / 4;   // 16-byte words a row
            for (int i = tid; i < HID * per; i += STEP_THREADS) {
                float4 w = *reinterpret_cast<const float4*>(stage + (i / per) * LD + 4 * (i % per));
                if (!set) {   // (the same thread's word of the last tile)
                    const float4 o = gw[i];
                    w = make_float4(o.x + w.x, o.y + w.y, o.z + w.z, o.w + w.w);
                }
                gw[i] = w;
            }
            __syncthreads();
        }
    };
    const long long ntile = (n + TM - 1) / TM;
    for (long long tile = blockIdx.x; tile < ntile && ok; tile += gridDim.x) {
        const long long m0 = tile * TM;
        load_image(S.wa, img + IW1, HID * HID);
        load_image(S.wb, img + IW2, HID * HID);
        // inputs: two threads per row, 16 columns each
        {
            const int r = tid >> 1, c0 = 16 * (tid & 1);
            const bool in = m0 + r < n;
            long long src = m0 + r;
            if (cur && in) src = (base + src) % n_total;
            __align__(16) __nv_bfloat16 o[16];
#pragma unroll
            for (int k = 0; k < 16; k++)
                o[k] = __float2bfloat16(in && c0 + k < n_in ? x[src * n_in + c0 + k] : 0.0f);
#pragma unroll
            for (int q = 0; q < 2; q++)
                *reinterpret_cast<uint4*>(at(S.x, r, c0 + 8 * q, NIN)) = reinterpret_cast<const uint4*>(o)[q];
            if (GRAD)
#pragma unroll
                for (int k = 0; k < 16; k++) *reinterpret_cast<__nv_bfloat16*>(at(S.xt, c0 + k, r, TM)) = o[k];
        }
        const bool live = m0 + m < n;
        cp_async_wait<2>();   // W0 (first tile)
        begin_mma();
        if (tid == 0) {
            issue(D, S.x, false, S.w0, false, NIN, HID);
            mma_commit(&S.bar);
        }
        end_mma();
        // hidden layers 0 and 1: bias, ReLU, BF16 (the loops over layers and
        // column halves stay rolled: 137 registers instead of 255, same time)
#pragma unroll 1
        for (int layer = 0; layer < 2; layer++) {
#pragma unroll 1
            for (int c = 0; c < 2; c++) {
                const int c0 = 64 * half + 32 * c;
                float v[32];
                tmem_ld32(T0 + D + tlane + (uint32_t)c0, v);
                __align__(16) __nv_bfloat16 o[32];
                uint32_t mk = 0;
#pragma unroll
                for (int k = 0; k < 32; k++) {
                    o[k] = __float2bfloat16(live ? fmaxf(v[k] + S.bias[layer][c0 + k], 0.0f) : 0.0f);
                    mk |= (__bfloat162float(o[k]) > 0.0f ? 1u : 0u) << k;
                }
                S.mask[layer][c][tid] = mk;
                if (GRAD) {
                    put_tile(S.row, layer == 0 ? S.h0t : S.h1t, m, c0, o);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; q++)
                        *reinterpret_cast<uint4*>(at(S.row, m, c0 + 8 * q, HID)) = reinterpret_cast<const uint4*>(o)[q];
                }
            }
            if (layer == 0) cp_async_wait<1>();   // W1
            else cp_async_wait<0>();              // W2 (and whatever was loaded behind it)
            begin_mma();
            if (tid == 0) {
                issue(D, S.row, false, layer == 0 ? S.wa : S.wb, false, HID, HID);
                mma_commit(&S.bar);
            }
            end_mma();
        }
        if (GRAD) load_image(S.wa, img + IW2T, HID * HID);   // W1 has been consumed
        // layer 2 and the head: the products with w3 in groups of four columns,
        // by row in the place of the consumed A operand, then added across the
        // groups 16, 8, 4, 2 and 1 apart.  The order is part of the result: dy's
        // last bit decides how dZ2 rounds to BF16, and another order moved the
        // gradients by 4e-5 in norm, where their own FP32 sums are good to 2e-7
        float* heads = reinterpret_cast<float*>(S.row);   // [32 groups][TM]
        static_assert(32 * TM * sizeof(float) <= sizeof(S.row), "heads");
#pragma unroll 1
        for (int c = 0; c < 2; c++) {
            const int c0 = 64 * half + 32 * c;
            float v[32];
            tmem_ld32(T0 + D + tlane + (uint32_t)c0, v);
            __align__(16) __nv_bfloat16 o[32];
            uint32_t mk = 0;
#pragma unroll
            for (int k = 0; k < 32; k++) {
                o[k] = __float2bfloat16(live ? fmaxf(v[k] + S.bias[2][c0 + k], 0.0f) : 0.0f);
                v[k] = __bfloat162float(o[k]);
                mk |= (v[k] > 0.0f ? 1u : 0u) << k;
            }
#pragma unroll
            for (int q = 0; q < 8; q++) {
                float s = __fmul_rn(v[4 * q], S.w3[c0 + 4 * q]);
#pragma unroll
                for (int z = 1; z < 4; z++) s = __fmaf_rn(v[4 * q + z], S.w3[c0 + 4 * q + z], s);
                heads[(c0 / 4 + q) * TM + m] = s;
            }
            S.mask[2][c][tid] = mk;
            if (GRAD) put_tile(nullptr, S.zt, m, c0, o);
        }
        if (GRAD) load_image(S.wb, img + IW1T, HID * HID);   // W2 has been consumed
        __syncthreads();
        if (half == 0) {
            float s[16];
#pragma unroll
            for (int q = 0; q < 16; q++) s[q] = heads[q * TM + m] + heads[(q + 16) * TM + m];
#pragma unroll
            for (int off = 8; off; off >>= 1)
#pragma unroll
                for (int q = 0; q < off; q++) s[q] += s[q + off];
            const float yr = s[0] + b3;
            if (y && live) y[m0 + m] = yr;
            if (GRAD) {
                long long src = m0 + m;
                if (cur && live) src = (base + src) % n_total;
                const float e = live ? yr - t[src] : 0.0f;
                const float d = 2.0f * e / (float)n;
                S.dy[m] = d;
                gb3 += d;
                lsum += e * e;
            }
        }
        if (!GRAD) {
            __syncthreads();   // the operands are rewritten by the next tile
            continue;
        }
        __syncthreads();
        gw3 += col_sum(true);
        const float dy = S.dy[m];
        __syncthreads();   // H2 has been read
#pragma unroll 1
        for (int c = 0; c < 2; c++) {
            const int c0 = 64 * half + 32 * c;
            const uint32_t mk = S.mask[2][c][tid];
            __align__(16) __nv_bfloat16 o[32];
#pragma unroll
            for (int k = 0; k < 32; k++) o[k] = __float2bfloat16((mk >> k) & 1u ? dy * S.w3[c0 + k] : 0.0f);
            put_tile(S.row, S.zt, m, c0, o);
        }
        // layers 2 and 1: weight gradient and input gradient in one batch
#pragma unroll 1
        for (int layer = 2; layer >= 1; layer--) {
            if (layer == 2) cp_async_wait<1>();   // W2^T
            else cp_async_wait<0>();              // W1^T
            begin_mma();
            if (tid == 0) {
                issue(D, S.row, false, layer == 2 ? S.wa : S.wb, false, HID, HID);
                issue(layer == 2 ? DW2 : DW1, S.zt, true, layer == 2 ? S.h1t : S.h0t, true, TM, HID);
                mma_commit(&S.bar);
            }
            const float cs = col_sum(false);   // beside the MMAs: both only read zt
            gb[2] += layer == 2 ? cs : 0.0f;
            gb[1] += layer == 2 ? 0.0f : cs;
            end_mma();
#pragma unroll 1
            for (int c = 0; c < 2; c++) {
                const int c0 = 64 * half + 32 * c;
                const uint32_t mk = S.mask[layer - 1][c][tid];
                float v[32];
                tmem_ld32(T0 + D + tlane + (uint32_t)c0, v);
                __align__(16) __nv_bfloat16 o[32];
#pragma unroll
                for (int k = 0; k < 32; k++) o[k] = __float2bfloat16((mk >> k) & 1u ? v[k] : 0.0f);
                put_tile(layer == 2 ? S.row : nullptr, S.zt, m, c0, o);
            }
        }
        begin_mma();
        if (tid == 0) {
            issue(DW0, S.zt, true, S.xt, false, TM, NIN);
            mma_commit(&S.bar);
        }
        gb[0] += col_sum(false);
        end_mma();
        if (ok) add_weights(blockIdx.x == tile);
    }
    cp_async_wait<0>();
    if (GRAD) {
        // the column sums of this CTA's partial gradient
        float* g = part + (long long)blockIdx.x * PSTRIDE;
        const int col = tid & 127;
        const float sums[4] = {gb[0], gb[1], gb[2], gw3};
        const long long to[4] = {OB0, OB1, OB2, OW3};
        for (int k = 0; k < 4; k++) {
            __syncthreads();
            if (tid >= 128) S.red[col] = sums[k];
            __syncthreads();
            if (tid < 128) g[to[k] + col] = sums[k] + S.red[col];
        }
        for (int off = 16; off; off >>= 1) {
            gb3 += __shfl_xor_sync(0xffffffffu, gb3, off);
            lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
        }
        __syncthreads();
        if (half == 0 && lane == 0) {
            S.red[quad] = gb3;
            S.lred[quad] = lsum;
        }
        __syncthreads();
        if (tid == 0) {
            g[OB3] = S.red[0] + S.red[1] + S.red[2] + S.red[3];
            g[NPARAM] = (S.lred[0] + S.lred[1] + S.lred[2] + S.lred[3]) / (float)n;
            // one more Adam step: read by k_adam only
            if (cur && blockIdx.x == 0) cur[1] += 1;
        }
    }
    if (!ok && tid == 0) atomicCAS(err, 0, (int)RPD_E_TIMEOUT);
    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(T0, 512);
}

// BF16 value of weight i of the master vector into its tile images.
__device__ __forceinline__ void put_weight(__nv_bfloat16* img, long long i, float w) {
    const __nv_bfloat16 b = __float2bfloat16(w);
    if (i < OB0) {
        *reinterpret_cast<__nv_bfloat16*>(at(img + IW0, (int)(i / NIN), (int)(i % NIN), NIN)) = b;
    } else if (i >= OW1 && i < OB1) {
        const int r = (int)((i - OW1) / HID), c = (int)((i - OW1) % HID);
        *reinterpret_cast<__nv_bfloat16*>(at(img + IW1, r, c, HID)) = b;
        *reinterpret_cast<__nv_bfloat16*>(at(img + IW1T, c, r, HID)) = b;
    } else if (i >= OW2 && i < OB2) {
        const int r = (int)((i - OW2) / HID), c = (int)((i - OW2) % HID);
        *reinterpret_cast<__nv_bfloat16*>(at(img + IW2, r, c, HID)) = b;
        *reinterpret_cast<__nv_bfloat16*>(at(img + IW2T, c, r, HID)) = b;
    }
}

__global__ void k_cast_weights(const float* __restrict__ p, __nv_bfloat16* __restrict__ img) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NPARAM) put_weight(img, i, p[i]);
}

// Sum of the CTAs' partial gradients for parameter i, loss at NPARAM: PGROUP
// threads each sum every PGROUP-th CTA's, then the first adds the groups' sums
// in order (only its result counts).  One thread summing all 64 waited for
// memory most of its 9.6 us (6.5 now).
constexpr int PGROUP = 8, PCOLS = 32;   // a block: 32 parameters x 8 groups
__device__ __forceinline__ float part_sum(const float* part, int np, long long i) {
    __shared__ float sums[PGROUP][PCOLS];
    const int col = threadIdx.x % PCOLS, grp = threadIdx.x / PCOLS;
    float s = 0.0f;
    if (i <= NPARAM) {
#pragma unroll 8
        for (int c = grp; c < np; c += PGROUP) s += part[(long long)c * PSTRIDE + i];
    }
    sums[grp][col] = s;
    __syncthreads();
    if (grp) return 0.0f;
    for (int g = 1; g < PGROUP; g++) s += sums[g][col];
    return s;
}
__device__ __forceinline__ long long part_param() {
    return (long long)blockIdx.x * PCOLS + threadIdx.x % PCOLS;
}

__global__ void __launch_bounds__(PGROUP* PCOLS) k_grad_sum(const float* __restrict__ part, int np,
                                                            float* __restrict__ g, float* __restrict__ loss) {
    const long long i = part_param();
    const float s = part_sum(part, np, i);
    if (threadIdx.x >= PCOLS) return;
    if (i < NPARAM) g[i] = s;
    if (i == NPARAM) *loss = s;
}

// Adam step on the FP32 master parameters: the gradient summed from the
// partials, step number cur[1] (bias corrections 1 - b^step), the BF16 tile
// images of the new weights, and the next batch's first row.
__global__ void __launch_bounds__(PGROUP* PCOLS)
    k_adam(float* p, const float* part, int np, float* g, float* m, float* v, __nv_bfloat16* img, float* loss, float lr,
           float b1, float b2, float eps, long long* cur, long long b, long long n_total) {
    cudaTriggerProgrammaticLaunchCompletion();
    // k_mlp_step's partials and cur[1], and through it the last k_adam's m, v and
    // cur[0] (no __restrict__ on any of them, see k_mlp_step)
    cudaGridDependencySynchronize();
    const long long i = part_param();
    const float gi = part_sum(part, np, i);
    if (threadIdx.x >= PCOLS) return;
    if (i == 0) cur[0] = (cur[0] + b) % n_total;   // read by k_mlp_step only
    if (i == NPARAM) *loss = gi;
    if (i >= NPARAM) return;
    const float step = (float)cur[1];
    const float c1 = 1.0f - powf(b1, step), c2 = 1.0f - powf(b2, step);
    const float mi = b1 * m[i] + (1.0f - b1) * gi, vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    g[i] = gi;
    m[i] = mi;
    v[i] = vi;
    const float w = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = w;
    put_weight(img, i, w);
}

}  // namespace

// ------------------------------------------------------------ host side
#define TRY_M(expr)                  \
    do {                             \
        rpd_status _s = (expr);      \
        if (_s != RPD_OK) return _s; \
    } while (0)

struct rpd_mlp {
    cudaStream_t stream = nullptr;
    int n_in = 0;
    char* mem = nullptr;  // one allocation for everything below
    float* p = nullptr;   // FP32 master parameters
    float* g = nullptr;   // gradient
    float* m = nullptr;   // Adam moments
    float* v = nullptr;
    __nv_bfloat16* img = nullptr;   // BF16 tile images of the hidden layers' weights
    int* err = nullptr;
    float* loss = nullptr;
    long long step = 0;
    long long* cur = nullptr;       // device: [next batch row, Adam steps taken]
    float* part = nullptr;          // partial gradients, one row per CTA
    int part_rows = 0;
};

namespace {

size_t step_smem() { return sizeof(StepSmem); }
static_assert(sizeof(StepSmem) <= 227 * 1024, "shared memory of one CTA");

int step_ctas(long long n) { return (int)std::min<long long>((n + TM - 1) / TM, MAX_CTAS); }

rpd_status ensure_part(rpd_mlp* q, long long n) {
    const int need = step_ctas(n);
    if (need <= q->part_rows) return RPD_OK;
    if (q->part) cudaFreeAsync(q->part, q->stream);
    q->part = nullptr;
    q->part_rows = 0;
    if (cudaMallocFromPoolAsync((void**)&q->part, sizeof(float) * PSTRIDE * need, library_pool(), q->stream) !=
        cudaSuccess) {
        cudaGetLastError();
        q->part = nullptr;
        return RPD_E_OOM;
    }
    q->part_rows = need;
    return RPD_OK;
}

rpd_status launch_check(rpd_mlp* q) {
    if (cudaGetLastError() != cudaSuccess) return RPD_E_CUDA;
    int e = 0;
    if (cudaMemcpyAsync(&e, q->err, sizeof(int), cudaMemcpyDeviceToHost, q->stream) != cudaSuccess ||
        cudaStreamSynchronize(q->stream) != cudaSuccess) {
        cudaGetLastError();
        return RPD_E_CUDA;
    }
    return e ? (rpd_status)e : RPD_OK;
}

// Forward, and with t backward into the partial gradients.  With n_total > 0
// the n rows are the training batch that starts at the device cursor's row of
// the n_total data rows (x and t are the whole data).
// One kernel behind the last one of the stream; with overlap its CTAs may
// become resident before that one has ended (programmatic dependent launch; the
// kernel itself waits for the end), which takes the launch gap and the prologue
// out of a run of dependent launches: 29.0 -> 24.3 us per training step.  Only for a kernel whose predecessor in the stream is one
// of these too.
template <class... P, class... A>
void launch_step(rpd_mlp* q, void (*kernel)(P...), int blocks, int threads, size_t smem, bool overlap, A... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = q->stream;
    cfg.attrs = &attr;
    cfg.numAttrs = overlap ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    note_launch();
}

void run_step(rpd_mlp* q, const float* x, const float* t, long long n, float* y, long long n_total = 0,
              bool overlap = false) {
    launch_step(q, t ? k_mlp_step<true> : k_mlp_step<false>, step_ctas(n), STEP_THREADS, step_smem(), overlap, x, t, n,
                q->n_in, n_total, n_total > 0 ? q->cur : nullptr, q->p, q->img, y, q->part, q->err);
}

void cast_weights(rpd_mlp* q) {
    k_cast_weights<<<nblk(NPARAM, 256), 256, 0, q->stream>>>(q->p, q->img);
    note_launch();
}

}  // namespace

extern "C" {

rpd_status rpd_mlp_create(int32_t n_in, uint64_t seed, void* cuda_stream, rpd_mlp** out) {
    if (!out) return RPD_E_INVALID;
    *out = nullptr;
    if (n_in < 1 || n_in > NIN) return RPD_E_INVALID;
    rpd_mlp* q = new rpd_mlp();
    q->stream = (cudaStream_t)cuda_stream;
    q->n_in = n_in;
    const int sm = (int)step_smem();
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t fb = al(sizeof(float) * NPARAM), ib = al(sizeof(__nv_bfloat16) * NIMG);
    cudaMemPool_t pool = library_pool();
    const bool ok =
        pool && cudaFuncSetAttribute(k_mlp_step<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm) == cudaSuccess &&
        cudaFuncSetAttribute(k_mlp_step<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm) == cudaSuccess &&
        cudaMallocFromPoolAsync((void**)&q->mem, 4 * fb + ib + 3 * 256, pool, q->stream) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        q->mem = nullptr;
        rpd_mlp_destroy(q);
        return RPD_E_OOM;
    }
    char* at = q->mem;
    for (float** b : {&q->p, &q->g, &q->m, &q->v}) {
        *b = (float*)at;
        at += fb;
    }
    q->img = (__nv_bfloat16*)at;
    at += ib;
    q->err = (int*)at;
    q->loss = (float*)(at + 256);
    q->cur = (long long*)(at + 512);
    // He-uniform weights from a 64-bit xorshift stream of the seed; zero biases
    std::vector<float> h(NPARAM, 0.0f);
    unsigned long long st = seed * 0x9E3779B97F4A7C15ull + 0xD1B54A32D192ED03ull;
    auto uni = [&]() {
        st ^= st << 13;
        st ^= st >> 7;
        st ^= st << 17;
        return (float)((st >> 11) * 0x1.0p-53) * 2.0f - 1.0f;
    };
    const float a0 = sqrtf(6.0f / (float)n_in), a1 = sqrtf(6.0f / HID);
    for (int r = 0; r < HID; r++)
        for (int c = 0; c < NIN; c++) h[OW0 + r * NIN + c] = c < n_in ? a0 * uni() : 0.0f;
    for (long long i = 0; i < HID * HID; i++) h[OW1 + i] = a1 * uni();
    for (long long i = 0; i < HID * HID; i++) h[OW2 + i] = a1 * uni();
    for (int k = 0; k < HID; k++) h[OW3 + k] = 0.1f * a1 * uni();
    cudaMemcpyAsync(q->p, h.data(), sizeof(float) * NPARAM, cudaMemcpyHostToDevice, q->stream);
    cudaMemsetAsync(q->m, 0, sizeof(float) * NPARAM, q->stream);
    cudaMemsetAsync(q->v, 0, sizeof(float) * NPARAM, q->stream);
    cudaMemsetAsync(q->err, 0, 3 * 256, q->stream);   // err, loss, cur
    cast_weights(q);
    const rpd_status s = launch_check(q);
    if (s != RPD_OK) {
        rpd_mlp_destroy(q);
        return s;
    }
    *out = q;
    return RPD_OK;
}

rpd_status rpd_mlp_params(rpd_mlp* q, float* d_out, int64_t cap, int64_t* n) {
    if (!q) return RPD_E_INVALID;
    if (n) *n = NPARAM;
    if (!d_out) return RPD_OK;
    if (cap < NPARAM) return RPD_E_INVALID;
    cudaMemcpyAsync(d_out, q->p, sizeof(float) * NPARAM, cudaMemcpyDeviceToDevice, q->stream);
    return launch_check(q);
}

rpd_status rpd_mlp_set_params(rpd_mlp* q, const float* d_in, int64_t n) {
    if (!q || !d_in || n != NPARAM) return RPD_E_INVALID;
    cudaMemcpyAsync(q->p, d_in, sizeof(float) * NPARAM, cudaMemcpyDeviceToDevice, q->stream);
    cast_weights(q);
    return launch_check(q);
}

rpd_status rpd_mlp_forward(rpd_mlp* q, const float* d_x, int64_t n, float* d_y) {
    if (!q || n < 0 || (n > 0 && (!d_x || !d_y))) return RPD_E_INVALID;
    if (n == 0) return RPD_OK;
    run_step(q, d_x, nullptr, n, d_y);
    return launch_check(q);
}

rpd_status rpd_mlp_grad(rpd_mlp* q, const float* d_x, const float* d_t, int64_t n, float* d_grad, float* h_loss) {
    if (!q || n < 1 || !d_x || !d_t) return RPD_E_INVALID;
    TRY_M(ensure_part(q, n));
    run_step(q, d_x, d_t, n, nullptr);
    k_grad_sum<<<nblk(NPARAM + 1, PCOLS), PGROUP * PCOLS, 0, q->stream>>>(q->part, step_ctas(n), q->g, q->loss);
    note_launch();
    if (d_grad) cudaMemcpyAsync(d_grad, q->g, sizeof(float) * NPARAM, cudaMemcpyDeviceToDevice, q->stream);
    if (h_loss) cudaMemcpyAsync(h_loss, q->loss, sizeof(float), cudaMemcpyDeviceToHost, q->stream);
    return launch_check(q);
}

rpd_status rpd_mlp_train(rpd_mlp* q, const float* d_x, const float* d_t, int64_t n, int32_t steps, int32_t batch,
                         float lr, float* h_loss) {
    if (!q || n < 1 || !d_x || !d_t || steps < 0 || batch < 1 || !(lr > 0)) return RPD_E_INVALID;
    const long long b = std::min<long long>(batch, n);
    if (steps > 0) {
        TRY_M(ensure_part(q, b));
        // consecutive batches of the (caller-shuffled) data, wrapping around:
        // the batch's rows come from the device cursor.  Two launches a step,
        // issued well ahead of the device (a step takes longer than they do).
        const long long c0[2] = {0, q->step};
        cudaMemcpyAsync(q->cur, c0, sizeof(c0), cudaMemcpyHostToDevice, q->stream);
        for (int it = 0; it < steps; it++) {
            run_step(q, d_x, d_t, b, nullptr, n, it > 0);
            launch_step(q, k_adam, nblk(NPARAM + 1, PCOLS), PGROUP * PCOLS, 0, true, q->p, q->part, step_ctas(b), q->g,
                        q->m, q->v, q->img, q->loss, lr, 0.9f, 0.999f, 1e-8f, q->cur, b, n);
        }
        q->step += steps;
    }
    if (h_loss) cudaMemcpyAsync(h_loss, q->loss, sizeof(float), cudaMemcpyDeviceToHost, q->stream);
    return launch_check(q);
}

void rpd_mlp_destroy(rpd_mlp* q) {
    if (!q) return;
    if (q->part) cudaFreeAsync(q->part, q->stream);
    if (q->mem) cudaFreeAsync(q->mem, q->stream);
    cudaStreamSynchronize(q->stream);
    cudaGetLastError();
    delete q;
}

}  // extern "C"
