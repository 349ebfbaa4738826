// Surrogate network inference on the 5th-generation tensor cores: BF16 operands in shared
// memory, FP32 accumulation in tensor memory (TMEM).
//
// A pair of SMs (a cluster of two CTAs, tcgen05 in cta_group::2) stays with one ensemble
// member and takes its share of the 256-sample tiles through the layers, two at a time, in
// ping-pong: while the tensor cores run one tile's products of a layer, the other tile's
// epilogue runs on the CUDA cores; a tile's place goes on to its next tile on its own.
//  * each CTA holds 128 rows of each tile's activations in shared memory, in the no-swizzle
//    K-major layout (8 x 8 core matrices of 16-byte rows, K-adjacent core matrices 128
//    bytes apart, 8-row groups K/8 x 128 bytes apart), and half of the layer's output rows
//    of the weights: at most 64 KB, so that a whole layer is resident and both tiles use
//    it.  It streams through two 32 KB buffers in chunks of 128 of K, each one contiguous run
//    of the packed weights (chunk_off) brought by one bulk copy from the load warp as soon
//    as the products that read the buffer have completed;
//  * one thread of the pair's first CTA issues tcgen05.mma (kind::f16, M = 256, N = the
//    layer's width, 16 of K at a time) into the tile's accumulator in TMEM (128 rows x 256
//    FP32 columns in each SM; the two tiles' fill TMEM's 512 columns), releasing a weight
//    buffer with a commit to both CTAs after the second tile's products and signalling
//    both CTAs' epilogues with another after a tile's last chunk;
//  * eight warps per tile and CTA (two per TMEM lane quadrant, each half the columns) read the
//    accumulator with tcgen05.ld, add the bias, apply the tanh-GELU (hidden layers) and
//    write the next layer's BF16 operand back into the tile, or write the FP32 outputs,
//    then tell the issuing thread that the tile is ready for its next layer.
// What bounds it: the instructions of the epilogues (135 per 16 columns of 32 samples, two
// tanh passes a pair among them: about 4.2k of a layer's 8k cycles, 256 wide) and the serial
// chain of a tile (epilogue 5.2k, then its product 3k); the tensor cores are busy a third of
// the time.  5 members of 6-256x4-33, 65536 samples, a call: 267 us with one CTA per two tiles of
// 128 (a layer's weights in two halves through one buffer, so that the tiles went through a
// layer together and only their epilogues overlapped), 258 us with pairs of SMs that take
// one pair of tiles and leave, 206 us with pairs that stay, 190 us with the outputs written by
// rows.  Streaming the weights once per tile instead had run into the 64 KB in flight; twelve
// warps a tile were no faster (206 us).
// The layer-0 operand is built by the epilogue warps from the FP32 queries.  Every
// mbarrier wait is bounded (timeout counted; the block then drains what it issued and
// still frees TMEM).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstddef>

#include "pic_internal.h"

namespace pic {

namespace {
constexpr int TM = 128;       // samples per tile and CTA
constexpr int NTILE = 2;      // tiles per CTA (ping-pong)
constexpr int EPI_WARPS = 8;  // per tile: two per TMEM lane quadrant, each half the columns
constexpr int PARTS = EPI_WARPS / 4;   // column parts per lane quadrant
constexpr int CTRL_WARP = NTILE * EPI_WARPS;   // lane 0 issues the pair's products (first CTA) or
                                               // passes on that its weights landed (second)
constexpr int LOAD_WARP = CTRL_WARP + 1;       // lane 0 streams the weights
constexpr int NTH = (LOAD_WARP + 1) * 32;
constexpr int KMAX = 256;
constexpr int NMAX = 256;
constexpr int WROWS = 128;    // output rows per weight chunk at most: half a layer's
constexpr int WK = 128;       // K columns per weight chunk
constexpr int NBUF = 2;       // weight buffers
constexpr int OCOLS = 4;      // output columns staged at a time (one 16-byte load of biases)
constexpr int TMEM_COLS = 512;    // training products
constexpr int MIN_BLOCKS = 1;     // inference blocks resident per SM
constexpr int INF_TMEM = NTILE * 256;   // inference accumulators: 256 columns a tile
constexpr int BIAS_MAX = MLP_MAX_LAYERS * NMAX;
constexpr long long WAIT_LIMIT = 1LL << 22;

struct PingSmem {
    uint16_t a[NTILE][TM * KMAX];        // activations of each tile, core-matrix layout
    uint16_t w[NBUF][WROWS * WK];        // weight chunks: this CTA's output rows x 128 of K
    alignas(16) float bias[BIAS_MAX];    // every layer's bias of the member (bmember used)
    float out[NTILE * EPI_WARPS][32 * (OCOLS + 1)];   // a warp's outputs on their way to memory
    unsigned long long wfull[NBUF];      // this CTA's part of a chunk landed
    unsigned long long wpeer[NBUF];      // (first CTA) the second CTA's part landed
    unsigned long long wempty[NBUF];     // the products that read a weight buffer completed
    unsigned long long accdone[NTILE];   // a tile's products of a layer completed
    unsigned long long ready[NTILE];     // (first CTA) a tile's operand for its next layer is
                                         // written, in both CTAs
    unsigned long long bbar;             // the biases landed
    unsigned long long drain;            // every product and arrival of the pair completed
    unsigned int tmem;
};
constexpr unsigned SMEM_ALIGN = 128;   // of operand tiles and bulk-copy destinations (16 needed)
static_assert(offsetof(PingSmem, w) % SMEM_ALIGN == 0 && offsetof(PingSmem, bias) % 16 == 0,
              "bulk-copy destinations and operand tiles must stay aligned");
static_assert(sizeof(PingSmem) + SMEM_ALIGN <= 227 * 1024, "shared memory of a block");

// element offset of (row r, column k) in a core-matrix tile with kp (padded) columns
__host__ __device__ __forceinline__ int core_off(int r, int k, int kp) {
    return ((r >> 3) * (kp >> 3) * 64) + ((k >> 3) * 64) + ((r & 7) * 8) + (k & 7);
}

// element offset of weight (row r, column k) of a layer's packed np x kp weights: half h of
// the rows (the CTA's of the pair), K chunk kc (columns [WK kc, WK kc + WK)) is one
// contiguous run, in core-matrix layout with its own width, so that one bulk copy brings it
// into shared memory
__host__ __device__ __forceinline__ long long chunk_off(int r, int k, int kp, int np) {
    const int rows = np / 2, h = r / rows, kc = k / WK;
    return (long long)h * rows * kp + (long long)rows * kc * WK +
           core_off(r - h * rows, k - kc * WK, min(WK, kp - kc * WK));
}

__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
// shared-memory matrix descriptor: start address, leading (K) and stride (8-row) byte
// offsets, descriptor version 1, no swizzle
__device__ __forceinline__ unsigned long long sdesc(unsigned addr, unsigned lbo, unsigned sbo) {
    return (unsigned long long)((addr >> 4) & 0x3FFFu) |
           ((unsigned long long)((lbo >> 4) & 0x3FFFu) << 16) |
           ((unsigned long long)((sbo >> 4) & 0x3FFFu) << 32) | (1ULL << 46);
}
// instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, N and M
__device__ __forceinline__ unsigned idesc_bf16(int n, int m) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(m >> 4) << 24);
}

__device__ __forceinline__ void fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void mma_bf16(unsigned d, unsigned long long a, unsigned long long b,
                                         unsigned idesc, int accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned long long *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(smem_u32(bar)) : "memory");
}
// the same of a pair of CTAs (issued by the first one's thread): A's 256 rows and B's rows lie
// half in each CTA's shared memory at the same places, D's rows half in each TMEM
__device__ __forceinline__ void mma2_bf16(unsigned d, unsigned long long a, unsigned long long b,
                                          unsigned idesc, int accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// arrives on both CTAs' barrier (the same place in each) once the products so far are done
__device__ __forceinline__ void mma2_commit(unsigned long long *bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 "
                 "[%0], %1;" ::"r"(smem_u32(bar)), "h"((unsigned short)3) : "memory");
}
// arrives on the first CTA's barrier at this place
__device__ __forceinline__ void arrive_first(unsigned long long *bar) {
    asm volatile(
        "{\n .reg .b32 r;\n mapa.shared::cluster.u32 r, %0, 0;\n"
        " mbarrier.arrive.release.cluster.shared::cluster.b64 _, [r];\n}\n"
        ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
// 16 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(unsigned taddr, float (&v)[16]) {
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}
// 16 consecutive FP32 columns of this thread's TMEM lane, issued without waiting: the
// registers are valid after tmem_wait16 on them (which waits for every load in flight)
__device__ __forceinline__ void tmem_issue16(unsigned taddr, unsigned (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait16(unsigned (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :: "memory");
}
__device__ __forceinline__ void mbar_init(unsigned long long *b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ bool mbar_wait(unsigned long long *b, unsigned parity,
                                          long long polls = WAIT_LIMIT) {
    for (long long k = 0; k < polls; k++) {
        unsigned ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok) : "r"(smem_u32(b)), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}

// the same for a barrier that the other CTA of the pair arrives on
__device__ __forceinline__ bool mbar_wait_cluster(unsigned long long *b, unsigned parity, long long polls) {
    for (long long k = 0; k < polls; k++) {
        unsigned ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok) : "r"(smem_u32(b)), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}

// 1-D bulk copy global -> shared completing on an mbarrier (16-byte aligned, size % 16 == 0)
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes,
                                          unsigned long long *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ uint16_t bf16_bits(float x) {
    return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}
// 8 values as 8 BF16 in one 16-byte word, two per conversion (element 0 lowest)
__device__ __forceinline__ unsigned bf16x2_bits(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned *>(&h);
}
__device__ __forceinline__ uint4 pack8x2(const float *v) {
    uint4 q;
    q.x = bf16x2_bits(v[0], v[1]);
    q.y = bf16x2_bits(v[2], v[3]);
    q.z = bf16x2_bits(v[4], v[5]);
    q.w = bf16x2_bits(v[6], v[7]);
    return q;
}

// Packed pairs of FP32 (element 0 in the low half): the bias is added two columns per
// instruction on the FP32 pipes.
__device__ __forceinline__ unsigned long long f2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_split(unsigned long long r, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// tanh-GELU of a pair, returned as two BF16 (element 0 low): 0.5 z (1 + tanh(w)),
// w = z (c0 + c1 z^2), c0 = sqrt(2/pi), c1 = 0.044715 sqrt(2/pi).  z is rounded to BF16
// once and the rest runs on BF16 pairs (the hardware tanh approximation included): the
// result is the next layer's BF16 operand, and the BF16 steps add about one rounding of
// it (relative 2^-8) to the one it takes anyway.
__device__ __forceinline__ unsigned gelu2_bf16(unsigned long long z) {
    float z0, z1;
    f2_split(z, z0, z1);
    unsigned zb, u, q, w, t, h, y;
    const unsigned c1 = 0x3D123D12u;   // BF16 pair of 0.044715 sqrt(2/pi) = 0.035677
    const unsigned c0 = 0x3F4C3F4Cu;   // BF16 pair of sqrt(2/pi) = 0.79788
    const unsigned half = 0x3F003F00u; // BF16 pair of 0.5
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(zb) : "f"(z1), "f"(z0));
    asm("mul.rn.bf16x2 %0, %1, %1;" : "=r"(u) : "r"(zb));
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(q) : "r"(u), "r"(c1), "r"(c0));
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(w) : "r"(zb), "r"(q));
    asm("tanh.approx.bf16x2 %0, %1;" : "=r"(t) : "r"(w));
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(h) : "r"(zb), "r"(half));
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(y) : "r"(h), "r"(t), "r"(h));
    return y;
}

// bias, GELU and BF16 of 16 accumulator columns c .. c+15 of row erow, written as the
// next layer's operand (core-matrix layout, np columns)
__device__ __forceinline__ void gelu_chunk(const unsigned (&r)[16], const float *bias, int c,
                                           uint16_t *act, int erow, int np) {
    const ulonglong2 *bias4 = reinterpret_cast<const ulonglong2 *>(bias + c);
    unsigned p[8];
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const ulonglong2 b = bias4[j];
        p[2 * j] = gelu2_bf16(add2(f2(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1])), b.x));
        p[2 * j + 1] = gelu2_bf16(
            add2(f2(__uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3])), b.y));
    }
    *reinterpret_cast<uint4 *>(act + core_off(erow, c, np)) = make_uint4(p[0], p[1], p[2], p[3]);
    *reinterpret_cast<uint4 *>(act + core_off(erow, c + 8, np)) = make_uint4(p[4], p[5], p[6], p[7]);
}

// the first 8 of a sample's inputs that this warp's part of the columns starts with
__device__ __forceinline__ void load_x(const float *X, long long row, long long n, int k0, int cc, float (&v)[8]) {
#pragma unroll
    for (int j = 0; j < 8; j++) v[j] = row < n && cc + j < k0 ? X[row * k0 + cc + j] : 0.f;
}

// blockIdx.x: 2 z + CTA of the pair, for member z; blockIdx.y: which of the member's gridDim.y
// pairs.  Pair y takes the 256-sample tiles y, y + gridDim.y, ..., two at a time.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NTH, MIN_BLOCKS)
k_mlp_tc(const __grid_constant__ MlpTc tc, const float *X, float *Y, long long n) {
    extern __shared__ unsigned char raw[];
    const unsigned pad = (SMEM_ALIGN - (smem_u32(raw) & (SMEM_ALIGN - 1u))) & (SMEM_ALIGN - 1u);
    PingSmem &sm = *reinterpret_cast<PingSmem *>(raw + pad);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // members run fastest along x, so that the blocks resident at one time read the
    // weights of every member rather than all the same member's (the same lines)
    const int z = blockIdx.x >> 1, rank = blockIdx.x & 1;
    const long long polls = tc.wait_polls;
    const long long all = (n + 2 * TM - 1) / (2 * TM);   // tiles
    const long long mine = (all - blockIdx.y + gridDim.y - 1) / gridDim.y;   // at least one

    if (tid == 0) {
        for (int b = 0; b < NBUF; b++) {
            mbar_init(&sm.wfull[b], 1);
            mbar_init(&sm.wpeer[b], 1);
            mbar_init(&sm.wempty[b], 1);
        }
        for (int t = 0; t < NTILE; t++) {
            mbar_init(&sm.accdone[t], 1);
            mbar_init(&sm.ready[t], 2 * EPI_WARPS);
        }
        mbar_init(&sm.bbar, 1);
        mbar_init(&sm.drain, 1);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&sm.tmem)), "r"(INF_TMEM) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    cluster_sync();   // both CTAs' barriers are there before either arrives on the other's
    fence_after();
    const unsigned tmem = sm.tmem;
    bool ok = true;

    // the weight chunks, numbered through the layers: chunk c sits in buffer c % NBUF
    if (warp == LOAD_WARP) {
        // ---- weights (and once, the biases) ------------------------------------------
        if (lane == 0) {
            const unsigned bb = (unsigned)(tc.bmember * 4);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                         ::"r"(smem_u32(&sm.bbar)), "r"(bb) : "memory");
            bulk_load(sm.bias, tc.b + (long long)z * tc.bmember, bb, &sm.bbar);
            unsigned c = 0;
            for (long long s = 0; s < mine && ok; s += NTILE)
                for (int l = 0; l < tc.L && ok; l++) {
                    const int kp = tc.kp[l], rows = tc.np[l] / 2;
                    for (int k = 0; k < kp; k += WK, c++) {
                        const unsigned b = c % NBUF;
                        // the products that read this buffer NBUF chunks ago have completed
                        if (c >= NBUF && !mbar_wait_cluster(&sm.wempty[b], (c / NBUF - 1) & 1, polls)) {
                            ok = false;
                            break;
                        }
                        const unsigned wb = (unsigned)(rows * min(WK, kp - k) * 2);
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                                     ::"r"(smem_u32(&sm.wfull[b])), "r"(wb) : "memory");
                        bulk_load(sm.w[b], tc.w + (long long)z * tc.wmember + tc.woff[l] +
                                               chunk_off(rank * rows, k, kp, tc.np[l]), wb, &sm.wfull[b]);
                    }
                }
            // before the block exits, every copy issued here has landed
            for (unsigned k = c > NBUF ? c - NBUF : 0; k < c; k++)
                mbar_wait(&sm.wfull[k % NBUF], (k / NBUF) & 1);
            mbar_wait(&sm.bbar, 0);
        }
    } else if (warp == CTRL_WARP) {
        if (lane == 0 && rank == 1) {
            // ---- the second CTA: its part of each chunk has landed ---------------------------
            unsigned c = 0;
            for (long long s = 0; s < mine && ok; s += NTILE)
                for (int l = 0; l < tc.L && ok; l++)
                    for (int k = 0; k < tc.kp[l]; k += WK, c++) {
                        if (!mbar_wait(&sm.wfull[c % NBUF], (c / NBUF) & 1, polls)) {
                            ok = false;
                            break;
                        }
                        arrive_first(&sm.wpeer[c % NBUF]);
                    }
        } else if (lane == 0) {
            // ---- products of the pair ----------------------------------------------------------
            unsigned c0 = 0, pass = 0;   // the layer's first chunk; each tile's layers so far
            for (long long s = 0; s < mine && ok; s += NTILE) {
                const int tiles = (int)min((long long)NTILE, mine - s);
                const bool last_pass = s + NTILE >= mine;
                unsigned left = 0;   // chunks of this pass that are still to come
                for (int l = 0; l < tc.L; l++) left += (tc.kp[l] + WK - 1) / WK;
                for (int l = 0; l < tc.L && ok; l++, pass++) {
                    const int kp = tc.kp[l], chunks = (kp + WK - 1) / WK;
                    const unsigned sbo_a = (unsigned)kp / 8u * 128u, id = idesc_bf16(tc.np[l], 2 * TM);
                    for (int t = 0; t < tiles && ok; t++) {
                        // the tile's operand is written and its accumulator has been read
                        if (!mbar_wait_cluster(&sm.ready[t], pass & 1, polls)) {
                            ok = false;
                            break;
                        }
                        for (int kc = 0; kc < chunks; kc++) {
                            const unsigned c = c0 + kc, b = c % NBUF, parity = (c / NBUF) & 1;
                            if (!mbar_wait(&sm.wfull[b], parity, polls) ||
                                !mbar_wait_cluster(&sm.wpeer[b], parity, polls)) {
                                ok = false;
                                break;
                            }
                            fence_after();
                            const int kw = min(WK, kp - kc * WK);
                            const unsigned w0 = smem_u32(sm.w[b]), sbo_w = (unsigned)kw / 8u * 128u;
                            const unsigned a0 = smem_u32(sm.a[t]) + (unsigned)(kc * (WK / 16)) * 256u;
                            for (int kk = 0; kk < kw / 16; kk++)
                                mma2_bf16(tmem + (unsigned)(t * 256), sdesc(a0 + kk * 256u, 128u, sbo_a),
                                          sdesc(w0 + kk * 256u, 128u, sbo_w), id, kc > 0 || kk > 0);
                            // a later chunk goes into this buffer
                            if (t == tiles - 1 && (!last_pass || left > (unsigned)(kc + NBUF)))
                                mma2_commit(&sm.wempty[b]);
                        }
                        if (ok) mma2_commit(&sm.accdone[t]);
                    }
                    c0 += chunks;
                    left -= chunks;
                }
            }
            mma2_commit(&sm.drain);
        }
        // the products in flight complete before either CTA leaves
        if (lane == 0) mbar_wait_cluster(&sm.drain, 0, WAIT_LIMIT);
    } else {
        // ---- epilogues: warps 8t .. 8t+7 own tile t ----------------------------------------
        const int t = warp / EPI_WARPS, w = warp % EPI_WARPS;
        const int quad = w & 3, part = w >> 2;
        const int erow = quad * 32 + lane, k0 = tc.k[0];
        const unsigned lane_base = tmem + ((unsigned)(quad * 32) << 16) + (unsigned)(t * 256);
        uint16_t *act = sm.a[t];
        float *stage = sm.out[warp];
        unsigned pass = 0;   // the tile's layers so far
        float x[8];
        long long tile = blockIdx.y + (long long)t * gridDim.y;
        if (t < mine) load_x(X, (2 * tile + rank) * TM + erow, n, k0, part * 8, x);
        ok = __all_sync(~0u, mbar_wait(&sm.bbar, 0, polls));
        for (long long s = t; s < mine && ok; s += NTILE, tile += NTILE * gridDim.y) {
            const long long row = (2 * tile + rank) * TM + erow;
            // layer-0 operand: the two warps of a quadrant split its 32 rows' columns
            for (int cc = part * 8; cc < tc.kp[0]; cc += 8 * PARTS) {
                if (cc != part * 8) load_x(X, row, n, k0, cc, x);
                *reinterpret_cast<uint4 *>(act + core_off(erow, cc, tc.kp[0])) = pack8x2(x);
            }
            for (int l = 0; l < tc.L; l++, pass++) {
                // the operand is written and the accumulator read: the tile's layer l
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                fence_before();
                __syncwarp();
                if (lane == 0) arrive_first(&sm.ready[t]);
                const bool last = l == tc.L - 1;
                const int np = last ? tc.np[l] : tc.kp[l + 1];   // columns that are wanted
                // the next tile's first inputs are on their way during the last layer
                if (last && s + NTILE < mine)
                    load_x(X, row + NTILE * (long long)gridDim.y * 2 * TM, n, k0, part * 8, x);
                if (!__all_sync(~0u, mbar_wait_cluster(&sm.accdone[t], pass & 1, polls))) {
                    ok = false;
                    break;
                }
                fence_after();
                const float *bias = sm.bias + tc.boff[l];
                // this warp's 16-column chunks: part p of PARTS (rounded so that two parts
                // split an odd count with the larger share first)
                const int chunks = np / 16;
                const int c0 = (chunks * part + PARTS - 1) / PARTS;
                const int c1 = (chunks * (part + 1) + PARTS - 1) / PARTS;
                // hidden layer (the next chunk's TMEM load in flight ahead of its use, or 32
                // columns a load, measured no faster: four warps a scheduler hide it)
                for (int ch = last ? c1 : c0; ch < c1; ch++) {
                    unsigned r[16];
                    tmem_issue16(lane_base + (unsigned)(ch * 16), r);
                    tmem_wait16(r);
                    gelu_chunk(r, bias, ch * 16, act, erow, np);
                }
                // outputs: a sample's lie nout floats behind the last one's, so that a lane's own
                // stores took a line each (5.4 M write requests for 5 x 32768 x 33 outputs, now
                // 0.8 M); through shared memory a warp writes OCOLS consecutive columns of
                // 32 / OCOLS samples at a time (2, 4, 8 columns: 200, 195, 202 us)
                for (int ch = last ? c0 : c1; ch < c1; ch++) {
                    const int nout = tc.n[l];
                    if (ch * 16 >= nout) break;
                    float v[16];
                    tmem_ld16(lane_base + (unsigned)(ch * 16), v);
#pragma unroll
                    for (int h = 0; h < 16 / OCOLS; h++) {
                        const float4 b = *reinterpret_cast<const float4 *>(bias + ch * 16 + h * OCOLS);
                        float *put = stage + lane * (OCOLS + 1);
                        __syncwarp();
                        put[0] = v[h * OCOLS] + b.x;
                        put[1] = v[h * OCOLS + 1] + b.y;
                        put[2] = v[h * OCOLS + 2] + b.z;
                        put[3] = v[h * OCOLS + 3] + b.w;
                        __syncwarp();
                        const int r0 = lane / OCOLS, c = ch * 16 + h * OCOLS + lane % OCOLS;
                        const long long left = n - (row - lane);
                        float *y = Y + ((long long)z * n + (row - lane) + r0) * nout + c;
#pragma unroll
                        for (int r = r0; r < 32; r += 32 / OCOLS, y += (32 / OCOLS) * nout)
                            if (r < left && c < nout) *y = stage[r * (OCOLS + 1) + lane % OCOLS];
                    }
                }
            }
        }
    }
    if (!ok) atomicAdd_system(tc.err, 1u);
    __syncwarp();
    fence_before();
    __syncthreads();
    cluster_sync();   // no product reads the other CTA's memory any more, no arrival is on its way
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(INF_TMEM) : "memory");
}

// ---- products of the training path ----
// Operand packing (many blocks per product): element (r, c) of the logical R x Cc matrix at
// src[r sR + c sC] (member stride sz) -> BF16 at core_off(r, c, Cp) of an Rp x Cp tile,
// zero-padded.  The index along which the source is contiguous runs fastest.
__global__ void k_tc_pack_op(const float *src, long long sz, int sR, int sC, int R, int Cc,
                             int Rp, int Cp, uint16_t *dst, long long dz) {
    const int z = blockIdx.y;
    const float *a = src + (long long)z * sz;
    uint16_t *d = dst + (long long)z * dz;
    const bool rows_fast = sR == 1 && sC != 1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Rp * Cp; i += gridDim.x * blockDim.x) {
        const int r = rows_fast ? i % Rp : i / Cp, c = rows_fast ? i / Rp : i % Cp;
        d[core_off(r, c, Cp)] =
            bf16_bits(r < R && c < Cc ? a[(long long)r * sR + (long long)c * sC] : 0.f);
    }
}

struct GemmSmem {
    uint16_t a[TM * KMAX];     // 128 rows of A, core-matrix layout
    uint16_t b[NMAX * KMAX];   // all of B
    unsigned long long mbar;   // products done
    unsigned long long lbar;   // operands landed
    unsigned int tmem;
};

struct TcGemmDev {
    const uint16_t *A, *B;     // packed operands
    long long sA, sB;          // their member strides (elements)
    float *C;
    long long sC;
    int ldc, M, N, Kp, Np, accumulate;
    unsigned int *err;
};

// One CTA: rows [128 x, 128 x + 128) of member y.  One thread brings both packed operands
// in with bulk copies and issues the products into TMEM; the four warps read their lane
// quadrants and write (or add to) C.
__global__ void __launch_bounds__(TM, 1) k_tc_gemm(TcGemmDev g) {
    extern __shared__ unsigned char raw[];
    const unsigned pad = (1024u - (smem_u32(raw) & 1023u)) & 1023u;
    GemmSmem &sm = *reinterpret_cast<GemmSmem *>(raw + pad);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int z = blockIdx.y, m0 = blockIdx.x * TM;
    if (tid == 0) {
        mbar_init(&sm.mbar, 1);
        mbar_init(&sm.lbar, 1);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&sm.tmem)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned tmem = sm.tmem;
    if (tid == 0) {
        const unsigned ab = (unsigned)(TM * g.Kp * 2), bb = (unsigned)(g.Np * g.Kp * 2);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                     ::"r"(smem_u32(&sm.lbar)), "r"(ab + bb) : "memory");
        bulk_load(sm.a, g.A + (long long)z * g.sA + (long long)m0 * g.Kp, ab, &sm.lbar);
        bulk_load(sm.b, g.B + (long long)z * g.sB, bb, &sm.lbar);
    }
    bool ok = __syncthreads_and(mbar_wait(&sm.lbar, 0u));
    if (ok) {
        if (tid == 0) {
            fence_after();
            const unsigned a0 = smem_u32(sm.a), b0 = smem_u32(sm.b);
            const unsigned sbo = (unsigned)g.Kp / 8u * 128u;
            const unsigned id = idesc_bf16(g.Np, TM);
            for (int kk = 0; kk < g.Kp / 16; kk++)
                mma_bf16(tmem, sdesc(a0 + kk * 256u, 128u, sbo), sdesc(b0 + kk * 256u, 128u, sbo),
                         id, kk > 0);
            mma_commit(&sm.mbar);
        }
        ok = __syncthreads_and(mbar_wait(&sm.mbar, 0u));
    }
    if (ok) {
        fence_after();
        const int m = m0 + warp * 32 + lane;
        float *c = g.C + (long long)z * g.sC + (long long)m * g.ldc;
        for (int c0 = 0; c0 < g.Np; c0 += 16) {
            float v[16];
            tmem_ld16(tmem + ((unsigned)(warp * 32) << 16) + (unsigned)c0, v);
            if (m < g.M) {
#pragma unroll
                for (int j = 0; j < 16; j++)
                    if (c0 + j < g.N) c[c0 + j] = g.accumulate ? c[c0 + j] + v[j] : v[j];
            }
        }
    } else {
        // a wait gave up: count it, give the copies and products in flight one more bounded
        // wait, free TMEM below
        if (tid == 0) {
            atomicAdd(g.err, 1u);
            mbar_wait(&sm.lbar, 0u);
            mbar_wait(&sm.mbar, 0u);
        }
        __syncthreads();
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(TMEM_COLS) : "memory");
}

// FP32 parameters -> BF16 core-matrix weights and FP32 biases, zero-padded
struct PackArgs {
    long long woff[MLP_MAX_LAYERS], boff[MLP_MAX_LAYERS];
};
__global__ void k_mlp_pack(MlpTc tc, const float *params, long long P, PackArgs pa) {
    const int z = blockIdx.y / tc.L, l = blockIdx.y % tc.L;
    const int kp = tc.kp[l], np = tc.np[l], k = tc.k[l], nn = tc.n[l];
    const float *W = params + (long long)z * P + pa.woff[l];
    uint16_t *dst = tc.w + (long long)z * tc.wmember + tc.woff[l];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np * kp; i += gridDim.x * blockDim.x) {
        const int r = i / kp, c = i % kp;
        dst[chunk_off(r, c, kp, np)] = bf16_bits(r < nn && c < k ? W[(long long)r * k + c] : 0.f);
    }
    const float *b = params + (long long)z * P + pa.boff[l];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x)
        tc.b[(long long)z * tc.bmember + tc.boff[l] + i] = i < nn ? b[i] : 0.f;
}
}  // namespace

void mlp_tc_pack(const MlpTc &tc, const float *params, long long P, const long long *woff,
                 const long long *boff, cudaStream_t s) {
    PackArgs pa;
    for (int l = 0; l < tc.L; l++) {
        pa.woff[l] = woff[l];
        pa.boff[l] = boff[l];
    }
    k_mlp_pack<<<dim3(64, tc.E * tc.L), 256, 0, s>>>(tc, params, P, pa);
    PIC_LAUNCHED();
}

bool mlp_tc_gemm(const TcGemmOp &g, int E, uint16_t *scratch_a, uint16_t *scratch_b,
                 unsigned int *err, cudaStream_t s) {
    if (g.N < 1 || g.N > NMAX || g.K < 1 || g.K > KMAX || g.M < 1) return false;
    static bool attr[64] = {};   // the shared-memory opt-in, once per device
    const int smem = (int)sizeof(GemmSmem) + 1024;
    int dev = 0;
    cudaGetDevice(&dev);
    if (!attr[dev & 63]) {
        if (cudaFuncSetAttribute(k_tc_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
            cudaSuccess)
            return false;
        attr[dev & 63] = true;
    }
    const int Mp = (g.M + TM - 1) / TM * TM, Kp = (g.K + 15) / 16 * 16, Np = (g.N + 15) / 16 * 16;
    // A as an M x K matrix; B as the N x K matrix of its transpose (both K-major)
    k_tc_pack_op<<<dim3(64, E), 256, 0, s>>>(g.A, g.sAz, g.sAm, g.sAk, g.M, g.K, Mp, Kp,
                                             scratch_a, (long long)Mp * Kp);
    PIC_LAUNCHED();
    k_tc_pack_op<<<dim3(64, E), 256, 0, s>>>(g.B, g.sBz, g.sBn, g.sBk, g.N, g.K, Np, Kp,
                                             scratch_b, (long long)Np * Kp);
    PIC_LAUNCHED();
    const TcGemmDev d{scratch_a, scratch_b, (long long)Mp * Kp, (long long)Np * Kp, g.C, g.sCz,
                      g.ldc, g.M, g.N, Kp, Np, g.accumulate, err};
    k_tc_gemm<<<dim3((unsigned)(Mp / TM), (unsigned)E), TM, smem, s>>>(d);
    PIC_LAUNCHED();
    return true;
}

// How many pairs of SMs share a member's `tiles`, of `slots` pairs that fit at a time: the
// count with the shortest time, taken as the rounds of pairs times a pair's time, in units of
// two tiles' pass through the layers.  A single tile's pass takes about 3/4 (nothing overlaps
// its epilogues), starting and leaving about 1/4.  Against the best of some 30 counts (us a
// call, this rule / best): 5 members of 4 x 256 at 4000, 20000, 65536, 131072 rows 51 / 49, 89 / 88,
// 199 / 199, 365 / 365; 8 of 2 x 100 at the same 39 / 39, 67 / 67, 135 / 135, 241 / 241; one of 4 x 256
// 48 / 46, 51 / 49, 71 / 68, 105 / 104; 5 of 4 x 64 40 / 38, 58 / 58, 112 / 112, 195 / 193.
static unsigned pairs_per_member(long long tiles, int E, int slots) {
    long long best = 1;
    double least = 0;
    for (int rounds = 1; rounds <= 8; rounds++) {
        const long long g = std::min(std::min(tiles, 65535LL), std::max(1LL, (long long)rounds * slots / E));
        const long long m = (tiles + g - 1) / g;
        const double t = (double)((E * g + slots - 1) / slots) * ((double)(m / 2) + 0.75 * (double)(m % 2) + 0.25);
        if (rounds == 1 || t < least) {
            best = g;
            least = t;
        }
    }
    return (unsigned)best;
}

pic_status mlp_tc_forward(const MlpTc &tc, const float *X, float *Y, int64_t n, cudaStream_t s) {
    if (n <= 0) return PIC_OK;
    if (tc.bmember > BIAS_MAX) {
        set_error("pic_mlp_forward: %lld biases per member, the tensor-core path holds %d",
                  tc.bmember, BIAS_MAX);
        return PIC_ERR_ARG;
    }
    const int smem = (int)(sizeof(PingSmem) + SMEM_ALIGN);
    static bool attr[64] = {};   // the shared-memory opt-in, once per device
    int dev = 0;
    PIC_CUDA_TRY(cudaGetDevice(&dev));
    if (!attr[dev & 63]) {
        PIC_CUDA_TRY(cudaFuncSetAttribute(k_mlp_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        PIC_CUDA_TRY(cudaFuncSetAttribute(k_mlp_tc, cudaFuncAttributePreferredSharedMemoryCarveout,
                                          (int)cudaSharedmemCarveoutMaxShared));
        attr[dev & 63] = true;
    }
    int sms = 0;
    PIC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const unsigned ny = pairs_per_member((n + 2 * TM - 1) / (2 * TM), tc.E, std::max(1, sms / 2));
    k_mlp_tc<<<dim3((unsigned)(2 * tc.E), ny), NTH, smem, s>>>(tc, X, Y, (long long)n);
    PIC_LAUNCHED();
    PIC_CUDA_TRY(cudaGetLastError());
    PIC_CUDA_TRY(cudaStreamSynchronize(s));
    const unsigned int err = *static_cast<volatile unsigned int *>(tc.err);
    *tc.err = 0;
    if (err) {
        set_error("pic_mlp_forward: %u tensor-core waits timed out", err);
        return PIC_ERR_TIMEOUT;
    }
    return PIC_OK;
}

}  // namespace pic
