// Surrogate networks in FP32 on CUDA cores: the layers' products with what follows each of
// them done in the product's own kernel (training, and inference on few rows), and whole
// networks in one kernel (inference on many rows).
#include <algorithm>

#include "mlp_math.h"
#include "pic_internal.h"

namespace pic {

namespace {

// =========================================================================================
// Layer products
// =========================================================================================
// C(z)[m][n] = sum_k A(z, m, k) B(z, k, n) over T x T tiles of C, one CTA a tile.  An
// operand is contiguous either along k or along its own index (m or n) and is staged as it
// lies: [index][k] or [k][index], rows padded by 4 floats, so that copies and reads are
// 16 bytes wide and free of bank conflicts in both layouts (reads take four k at a time
// from the first layout and a thread's whole row or column group from the second).
//
// At training's sizes (128 x 256 x 256 for five members) a product is 40 tiles of 64 x 64
// or 160 of 32 x 32 for 152 SMs, and what counts is the chain of the step's ten dependent
// products: 32 x 32 tiles keep every SM busy, and each launch begins while the one before
// it drains.  The eight warps of a 32 x 32 tile split k (a warp takes the whole tile, four
// of every 32 k, 8 x 4 elements a thread) and their partial sums are added in a fixed
// order: splitting the tile instead leaves each thread 2 x 2 elements, which ask 2.7 times
// the shared-memory reads (1.05M wavefronts, 6.9k of a tile's 15k cycles).  64 x 64 tiles
// (4 x 4 elements a thread, the tile split over the warps) ask half the L2 bandwidth a
// flop and take over once they fill the SMs twice (mlp_jobs).
//
// Measured, a training step of 5 x 6 -> 4 x 256 -> 33 at batch 128: 84 us in 11 launches (335 us
// in 31 with 16 x 16 tiles of one element a thread and separate bias, activation, column-sum
// and Adam kernels; 67 us with all but the weight gradients in one kernel, k_mlp_chain.cu);
// batch 256: 128 us.
constexpr int BK = 32;

template <int T>
struct Shape;
template <>
struct Shape<32> {
    // threads; a thread's elements; stages; warps along k, m, n; lanes along n
    static constexpr int NT = 256, RM = 8, RN = 4, STG = 6, WK = 8, WM = 1, WN = 1, LN = 8;
};
template <>
struct Shape<64> {
    static constexpr int NT = 256, RM = 4, RN = 4, STG = 3, WK = 1, WM = 4, WN = 2, LN = 8;
};

template <int T>
struct alignas(16) TileSmem {
    static constexpr int OPER = T * (BK + 4) > BK * (T + 4) ? T * (BK + 4) : BK * (T + 4);
    static constexpr int CLD = T + 8;    // row stride of the sums: 8 mod 32, free of conflicts
    union {
        struct {
            float a[Shape<T>::STG][OPER], b[Shape<T>::STG][OPER];
        };
        float c[Shape<T>::WK][T * CLD];  // the warps' sums, after the last stage
    };
};

// One operand's copies into its stages: BK of k by T of the operand's index, zero outside
// K x I.  KC: contiguous along k.  16 bytes at a time where base and stride allow it: each
// thread then keeps its few addresses and steps them from stage to stage.
template <int T, bool KC>
struct Operand {
    static constexpr int NT = Shape<T>::NT;
    static constexpr int FAST = KC ? BK : T, SLOW = KC ? T : BK;   // contiguous and strided extents
    static constexpr int PER = SLOW * FAST / 4 / NT;
    static_assert(SLOW * FAST / 4 % NT == 0 && NT % (FAST / 4) == 0, "whole rounds of copies");
    const float *p, *at;
    int ld, i0, I, K, s, f, vec;
    __device__ __forceinline__ Operand(const float *p_, int ld_, int i0_, int I_, int K_, int tid)
        : p(p_), ld(ld_), i0(i0_), I(I_), K(K_) {
        vec = ((size_t)p & 15) == 0 && ld % 4 == 0;
        s = tid / (FAST / 4);
        f = tid % (FAST / 4) * 4;
        at = KC ? p + (long long)(i0 + s) * ld + f : p + (long long)s * ld + i0 + f;
    }
    __device__ __forceinline__ void load(float *S, int k0, int tid) const {
        constexpr int ROWS = NT / (FAST / 4);   // strided indices a round of copies covers
        if (vec) {
            const float *src = at + (KC ? (long long)k0 : (long long)k0 * ld);
            float *dst = S + s * (FAST + 4) + f;
            const int left = KC ? K - k0 - f : I - i0 - f, slow = KC ? I - i0 - s : K - k0 - s;
            const int bytes = min(max(left * 4, 0), 16);
#pragma unroll
            for (int r = 0; r < PER; r++) {
                const int n = r * ROWS < slow ? bytes : 0;
                cp16(dst + r * ROWS * (FAST + 4), n > 0 ? src + (long long)r * ROWS * ld : p, n);
            }
        } else {
            for (int e = tid; e < SLOW * FAST; e += NT) {
                const int si = e / FAST, fi = e % FAST;
                const int k = k0 + (KC ? fi : si), i = i0 + (KC ? si : fi);
                const bool in = k < K && i < I;
                cp4(S + si * (FAST + 4) + fi,
                    in ? (KC ? p + (long long)i * ld + k : p + (long long)k * ld + i) : p, in ? 4 : 0);
            }
        }
    }
};

// R values of an operand at four consecutive k: [R][4]; the element i of a lane group g is
// base + g + G i (KC) or base + g R + i
template <int T, bool KC, int R, int G>
__device__ __forceinline__ void fetch(const float *S, int k, int base, int g, float (&v)[R][4]) {
    if constexpr (KC) {
#pragma unroll
        for (int i = 0; i < R; i++) {
            const float4 q = *reinterpret_cast<const float4 *>(S + (base + g + G * i) * (BK + 4) + k);
            v[i][0] = q.x;
            v[i][1] = q.y;
            v[i][2] = q.z;
            v[i][3] = q.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 4; j++)
#pragma unroll
            for (int h = 0; h < R; h += 4) {
                const float4 q = *reinterpret_cast<const float4 *>(S + (k + j) * (T + 4) + base + g * R + h);
                v[h][j] = q.x;
                v[h + 1][j] = q.y;
                v[h + 2][j] = q.z;
                v[h + 3][j] = q.w;
            }
    }
}

// The tile's sums into sm.c, one part per warp along k.  SUM: column sums over k of A (the
// bias gradient), one per thread below T of the first column of tiles.
template <int T, bool AKC, bool BKC, bool SUM>
__device__ __forceinline__ void product(TileSmem<T> &sm, const MlpJob &g, const float *A, const float *B,
                                        int m0, int n0, float &sum) {
    using S = Shape<T>;
    constexpr int LM = 32 / S::LN;
    constexpr int TM = T / S::WM, TN = T / S::WN;       // a warp's tile
    static_assert(LM * S::RM == TM && S::LN * S::RN == TN, "lanes cover the warp's tile");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ln = lane % S::LN, lm = lane / S::LN;
    const int wk = warp % S::WK, wm = warp / S::WK % S::WM * TM, wn = warp / S::WK / S::WM * TN;
    const int nk = (g.K + BK - 1) / BK;
    const Operand<T, AKC> oa(A, g.lda, m0, g.M, g.K, tid);
    const Operand<T, BKC> ob(B, g.ldb, n0, g.N, g.K, tid);
    auto load = [&](int kt) {
        if (kt < nk) {
            oa.load(sm.a[kt % S::STG], kt * BK, tid);
            ob.load(sm.b[kt % S::STG], kt * BK, tid);
        }
        cp_commit();
    };
    float acc[S::RM][S::RN] = {};
    for (int s = 0; s < S::STG - 1; s++) load(s);
    for (int kt = 0; kt < nk; kt++) {
        cp_wait<S::STG - 2>();
        __syncthreads();
        load(kt + S::STG - 1);
        const float *a = sm.a[kt % S::STG], *b = sm.b[kt % S::STG];
#pragma unroll
        for (int k = 0; k < BK / S::WK; k += 4) {
            float bv[S::RN][4];
            fetch<T, BKC, S::RN, S::LN>(b, wk * (BK / S::WK) + k, wn, ln, bv);
#pragma unroll
            for (int h = 0; h < S::RM; h += 4) {   // four rows at a time: fewer registers
                float av[4][4];
                // lane group lm's rows h ..: (lm + LM h) + LM i, or lm RM + h + i
                fetch<T, AKC, 4, LM>(a, wk * (BK / S::WK) + k, wm + (AKC ? LM * h : lm * (S::RM - 4) + h), lm, av);
#pragma unroll
                for (int q = 0; q < 4; q++)
#pragma unroll
                    for (int i = 0; i < 4; i++)
#pragma unroll
                        for (int j = 0; j < S::RN; j++)
                            acc[h + i][j] = fmaf(av[i][q], bv[j][q], acc[h + i][j]);
            }
        }
        if constexpr (SUM)
            if (n0 == 0 && tid < T) {
#pragma unroll
                for (int k = 0; k < BK; k++) sum += a[k * (T + 4) + tid];
            }
    }
    cp_wait<0>();
    __syncthreads();   // the stages are read: their memory takes the sums
    float *c = sm.c[wk];
#pragma unroll
    for (int i = 0; i < S::RM; i++) {
        const int m = wm + (AKC ? lm + LM * i : lm * S::RM + i);
#pragma unroll
        for (int j = 0; j < S::RN; j++) c[m * sm.CLD + wn + (BKC ? ln + S::LN * j : ln * S::RN + j)] = acc[i][j];
    }
    __syncthreads();
}

// four consecutive elements of a row, as far as it goes
__device__ __forceinline__ float4 row4(const float *p, int left, bool vec) {
    if (vec) return *reinterpret_cast<const float4 *>(p);
    return make_float4(p[0], left > 1 ? p[1] : 0.f, left > 2 ? p[2] : 0.f, left > 3 ? p[3] : 0.f);
}
__device__ __forceinline__ void put4(float *p, const float (&v)[4], int left, bool vec) {
    if (vec) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
        return;
    }
    for (int q = 0; q < 4 && q < left; q++) p[q] = v[q];
}
__device__ __forceinline__ void list4(float4 q, float (&v)[4]) {
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
}

// Two blocks an SM: three cap the registers at 80, and the spills cost a training step
// 113 us instead of 86.
template <int T>
__global__ void __launch_bounds__(Shape<T>::NT, 2) k_mlp_jobs(const __grid_constant__ MlpJobs jobs) {
    using S = Shape<T>;
    extern __shared__ __align__(16) unsigned char raw[];
    TileSmem<T> &sm = *reinterpret_cast<TileSmem<T> *>(raw);
    chain_wait();
    int j = 0, blk = blockIdx.x;
    while (j + 1 < jobs.n && blk >= jobs.blocks[j]) blk -= jobs.blocks[j++];
    const MlpJob &g = jobs.job[j];
    const int tn = (g.N + T - 1) / T, tiles = tn * ((g.M + T - 1) / T);
    const int z = blk / tiles, m0 = (blk % tiles) / tn * T, n0 = (blk % tiles) % tn * T;
    const float *A = g.A + z * g.sA, *B = g.B + z * g.sB;
    const int tid = threadIdx.x;
    const bool adam = g.epi == MLP_EPI_ADAM;
    // the epilogue's elements of a thread: four of a row, of every (T / PASS)-th row.  What
    // it reads is loaded ahead of the product for the one row of a 32 x 32 tile (loaded
    // after it, element by element, the epilogue cost as much as the product of 256 k).
    constexpr int PASS = T * T / 4 / S::NT, ROWS = T / PASS;
    const int r = tid / (T / 4), n = n0 + tid % (T / 4) * 4, left = g.N - n;
    float *C = g.C + z * g.sC, *Z = g.Z ? g.Z + z * g.sZ : nullptr;
    float *am = adam ? g.am + z * g.sC : nullptr, *av = adam ? g.av + z * g.sC : nullptr;
    const float *e = adam ? C : g.epi >= MLP_EPI_LOSS ? Z : nullptr;
    const bool whole = left >= 4 && g.ldc % 4 == 0;
    const bool vc = whole && ((size_t)C & 15) == 0, vz = whole && ((size_t)Z & 15) == 0;
    const bool ve = adam ? vc : vz;
    const bool vm = whole && ((size_t)am & 15) == 0 && ((size_t)av & 15) == 0;
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 e0 = none, e1 = none, e2 = none;
    float bias[4] = {};
    if (g.bias && left > 0)
        list4(row4(g.bias + z * g.sbias + n, left, left >= 4 && ((size_t)(g.bias + z * g.sbias) & 15) == 0), bias);
    const auto ahead = [&](int m) {
        if (m >= g.M || left <= 0) return;
        const long long at = (long long)m * g.ldc + n;
        if (e) e0 = row4(e + at, left, ve);
        if (adam) {
            e1 = row4(am + at, left, vm);
            e2 = row4(av + at, left, vm);
        }
    };
    if constexpr (PASS == 1) ahead(m0 + r);
    const bool colsum = g.kind == MLP_DW && n0 == 0 && tid < T && m0 + tid < g.M && g.db;
    const long long cs = z * g.sC + m0 + tid;
    float sum = 0.f, s0 = 0.f, s1 = 0.f, s2 = 0.f;
    if (colsum && adam) {
        s0 = g.db[cs];
        s1 = g.dbm[cs];
        s2 = g.dbv[cs];
    }
    // what an operand is contiguous along goes with the product: forward A and B along k,
    // dX = G W: A along k, B along n; dW = G^T A: both along their own index
    if (g.kind == MLP_FWD) product<T, true, true, false>(sm, g, A, B, m0, n0, sum);
    else if (g.kind == MLP_DX) product<T, true, false, false>(sm, g, A, B, m0, n0, sum);
    else product<T, false, false, true>(sm, g, A, B, m0, n0, sum);

    float lsum = 0.f;
#pragma unroll 1
    for (int p = 0; p < PASS; p++) {
        const int m = m0 + r + p * ROWS;
        if constexpr (PASS > 1) ahead(m);
        if (m >= g.M || left <= 0) continue;
        const long long at = (long long)m * g.ldc + n;
        float x[4], v[4], w[4], y[4];
        list4(*reinterpret_cast<const float4 *>(sm.c[0] + (m - m0) * sm.CLD + n - n0), x);
#pragma unroll
        for (int k = 1; k < S::WK; k++) {
            list4(*reinterpret_cast<const float4 *>(sm.c[k] + (m - m0) * sm.CLD + n - n0), v);
#pragma unroll
            for (int q = 0; q < 4; q++) x[q] += v[q];
        }
        list4(e0, v);
        if (g.epi == MLP_EPI_BIAS || g.epi == MLP_EPI_GELU) {
#pragma unroll
            for (int q = 0; q < 4; q++) x[q] += bias[q];
            if (Z) put4(Z + at, x, left, vz);
            if (g.epi == MLP_EPI_GELU)
#pragma unroll
                for (int q = 0; q < 4; q++) x[q] = gelu(x[q]);
        } else if (g.epi == MLP_EPI_LOSS) {
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float d = q < left ? (x[q] + bias[q]) - v[q] : 0.f;
                x[q] = g.scale * d;
                lsum += d * d;
            }
        } else if (g.epi == MLP_EPI_GELU_GRAD) {
#pragma unroll
            for (int q = 0; q < 4; q++) x[q] *= gelu_grad(v[q]);
        } else if (adam) {
            list4(e1, w);
            list4(e2, y);
#pragma unroll
            for (int q = 0; q < 4; q++) {
                adam_step(g.adam, x[q], v[q], w[q], y[q]);
                x[q] = v[q];
            }
            put4(am + at, w, left, vm);
            put4(av + at, y, left, vm);
        }
        put4(C + at, x, left, vc);
    }
    if (colsum) {
        if (adam) {
            adam_step(g.adam, sum, s0, s1, s2);
            g.db[cs] = s0;
            g.dbm[cs] = s1;
            g.dbv[cs] = s2;
        } else {
            g.db[cs] = sum;
        }
    }
    if (g.epi == MLP_EPI_LOSS && g.loss) {
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (tid % 32 == 0 && lsum != 0.f) atomicAdd(g.loss + z, lsum / ((float)g.M * (float)g.N));
    }
}

int sm_count() {
    static thread_local int dev_of = -1, sms = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != dev_of) {
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        dev_of = dev;
    }
    return sms > 0 ? sms : 1;
}

// =========================================================================================
// Whole networks
// =========================================================================================
// A CTA takes ROWS rows of one member through every layer; the activations stay in shared
// memory ([unit][row], 64 KB) and the weights, packed k-major (pack below), stream through
// three 16 KB stages of 16 k each.  A thread owns TR rows x 8 columns: per k it reads TR
// activations and 8 weights and issues 4 TR packed FMAs (fma.rn.f32x2: two rows an
// instruction, which leaves issue slots for the shared-memory reads).  TR follows the
// layer's width, so that a narrow output layer is spread over all threads too.  Each
// element's sum runs over k in order, as in the 64 x 64 tiles of the layer products; the
// 32 x 32 tiles add eight partial sums, so that a row's last bits depend on the path that the
// number of rows takes.
constexpr int FNT = 256;      // threads
constexpr int FK = 16;        // k a stage
constexpr int FSTG = 3;
constexpr int FW = FK * 256;  // floats a stage holds at most

template <int NW>
struct FusedSmem {
    static constexpr int ROWS = 64 * 256 / NW;
    float act[NW * ROWS];
    float w[FSTG][FW];
};

__device__ __forceinline__ unsigned long long dup2(float x) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ void fma2(unsigned long long &c, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 split2(unsigned long long x) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x));
    return r;
}

// the stream of weight stages: layer by layer, FK rows of the packed weights each
struct Stream {
    const MlpF32 *net;
    const float *w;     // the member's packed weights from here on
    int l, k;
    __device__ __forceinline__ void next(float *dst, int tid) {
        if (l < net->L) {
            const int n = FK * net->np[l];
            for (int e = tid * 4; e < n; e += FNT * 4) cp16(dst + e, w + e, 16);
            w += n;
            k += FK;
            if (k >= net->kp[l]) {
                k = 0;
                l++;
            }
        }
        cp_commit();
    }
};

template <int NW, int TR>
__device__ __forceinline__ void fused_layer(FusedSmem<NW> &sm, const MlpF32 &net, int l, int z, Stream &st,
                                            int &c, long long row0, long long n, float *Y) {
    constexpr int ROWS = FusedSmem<NW>::ROWS;
    constexpr int CG = NW * TR / 64;                  // column groups of 8
    constexpr int CPW = CG < 8 ? CG : 8, RPW = 32 / CPW;
    constexpr int WC = CG / CPW;                      // warps across the columns
    constexpr int np = CG * 8;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cg = lane % CPW, rg = (warp / WC) * RPW + lane / CPW;
    const int cb = (warp % WC) * CPW * 8 + cg * 4;    // columns cb + j, cb + 4 CPW + j
    const int r0 = rg * TR;
    unsigned long long acc[TR / 2][8];
#pragma unroll
    for (int p = 0; p < TR / 2; p++)
#pragma unroll
        for (int j = 0; j < 8; j++) acc[p][j] = 0ULL;
    for (int k0 = 0; k0 < net.kp[l]; k0 += FK, c++) {
        cp_wait<FSTG - 2>();
        __syncthreads();
        st.next(sm.w[(c + FSTG - 1) % FSTG], tid);
        const float *w = sm.w[c % FSTG] + cb;
        const float *a = sm.act + k0 * ROWS + r0;
#pragma unroll 8
        for (int k = 0; k < FK; k++) {
            unsigned long long av[TR / 2];
            if constexpr (TR >= 4) {
#pragma unroll
                for (int p = 0; p < TR / 4; p++) {
                    const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(a + k * ROWS + 4 * p);
                    av[2 * p] = q.x;
                    av[2 * p + 1] = q.y;
                }
            } else {
                av[0] = *reinterpret_cast<const unsigned long long *>(a + k * ROWS);
            }
            const float4 b0 = *reinterpret_cast<const float4 *>(w + k * np);
            const float4 b1 = *reinterpret_cast<const float4 *>(w + k * np + 4 * CPW);
            const unsigned long long bv[8] = {dup2(b0.x), dup2(b0.y), dup2(b0.z), dup2(b0.w),
                                              dup2(b1.x), dup2(b1.y), dup2(b1.z), dup2(b1.w)};
#pragma unroll
            for (int p = 0; p < TR / 2; p++)
#pragma unroll
                for (int j = 0; j < 8; j++) fma2(acc[p][j], av[p], bv[j]);
        }
    }
    const bool last = l == net.L - 1;
    const float *bias = net.b + (long long)z * net.bmember + net.boff[l];
    __syncthreads();   // every thread has read the layer's input
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const int col = cb + (j < 4 ? j : 4 * CPW + j - 4);
        const float b = __ldg(bias + col);
        if (!last) {
            const bool unit = col < net.n[l];   // padding stays zero whatever the inputs are
#pragma unroll
            for (int p = 0; p < TR / 2; p++) {
                const float2 v = split2(acc[p][j]);
                *reinterpret_cast<float2 *>(sm.act + col * ROWS + r0 + 2 * p) =
                    unit ? make_float2(gelu(v.x + b), gelu(v.y + b)) : make_float2(0.f, 0.f);
            }
        } else if (col < net.n[l]) {
#pragma unroll
            for (int p = 0; p < TR / 2; p++) {
                const float2 v = split2(acc[p][j]);
                const long long row = row0 + r0 + 2 * p;
                float *y = Y + ((long long)z * n + row) * net.n[l] + col;
                if (row < n) y[0] = v.x + b;
                if (row + 1 < n) y[net.n[l]] = v.y + b;
            }
        }
    }
}

template <int NW>
__global__ void __launch_bounds__(FNT, 2) k_mlp_fused(MlpF32 net, const float *X, float *Y, long long n) {
    extern __shared__ __align__(16) unsigned char raw[];
    FusedSmem<NW> &sm = *reinterpret_cast<FusedSmem<NW> *>(raw);
    constexpr int ROWS = FusedSmem<NW>::ROWS;
    const int tid = threadIdx.x, z = blockIdx.x % net.E;
    const long long row0 = (long long)(blockIdx.x / net.E) * ROWS;
    Stream st{&net, net.w + (long long)z * net.wmember, 0, 0};
    for (int s = 0; s < FSTG - 1; s++) st.next(sm.w[s], tid);
    const int k0 = net.k[0];
    for (int e = tid; e < net.kp[0] * ROWS; e += FNT) {
        const int k = e / ROWS, r = e % ROWS;
        sm.act[e] = k < k0 && row0 + r < n ? X[(row0 + r) * k0 + k] : 0.f;
    }
    int c = 0;
    for (int l = 0; l < net.L; l++) {
        const int np = net.np[l];
        if (np == NW) fused_layer<NW, 8>(sm, net, l, z, st, c, row0, n, Y);
        else if (np == NW / 2) fused_layer<NW, 4>(sm, net, l, z, st, c, row0, n, Y);
        else fused_layer<NW, 2>(sm, net, l, z, st, c, row0, n, Y);
    }
    cp_wait<0>();
}

// FP32 parameters -> k-major weights and biases, zero-padded to the kernel's shapes
__global__ void k_mlp_f32_pack(MlpF32 net, const float *params, long long P, MlpOffsets o) {
    const int z = blockIdx.y / net.L, l = blockIdx.y % net.L;
    const int kp = net.kp[l], np = net.np[l], k = net.k[l], nn = net.n[l];
    const float *W = params + (long long)z * P + o.w[l];
    float *dst = net.w + (long long)z * net.wmember + net.woff[l];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np * kp; i += gridDim.x * blockDim.x) {
        const int c = i % np, r = i / np;
        dst[i] = c < nn && r < k ? W[(long long)c * k + r] : 0.f;
    }
    const float *b = params + (long long)z * P + o.b[l];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x)
        net.b[(long long)z * net.bmember + net.boff[l] + i] = i < nn ? b[i] : 0.f;
}

template <int NW>
pic_status launch_fused(const MlpF32 &net, const float *X, float *Y, int64_t n, cudaStream_t s) {
    const int smem = (int)sizeof(FusedSmem<NW>);
    PIC_CUDA_TRY(cudaFuncSetAttribute(k_mlp_fused<NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const int64_t rows = FusedSmem<NW>::ROWS;
    k_mlp_fused<NW><<<(unsigned)((n + rows - 1) / rows * net.E), FNT, smem, s>>>(net, X, Y, n);
    PIC_LAUNCHED();
    PIC_CUDA_TRY(cudaGetLastError());
    return PIC_OK;
}

}  // namespace

template <int T>
static void launch_jobs(const MlpJobs &jobs, unsigned blocks, bool chain, cudaStream_t s) {
    const int smem = (int)sizeof(TileSmem<T>);
    static bool attr[64] = {};   // the shared-memory opt-in, once per device
    int dev = 0;
    cudaGetDevice(&dev);
    if (!attr[dev & 63]) {
        cudaFuncSetAttribute(k_mlp_jobs<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        attr[dev & 63] = true;
    }
    launch_chained(chain, k_mlp_jobs<T>, blocks, Shape<T>::NT, smem, s, jobs);
}

int mlp_f32_shape(int maxw, int width) {
    const int NW = maxw <= 64 ? 64 : maxw <= 128 ? 128 : 256;
    return width <= NW / 4 ? NW / 4 : width <= NW / 2 ? NW / 2 : NW;
}

void mlp_f32_pack(const MlpF32 &net, const float *params, long long P, const MlpOffsets &o,
                  cudaStream_t s) {
    k_mlp_f32_pack<<<dim3(64, net.E * net.L), 256, 0, s>>>(net, params, P, o);
    PIC_LAUNCHED();
}

pic_status mlp_f32_forward(const MlpF32 &net, const float *X, float *Y, int64_t n, cudaStream_t s) {
    if (net.NW == 64) return launch_fused<64>(net, X, Y, n, s);
    if (net.NW == 128) return launch_fused<128>(net, X, Y, n, s);
    return launch_fused<256>(net, X, Y, n, s);
}

void mlp_jobs(MlpJobs &jobs, int E, bool chain, cudaStream_t s) {
    long long big = 0;
    for (int j = 0; j < jobs.n; j++)
        big += (long long)((jobs.job[j].M + 63) / 64) * ((jobs.job[j].N + 63) / 64) * E;
    // one block an SM and a half are enough behind nothing that waits for the last of them: all
    // weight gradients in one launch (a step of 5 x 4 x 256 at batch 128 / 64 / 16 with 280 blocks
    // of 64 x 64: 67.4 / 55.3 / 46.7 us, 32 x 32: 69.7 / 57.2 / 48.1; with 160 blocks 46.9 and 42.2)
    const int T = 2 * big >= (jobs.n > 2 ? 3 : 4) * sm_count() ? 64 : 32;
    long long blocks = 0;
    for (int j = 0; j < jobs.n; j++) {
        jobs.blocks[j] = (int)((long long)((jobs.job[j].M + T - 1) / T) * ((jobs.job[j].N + T - 1) / T) * E);
        blocks += jobs.blocks[j];
    }
    if (T == 64) launch_jobs<64>(jobs, (unsigned)blocks, chain, s);
    else launch_jobs<32>(jobs, (unsigned)blocks, chain, s);
}

}  // namespace pic
