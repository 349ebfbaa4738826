// Surrogate network training in FP32: a batch's way forward through all layers, its loss and
// the gradients' way back to the first layer's sums in one kernel.
//
// A row of the batch needs no other row until the weight gradients are summed, so a cluster
// of four CTAs takes 4 RT rows of one member through the whole chain of 2 L - 1 products
// with no launch in between; what the weight gradients need (activations, and the gradients
// by the layers' sums in the place of the sums) goes to memory on the way.  Each CTA
// computes a quarter of a layer's columns for all the rows and writes them into the four
// CTAs' copies of the next product's input (distributed shared memory); one cluster barrier
// a product.  Eight pairs of warps split the product's k, a pair's lanes take RT rows by 4
// columns each; a pair brings its slice of the next product's weights while this one's
// results are summed and exchanged, and the slices' sums are added in a fixed order.
//
// What bounds it: of a product's 12k cycles at 24 rows and 256 x 256, the product 5.7k
// (shared-memory reads: ten 16-byte loads a lane for 96 FMAs, 5.1k), the copies of 64 KB of weights a
// CTA 2.4k, sums, activation and exchange 2.8k, the barrier 1k.  A step of five members of
// 6 -> 4 x 256 -> 33 at batch 128 takes 67 us in 3 launches (84 us in 11 layer by layer), 48 of
// them here.  Unrolled twice over k, with spills: 2 us more; results written to memory ahead
// of the barrier's arrival: 3 more; eight warps with twice the rows a thread: 7 more; sixteen
// slices of k, 10 rows a thread: as fast, but narrow layers slower by a tenth; 8 columns a
// thread and two warps that bring the weights: 16 more; the warps that have no results to
// finish bringing the weights meanwhile: 4 more.
#include "mlp_math.h"
#include "pic_internal.h"

namespace pic {

namespace {

constexpr int CS = 4;           // CTAs a cluster
constexpr int NT = 512, NW = 8, RG = NT / 32 / NW * 2;   // threads; warps along k; row groups
constexpr int COLS = 256 / CS;  // columns of a layer a CTA computes at most
constexpr int KS = 256 / NW;    // k of a product a warp takes at most
constexpr int LDA = 256 + 4;    // row strides, 4 mod 32: free of bank conflicts
constexpr int LDR = COLS + 4;
constexpr int LDK = KS + 4;     // forward: weights [column][k]; back: [k][column], LDR

template <int RT>
struct alignas(16) ChainSmem {
    float in[2][RG * RT * LDA];       // a product's input, and the next one's
    float w[NW][COLS * LDK];         // a slice's weights
    float sum[NW][RG * RT * LDR];    // a slice's partial sums
};
static_assert(KS * LDR <= COLS * LDK, "both layouts of the weights fit");

__device__ __forceinline__ unsigned smem_at(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void put_peer(const float *own, int cta, const float (&v)[4]) {
    asm volatile(
        "{\n .reg .b32 r;\n mapa.shared::cluster.u32 r, %0, %1;\n"
        " st.shared::cluster.v4.f32 [r], {%2, %3, %4, %5};\n}\n"
        ::"r"(smem_at(own)), "r"(cta), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
__device__ __forceinline__ int up4(int x) { return (x + 3) & ~3; }

// The products in order: forward 0 .. L-1, then back L-1 .. 1.
struct Stage {
    bool fwd;
    int l, K, N;   // inputs and columns of the product
    __device__ __forceinline__ Stage(const MlpChain &a, int s)
        : fwd(s < a.L), l(fwd ? s : 2 * a.L - 1 - s), K(a.sz[fwd ? l : l + 1]), N(a.sz[fwd ? l + 1 : l]) {}
    __device__ __forceinline__ int share() const { return up4((N + CS - 1) / CS); }   // columns a CTA
    __device__ __forceinline__ int slice() const { return up4((K + NW - 1) / NW); }   // k a warp
};

// slice `sl` of a product's weights (n x k in memory), half h of it: zero outside.  A lane
// keeps its place in a row of 32 k (forward) or 64 columns (back).
__device__ __forceinline__ void load_weights(const MlpChain &a, const Stage &st, const float *params, int rank,
                                             int sl, int h, int lane, float *w) {
    const float *W = params + a.woff[st.l];
    const int share = st.share(), c0 = rank * share, ks = st.slice(), k0 = sl * ks, ld = a.sz[st.l];
    const bool vec = ld % 4 == 0;   // the parameters of a layer lie on 16-byte boundaries
    constexpr int KQ = KS / 4, CQ = COLS / 4;
    const int slow = st.fwd ? h * (32 / KQ) + lane / KQ : h * (32 / CQ) + lane / CQ;
    const int fast = st.fwd ? lane % KQ * 4 : lane % CQ * 4, step = st.fwd ? 2 * (32 / KQ) : 2 * (32 / CQ);
    const int end = st.fwd ? min(share, st.N - c0) : ks;
    const int in = st.fwd ? st.N - c0 : st.K - k0;          // strided indices that exist
    const int left = (st.fwd ? st.K - k0 : st.N - c0) - fast, n = min(max(left, 0), 4);
    if (fast >= (st.fwd ? ks : share)) return;
    const float *src = W + (long long)((st.fwd ? c0 : k0) + slow) * ld + (st.fwd ? k0 : c0) + fast;
    float *dst = w + slow * (st.fwd ? LDK : LDR) + fast;
    for (int i = slow; i < end; i += step, src += (long long)step * ld, dst += step * (st.fwd ? LDK : LDR)) {
        const int m = i < in ? n : 0;
        if (vec) cp16(dst, m > 0 ? src : W, 4 * m);
        else
            for (int q = 0; q < 4; q++) cp4(dst + q, q < m ? src + q : W, q < m ? 4 : 0);
    }
}

__device__ __forceinline__ float4 at4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// RT rows by 4 columns of the product over the warp's k: rows RT g ..; columns cg + 16 i
// forward, 4 cg + i back (cg: of 16 lanes).  Its partial sums into `out`.
template <int RT, bool FWD>
__device__ __forceinline__ void partial(const float *in, const float *w, int quads, int g, int cg, float *out) {
    float acc[RT][4] = {};
#pragma unroll 1
    for (int q = 0; q < quads; q++) {
        float4 b[4];
#pragma unroll
        for (int i = 0; i < 4; i++) b[i] = at4(FWD ? w + (cg + 16 * i) * LDK + 4 * q : w + (4 * q + i) * LDR + 4 * cg);
#pragma unroll
        for (int r = 0; r < RT; r++) {
            const float4 x = at4(in + (g * RT + r) * LDA + 4 * q);
            if constexpr (FWD) {
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    acc[r][i] = fmaf(x.x, b[i].x, acc[r][i]);
                    acc[r][i] = fmaf(x.y, b[i].y, acc[r][i]);
                    acc[r][i] = fmaf(x.z, b[i].z, acc[r][i]);
                    acc[r][i] = fmaf(x.w, b[i].w, acc[r][i]);
                }
            } else {
                const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    acc[r][0] = fmaf(v[i], b[i].x, acc[r][0]);
                    acc[r][1] = fmaf(v[i], b[i].y, acc[r][1]);
                    acc[r][2] = fmaf(v[i], b[i].z, acc[r][2]);
                    acc[r][3] = fmaf(v[i], b[i].w, acc[r][3]);
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < RT; r++) {
        float *o = out + (g * RT + r) * LDR;
        if constexpr (FWD) {
#pragma unroll
            for (int i = 0; i < 4; i++) o[cg + 16 * i] = acc[r][i];
        } else {
            *reinterpret_cast<float4 *>(o + 4 * cg) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
        }
    }
}

template <int RT>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(NT, 1) k_mlp_chain(const __grid_constant__ MlpChain a) {
    extern __shared__ __align__(16) unsigned char raw[];
    ChainSmem<RT> &sm = *reinterpret_cast<ChainSmem<RT> *>(raw);
    constexpr int R = RG * RT;
    constexpr int EPI = (R * COLS / 4 + NT - 1) / NT;   // groups of four results a thread finishes
    const int tid = threadIdx.x, lane = tid & 31, sl = tid / 32 % NW, half = tid / 32 / NW;
    const int rank = blockIdx.x % CS, z = blockIdx.x / CS % a.E, row0 = blockIdx.x / CS / a.E * R;
    for (int e = tid; e < 2 * R * LDA; e += NT) sm.in[0][e] = 0.f;
    __syncthreads();
    chain_wait();
    const float *params = a.params + z * a.P;
    const int last = 2 * a.L - 2;
    load_weights(a, Stage(a, 0), params, rank, sl, half, lane, sm.w[sl]);
    cp_commit();
    {
        const int K = a.sz[0];
        const float *x = a.act[0] + z * a.batch * K;
        for (int e = tid; e < R * K; e += NT) {
            const int r = e / K, k = e % K;
            if (row0 + r < a.rows) sm.in[0][r * LDA + k] = x[(long long)(row0 + r) * K + k];
        }
    }
    cp_wait<0>();
    cluster_arrive();
    cluster_wait();   // every CTA of the cluster runs and has cleared its inputs
    float lsum = 0.f;
    for (int s = 0; s <= last; s++) {
        const Stage st(a, s);
        const int ks = st.slice(), k0 = sl * ks, N = st.N;
        const int quads = min(max(up4(st.K) - k0, 0), ks) / 4;
        const int share = st.share(), c0 = rank * share;
        const bool out = s == a.L - 1;
        // what the results are combined with, on its way during the product
        float e[EPI][4], b[EPI][4];
        const float *with = st.fwd ? (out ? a.T + z * a.batch * N : nullptr) : a.pre[st.l - 1] + z * a.batch * N;
        const float *bias = st.fwd ? params + a.boff[st.l] : nullptr;
#pragma unroll
        for (int u = 0; u < EPI; u++) {
            const int idx = tid + u * NT, row = row0 + idx / (COLS / 4), c = idx % (COLS / 4) * 4;
            const bool in = idx / (COLS / 4) < R && c < share;
            const bool have = in && with && row < a.rows;
            if (N % 4 == 0) {
                const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
                const float4 x = have && c0 + c < N ? at4(with + (long long)row * N + c0 + c) : none;
                const float4 y = in && bias && c0 + c < N ? at4(bias + c0 + c) : none;
                e[u][0] = x.x, e[u][1] = x.y, e[u][2] = x.z, e[u][3] = x.w;
                b[u][0] = y.x, b[u][1] = y.y, b[u][2] = y.z, b[u][3] = y.w;
            } else {
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    e[u][q] = have && c0 + c + q < N ? with[(long long)row * N + c0 + c + q] : 0.f;
                    b[u][q] = in && bias && c0 + c + q < N ? bias[c0 + c + q] : 0.f;
                }
            }
        }
        const float *in = sm.in[s & 1] + k0;
        if (st.fwd) partial<RT, true>(in, sm.w[sl], quads, 2 * half + lane / 16, lane % 16, sm.sum[sl]);
        else partial<RT, false>(in, sm.w[sl], quads, 2 * half + lane / 16, lane % 16, sm.sum[sl]);
        __syncthreads();
        if (s < last) load_weights(a, Stage(a, s + 1), params, rank, sl, half, lane, sm.w[sl]);
        cp_commit();
        float *next = sm.in[(s + 1) & 1];
        // results for memory are kept until the cluster knows of the exchanged ones: its
        // barrier would wait for the stores too
        float x[EPI][4], y[EPI][4];   // for the next product (activation or gradient); the layer's sum
#pragma unroll
        for (int u = 0; u < EPI; u++) {
            const int idx = tid + u * NT, r = idx / (COLS / 4), c = idx % (COLS / 4) * 4, col = c0 + c;
            if (r >= R || c >= share || col >= N) continue;
            float4 p = at4(sm.sum[0] + r * LDR + c);
            x[u][0] = p.x, x[u][1] = p.y, x[u][2] = p.z, x[u][3] = p.w;
#pragma unroll
            for (int w = 1; w < NW; w++) {
                p = at4(sm.sum[w] + r * LDR + c);
                x[u][0] += p.x;
                x[u][1] += p.y;
                x[u][2] += p.z;
                x[u][3] += p.w;
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const bool in = col + q < N;
                if (st.fwd && !out) {
                    y[u][q] = x[u][q] + b[u][q];
                    x[u][q] = in ? gelu(y[u][q]) : 0.f;
                } else if (out) {
                    const float d = in && row0 + r < a.rows ? (x[u][q] + b[u][q]) - e[u][q] : 0.f;
                    x[u][q] = a.scale * d;
                    lsum += d * d;
                } else {
                    x[u][q] = in ? x[u][q] * gelu_grad(e[u][q]) : 0.f;
                }
            }
            if (s < last)
#pragma unroll
                for (int cta = 0; cta < CS; cta++) put_peer(next + r * LDA + col, cta, x[u]);
        }
        cluster_arrive();
        const auto put = [&](float *p, const float (&v)[4], long long at, int left) {
            if (N % 4 == 0) {
                *reinterpret_cast<float4 *>(p + at) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (q < left) p[at + q] = v[q];
            }
        };
#pragma unroll
        for (int u = 0; u < EPI; u++) {
            const int idx = tid + u * NT, r = idx / (COLS / 4), c = idx % (COLS / 4) * 4, col = c0 + c;
            if (r >= R || c >= share || col >= N || row0 + r >= a.rows) continue;
            const long long at = z * a.batch * N + (long long)(row0 + r) * N + col;
            if (st.fwd && !out) {
                put(a.pre[st.l], y[u], at, N - col);
                put(a.act[st.l + 1], x[u], at, N - col);
            } else {
                put(a.pre[out ? st.l : st.l - 1], x[u], at, N - col);
            }
        }
        cp_wait<0>();
        // the next product's inputs are there, this one's have been read (and on the last
        // one, no CTA leaves before its peers are done)
        cluster_wait();
        __syncthreads();
    }
    if (a.loss) {
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0 && lsum != 0.f) atomicAdd(a.loss + z, lsum / ((float)a.rows * (float)a.sz[a.L]));
    }
}

// clusters that the device holds at a time
template <int RT>
int slots() {
    static int cap[64] = {};   // per device, with the shared-memory opt-in
    int dev = 0;
    cudaGetDevice(&dev);
    int &n = cap[dev & 63];
    if (n == 0) {
        const int smem = (int)sizeof(ChainSmem<RT>);
        if (cudaFuncSetAttribute(k_mlp_chain<RT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
            return 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(CS);
        cfg.blockDim = dim3(NT);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute at = {};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = CS;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int c = 0;
        if (cudaOccupancyMaxActiveClusters(&c, k_mlp_chain<RT>, &cfg) != cudaSuccess) return 0;
        n = c;
    }
    return n;
}

template <int RT>
void launch(const MlpChain &a, bool chain, cudaStream_t s) {
    const long long slabs = (a.rows + RG * RT - 1) / (RG * RT);
    launch_chained(chain, k_mlp_chain<RT>, (unsigned)(CS * a.E * slabs), NT, sizeof(ChainSmem<RT>), s, a);
}
}  // namespace

// The fewest rows a CTA with which one round of clusters does: more rounds, or layers of which
// the product's columns fill little, go faster layer by layer (us a step, here and there:
// 5 members of 4 x 256, batch 128: 67 / 84, 512: 231 / 210; of 4 x 64, batch 128: 33 / 44, 1024:
// 179 / 135; 8 of 5 x 100, batch 64: 42 / 58, 256: 141 / 98; one of 4 x 256, batch 700: 69 / 112).
bool mlp_chain(const MlpChain &a, bool chain, cudaStream_t s) {
    const auto fits = [&](int rt, int cap) { return a.E * (((long long)a.rows + RG * rt - 1) / (RG * rt)) <= cap; };
    if (fits(2, slots<2>())) launch<2>(a, chain, s);
    else if (fits(4, slots<4>())) launch<4>(a, chain, s);
    else if (fits(6, slots<6>())) launch<6>(a, chain, s);
    else return false;
    return true;
}

}  // namespace pic
