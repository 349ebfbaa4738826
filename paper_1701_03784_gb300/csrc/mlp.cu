// Surrogate network ensemble: small multilayer perceptrons (tanh-GELU hidden layers, linear
// output) that map sweep parameters to simulation outputs, trained and evaluated on the
// GPU by the kernels in k_mlp_f32.cu (FP32 on CUDA cores) and k_mlp_tc.cu (BF16 tensor-core
// inference, and optionally the training products: pic_mlp_set_training).  The paper has
// no counterpart.
//
// Layout: per member, the layers' parameters one after another, W_l (n_out x n_in,
// row-major) then b_l, each starting on a 16-byte boundary (the copies into shared memory
// are 16 bytes wide); members follow each other at a fixed stride.  The caller's arrays
// are without the padding.  Activations are
// row-major (sample x unit) per member.  Minibatch indices come from a counter-based hash
// of (seed, member, step, row), so a training run is reproducible.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "mlp_math.h"
#include "pic_internal.h"

namespace pic {

namespace {
// C(z)[m][n] (+)= sum_k A(z, m, k) B(z, k, n), operands addressed by strides; z = member
struct GemmArgs {
    const float *A, *B;
    float *C;
    int M, N, K;
    long long sAz, sBz, sCz;
    int sAm, sAk, sBk, sBn, ldc;
    int accumulate;
};

// Z += b (per column); A = gelu(Z) for hidden layers, A = Z for the output layer
__global__ void k_bias_act(float *Z, float *A, const float *b, long long bz, int rows, int cols,
                           long long sz, int act) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int z = blockIdx.y;
    if (i >= (long long)rows * cols) return;
    const float v = Z[z * sz + i] + b[z * bz + (int)(i % cols)];
    Z[z * sz + i] = v;
    if (A) A[z * sz + i] = act ? gelu(v) : v;
}

// G = scale (Y - T); loss[z] += sum (Y - T)^2 / count
__global__ void k_loss_grad(const float *Y, const float *T, float *G, long long n, long long sY,
                            long long sT, long long sG, float scale, float *loss) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int z = blockIdx.y;
    float e = 0.f;
    if (i < n) {
        e = Y[z * sY + i] - T[z * sT + i];
        G[z * sG + i] = scale * e;
    }
    float s = e * e;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (loss && (threadIdx.x & 31) == 0 && s != 0.f) atomicAdd(loss + z, s / (float)n);
}

__global__ void k_gelu_back(float *G, const float *Z, long long n, long long sG, long long sZ) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) G[blockIdx.y * sG + i] *= gelu_grad(Z[blockIdx.y * sZ + i]);
}

// db[j] = sum_i G[i][j]
__global__ void k_colsum(const float *G, float *db, int rows, int cols, long long sg, long long sb) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int z = blockIdx.y;
    if (j >= cols) return;
    float s = 0.f;
    for (int i = 0; i < rows; i++) s += G[z * sg + (long long)i * cols + j];
    db[z * sb + j] = s;
}

__global__ void k_adam(float *p, const float *g, float *m, float *v, long long n, AdamArgs a) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) adam_step(a, g[i], p[i], m[i], v[i]);
}

__device__ __forceinline__ unsigned long long mix64(unsigned long long x) {
    // splitmix64 finaliser
    x += 0x9E3779B97F4A7C15ULL;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
    return x ^ (x >> 31);
}

// `rows` samples per member into the member's batch buffers (row stride mrows): drawn from
// n with replacement (random = 1) or rows 0.. of X and T (random = 0).  One thread a value:
// one thread a row, looping over its 6 + 33 values, took 8.4 us for 5 x 128 rows.  Clears the
// members' losses for the kernels behind it, where they are wanted.
__global__ void k_gather(const float *X, const float *T, float *Xb, float *Tb, long long n, int rows,
                         int mrows, int din, int dout, unsigned long long seed, long long step,
                         int random, float *loss) {
    chain_wait();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int z = blockIdx.y, w = din + dout;
    if (loss && i == 0) loss[z] = 0.f;
    const int r = (int)(i / w), k = (int)(i % w);
    if (r >= rows) return;
    long long s = r;
    if (random) {
        const unsigned long long h = mix64(
            seed ^ mix64(((unsigned long long)z << 48) ^ ((unsigned long long)step << 20) ^ r));
        s = (long long)(h % (unsigned long long)n);
    }
    const long long o = (long long)z * mrows + r;
    if (k < din) Xb[o * din + k] = X[s * din + k];
    else Tb[o * dout + k - din] = T[s * dout + k - din];
}

// the caller's parameters (members at stride cP, packed) into the padded layout
__global__ void k_params_in(const double *src, float *dst, MlpOffsets from, MlpOffsets to, MlpOffsets len,
                            int L, long long cP, long long P) {
    const int z = blockIdx.y / L, l = blockIdx.y % L;
    const double *s = src + z * cP;
    float *d = dst + z * P;
    for (long long i = blockIdx.x * blockDim.x + threadIdx.x; i < len.w[l] + len.b[l];
         i += (long long)gridDim.x * blockDim.x) {
        if (i < len.w[l]) d[to.w[l] + i] = (float)s[from.w[l] + i];
        else d[to.b[l] + i - len.w[l]] = (float)s[from.b[l] + i - len.w[l]];
    }
}

// and the way back
__global__ void k_params_out(const float *src, double *dst, MlpOffsets from, MlpOffsets to, MlpOffsets len,
                             int L, long long P, long long cP) {
    const int z = blockIdx.y / L, l = blockIdx.y % L;
    const float *s = src + z * P;
    double *d = dst + z * cP;
    for (long long i = blockIdx.x * blockDim.x + threadIdx.x; i < len.w[l] + len.b[l];
         i += (long long)gridDim.x * blockDim.x) {
        if (i < len.w[l]) d[to.w[l] + i] = s[from.w[l] + i];
        else d[to.b[l] + i - len.w[l]] = s[from.b[l] + i - len.w[l]];
    }
}

inline unsigned blocks(long long n, int b = 256) { return (unsigned)((n + b - 1) / b); }
}  // namespace


struct MlpImpl {
    int device = 0;
    Allocator al;
    std::vector<void *> allocs;
    int E = 0, L = 0, max_batch = 0, maxw = 0;
    std::vector<int> sz;
    std::vector<long long> woff, boff;
    long long P = 0, cP = 0;       // parameters of a member: stride here, the caller's count
    MlpOffsets off{}, coff{}, len{};   // here, in the caller's arrays, and how many
    float *params = nullptr, *grads = nullptr, *am = nullptr, *av = nullptr, *Tb = nullptr,
          *loss = nullptr;
    double *stage = nullptr;
    std::vector<float *> act, pre;
    float *gbuf[3] = {nullptr, nullptr, nullptr};
    long long adam_step = 0;
    MlpTc tc;               // BF16 tensor-core copy of the parameters
    MlpF32 f32;             // packed FP32 copy of the parameters for whole-network inference,
                            // as current as they are: see changed()
    bool tc_dirty = true;   // parameters changed since it was packed
    // training products on the tensor cores (pic_mlp_set_training): packed BF16 operand
    // scratch and the bounded-wait counter
    bool train_tc = false;
    uint16_t *tsa = nullptr, *tsb = nullptr;
    unsigned int *terr = nullptr;

    ~MlpImpl() {
        cudaSetDevice(device);
        cudaDeviceSynchronize();
        if (tc.err) cudaFreeHost(tc.err);
        for (void *p : allocs) {
            if (al.free) al.free(p, al.ctx);
            else cudaFree(p);
        }
    }
    template <class T>
    pic_status dalloc(T *&p, long long n) {
        const size_t bytes = sizeof(T) * (size_t)std::max<long long>(n, 1);
        void *v = nullptr;
        if (al.alloc) v = al.alloc(bytes, al.ctx);
        else if (cudaMalloc(&v, bytes) != cudaSuccess) v = nullptr;
        if (!v) {
            set_error("pic_mlp_create: device allocation of %zu bytes failed", bytes);
            return PIC_ERR_OOM;
        }
        allocs.push_back(v);
        p = static_cast<T *>(v);
        return PIC_OK;
    }

    // places of arrays in one allocation
    struct Carver {
        std::vector<std::pair<void **, size_t>> at;
        size_t bytes = 0;
        template <class T>
        void want(T *&p, long long n) {
            at.push_back({reinterpret_cast<void **>(&p), bytes});
            bytes += (sizeof(T) * (size_t)std::max<long long>(n, 1) + 255) / 256 * 256;
        }
    };

    pic_status init(int members, int layers, const int32_t *sizes, int batch) {
        E = members;
        L = layers;
        max_batch = batch;
        sz.assign(sizes, sizes + layers + 1);
        maxw = *std::max_element(sz.begin(), sz.end());
        for (int l = 0; l < L; l++) {
            len.w[l] = (long long)sz[l + 1] * sz[l];
            len.b[l] = sz[l + 1];
            off.w[l] = P;
            P += (len.w[l] + 3) / 4 * 4;
            off.b[l] = P;
            P += (len.b[l] + 3) / 4 * 4;
            coff.w[l] = cP;
            coff.b[l] = cP + len.w[l];
            cP += len.w[l] + len.b[l];
            woff.push_back(off.w[l]);
            boff.push_back(off.b[l]);
        }
        // everything in one allocation, each array on a 256-byte boundary
        Carver carve;
        carve.want(params, E * P);   // these are cleared together
        carve.want(grads, E * P);
        carve.want(am, E * P);
        carve.want(av, E * P);
        // whole-network FP32 inference: every width at most 256
        f32.ok = maxw <= 256;
        if (f32.ok) {
            f32.E = E;
            f32.L = L;
            f32.NW = maxw <= 64 ? 64 : maxw <= 128 ? 128 : 256;
            for (int l = 0; l < L; l++) {
                f32.k[l] = sz[l];
                f32.n[l] = sz[l + 1];
                f32.kp[l] = (sz[l] + 15) / 16 * 16;
                f32.np[l] = mlp_f32_shape(maxw, sz[l + 1]);
                f32.woff[l] = f32.wmember;
                f32.wmember += (long long)f32.kp[l] * f32.np[l];
                f32.boff[l] = f32.bmember;
                f32.bmember += f32.np[l];
            }
            carve.want(f32.w, E * f32.wmember);
            carve.want(f32.b, E * f32.bmember);
        }
        const size_t cleared = carve.bytes;
        carve.want(stage, E * cP);
        carve.want(Tb, (long long)E * batch * sz[L]);
        carve.want(loss, E);
        for (float *&g : gbuf) carve.want(g, (long long)E * batch * maxw);
        act.assign(L + 1, nullptr);
        pre.assign(L, nullptr);
        for (int l = 0; l <= L; l++) carve.want(act[l], (long long)E * batch * sz[l]);
        for (int l = 0; l < L; l++) carve.want(pre[l], (long long)E * batch * sz[l + 1]);
        // tensor-core inference: every width at most 256
        tc.ok = L <= MLP_MAX_LAYERS && maxw <= 256;
        if (tc.ok) {
            tc.E = E;
            tc.L = L;
            for (int l = 0; l < L; l++) {
                tc.k[l] = sz[l];
                tc.n[l] = sz[l + 1];
                tc.kp[l] = (sz[l] + 15) / 16 * 16;
                tc.np[l] = (sz[l + 1] + 31) / 32 * 32;   // half in each CTA of a pair
                tc.woff[l] = tc.wmember;
                tc.wmember += (long long)tc.kp[l] * tc.np[l];
                tc.boff[l] = tc.bmember;
                tc.bmember += tc.np[l];
            }
            carve.want(tc.w, E * tc.wmember);
            carve.want(tc.b, E * tc.bmember);
            const long long mp = (std::max(max_batch, maxw) + 127) / 128 * 128;
            carve.want(tsa, (long long)E * mp * 256);
            carve.want(tsb, (long long)E * 256 * 256);
            carve.want(terr, 1);
        }
        unsigned char *base = nullptr;
        pic_status st = dalloc(base, (long long)carve.bytes);
        if (st != PIC_OK) return st;
        for (const auto &x : carve.at) *x.first = base + x.second;
        PIC_CUDA_TRY(cudaMemset(base, 0, cleared));
        if (terr) PIC_CUDA_TRY(cudaMemset(terr, 0, sizeof(unsigned int)));
        if (tc.ok) {
            // read by the host once the stream is done, without a copy
            PIC_CUDA_TRY(cudaHostAlloc(&tc.err, sizeof(unsigned int), cudaHostAllocMapped | cudaHostAllocPortable));
            *tc.err = 0;
        }
        return PIC_OK;
    }

    // timeouts of the training products since the last check (synchronises when the
    // tensor-core products were on)
    pic_status tc_errors(const char *who, cudaStream_t s) {
        if (!train_tc || !terr) return PIC_OK;
        unsigned int e = 0;
        PIC_CUDA_TRY(cudaMemcpyAsync(&e, terr, sizeof e, cudaMemcpyDeviceToHost, s));
        PIC_CUDA_TRY(cudaStreamSynchronize(s));
        if (e) {
            PIC_CUDA_TRY(cudaMemsetAsync(terr, 0, sizeof e, s));
            set_error("%s: %u tensor-core waits timed out", who, e);
            return PIC_ERR_TIMEOUT;
        }
        return PIC_OK;
    }

    // one product of the tensor-core training path; its K may exceed what that takes
    void gemm(const GemmArgs &g, cudaStream_t s) {
        const TcGemmOp op{g.A, g.B, g.C, g.M, g.N, g.K, g.sAz, g.sBz, g.sCz,
                          g.sAm, g.sAk, g.sBk, g.sBn, g.ldc, g.accumulate};
        if (mlp_tc_gemm(op, E, tsa, tsb, terr, s)) return;
        MlpJobs jobs;
        MlpJob &j = jobs.job[jobs.n++];
        j = MlpJob{};
        j.kind = g.sAm == 1 && g.sBn == 1 ? MLP_DW : g.sBn == 1 ? MLP_DX : MLP_FWD;
        j.epi = MLP_EPI_STORE;
        j.M = g.M;
        j.N = g.N;
        j.K = g.K;
        j.A = g.A;
        j.B = g.B;
        j.C = g.C;
        j.sA = g.sAz;
        j.sB = g.sBz;
        j.sC = g.sCz;
        j.lda = j.kind == MLP_DW ? g.sAk : g.sAm;
        j.ldb = j.kind == MLP_FWD ? g.sBn : g.sBk;
        j.ldc = g.ldc;
        mlp_jobs(jobs, E, false, s);
    }

    // ---- the FP32 path: every product with what follows it (k_mlp_f32.cu) ----
    // layer l for `rows` samples of A; C: where its outputs go (member stride sC)
    MlpJob forward_job(int l, int rows, const float *A, long long sA, float *C, long long sC) {
        MlpJob j{};
        j.kind = MLP_FWD;
        j.epi = l < L - 1 ? MLP_EPI_GELU : MLP_EPI_BIAS;
        j.M = rows;
        j.N = j.ldc = sz[l + 1];
        j.K = j.lda = j.ldb = sz[l];
        j.A = A;
        j.sA = sA;
        j.B = params + woff[l];
        j.sB = j.sbias = P;
        j.bias = params + boff[l];
        j.C = C;
        j.sC = sC;
        return j;
    }
    // `rows` samples of X (every member the same) through all layers into Y (n rows a
    // member), from row c0 on
    void infer(int rows, const float *X, float *Y, long long n, long long c0, cudaStream_t s) {
        const float *A = X;
        long long sA = 0;
        for (int l = 0; l < L; l++) {
            const bool last = l == L - 1;
            MlpJobs jobs;
            jobs.job[jobs.n++] = forward_job(l, rows, A, sA, last ? Y + c0 * sz[L] : act[l + 1],
                                             last ? n * sz[L] : (long long)max_batch * sz[l + 1]);
            mlp_jobs(jobs, E, l > 0 || c0 > 0, s);
            A = act[l + 1];
            sA = (long long)max_batch * sz[l + 1];
        }
    }
    // the batch in act[0], Tb: losses (where asked for), gradients, and with `adam` the
    // parameters' step in the place of the gradients' storing.  The weight gradients of a
    // layer go with the next input gradient, which reads other weights.
    void fused_step(int rows, float *loss_out, const AdamArgs *adam, cudaStream_t s) {
        bool whole = false;
        if (f32.ok) {
            MlpChain c{};
            c.E = E;
            c.L = L;
            c.rows = rows;
            c.batch = max_batch;
            c.P = P;
            c.params = params;
            c.T = Tb;
            for (int l = 0; l <= L; l++) c.sz[l] = sz[l];
            for (int l = 0; l < L; l++) {
                c.woff[l] = woff[l];
                c.boff[l] = boff[l];
                c.act[l] = act[l];
                c.pre[l] = pre[l];
            }
            c.scale = 2.f / (float)((long long)rows * sz[L]);
            c.loss = loss_out;
            whole = mlp_chain(c, true, s);
        }
        const long long sg = (long long)max_batch * maxw;
        const auto sa = [&](int l) { return (long long)max_batch * sz[l]; };
        const auto dw = [&](int l) {
            MlpJob j{};
            j.kind = MLP_DW;
            j.M = j.lda = sz[l + 1];
            j.N = j.ldb = j.ldc = sz[l];
            j.K = rows;
            j.A = whole ? pre[l] : gbuf[l % 3];
            j.sA = whole ? sa(l + 1) : sg;
            j.B = act[l];
            j.sB = sa(l);
            j.sC = P;
            if (adam) {
                j.epi = MLP_EPI_ADAM;
                j.adam = *adam;
                j.C = params + woff[l];
                j.am = am + woff[l];
                j.av = av + woff[l];
                j.db = params + boff[l];
                j.dbm = am + boff[l];
                j.dbv = av + boff[l];
            } else {
                j.epi = MLP_EPI_STORE;
                j.C = grads + woff[l];
                j.db = grads + boff[l];
            }
            return j;
        };
        if (whole) {   // pre: the gradients by the layers' sums
            MlpJobs jobs;
            for (int l = L - 1; l >= 0; l--) jobs.job[jobs.n++] = dw(l);
            mlp_jobs(jobs, E, true, s);
            return;
        }
        for (int l = 0; l < L; l++) {
            MlpJobs jobs;
            const bool last = l == L - 1;
            MlpJob &j = jobs.job[jobs.n++];
            j = forward_job(l, rows, act[l], sa(l), last ? gbuf[l % 3] : act[l + 1], last ? sg : sa(l + 1));
            if (last) {
                j.epi = MLP_EPI_LOSS;
                j.Z = Tb;
                j.sZ = sa(L);
                j.scale = 2.f / (float)((long long)rows * sz[L]);
                j.loss = loss_out;
            } else {
                j.Z = pre[l];
                j.sZ = sa(l + 1);
            }
            mlp_jobs(jobs, E, true, s);
        }
        const auto dx = [&](int l) {
            MlpJob j{};
            j.kind = MLP_DX;
            j.epi = MLP_EPI_GELU_GRAD;
            j.M = rows;
            j.N = j.ldb = j.ldc = sz[l];
            j.K = j.lda = sz[l + 1];
            j.A = gbuf[l % 3];
            j.sA = j.sC = sg;
            j.B = params + woff[l];
            j.sB = P;
            j.C = gbuf[(l - 1) % 3];
            j.Z = pre[l - 1];
            j.sZ = sa(l);
            return j;
        };
        for (int l = L - 1; l >= 1; l--) {
            MlpJobs jobs;
            jobs.job[jobs.n++] = dx(l);
            if (l + 1 < L) jobs.job[jobs.n++] = dw(l + 1);
            mlp_jobs(jobs, E, true, s);
        }
        MlpJobs jobs;
        if (L > 1) jobs.job[jobs.n++] = dw(1);
        jobs.job[jobs.n++] = dw(0);
        mlp_jobs(jobs, E, true, s);
    }

    void gather(int rows, const float *X, const float *T, long long n, unsigned long long seed,
                long long step, int random, float *loss_out, bool chain, cudaStream_t s) {
        launch_chained(chain, k_gather, dim3(blocks((long long)rows * (sz[0] + sz[L])), E), 256, 0, s, X, T, act[0],
                       Tb, n, rows, max_batch, sz[0], sz[L], seed, step, random, loss_out);
    }
    // FP32 inference on n rows by the whole-network kernel, or layer by layer in batches of
    // max_batch.  A block of the whole-network kernel takes as long for one row as for its
    // 64 to 256 (us for 6 -> 4 x 256 -> 33: 105, with 4 x 128: 64, with 4 x 64: 43), and
    // 300 blocks run side by side; a batch of 256 rows layer by layer takes 49, 27 and 27 us
    // for five members.  Measured, five members: 512 rows 105 / 64 / 43 against 97 / 52 / 38,
    // 768 rows 105 / 64 / 43 against 145 / 78 / 54; one member of 4 x 256: 1024 rows 105
    // against 101.
    bool whole_network(long long n) const {
        return f32.ok && n > std::min<long long>(2LL * max_batch, 1024);
    }
    // Work on s has changed the parameters: what waits for that work finds the FP32 copy
    // packed too.  A forward call only reads it, so that calls on several streams, and replays
    // of a recorded one, need no more order than the parameters themselves ask for (packed by
    // the first forward call after a change, a call on another stream could read the copy
    // half written, and a replay never packed it).  A call that trains five members of
    // 6 -> 4 x 256 -> 33 for one step takes 111 us instead of 103 with it, of 100 steps 7.36
    // instead of 7.34 ms.  The BF16 copy is packed by the forward call, which synchronises.
    void changed(cudaStream_t s) {
        tc_dirty = true;
        if (f32.ok) mlp_f32_pack(f32, params, P, off, s);
    }
    // E x P floats (parameters or gradients) as E x cP doubles into a host array: converted
    // on the device (as a vector converted on the host, 1.1M parameters took 1151 us)
    pic_status to_host(const float *src, double *out, cudaStream_t s) {
        k_params_out<<<dim3(64, E * L), 256, 0, s>>>(src, stage, off, coff, len, L, P, cP);
        PIC_LAUNCHED();
        PIC_CUDA_TRY(cudaMemcpyAsync(out, stage, sizeof(double) * E * cP, cudaMemcpyDeviceToHost, s));
        PIC_CUDA_TRY(cudaStreamSynchronize(s));
        return PIC_OK;
    }

    // ---- the tensor-core training path: products, then elementwise kernels ----
    // all layers for `rows` samples; the input of member z is X0 + z * sX0z (row-major)
    void forward(int rows, const float *X0, long long sX0z, cudaStream_t s) {
        const float *A = X0;
        long long sAz = sX0z;
        for (int l = 0; l < L; l++) {
            const int K = sz[l], N = sz[l + 1];
            GemmArgs g{A, params + woff[l], pre[l], rows, N, K, sAz, P,
                       (long long)max_batch * N, K, 1, 1, K, N, 0};
            gemm(g, s);
            k_bias_act<<<dim3(blocks((long long)rows * N), E), 256, 0, s>>>(
                pre[l], act[l + 1], params + boff[l], P, rows, N, (long long)max_batch * N,
                l < L - 1);
            PIC_LAUNCHED();
            A = act[l + 1];
            sAz = (long long)max_batch * N;
        }
    }

    // gradients of the mean squared error of act[L] against Tb (rows samples), inputs act[0]
    void backward(int rows, float *loss_out, cudaStream_t s) {
        const int dout = sz[L];
        float *G = gbuf[0], *Gn = gbuf[1];
        const long long sg = (long long)max_batch * maxw;
        k_loss_grad<<<dim3(blocks((long long)rows * dout), E), 256, 0, s>>>(
            act[L], Tb, G, (long long)rows * dout, (long long)max_batch * dout,
            (long long)max_batch * dout, sg, 2.f / (float)((long long)rows * dout), loss_out);
        PIC_LAUNCHED();
        // G is stored with the layer's width as row stride, member stride sg
        for (int l = L - 1; l >= 0; l--) {
            const int K = sz[l], N = sz[l + 1];
            if (l < L - 1) {
                k_gelu_back<<<dim3(blocks((long long)rows * N), E), 256, 0, s>>>(
                    G, pre[l], (long long)rows * N, sg, (long long)max_batch * N);
                PIC_LAUNCHED();
            }
            GemmArgs dw{G, act[l], grads + woff[l], N, K, rows, sg, (long long)max_batch * K, P,
                        1, N, K, 1, K, 0};
            gemm(dw, s);
            k_colsum<<<dim3(blocks(N), E), 256, 0, s>>>(G, grads + boff[l], rows, N, sg, P);
            PIC_LAUNCHED();
            if (l > 0) {
                GemmArgs dx{G, params + woff[l], Gn, rows, K, N, sg, P, sg, N, 1, K, 1, K, 0};
                gemm(dx, s);
                std::swap(G, Gn);
            }
        }
    }
};

}  // namespace pic

using namespace pic;

struct pic_mlp {
    MlpImpl *impl = nullptr;
    ~pic_mlp() { delete impl; }
};

#define MLP_CHECK(m, name)                                   \
    do {                                                     \
        if (!(m) || !(m)->impl) {                            \
            pic::set_error("%s: null network", name);        \
            return PIC_ERR_ARG;                              \
        }                                                    \
        cudaError_t e__ = cudaSetDevice((m)->impl->device);  \
        if (e__ != cudaSuccess) {                            \
            pic::set_error("%s: %s", name, cudaGetErrorString(e__)); \
            return PIC_ERR_CUDA;                             \
        }                                                    \
    } while (0)

extern "C" pic_status pic_mlp_create(int32_t n_members, int32_t n_layers, const int32_t *sizes,
                                     int32_t max_batch, pic_mlp **out) try {
    if (!sizes || !out || n_members < 1 || n_members > 64 || n_layers < 1 || n_layers > 16 ||
        max_batch < 1 || max_batch > (1 << 20)) {
        set_error("pic_mlp_create: bad arguments");
        return PIC_ERR_ARG;
    }
    for (int l = 0; l <= n_layers; l++)
        if (sizes[l] < 1 || sizes[l] > 4096) {
            set_error("pic_mlp_create: layer width %d out of range", sizes[l]);
            return PIC_ERR_ARG;
        }
    std::unique_ptr<pic_mlp> m(new (std::nothrow) pic_mlp);
    if (!m || !(m->impl = new (std::nothrow) MlpImpl)) {
        set_error("pic_mlp_create: out of host memory");
        return PIC_ERR_OOM;
    }
    PIC_CUDA_TRY(cudaGetDevice(&m->impl->device));
    m->impl->al = current_allocator();
    pic_status st = m->impl->init(n_members, n_layers, sizes, max_batch);
    if (st != PIC_OK) return st;
    *out = m.release();
    return PIC_OK;
}
PIC_CATCH("pic_mlp_create")

extern "C" pic_status pic_mlp_param_count(pic_mlp *m, int64_t *per_member) try {
    MLP_CHECK(m, "pic_mlp_param_count");
    if (!per_member) {
        set_error("pic_mlp_param_count: null output");
        return PIC_ERR_ARG;
    }
    *per_member = m->impl->cP;
    return PIC_OK;
}
PIC_CATCH("pic_mlp_param_count")

extern "C" pic_status pic_mlp_params_set(pic_mlp *m, const double *params) try {
    MLP_CHECK(m, "pic_mlp_params_set");
    MlpImpl &x = *m->impl;
    if (!params) {
        set_error("pic_mlp_params_set: null parameters");
        return PIC_ERR_ARG;
    }
    const long long n = x.E * x.P;
    PIC_CUDA_TRY(cudaMemcpy(x.stage, params, sizeof(double) * x.E * x.cP, cudaMemcpyHostToDevice));
    k_params_in<<<dim3(64, x.E * x.L), 256>>>(x.stage, x.params, x.coff, x.off, x.len, x.L, x.cP, x.P);
    PIC_LAUNCHED();
    PIC_CUDA_TRY(cudaMemset(x.am, 0, sizeof(float) * n));
    PIC_CUDA_TRY(cudaMemset(x.av, 0, sizeof(float) * n));
    x.adam_step = 0;
    x.changed(nullptr);
    PIC_CUDA_TRY(cudaDeviceSynchronize());
    return PIC_OK;
}
PIC_CATCH("pic_mlp_params_set")

extern "C" pic_status pic_mlp_params_get(pic_mlp *m, double *params) try {
    MLP_CHECK(m, "pic_mlp_params_get");
    MlpImpl &x = *m->impl;
    if (!params) {
        set_error("pic_mlp_params_get: null output");
        return PIC_ERR_ARG;
    }
    PIC_CUDA_TRY(cudaDeviceSynchronize());
    return x.to_host(x.params, params, nullptr);
}
PIC_CATCH("pic_mlp_params_get")

extern "C" pic_status pic_mlp_grad(pic_mlp *m, const float *X, const float *T, int64_t n,
                                   double *grads, double *loss, void *st) try {
    MLP_CHECK(m, "pic_mlp_grad");
    MlpImpl &x = *m->impl;
    if (!X || !T || !grads || n < 1 || n > x.max_batch) {
        set_error("pic_mlp_grad: bad arguments (n must be 1..max_batch)");
        return PIC_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)st;
    const int rows = (int)n;
    x.gather(rows, X, T, n, 0, 0, 0, x.loss, false, s);
    if (x.train_tc) {
        x.forward(rows, x.act[0], (long long)x.max_batch * x.sz[0], s);
        x.backward(rows, x.loss, s);
    } else {
        x.fused_step(rows, x.loss, nullptr, s);
    }
    PIC_CUDA_TRY(cudaGetLastError());
    pic_status ts = x.tc_errors("pic_mlp_grad", s);
    if (ts != PIC_OK) return ts;
    std::vector<float> hl(x.E);
    PIC_CUDA_TRY(cudaMemcpyAsync(hl.data(), x.loss, sizeof(float) * x.E, cudaMemcpyDeviceToHost, s));
    if ((ts = x.to_host(x.grads, grads, s)) != PIC_OK) return ts;
    if (loss)
        for (int z = 0; z < x.E; z++) loss[z] = hl[z];
    return PIC_OK;
}
PIC_CATCH("pic_mlp_grad")

extern "C" pic_status pic_mlp_train(pic_mlp *m, const float *X, const float *T, int64_t n,
                                    int32_t batch, int64_t steps, double lr, uint64_t seed,
                                    double *last_loss, void *st) try {
    MLP_CHECK(m, "pic_mlp_train");
    MlpImpl &x = *m->impl;
    if (!X || !T || n < 1 || batch < 1 || batch > x.max_batch || steps < 0 || !(lr > 0)) {
        set_error("pic_mlp_train: bad arguments (batch must be 1..max_batch)");
        return PIC_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)st;
    const long long np = x.E * x.P;
    x.tc_dirty = true;
    for (long long k = 0; k < steps; k++) {
        const bool last = k == steps - 1;
        x.gather(batch, X, T, n, seed, x.adam_step, 1, last ? x.loss : nullptr, k > 0, s);
        x.adam_step++;
        const float b1 = 0.9f, b2 = 0.999f;
        const AdamArgs adam{(float)lr, b1, b2, 1e-8f, 1.f - std::pow(b1, (float)x.adam_step),
                            1.f - std::pow(b2, (float)x.adam_step)};
        if (x.train_tc) {
            x.forward(batch, x.act[0], (long long)x.max_batch * x.sz[0], s);
            x.backward(batch, last ? x.loss : nullptr, s);
            k_adam<<<blocks(np), 256, 0, s>>>(x.params, x.grads, x.am, x.av, np, adam);
            PIC_LAUNCHED();
        } else {
            x.fused_step(batch, last ? x.loss : nullptr, &adam, s);
        }
    }
    if (steps > 0) x.changed(s);
    PIC_CUDA_TRY(cudaGetLastError());
    pic_status ts = x.tc_errors("pic_mlp_train", s);
    if (ts != PIC_OK) return ts;
    if (last_loss) {
        std::vector<float> hl(x.E, 0.f);
        if (steps > 0)
            PIC_CUDA_TRY(cudaMemcpyAsync(hl.data(), x.loss, sizeof(float) * x.E,
                                         cudaMemcpyDeviceToHost, s));
        PIC_CUDA_TRY(cudaStreamSynchronize(s));
        for (int z = 0; z < x.E; z++) last_loss[z] = hl[z];
    }
    return PIC_OK;
}
PIC_CATCH("pic_mlp_train")

extern "C" pic_status pic_mlp_forward(pic_mlp *m, const float *X, float *Y, int64_t n,
                                      int32_t tensor_cores, void *st) try {
    MLP_CHECK(m, "pic_mlp_forward");
    MlpImpl &x = *m->impl;
    if (!X || !Y || n < 0) {
        set_error("pic_mlp_forward: bad arguments");
        return PIC_ERR_ARG;
    }
    if (tensor_cores) {
        if (!x.tc.ok) {
            set_error("pic_mlp_forward: the tensor-core path needs layer widths of at most 256");
            return PIC_ERR_ARG;
        }
        if (x.tc_dirty) {
            mlp_tc_pack(x.tc, x.params, x.P, x.woff.data(), x.boff.data(), (cudaStream_t)st);
            x.tc_dirty = false;
        }
        return mlp_tc_forward(x.tc, X, Y, n, (cudaStream_t)st);
    }
    if (n == 0) return PIC_OK;
    cudaStream_t s = (cudaStream_t)st;
    if (x.whole_network(n)) return mlp_f32_forward(x.f32, X, Y, n, s);
    for (long long c0 = 0; c0 < n; c0 += x.max_batch)
        x.infer((int)std::min<long long>(x.max_batch, n - c0), X + c0 * x.sz[0], Y, n, c0, s);
    PIC_CUDA_TRY(cudaGetLastError());
    return PIC_OK;
}
PIC_CATCH("pic_mlp_forward")

extern "C" pic_status pic_mlp_set_training(pic_mlp *m, int32_t tensor_cores) try {
    MLP_CHECK(m, "pic_mlp_set_training");
    MlpImpl &x = *m->impl;
    if (tensor_cores && !x.tc.ok) {
        set_error("pic_mlp_set_training: tensor-core products need widths of at most 256");
        return PIC_ERR_ARG;
    }
    x.train_tc = tensor_cores != 0;
    return PIC_OK;
}
PIC_CATCH("pic_mlp_set_training")

extern "C" pic_status pic_mlp_set_wait_limit(pic_mlp *m, int64_t polls) try {
    MLP_CHECK(m, "pic_mlp_set_wait_limit");
    if (polls < 0) {
        set_error("pic_mlp_set_wait_limit: negative poll count");
        return PIC_ERR_ARG;
    }
    m->impl->tc.wait_polls = polls;
    return PIC_OK;
}
PIC_CATCH("pic_mlp_set_wait_limit")

extern "C" void pic_mlp_destroy(pic_mlp *m) { delete m; }
