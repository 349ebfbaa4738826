// Internal declarations of the GB300 PIC library: host mesh, device record layouts,
// precision policies and kernel launchers.  Not part of the C ABI.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <exception>
#include <new>
#include <string>
#include <thread>
#include <vector>

#include "../../include/pic.h"

namespace pic {

// ---------------------------------------------------------------------------------
// errors
// ---------------------------------------------------------------------------------
void set_error(const char *fmt, ...);

// Handlers closing the function-try-block of every status-returning entry point, so that
// no C++ exception (a failed host allocation, a thread that cannot start) crosses the C
// ABI: the call returns a status and leaves its message instead.
#define PIC_CATCH(name)                                                    \
    catch (const std::bad_alloc &) {                                       \
        ::pic::set_error("%s: out of host memory", name);                  \
        return PIC_ERR_OOM;                                                \
    }                                                                      \
    catch (const std::exception &ex__) {                                   \
        ::pic::set_error("%s: %s", name, ex__.what());                     \
        return PIC_ERR_ARG;                                                \
    }                                                                      \
    catch (...) {                                                          \
        ::pic::set_error("%s: unexpected error", name);                    \
        return PIC_ERR_ARG;                                                \
    }

// device-memory hooks installed by pic_set_allocator (nulls: cudaMalloc / cudaFree)
struct Allocator {
    pic_alloc_fn alloc = nullptr;
    pic_free_fn free = nullptr;
    void *ctx = nullptr;
};
Allocator current_allocator();

// Tensor-core inference state of a surrogate network (k_mlp_tc.cu): BF16 weights of every
// member and layer, zero-padded (inputs to multiples of 16, outputs to multiples of 32: a pair
// of SMs takes half each) and stored in the tensor core's no-swizzle K-major layout (8 x 8 core
// matrices, K-adjacent ones contiguous), and FP32 biases.  Usable when every layer width is at most 256.
constexpr int MLP_MAX_LAYERS = 16;
struct MlpTc {
    int E = 0, L = 0;
    int k[MLP_MAX_LAYERS] = {}, n[MLP_MAX_LAYERS] = {};    // widths: in, out
    int kp[MLP_MAX_LAYERS] = {}, np[MLP_MAX_LAYERS] = {};  // padded to 16 and 32
    long long woff[MLP_MAX_LAYERS] = {}, boff[MLP_MAX_LAYERS] = {};
    long long wmember = 0, bmember = 0;                     // elements per member
    uint16_t *w = nullptr;                                  // E * wmember BF16
    float *b = nullptr;                                     // E * bmember
    unsigned int *err = nullptr;                            // bounded-wait timeouts: a word of
                                                            // mapped host memory, zero between calls
    long long wait_polls = 1LL << 22;                       // polls of a pipeline wait
    bool ok = false;
};
// FP32 parameters (per member: W_l (n x k), b_l at woff / boff, member stride P) -> tc
void mlp_tc_pack(const MlpTc &tc, const float *params, long long P, const long long *woff,
                 const long long *boff, cudaStream_t s);
// Y (E x n x outputs, FP32) from X (n x inputs, FP32); PIC_ERR_TIMEOUT if a wait gave up
pic_status mlp_tc_forward(const MlpTc &tc, const float *X, float *Y, int64_t n, cudaStream_t s);
// One product of the training path on the tensor cores, per member z of E:
// C(z)[m][n] (+)= sum_k A(z, m, k) B(z, k, n), operands FP32 addressed by strides (as the
// CUDA-core GEMM takes them), rounded to BF16 into the packed scratch buffers (A: E x
// roundup(M, 128) x roundup(K, 16), B: E x roundup(N, 16) x roundup(K, 16) elements), FP32
// accumulation in TMEM.  Needs N <= 256 and K <= 256 (false: not done).  Bounded waits
// that give up are counted in *err.
struct TcGemmOp {
    const float *A, *B;
    float *C;
    int M, N, K;
    long long sAz, sBz, sCz;
    int sAm, sAk, sBk, sBn, ldc;
    int accumulate;
};
bool mlp_tc_gemm(const TcGemmOp &g, int E, uint16_t *scratch_a, uint16_t *scratch_b,
                 unsigned int *err, cudaStream_t s);

// ---- FP32 networks (k_mlp_f32.cu) ----
// One product of a layer for every member, and what is done with each element of it.
enum { MLP_FWD, MLP_DX, MLP_DW };   // A W^T, G W, G^T A
enum {
    MLP_EPI_STORE,      // C = x (DW: db = column sums of G, where db is set)
    MLP_EPI_BIAS,       // v = x + bias; C = v (and Z = v, where Z is set)
    MLP_EPI_GELU,       // the same with C = gelu(v)
    // from here on Z or C is read:
    MLP_EPI_LOSS,       // e = x + bias - Z; C = scale e; loss += e^2 / (M N), where loss is set
    MLP_EPI_GELU_GRAD,  // C = x gelu'(Z)
    MLP_EPI_ADAM,       // x is the gradient of C (am, av its moments), the column sums that of db
};
struct AdamArgs {
    float lr, b1, b2, eps, c1, c2;   // c1, c2: the bias corrections of this step
};
struct MlpJob {
    int kind, epi;
    int M, N, K;
    const float *A, *B;         // lda, ldb: stride of the index the operand is not contiguous along
    float *C;
    long long sA, sB, sC;       // member strides; db's is sC
    int lda, ldb, ldc;
    const float *bias;
    float *Z;                   // laid out like C, member stride sZ
    long long sbias, sZ;
    float *db, *am, *av, *dbm, *dbv;
    float scale;
    float *loss;
    AdamArgs adam;
};
constexpr int MLP_MAX_JOBS = MLP_MAX_LAYERS;
struct MlpJobs {
    MlpJob job[MLP_MAX_JOBS];   // in the order that the blocks take them
    int blocks[MLP_MAX_JOBS];
    int n = 0;
};
// the jobs in one launch (their results must not depend on each other)
void mlp_jobs(MlpJobs &jobs, int E, bool chain, cudaStream_t s);

// A batch's forward products, loss and gradients by the layers' sums (k_mlp_chain.cu): every
// width at most 256.
struct MlpChain {
    int E, L, rows;
    int sz[MLP_MAX_LAYERS + 1];
    long long batch, P;                                    // rows the arrays hold; member stride
    const float *params, *T;                               // parameters; targets (batch x outputs)
    long long woff[MLP_MAX_LAYERS], boff[MLP_MAX_LAYERS];
    float *act[MLP_MAX_LAYERS];                            // layer l's inputs; act[0] is read
    float *pre[MLP_MAX_LAYERS];                            // gradients by layer l's sums, on return
    float scale;                                           // of the gradient by the outputs
    float *loss;                                           // per member, added to; or null
};
// false: not for this many rows, nothing launched
bool mlp_chain(const MlpChain &a, bool chain, cudaStream_t s);

// Parameters as the whole-network kernel reads them: per member and layer the weights
// k-major (kp x np: kp the inputs up to a multiple of 16, np by mlp_f32_shape) and np biases.
struct MlpF32 {
    int E = 0, L = 0, NW = 0;                              // NW: 64, 128 or 256 units at most
    int k[MLP_MAX_LAYERS] = {}, n[MLP_MAX_LAYERS] = {};
    int kp[MLP_MAX_LAYERS] = {}, np[MLP_MAX_LAYERS] = {};
    long long woff[MLP_MAX_LAYERS] = {}, boff[MLP_MAX_LAYERS] = {};
    long long wmember = 0, bmember = 0;
    float *w = nullptr, *b = nullptr;
    bool ok = false;
};
struct MlpOffsets {
    long long w[MLP_MAX_LAYERS], b[MLP_MAX_LAYERS];        // in a member's parameters
};
int mlp_f32_shape(int maxw, int width);
void mlp_f32_pack(const MlpF32 &net, const float *params, long long P, const MlpOffsets &o,
                  cudaStream_t s);
// Y (E x n x outputs) from X (n x inputs)
pic_status mlp_f32_forward(const MlpF32 &net, const float *X, float *Y, int64_t n, cudaStream_t s);

#define PIC_CUDA_TRY(expr)                                                              \
    do {                                                                                \
        cudaError_t err__ = (expr);                                                     \
        if (err__ != cudaSuccess) {                                                     \
            ::pic::set_error("%s failed: %s (%s:%d)", #expr, cudaGetErrorString(err__), \
                             __FILE__, __LINE__);                                       \
            return PIC_ERR_CUDA;                                                        \
        }                                                                               \
    } while (0)

// ---------------------------------------------------------------------------------
// fixed point of the FP32 build
// ---------------------------------------------------------------------------------
// Barycentric coordinates are stored as integers in units of 2^-22 that sum to exactly
// 2^22.  The current of a segment, lambda_a^s lambda_b^e - lambda_b^s lambda_a^e, is then
// an exact integer in units of 2^-44 and node charges are integers in units of 2^-22:
// every scatter sum is exact and independent of summation order, and the discrete
// continuity equation holds identically in integers.
constexpr int LAM_BITS = 22;
constexpr int32_t LAM_ONE = 1 << LAM_BITS;
constexpr double LAM_INV = 1.0 / (double)LAM_ONE;
constexpr double J_INV = LAM_INV * LAM_INV;  // 2^-44

// ---------------------------------------------------------------------------------
// host mesh and operators
// ---------------------------------------------------------------------------------
struct HostMesh {
    pic_units units{};
    int64_t N0 = 0, N1 = 0, N2 = 0;
    std::vector<double> zr;            // N0 x 2 (z, rho)
    std::vector<int32_t> tri;          // N2 x 3, counter-clockwise in (z, rho)
    std::vector<int32_t> tri_edge;     // N2 x 3, local edge k opposite local node k
    std::vector<int32_t> tri_nbr;      // N2 x 3, neighbour across local edge k or -1
    std::vector<int32_t> edge_nodes;   // N1 x 2 (tail = lower index, head)
    std::vector<int32_t> edge_tag;     // N1: 0 interior or PIC_BC_*
    std::vector<int32_t> edge_face;    // N1 x 2 faces (or -1)
    std::vector<int8_t> edge_face_sign;// N1 x 2: D_curl entry of (face, edge)
    std::vector<double> area;          // N2
    std::vector<double> grad;          // N2 x 3 x 2: grad(lambda_k) (d/dz, d/drho)
    std::vector<double> mu_inv;        // N2: diagonal of star_mu^-1
    std::vector<int64_t> eps_ptr;      // star_eps in CSR, N1 rows
    std::vector<int32_t> eps_idx;
    std::vector<double> eps_val;
    std::vector<int32_t> free_edges;   // non-PEC edges, ascending
    std::vector<int32_t> free_of_edge; // N1: index in free_edges or -1
    std::vector<uint8_t> node_on_pec;  // N0
    bool have_spai = false;
    std::vector<int64_t> M_ptr;        // SPAI M in CSR over free edges
    std::vector<int32_t> M_idx;
    std::vector<double> M_val;
    double dt_stable = 0.0;
    double lambda_max = 0.0;
    // uniform bucket grid over triangle bounding boxes, for point location
    double bb_z0 = 0, bb_r0 = 0, bb_h = 1;
    int64_t bb_nz = 0, bb_nr = 0;
    std::vector<int64_t> bb_ptr;
    std::vector<int32_t> bb_tri;
};

// local edge k joins local nodes (k+1)%3 and (k+2)%3; its tail is the lower node index
inline void edge_tail_head(const int32_t *n3, int k, int *a, int *b) {
    int i = (k + 1) % 3, j = (k + 2) % 3;
    if (n3[i] < n3[j]) { *a = i; *b = j; } else { *a = j; *b = i; }
}

// run f(begin, end) over [0, n) on the host's cores, at least `grain` items a thread: a
// thread takes some 30 us to start, so light loops ask for thousands.  The caller takes a part
// too, and the parts of threads that do not start.  An exception thrown by f is thrown on
// once every thread is done (the first part's of several).
template <class F>
void parallel_for(int64_t n, F &&f, int64_t grain = 1) {
    unsigned nt = std::max(1u, std::min(64u, std::thread::hardware_concurrency()));
    nt = (unsigned)std::max<int64_t>(1, std::min<int64_t>(nt, n / grain));
    if (n < 4096 || nt == 1) {
        f((int64_t)0, n);
        return;
    }
    const int64_t chunk = (n + nt - 1) / nt;
    std::vector<std::exception_ptr> thrown(nt);
    const auto part = [&](unsigned i) {
        const int64_t a = std::min(n, (int64_t)i * chunk), b = std::min(n, a + chunk);
        if (a >= b) return;
        try {
            f(a, b);
        } catch (...) {
            thrown[i] = std::current_exception();
        }
    };
    std::vector<std::thread> th;
    th.reserve(nt);   // nothing below throws but the start of a thread
    unsigned started = 1;
    try {
        for (; started < nt; started++) th.emplace_back(part, started);
    } catch (...) {
    }
    part(0);
    for (unsigned i = started; i < nt; i++) part(i);
    for (auto &t : th) t.join();
    for (const auto &e : thrown)
        if (e) std::rethrow_exception(e);
}

void build_locator(HostMesh &m);
// containing triangle (largest smallest barycentric coordinate) or -1; lam[3] out
int32_t locate_point(const HostMesh &m, double z, double rho, double lam[3]);
// intervals of the line z = z0, rho in [rho0, rho1], per triangle crossed (sorted, with
// the barycentric coordinates at both ends); false if the line leaves the mesh, passes
// through a node's z or the intervals do not tile [rho0, rho1]
bool build_emit_line(const HostMesh &m, double z0, double rho0, double rho1,
                     std::vector<double> &rho_a, std::vector<double> &rho_b,
                     std::vector<double> &lam_a, std::vector<double> &lam_b,
                     std::vector<int32_t> &tri);

// Kernels the library has enqueued for execution in this process.  Every launch site adds
// one; a stream capture runs nothing, so the kernels it recorded are taken back out and
// added again at each replay of the graph.
void note_launches(long long k);
long long launches_this_thread();
#define PIC_LAUNCHED() ::pic::note_launches(1)

// Launch of a kernel of a dependent chain: its blocks may take their places before the
// kernel ahead of it has completed and its writes are visible, and wait for that
// (griddepcontrol.wait, in chain_wait, ahead of which a kernel only reads what no kernel of
// the chain writes).
//
// When the blocks of the kernel behind may come is the kernel ahead's choice, made after its
// own wait, so that whatever a kernel has waited for has completed before its successor
// starts.  A small grid (at most CHAIN_EARLY threads) leaves most SMs idle and lets them come
// at once; a large one as its own blocks finish, because blocks that wait hold places and
// registers that working ones could use.  Measured, at once / as blocks finish / by this
// rule: 200 FP64 steps on 2000 triangles with 10,000 particles 1971 / 2075 /
// 2001 us, 8 of 1M FP64 particles on 199k triangles 3267 / 2827 / 2842 us, 64 of eight
// surrogate instances 2600 / 2327 / 2283 us, 16M particles 290 / 285 / 284 us a step.
//
// chain = false: an ordinary launch, for the first kernel of a call and for one that
// follows an event wait (what it depends on is then not a kernel of this stream).
constexpr unsigned CHAIN_EARLY = 32768;
#ifdef __CUDACC__
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (gridDim.x * gridDim.y * blockDim.x <= CHAIN_EARLY)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif
template <class... Params, class... Args>
void launch_chained(bool chain, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem,
                    cudaStream_t s, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = chain ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
    PIC_LAUNCHED();
}

// ---------------------------------------------------------------------------------
// device layouts
// ---------------------------------------------------------------------------------
// One record per triangle, read by the particle kernel: static geometry and topology,
// plus the per-step field coefficients written by the field kernel.  The E field inside
// the triangle is linear in lambda: E(lambda) = sum_k lambda_k c_k (components z, rho);
// bphi = (B^{n+1/2} + B^{n-1/2}) / (2 A) is the time-centred B_phi (W2 = 1/A).
template <class R>
struct alignas(sizeof(R) == 4 ? 128 : 64) TriRec {
    R g[4];       // grad lambda_0 (z, rho), grad lambda_1 (z, rho); grad lambda_2 = -g0 - g1
    R rho[3];     // node rho
    R inv_area;
    R c[6];       // c_0 (z, rho), c_1, c_2
    R bphi;
    R pad;
    int32_t node[3];
    int32_t flags; // bit k: local edge k runs (k+1)%3 -> (k+2)%3 (D_curl entry +1)
    int32_t edge[3];
    int32_t eflags; // = flags, beside the edges: one 16-byte load gives both
    int32_t nbr[3]; // neighbour triangle, or -(PIC_BC_* tag) on the boundary
    int32_t entry;  // bits 2k, 2k+1: local index, in nbr[k], of the node opposite the
                    // shared edge (the mesh is conforming and counter-clockwise, so the
                    // neighbour runs that edge the other way: its node entry+1 is this
                    // triangle's node k+2, its node entry+2 is node k+1)
};

// FP32 build: the currents of a step are summed per triangle and taken apart into edge
// currents once, by the residual kernel.  With the local edges oriented counter-clockwise
// (edge 0: 1->2, 1: 2->0, 2: 0->1) a segment s -> e in one triangle carries (Eq. current)
//   A0 = s1 e2 - s2 e1,  A1 = s2 e0 - s0 e2,  A2 = s0 e1 - s1 e0,
// and because s and e both sum to 2^22, the net outflow at each node is
//   A2 - A1 = 2^22 (s0 - e0),  A0 - A2 = 2^22 (s1 - e1)   (the identity behind Eq. DCE),
// so one product pair (A1) and two differences determine all three, also after summing
// over the segments in the triangle; and the charge that leaves node k through the
// triangle is the sum of s_k - e_k.  Beside the sums, in the same 32-byte sector, what the
// residual kernel needs of the triangle's B.  Read and written in 16-byte words.
struct alignas(32) FaceSum {
    unsigned long long d0, d1;   // sums of s0 - e0 and s1 - e1 (two's complement)
    unsigned long long a1;       // sum of A1
    double h;                    // star_mu^-1 B^{n+1/2}
};
static_assert(offsetof(FaceSum, d0) == 0 && offsetof(FaceSum, d1) == 8 && offsetof(FaceSum, a1) == 16 &&
                  offsetof(FaceSum, h) == 24 && sizeof(FaceSum) == 32,
              "d0, d1 and a1, h are a 16-byte word each");

struct PF32 {
    using R = float;
    using Lam = int32_t;
    using Acc = unsigned long long;  // two's-complement int64 accumulators
    static constexpr bool fixed = true;
};
struct PF64 {
    using R = double;
    using Lam = double;
    using Acc = double;
    static constexpr bool fixed = false;
};

template <class P>
struct Particles {
    int32_t *tri = nullptr;
    typename P::Lam *l0 = nullptr, *l1 = nullptr;
    typename P::R *ur = nullptr, *up = nullptr, *uz = nullptr;
    int32_t *pid = nullptr;
};

enum {
    CNT_ABSORBED = 0,
    CNT_OVERFLOW = 1,
    CNT_CROSSINGS = 2,
    CNT_TILE = 3,       // FP32 particle kernel: tiles taken so far from the shared end (zeroed per step)
    CNT_TIMEOUT = 4,    // bounded device waits that gave up (must stay 0)
    CNT_EMITTED = 5,    // particles born by the emitter
    CNT_NEXT_PID = 6,   // next particle id once an emitter was set
    CNT_EMIT_DROPPED = 7,   // particles the emitter did not make for lack of room
    CNT_EMIT_TICKET = 8,    // emission blocks done in this step
    CNT_N = 9
};
// slots past the capacity that the particle arrays keep for 16-byte bulk-copy rounding
constexpr int64_t SLOT_PAD = 8;

template <class P>
struct PushArgs {
    const TriRec<typename P::R> *rec;
    Particles<P> p;
    // device count of slots; behind it how many of them the last re-sort ordered (births
    // since then follow them), unless `sorted` says that all are in order
    const int64_t *n_slots;
    bool sorted = false;
    typename P::Acc *J;         // FP64: N1 edge currents, units q_src/dt
    FaceSum *face;              // FP32: N2 current sums, units 2^-44 and 2^-22 of q_src/dt
    typename P::Acc *Q;         // N0, Q^{n+1}, units 2^-22 / 1 of q_src
    typename P::Acc *Qabs;      // N0
    unsigned long long *counters;
    typename P::R qmdt2;        // q dt / (2 m)
    typename P::R dt;
    typename P::R inv_c2;
    typename P::R bz;
    int32_t walk_cap;
    int32_t ctas_per_sm;        // launch shape: persistent CTAs per SM (0: as many as fit)
    int32_t pusher;             // PIC_PUSHER_BORIS or PIC_PUSHER_VAY (Eq. DLE)
    int64_t wait_polls;         // FP32 kernel: polls before a tile-pipeline wait gives up
    bool chain = true;          // launched behind a kernel of the step (launch_chained)
};
// default of PushArgs::wait_polls (each poll suspends the thread for at most 100 us)
constexpr int64_t PUSH_WAIT_POLLS = 1LL << 14;

// Emission line z = const, cut into the triangles it crosses: interval k spans
// rho in [rho_a[k], rho_b[k]] inside triangle tri[k], with barycentric coordinates lam_a
// and lam_b (3 each) at its ends (linear in between).
struct EmitLine {
    const double *rho_a, *rho_b, *lam_a, *lam_b;
    const int32_t *tri;
    int32_t n;
};

template <class P>
struct EmitArgs {
    EmitLine line;
    Particles<P> p;
    const TriRec<typename P::R> *rec;
    int64_t *n_slots;
    unsigned long long *counters;
    typename P::Acc *Qn;        // Q^n: the births' charge is added here
    typename P::Acc *Qwall;     // and taken out of the Gauss-law bookkeeping here
    int64_t cap, per_step;
    double rho0, rho1, u_normal, u_thermal;
    unsigned long long seed;
};

// field probes: group g owns entries [ptr[g], ptr[g+1]) of (face, weight); state[0] is
// the step phase, state[1] the records written, state[2] the records dropped
template <class P>
struct ProbeArgs {
    const typename P::R *B;
    const int64_t *ptr;
    const int32_t *face;
    const double *weight;
    const int32_t *power;
    double *buf;            // capacity x n_groups
    long long *state;
    unsigned *done;
    int32_t n_groups = 0, every = 1;
    long long capacity = 0;
};

// output ports: port k owns entries [ptr[k], ptr[k+1]) of (triangle, barycentric point,
// quadrature weight); between the face kernels of two steps, P_k = sum w E_rho(lambda) B_phi
// from the triangle records (E^n and the time-centred B_phi); every `every` steps the
// ports' values are appended to a device buffer; state as for the probes
template <class P>
struct PortArgs {
    const TriRec<typename P::R> *rec;
    const int64_t *ptr;
    const int32_t *tri;
    const double *lam;      // 3 per entry
    const double *weight;
    double *buf;            // capacity x n_ports
    long long *state;
    unsigned *done;
    int32_t n_ports = 0, every = 1;
    long long capacity = 0;
};

template <class P>
struct FieldArgs {
    TriRec<typename P::R> *rec;
    typename P::R *E;           // N1
    const typename P::R *Es;    // N1 static field added at the gather only, or null
    // lossy (absorbing) layer, or null: per free-edge row (a, b) with
    // E <- a E + b dt (M r), per face (a, b) with B <- a B - b dt (D_curl E)
    const typename P::R *loss_e;  // nf x 2
    const typename P::R *loss_f;  // N2 x 2
    typename P::R *B;           // N2, B^{n-1/2} in, B^{n+1/2} out
    const typename P::R *mu_inv;// N2
    const int32_t *edge_face;   // N1 x 2, per edge: (4 face + local edge + 1) * sign, 0 if none
    const int32_t *free_edges;  // nf
    const int32_t *free_of_edge;// N1: index in free_edges or -1
    // FP64: edge currents, zeroed by the face kernel before the particle step; FP32: written
    // by the residual kernel from the triangles' sums, which the face kernel zeroes
    typename P::Acc *J;
    FaceSum *face;
    double *D;                  // N1 auxiliary dual flux (DGL)
    typename P::R *r;           // nf scratch: D_curl^T star_mu^-1 B - J
    // M in sliced ELL: slices of 32 rows, column-major inside a slice
    const int64_t *ell_off;     // n_slices + 1, element offset of each slice
    const int32_t *ell_col;
    const typename P::R *ell_val;
    int64_t N1, N2, nf;
    typename P::R dt;
    double dt64;                // dt as the fields see it: (double)dt
    double j_scale;             // physical J = J_acc * j_scale
    // FP32 build: Q^{n+1} = Q^n - D_div J / 2^22 - Q_absorbed per node (exact)
    const int32_t *face_ptr;    // N0 + 1: node -> incident triangles
    const int32_t *node_face;   // 4 triangle + local node
    const typename P::Acc *Qn;
    typename P::Acc *Qabs;      // N0 (zeroed by the face kernel before the particle step)
    typename P::Acc *Qnext;
    typename P::Acc *Qwall;     // N0: charge removed at walls since the Gauss-law reference
    unsigned long long *counters;
    int64_t N0;
    int32_t block;              // launch shape: threads per block (<= 512)
    bool chain = true;          // the face kernel is launched behind a kernel of the last step
};

template <class P> void launch_push(const PushArgs<P> &a, int64_t n_bound, cudaStream_t s);
void launch_push_f32(const PushArgs<PF32> &a, int64_t n_bound, cudaStream_t s);
// emit: births to make beside the face kernel, or null
template <class P>
void launch_field_b(const FieldArgs<P> &a, const EmitArgs<P> *emit, cudaStream_t s);
// probe, port: recorded beside the residual kernel; no groups, no ports: none
template <class P>
void launch_field_e(const FieldArgs<P> &a, const ProbeArgs<P> &probe, const PortArgs<P> &port,
                    cudaStream_t s);
template <class P>
void launch_deposit_q(const TriRec<typename P::R> *rec, Particles<P> p, int64_t first,
                      int64_t count, const int64_t *n_slots, typename P::Acc *Q, cudaStream_t s);

struct SortScratch {
    int32_t *cnt = nullptr;      // N2: counts, zero between re-sorts
    int32_t *cursor = nullptr;   // N2: write cursors
    int32_t *blk = nullptr;      // scan chunk sums
    int64_t *n_old = nullptr;    // slot count before the sort
};
// stable-enough counting sort by triangle; drops removed particles; writes the new
// slot count to n_slots[0] and n_slots[1] (device)
template <class P>
void launch_resort(Particles<P> src, Particles<P> dst, int64_t *n_slots, int64_t n_bound,
                   int64_t N2, const SortScratch &sc, bool chain, cudaStream_t s);

// diagnostics, FP64 reductions on the device
struct DiagDev {
    const int64_t *node_ptr;     // N0 + 1: node -> incident edges (CSR)
    const int32_t *node_edge;    // incident edge
    const int8_t *node_sign;     // D_div entry: +1 tail, -1 head
    const uint8_t *node_on_pec;  // N0
    const int64_t *eps_ptr;      // star_eps CSR
    const int32_t *eps_idx;
    const double *eps_val;
    int64_t N0, N1, N2;
};
// out[0]: max |dce| (units of q_src), out[1]: count of nonzero dce (fixed: exact),
// out[2]: max |NR_DCE|, out[3]: max |dgl - ref|, out[4]: max |Q|, out[5]: field energy,
// out[6]: sum (gamma - 1) over live particles
template <class P>
void launch_diag(const DiagDev &d, const typename P::Acc *J, const typename P::Acc *Qn,
                 const typename P::Acc *Qp, const typename P::Acc *Qabs,
                 const typename P::Acc *Qpos, const typename P::Acc *Qwall, const double *D,
                 double *dgl_ref, int set_ref, const typename P::R *E,
                 const typename P::R *B, const typename P::R *mu_inv, Particles<P> p,
                 const int64_t *n_slots, int64_t n_bound, double q_scale, double inv_c2,
                 double *out, cudaStream_t s);
template <class P>
void launch_export(Particles<P> p, int64_t n, const TriRec<typename P::R> *rec,
                   double *lam3, double *u3, int64_t *pid, cudaStream_t s);
// arrays to be read back as FP64: fields as they are, accumulators times a scale; array q's
// n[q] values go to out + at[q]
template <class P>
struct ReadArgs {
    const typename P::R *field[4] = {};
    const typename P::Acc *acc[4] = {};
    double scale[4] = {};
    int64_t n[4] = {}, at[4] = {};
    int count = 0;
    int64_t total = 0;
    int64_t add(const typename P::R *f, const typename P::Acc *x, double sc, int64_t m) {
        field[count] = f;
        acc[count] = x;
        scale[count] = sc;
        n[count] = m;
        at[count] = total;
        total += m;
        return at[count++];
    }
};
template <class P>
void launch_read(const ReadArgs<P> &a, double *out, cudaStream_t s);

}  // namespace pic

struct pic_mesh {
    pic::HostMesh h;
};
