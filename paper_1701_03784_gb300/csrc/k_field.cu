// Field update of the mixed E-B leapfrog (Eqs. full_d_dfl, full_d_dal) and the per-step
// triangle field records read by the particle kernel.
#include <algorithm>
#include <type_traits>

#include "emit.h"
#include "pic_internal.h"
#include "record.h"

namespace pic {

// The kernels of a step are chained (launch_chained): a kernel's blocks take their places
// while the one before it drains, load what never changes after creation (geometry,
// incidence, matrix entries), wait, and only then touch anything that a kernel writes.
// Measured with graph replay on 2000 triangles and 10,000 particles (FP64): 12.8 -> 9.5 us
// a step; 32 steps enqueued one by one on 47k triangles and 500k particles: 1824 -> 1737 us.

// s flipped where the edge runs against the counter-clockwise boundary
template <class R>
__device__ __forceinline__ R along(R e, bool fwd) { return fwd ? e : -e; }

// K3, one thread per face: B^{n+1/2} = B^{n-1/2} - dt (D_curl E^n)_f, and the record's
// field coefficients: E(lambda) = sum_k E_k (lambda_a grad lambda_b - lambda_b grad
// lambda_a) = sum_m lambda_m c_m (E_k plus the static field's edge value when one is set:
// it drives the particles but takes no part in the leapfrog), and
// B_phi = (B^{n+1/2} + B^{n-1/2}) / (2A) (W2 = 1/A).  In a lossy layer
// B^{n+1/2} = a_f B^{n-1/2} - b_f dt (D_curl E^n)_f.
// The same launch clears the step's accumulators (the current sums per triangle, in the
// FP64 build J per edge; Q_abs per node; and in the FP64 build Q^{n+1}, which the particle
// kernel accumulates).  Its first emit_blocks blocks
// make the step's births (emit.h).
// The record is read and written in 16-byte words (g | rho, 1/A | c0 c1 c2, B_phi, pad |
// nodes, flags | edges, flags); in 8-byte ones the FP64 build's stores alone kept a launch
// on 199k faces at 27 us.
template <class P, bool STATIC, bool LOSS, bool EMIT>
__global__ void __launch_bounds__(512) k_field_b(const __grid_constant__ FieldArgs<P> a,
                                                 const __grid_constant__ EmitArgs<P> em, int emit_blocks) {
    using R = typename P::R;
    using R4 = typename std::conditional<sizeof(R) == 4, float4, double2>::type;   // 16 bytes
    constexpr int W = 16 / sizeof(R);
    if constexpr (EMIT) {
        if ((int)blockIdx.x < emit_blocks) {
            chain_wait();
            emit_block<P>(em, blockIdx.x, emit_blocks);
            return;
        }
    }
    const int64_t f = (int64_t)(blockIdx.x - (EMIT ? emit_blocks : 0)) * blockDim.x + threadIdx.x;
    const bool face = f < a.N2;
    R g[2][2] = {}, inv_area = 0, mu = 0;
    int4 EG = make_int4(0, 0, 0, 0);
    if (face) {
        const R *rc = reinterpret_cast<const R *>(a.rec + f);
        R w[8];   // g (4), rho (3), 1/A
#pragma unroll
        for (int k = 0; k < 8; k += W) *reinterpret_cast<R4 *>(w + k) = *reinterpret_cast<const R4 *>(rc + k);
        g[0][0] = w[0];
        g[0][1] = w[1];
        g[1][0] = w[2];
        g[1][1] = w[3];
        inv_area = w[7];
        EG = *reinterpret_cast<const int4 *>(a.rec[f].edge);
        if constexpr (P::fixed) mu = a.mu_inv[f];
    }
    chain_wait();
    if constexpr (!P::fixed) {
        if (f < a.N1) a.J[f] = 0;
    } else if (f == 0) {
        a.counters[CNT_TILE] = 0;
    }
    if (f < a.N0) {
        a.Qabs[f] = 0;
        if constexpr (!P::fixed) a.Qnext[f] = 0;
    }
    if (!face) return;
    // edge values along the counter-clockwise boundary (edge k: local node k+1 -> k+2)
    const int e3[3] = {EG.x, EG.y, EG.z};
    R E3[3], s[3];
#pragma unroll
    for (int k = 0; k < 3; k++) E3[k] = a.E[e3[k]];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const bool fwd = (EG.w >> k) & 1;
        s[k] = along<R>(STATIC ? E3[k] + a.Es[e3[k]] : E3[k], fwd);   // the gather sees the static field
        E3[k] = along<R>(E3[k], fwd);
    }
    const R Bold = a.B[f];
    const R curl = (E3[0] + E3[1]) + E3[2];
    R Bnew = Bold - a.dt * curl;
    if constexpr (LOSS) Bnew = a.loss_f[2 * f] * Bold - a.loss_f[2 * f + 1] * (a.dt * curl);
    a.B[f] = Bnew;
    if constexpr (P::fixed) {
        FaceSum &fs = a.face[f];
        *reinterpret_cast<longlong2 *>(&fs.d0) = make_longlong2(0, 0);
        *reinterpret_cast<longlong2 *>(&fs.a1) = make_longlong2(0, __double_as_longlong((double)mu * (double)Bnew));
    }
    R w[8];
#pragma unroll
    for (int d = 0; d < 2; d++) {
        const R g0 = g[0][d], g1 = g[1][d], g2 = -g0 - g1;
        w[d] = fma(s[2], g1, -(s[1] * g2));
        w[2 + d] = fma(-s[2], g0, s[0] * g2);
        w[4 + d] = fma(s[1], g0, -(s[0] * g1));
    }
    w[6] = R(0.5) * (Bnew + Bold) * inv_area;
    w[7] = 0;
    R *out = reinterpret_cast<R *>(a.rec + f) + 8;
#pragma unroll
    for (int k = 0; k < 8; k += W) *reinterpret_cast<R4 *>(out + k) = *reinterpret_cast<R4 *>(w + k);
}

// A 64-bit integer as a double in two FP64 additions: each half becomes the low bits of a
// double's mantissa (at 2^52 and 2^84), whose offsets are then taken out.  The first addition
// is exact (multiples of 2^32 that come out below 2^64), the second rounds once: the nearest
// double.
__device__ __forceinline__ double to_double(long long v) {
    const double lo = __hiloint2double(0x43300000, (int)v);                                   // 2^52 + low
    const double hi = __hiloint2double(0x45300000, (int)((unsigned)(v >> 32) ^ 0x80000000u)); // 2^84 + (high + 2^31) 2^32
    return (hi - (0x1.0p84 + 0x1.0p63 + 0x1.0p52)) + lo;
}

// K4a, one thread per edge: in the FP32 build its current from the sums of its triangles;
// on free edges r = D_curl^T star_mu^-1 B^{n+1/2} - J^{n+1/2} and the DGL auxiliary flux
// D += dt r.  The first blocks record probes and ports (record.h).
//
// One thread per node, in the same launch: in the FP32 build Q^{n+1} = Q^n - (D_div J)/2^22
// - Q_absorbed, where (D_div J)/2^22 is the charge that left the node through its triangles
// (FaceSum), which equals Eq. charge evaluated at the new positions exactly (the
// diagnostics compare); in both builds the charge removed at walls is summed since the
// Gauss-law reference.
//
// FP64 instructions take 16 cycles of an SM each (49% of its time on the 200k-triangle mesh
// with the integer and dt converted by the compiler's rules): r and D need five.
// Bound by the sectors it gathers from triangles that lie anywhere in memory: two an edge
// and six a node, of 32 bytes each (with B, star_mu^-1 and the sums in arrays of their own
// it was six an edge, and eight surrogate instances' 64 steps took 2956 us instead of 2676).
template <class P, bool REC>
__global__ void __launch_bounds__(512) k_field_r(const __grid_constant__ FieldArgs<P> a,
                                                 const __grid_constant__ ProbeArgs<P> probe,
                                                 const __grid_constant__ PortArgs<P> port) {
    using R = typename P::R;
    int blk = blockIdx.x;
    if constexpr (REC) {
        if (blk < probe.n_groups + port.n_ports) {
            chain_wait();
            if (blk < probe.n_groups) probe_block<P>(probe, blk);
            else port_block<P>(port, blk - probe.n_groups);
            return;
        }
        blk -= probe.n_groups + port.n_ports;
    }
    const int64_t e = (int64_t)blk * blockDim.x + threadIdx.x;
    int fs[2] = {0, 0}, i = -1;
    R mu[2] = {0, 0};
    if (e < a.N1) {
        const int2 ef = reinterpret_cast<const int2 *>(a.edge_face)[e];
        fs[0] = ef.x;
        fs[1] = ef.y;
        i = a.free_of_edge[e];
    }
    // a node's triangles: the first NEAR of them before the wait (six on average)
    constexpr int NEAR = P::fixed ? 7 : 1;
    int near[NEAR], q0 = 0, q1 = 0;
    if constexpr (P::fixed) {
        if (e < a.N0) {
            q0 = a.face_ptr[e];
            q1 = a.face_ptr[e + 1];
        }
#pragma unroll
        for (int q = 0; q < NEAR; q++)
            if (q0 + q < q1) near[q] = a.node_face[q0 + q];
    } else {
#pragma unroll
        for (int q = 0; q < 2; q++)
            if (fs[q] != 0) mu[q] = a.mu_inv[(abs(fs[q]) - 1) >> 2];
    }
    chain_wait();
    if (e < a.N1) {
        double h[2] = {0.0, 0.0};
        long long J = 0;
#pragma unroll
        for (int q = 0; q < 2; q++) {
            if (fs[q] == 0) continue;
            const int fk = abs(fs[q]) - 1, f = fk >> 2;
            if constexpr (P::fixed) {
                const FaceSum &sum = a.face[f];
                const longlong2 d = *reinterpret_cast<const longlong2 *>(&sum.d0);
                const longlong2 ah = *reinterpret_cast<const longlong2 *>(&sum.a1);
                long long A = ah.x;                                  // edge 1
                if ((fk & 3) != 1) A += d.x << LAM_BITS;             // edge 2
                if ((fk & 3) == 0) A += d.y << LAM_BITS;             // edge 0
                J += fs[q] > 0 ? A : -A;
                h[q] = __longlong_as_double(ah.y);
            } else {
                h[q] = mu[q] * a.B[f];
            }
            if (fs[q] < 0) h[q] = -h[q];
        }
        if constexpr (P::fixed) a.J[e] = (unsigned long long)J;
        if (i >= 0) {
            double r = h[0] + h[1];
            if constexpr (P::fixed) {
                if (J != 0) r -= to_double(J) * a.j_scale;   // no beam over most of a mesh
            } else {
                r -= a.J[e] * a.j_scale;
            }
            a.D[e] += a.dt64 * r;
            a.r[i] = (R)r;
        }
    }
    if (e >= a.N0) return;
    const typename P::Acc gone = a.Qabs[e];
    if constexpr (P::fixed) {
        long long out = 0;
        const auto left = [&](int fk) {
            const longlong2 d = *reinterpret_cast<const longlong2 *>(&a.face[fk >> 2].d0);
            const int k = fk & 3;
            out += k == 0 ? d.x : k == 1 ? d.y : -(d.x + d.y);
        };
#pragma unroll
        for (int q = 0; q < NEAR; q++)
            if (q0 + q < q1) left(near[q]);
        for (int q = q0 + NEAR; q < q1; q++) left(a.node_face[q]);
        a.Qnext[e] = a.Qn[e] - (unsigned long long)out - gone;
    }
    a.Qwall[e] += gone;
}

// K4b, sliced ELL SpMV over free edges: E_e += dt (M r)_i (in a lossy layer
// E_e <- a_e E_e + b_e dt (M r)_i, a = (1 - s)/(1 + s), b = 1/(1 + s), s = sigma dt/(2 eps0)).  A warp owns a slice of 32 rows
// stored column-major, so each step of the row loop reads 32 consecutive values.  FP32: at
// most 32 registers, so that 300k rows are one wave (40 took 1% of a step more).
template <class P, bool LOSS>
__global__ void __launch_bounds__(512, sizeof(typename P::R) == 4 ? 4 : 1) k_field_spmv(const __grid_constant__ FieldArgs<P> a) {
    using R = typename P::R;
    int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t slice = row >> 5;
    int lane = (int)(row & 31);
    int64_t n_slices = (a.nf + 31) >> 5;
    if (slice >= n_slices) {
        chain_wait();
        return;
    }
    const int64_t off = a.ell_off[slice];
    const int width = (int)((a.ell_off[slice + 1] - off) >> 5);
    const int32_t *cols = a.ell_col + off + lane;
    const R *vals = a.ell_val + off + lane;
    // HEAD columns' indices and values are in flight before the wait, four at a time after
    // (the sum keeps the column order).  More of them ahead cost occupancy: 12 take 78
    // registers, and 32 steps of the 200k-triangle BWO 12.14 ms; 8 12.03 ms; 4 11.98 ms
    constexpr int HEAD = 4;
    int32_t col[HEAD];
    R val[HEAD];
#pragma unroll
    for (int u = 0; u < HEAD; u++)
        if (u < width) {
            col[u] = cols[u * 32];
            val[u] = vals[u * 32];
        }
    const int32_t e = row < a.nf ? a.free_edges[row] : 0;
    chain_wait();
    R acc = 0;
    {
        R rv[HEAD];
#pragma unroll
        for (int u = 0; u < HEAD; u++)
            if (u < width) rv[u] = a.r[col[u]];
#pragma unroll
        for (int u = 0; u < HEAD; u++)
            if (u < width) acc += val[u] * rv[u];
    }
    int k = HEAD;
    for (; k + 4 <= width; k += 4) {
        int32_t c4[4];
        R v4[4], r4[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            c4[u] = cols[(int64_t)(k + u) * 32];
            v4[u] = vals[(int64_t)(k + u) * 32];
        }
#pragma unroll
        for (int u = 0; u < 4; u++) r4[u] = a.r[c4[u]];
#pragma unroll
        for (int u = 0; u < 4; u++) acc += v4[u] * r4[u];
    }
    for (; k < width; k++) acc += vals[(int64_t)k * 32] * a.r[cols[(int64_t)k * 32]];
    if (row < a.nf) {
        if constexpr (LOSS) a.E[e] = a.loss_e[2 * row] * a.E[e] + a.loss_e[2 * row + 1] * (a.dt * acc);
        else a.E[e] += a.dt * acc;
    }
}

template <class P>
void launch_field_b(const FieldArgs<P> &a, const EmitArgs<P> *emit, cudaStream_t s) {
    const int64_t n = std::max(a.N2, P::fixed ? a.N0 : std::max(a.N1, a.N0));
    const int b = a.block;
    const bool births = emit && emit->per_step > 0 && emit->line.n > 0;
    const EmitArgs<P> em = births ? *emit : EmitArgs<P>{};
    // a birth a thread, up to one block an SM or so: beyond that the threads take several
    const int eb = births ? (int)std::min<int64_t>((em.per_step + b - 1) / b, 1024) : 0;
    const unsigned g = (unsigned)((n + b - 1) / b + eb);
    // the optional static field, lossy layer and emission as instantiations: none costs the
    // common case anything
    const auto go = [&](auto kernel) { launch_chained(a.chain, kernel, g, b, 0, s, a, em, eb); };
    if (births) {
        if (a.Es && a.loss_f) go(k_field_b<P, true, true, true>);
        else if (a.Es) go(k_field_b<P, true, false, true>);
        else if (a.loss_f) go(k_field_b<P, false, true, true>);
        else go(k_field_b<P, false, false, true>);
    } else {
        if (a.Es && a.loss_f) go(k_field_b<P, true, true, false>);
        else if (a.Es) go(k_field_b<P, true, false, false>);
        else if (a.loss_f) go(k_field_b<P, false, true, false>);
        else go(k_field_b<P, false, false, false>);
    }
}

template <class P>
void launch_field_e(const FieldArgs<P> &a, const ProbeArgs<P> &probe, const PortArgs<P> &port,
                    cudaStream_t s) {
    const int64_t n = std::max(a.N1, a.N0);
    const int b = a.block, nr = probe.n_groups + port.n_ports;
    const unsigned g = (unsigned)((n + b - 1) / b + nr);
    if (nr > 0) launch_chained(true, k_field_r<P, true>, g, b, 0, s, a, probe, port);
    else launch_chained(true, k_field_r<P, false>, g, b, 0, s, a, probe, port);
    int64_t rows = ((a.nf + 31) / 32) * 32;
    const unsigned gs = (unsigned)((rows + b - 1) / b);
    if (a.loss_e) launch_chained(true, k_field_spmv<P, true>, gs, b, 0, s, a);
    else launch_chained(true, k_field_spmv<P, false>, gs, b, 0, s, a);
}

template void launch_field_b<PF32>(const FieldArgs<PF32> &, const EmitArgs<PF32> *, cudaStream_t);
template void launch_field_b<PF64>(const FieldArgs<PF64> &, const EmitArgs<PF64> *, cudaStream_t);
template void launch_field_e<PF32>(const FieldArgs<PF32> &, const ProbeArgs<PF32> &, const PortArgs<PF32> &,
                                   cudaStream_t);
template void launch_field_e<PF64>(const FieldArgs<PF64> &, const ProbeArgs<PF64> &, const PortArgs<PF64> &,
                                   cudaStream_t);

}  // namespace pic
