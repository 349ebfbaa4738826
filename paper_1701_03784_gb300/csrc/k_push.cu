// K1, FP64 build: fused particle step -- Whitney gather, relativistic push, rotate-back to the
// meridian plane, triangle walk with segment splitting, charge-conserving scatter.  (The
// FP32 build's kernel is k_push_f32.cu; the charge deposit of both builds is here.)
//
// Bound by the FP64 units: two lanes a clock and SM on this GPU, so a warp-wide FP64
// instruction takes 16 cycles of the SM whatever it does and however many lanes need it.
// Comparisons, conversions and selections of doubles are FP64 instructions too unless they
// are done on the bits.  Hence:
//  * a warp takes its slots 32 at a time (sorted by triangle: coalesced loads, records from
//    L1) through the part that every particle needs -- gather, push, move, end point,
//    current and charge of those that stay in their triangle -- and puts the one in five
//    that leaves on a ring in shared memory; the walk over edges runs 32 ring entries at
//    a time, instead of in every warp for the few lanes that need it;
//  * 1/gamma and 1/rho are reciprocal square roots, the exit edge is found by products
//    (one division per crossing, not one per edge), signs and orders of non-negative
//    numbers are integer comparisons.
// Scatter (Eq. current, Eq. charge): atomics per particle and edge or node.
//
// Measured, 1M particles on 199k triangles, Boris: 475 -> 275 us a launch, 54M -> 29M warp
// instructions, FP64 units 86% -> 83% busy (one thread per particle walking in place, a
// division per edge, square roots and divisions for 1/gamma and the rotation, before).
#include "pic_internal.h"

namespace pic {

namespace {

__device__ __forceinline__ void atomic_acc(unsigned long long *p, long long v) {
    if (v != 0) atomicAdd(p, (unsigned long long)v);
}
__device__ __forceinline__ void atomic_acc(double *p, double v) { atomicAdd(p, v); }

// x < 0 on the bits: not for -0 and NaN
__device__ __forceinline__ bool negative(double x) {
    return (unsigned long long)__double_as_longlong(x) - 0x8000000000000001ULL <= 0x7FEFFFFFFFFFFFFFULL;
}
// a < b for numbers that are not negative
__device__ __forceinline__ bool below(double a, double b) {
    return __double_as_longlong(a) < __double_as_longlong(b);
}
__device__ __forceinline__ double sel3(int k, double a, double b, double c) {
    return k == 0 ? a : (k == 1 ? b : c);
}
__device__ __forceinline__ int sel3(int k, int a, int b, int c) { return k == 0 ? a : (k == 1 ? b : c); }

constexpr int PW = 2;        // warps per block: few particles spread over all SMs' FP64 units
constexpr int QCAP = 64;     // ring entries per warp (at most 31 + 32 used)
constexpr int ROUNDS = 8;    // 32 ROUNDS slots a warp are enough to fill its ring
constexpr int BPS = 16;      // blocks resident per SM (at most 64 registers a thread)

// particles whose displacement (d0, d1) leaves triangle t, at l = (l0, l1, 1 - l0 - l1)
struct Ring {
    int slot[QCAP], t[QCAP];
    double l0[QCAP], l1[QCAP], d0[QCAP], d1[QCAP];
};

// Eq. current of a segment l -> e: lam_a^s lam_b^e - lam_b^s lam_a^e for each local edge with
// tail a and head b (the line integral of W1); flags bit k: edge k runs k+1 -> k+2
__device__ __forceinline__ void deposit_current(double *J, const int4 EG, const double (&l)[3],
                                                const double (&e)[3]) {
    const int edge[3] = {EG.x, EG.y, EG.z};
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const int i = (k + 1) % 3, j = (k + 2) % 3;
        const double c = l[i] * e[j] - l[j] * e[i];
        atomic_acc(J + edge[k], (EG.w >> k) & 1 ? c : -c);
    }
}
__device__ __forceinline__ void deposit_charge(double *Q, const int4 ND, const double (&l)[3]) {
    atomic_acc(Q + ND.x, l[0]);
    atomic_acc(Q + ND.y, l[1]);
    atomic_acc(Q + ND.z, l[2]);
}

__device__ __forceinline__ const double2 *rec2(const TriRec<double> *rec, int t) {
    return reinterpret_cast<const double2 *>(rec + t);
}
// node, flags | edge, flags | neighbour, entries
__device__ __forceinline__ int4 ids(const TriRec<double> *rec, int t, int k) {
    return __ldg(reinterpret_cast<const int4 *>(rec[t].node) + k);
}

// Eq. DLE.  Boris: half electric kick, rotation by t = h B / gamma(u-), half kick.  Vay (2008,
// the correction cited in Sec. 3.3): the magnetic term read as the mean of the velocities
// v^{n-1/2} and v^{n+1/2}, solved in closed form.  Fields in the local frame:
// E = (Er, 0, Ez), B = (0, bphi, bz); h = q dt / (2 m).
//   u' = u + 2h E + h (u / gamma(u)) x B,  tau = h B,
//   gamma_new^2 = (sigma + sqrt(sigma^2 + 4 (tau^2 + (u'.tau)^2 / c^2))) / 2,
//   sigma = gamma(u')^2 - tau^2 (the other form of the root when sigma < 0),
//   t = tau / gamma_new,  u_new = (u' + (u'.t) t + u' x t) / (1 + t^2).
template <bool VAY>
__device__ __forceinline__ void kick(double &ur, double &up, double &uz, double Er, double Ez, double bphi,
                                     double bz, double h, double inv_c2) {
    const double tau_p = h * bphi, tau_z = h * bz;
    if constexpr (VAY) {
        const double gi = rsqrt(fma(fma(ur, ur, fma(up, up, uz * uz)), inv_c2, 1.0));
        const double vr = gi * ur;
        const double pr = fma(2.0 * h, Er, ur) + gi * (up * tau_z - uz * tau_p);
        const double pp = up - vr * tau_z;
        const double pz = fma(2.0 * h, Ez, uz) + vr * tau_p;
        const double tau2 = tau_p * tau_p + tau_z * tau_z;
        const double ut0 = pp * tau_p + pz * tau_z;
        const double x = tau2 + ut0 * ut0 * inv_c2;
        const double sigma = 1.0 + (pr * pr + pp * pp + pz * pz) * inv_c2 - tau2;
        const double disc = sqrt(sigma * sigma + 4.0 * x);
        const double g2 = negative(sigma) ? 2.0 * x / (disc - sigma) : 0.5 * (sigma + disc);
        const double gn = rsqrt(g2);
        const double qp = tau_p * gn, qz = tau_z * gn;
        const double ut = pp * qp + pz * qz;
        const double sf = 1.0 / (1.0 + qp * qp + qz * qz);
        ur = sf * (pr + pp * qz - pz * qp);
        up = sf * (pp + ut * qp - pr * qz);
        uz = sf * (pz + ut * qz + pr * qp);
    } else {
        const double er = h * Er, ez = h * Ez;
        ur += er;
        uz += ez;
        const double gi = rsqrt(fma(fma(ur, ur, fma(up, up, uz * uz)), inv_c2, 1.0));
        const double tp = tau_p * gi, tz = tau_z * gi;
        const double sf = 2.0 / fma(tp, tp, fma(tz, tz, 1.0));
        const double pr = ur + (up * tz - uz * tp);   // u' = u- + u- x t
        const double pp = up - ur * tz;
        const double pz = uz + ur * tp;
        const double sp = sf * tp, sz = sf * tz;
        ur = (ur + (pp * sz - pz * sp)) + er;         // u+ = u- + u' x (sf t), half kick
        up -= pr * sz;
        uz = (uz + pr * sp) + ez;
    }
}

// Walk one ring entry along its straight meridian segment: per triangle the part to the
// first edge reached (smallest crossing parameter, between 0 and 1; ties to the lower edge,
// never the edge just entered), its current, then the neighbour, where the two shared nodes
// keep their coordinates; until the end point, the axis, a wall or the walk cap.  Returns the
// edges reached.
__device__ __forceinline__ unsigned walk(const PushArgs<PF64> &a, int slot, int t, double l0, double l1,
                                         double d0, double d1) {
    double l[3] = {l0, l1, 1.0 - l0 - l1};
    int entered = -1;
    for (int ncross = 0;; ncross++) {
        const double2 g0 = __ldg(rec2(a.rec, t)), g1 = __ldg(rec2(a.rec, t) + 1);
        const int4 EG = ids(a.rec, t, 1);
        double dl[3], e[3];
        dl[0] = g0.x * d0 + g0.y * d1;
        dl[1] = g1.x * d0 + g1.y * d1;
        dl[2] = -(dl[0] + dl[1]);
        int kx = -1;
        double lb = 0.0, wb = 0.0;   // crossing parameter of kx: lb / wb
#pragma unroll
        for (int k = 0; k < 3; k++) {
            e[k] = l[k] + dl[k];
            // a coordinate that rounding left below zero and that does not fall is no exit
            if (k == entered || !negative(e[k]) || !negative(dl[k])) continue;
            const double b = __double_as_longlong(l[k]) < 0 ? 0.0 : l[k], w = -dl[k];
            if (kx < 0 || below(b * wb, lb * w)) {
                kx = k;
                lb = b;
                wb = w;
            }
        }
        if (kx < 0) {
            if (entered >= 0 && negative(sel3(entered, e[0], e[1], e[2]))) {
                // a round-off negative on the entry edge
#pragma unroll
                for (int k = 0; k < 3; k++)
                    if (k == entered) e[k] = 0.0;
                const double inv = 1.0 / (e[0] + e[1] + e[2]);
#pragma unroll
                for (int k = 0; k < 3; k++) e[k] *= inv;
            }
            deposit_current(a.J, EG, l, e);
            deposit_charge(a.Q, ids(a.rec, t, 0), e);
            a.p.tri[slot] = t;
            a.p.l0[slot] = e[0];
            a.p.l1[slot] = e[1];
            return (unsigned)ncross;
        }
        const double sx = lb / wb;
        const double ci = fma(sx, sel3(kx, dl[1], dl[2], dl[0]), sel3(kx, l[1], l[2], l[0]));
        const double cj = fma(sx, sel3(kx, dl[2], dl[0], dl[1]), sel3(kx, l[2], l[0], l[1]));
        const double inv = 1.0 / (ci + cj), ea = ci * inv, eb = cj * inv;   // at nodes kx+1, kx+2
        e[0] = sel3(kx, 0.0, eb, ea);
        e[1] = sel3(kx, ea, 0.0, eb);
        e[2] = sel3(kx, eb, ea, 0.0);
        deposit_current(a.J, EG, l, e);
        const int4 NB = ids(a.rec, t, 2);
        const int nb = sel3(kx, NB.x, NB.y, NB.z);
        if (nb < 0 && -nb == PIC_BC_AXIS) {   // stays on the axis edge
            deposit_charge(a.Q, ids(a.rec, t, 0), e);
            a.p.tri[slot] = t;
            a.p.l0[slot] = e[0];
            a.p.l1[slot] = e[1];
            return (unsigned)ncross + 1;
        }
        if (nb < 0 || ncross + 1 >= a.walk_cap) {
            // absorbed at the wall (or walk cap): its charge leaves the grid
            deposit_charge(a.Qabs, ids(a.rec, t, 0), e);
            if (nb >= 0) atomicAdd(a.counters + CNT_OVERFLOW, 1ULL);
            atomicAdd(a.counters + CNT_ABSORBED, 1ULL);
            a.p.tri[slot] = -1;
            return (unsigned)ncross + 1;
        }
        // nb's local edge j (opposite its node j): its node j+2 is node kx+1 of t, its node
        // j+1 is node kx+2
        const int j = (NB.w >> (2 * kx)) & 3;
        l[0] = sel3(j, 0.0, ea, eb);
        l[1] = sel3(j, eb, 0.0, ea);
        l[2] = sel3(j, ea, eb, 0.0);
        entered = j;
        const double rest = 1.0 - sx;
        d0 *= rest;
        d1 *= rest;
        t = nb;
    }
}

}  // namespace

template <bool VAY>
__global__ void __launch_bounds__(32 * PW, BPS) k_push_f64(const __grid_constant__ PushArgs<PF64> a) {
    __shared__ Ring rings[PW];
    chain_wait();
    const int64_t n = *a.n_slots;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned full = 0xffffffffu, before = (1u << lane) - 1;
    Ring &ring = rings[warp];
    unsigned head = 0, tail = 0, cx = 0;   // warp-uniform, ring index = value & (QCAP - 1)
    const auto pass = [&](bool valid) {
        __syncwarp();
        const int q = (head + lane) & (QCAP - 1);
        if (valid) cx += walk(a, ring.slot[q], ring.t[q], ring.l0[q], ring.l1[q], ring.d0[q], ring.d1[q]);
        __syncwarp();
    };
    // the rounds of 32 slots in use are dealt out evenly: of the slots that the launch allows
    // for there may be few (with an emitter, it allows for the capacity)
    const unsigned long long all = (unsigned long long)(n + 31) / 32, warps = (unsigned long long)gridDim.x * PW;
    const unsigned me = blockIdx.x * PW + warp;
    const int64_t last = (int64_t)(32 * ((me + 1) * all / warps));
    for (int64_t base = (int64_t)(32 * (me * all / warps)); base < last; base += 32) {
        const int64_t i = base + lane;
        const int t = i < n ? a.p.tri[i] : -1;
        bool leaves = false;
        double l[3] = {0, 0, 0}, d0 = 0, d1 = 0;
        if (t >= 0) {
            const double2 *R = rec2(a.rec, t);
            l[0] = a.p.l0[i];
            l[1] = a.p.l1[i];
            l[2] = 1.0 - l[0] - l[1];
            double ur = a.p.ur[i], up = a.p.up[i], uz = a.p.uz[i];
            // gather (Sec. 3.2): E(lambda) = sum_k lambda_k c_k; B_phi time-centred; guide B_z
            const double2 c0 = R[4], c1 = R[5], c2 = R[6], rh = R[2];
            const double Ez = fma(l[0], c0.x, fma(l[1], c1.x, l[2] * c2.x));
            const double Er = fma(l[0], c0.y, fma(l[1], c1.y, l[2] * c2.y));
            const double rho = fma(l[0], rh.x, fma(l[1], rh.y, l[2] * R[3].x));
            kick<VAY>(ur, up, uz, Er, Ez, R[7].x, a.bz, a.qmdt2, a.inv_c2);
            // move (Eq. DNE) in the ring's Cartesian frame, rotate back to the meridian plane
            const double gi = rsqrt(fma(fma(ur, ur, fma(up, up, uz * uz)), a.inv_c2, 1.0)) * a.dt;
            const double xr = ur * gi, yp = up * gi;
            d0 = uz * gi;
            const double x = rho + xr;
            const double rn2 = fma(x, x, yp * yp);
            double inv = 0.0;   // 1 / rn, for rn > 0
            if (rn2 > 0.0) {
                inv = rsqrt(rn2);
                const double cs = x * inv, sn = yp * inv;
                const double nr = cs * ur + sn * up;
                up = cs * up - sn * ur;
                ur = nr;
            }
            // rn - rho without cancellation, on the axis (rn = 0) too; rounding can leave rho
            // just below zero, and then rn + rho at or below it
            const double both = fma(rn2, inv, rho);
            if (__double_as_longlong(both) > 0) d1 = fma(xr, fma(2.0, rho, xr), yp * yp) / both;
            a.p.ur[i] = ur;
            a.p.up[i] = up;
            a.p.uz[i] = uz;
            // end point in the start triangle
            const double2 g0 = R[0], g1 = R[1];
            const double dl0 = g0.x * d0 + g0.y * d1, dl1 = g1.x * d0 + g1.y * d1;
            const double e[3] = {l[0] + dl0, l[1] + dl1, l[2] - (dl0 + dl1)};
            leaves = negative(e[0]) || negative(e[1]) || negative(e[2]);
            if (!leaves) {
                deposit_current(a.J, ids(a.rec, t, 1), l, e);
                deposit_charge(a.Q, ids(a.rec, t, 0), e);
                a.p.l0[i] = e[0];
                a.p.l1[i] = e[1];
            }
        }
        const unsigned mask = __ballot_sync(full, leaves);
        if (leaves) {
            const int q = (tail + __popc(mask & before)) & (QCAP - 1);
            ring.slot[q] = (int)i;
            ring.t[q] = t;
            ring.l0[q] = l[0];
            ring.l1[q] = l[1];
            ring.d0[q] = d0;
            ring.d1[q] = d1;
        }
        tail += __popc(mask);
        if (tail - head >= 32) {
            pass(true);
            head += 32;
        }
    }
    pass(lane < (int)(tail - head));
    const unsigned sx = __reduce_add_sync(full, cx);
    if (lane == 0 && sx) atomicAdd(a.counters + CNT_CROSSINGS, (unsigned long long)sx);
}

static void launch_push_f64(const PushArgs<PF64> &a, int64_t n_bound, cudaStream_t s) {
    if (n_bound <= 0) return;
    static int sms[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    int &sm = sms[dev & 63];
    if (sm == 0) cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev);
    // As many slots a warp as keep 16 warps on every SM, up to ROUNDS of 32: more of them
    // fill the last ring pass better, fewer spread a small simulation over the SMs; and no
    // more blocks than fit at a time.  Room for 3M, us a launch with 1000, 50,000, 1M slots in
    // use: ROUNDS in a row for each warp 47, 50, 266; dealt out over as many warps as ROUNDS for
    // 3M ask 18, 34, 286; over those that fit 17, 31, 262.  All slots in use, launches of 1.25M,
    // 4M, 12M: 307, 896, 2637 -> 291, 883, 2585
    const int64_t all = (n_bound + 31) / 32, spread = 16 * std::max(sm, 1);
    const int64_t rounds = std::min<int64_t>(ROUNDS, std::max<int64_t>(1, all / spread));
    const int64_t blocks = ((all + rounds - 1) / rounds + PW - 1) / PW;
    const unsigned grid = (unsigned)std::min<int64_t>(blocks, (int64_t)BPS * std::max(sm, 1));
    if (a.pusher == PIC_PUSHER_VAY) launch_chained(a.chain, k_push_f64<true>, grid, 32 * PW, 0, s, a);
    else launch_chained(a.chain, k_push_f64<false>, grid, 32 * PW, 0, s, a);
}

template <class P>
void launch_push(const PushArgs<P> &a, int64_t n_bound, cudaStream_t s) {
    if constexpr (P::fixed) launch_push_f32(a, n_bound, s);
    else launch_push_f64(a, n_bound, s);
}

// Eq. charge of the particles in slots [first, first + count) (new particles at
// injection; all of them, as far as *n_slots goes, for the diagnostics).  FP32 build: the fixed-point coordinates of
// the lanes that share a triangle are summed first (sorted slots: most lanes of a warp do),
// one set of atomics per triangle; sums of at most 32 coordinates < 2^23 fit in 32 bits.
template <class P>
__global__ void k_deposit_q(const TriRec<typename P::R> *rec, Particles<P> p, int64_t first,
                            int64_t count, const int64_t *n_slots, typename P::Acc *Q) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = first + k;
    const int t = k < count && (!n_slots || i < *n_slots) ? p.tri[i] : -1;
    if constexpr (P::fixed) {
        const unsigned grp = __match_any_sync(0xffffffffu, t);
        if (t < 0) return;
        const unsigned a = (unsigned)p.l0[i], b = (unsigned)p.l1[i];
        const unsigned sa = __reduce_add_sync(grp, a), sb = __reduce_add_sync(grp, b);
        if ((threadIdx.x & 31) == __ffs(grp) - 1) {
            const long long sc = (long long)__popc(grp) * LAM_ONE - (long long)sa - (long long)sb;
            atomic_acc(Q + rec[t].node[0], (long long)sa);
            atomic_acc(Q + rec[t].node[1], (long long)sb);
            atomic_acc(Q + rec[t].node[2], sc);
        }
    } else {
        if (t < 0) return;
        const double l0 = p.l0[i], l1 = p.l1[i];
        atomic_acc(Q + rec[t].node[0], l0);
        atomic_acc(Q + rec[t].node[1], l1);
        atomic_acc(Q + rec[t].node[2], 1.0 - l0 - l1);
    }
}

template <class P>
void launch_deposit_q(const TriRec<typename P::R> *rec, Particles<P> p, int64_t first,
                      int64_t count, const int64_t *n_slots, typename P::Acc *Q, cudaStream_t s) {
    if (count <= 0) return;
    k_deposit_q<P><<<(unsigned)((count + 255) / 256), 256, 0, s>>>(rec, p, first, count, n_slots, Q);
    PIC_LAUNCHED();
}

template void launch_push<PF32>(const PushArgs<PF32> &, int64_t, cudaStream_t);
template void launch_push<PF64>(const PushArgs<PF64> &, int64_t, cudaStream_t);
template void launch_deposit_q<PF32>(const TriRec<float> *, Particles<PF32>, int64_t, int64_t,
                                     const int64_t *, unsigned long long *, cudaStream_t);
template void launch_deposit_q<PF64>(const TriRec<double> *, Particles<PF64>, int64_t, int64_t,
                                     const int64_t *, double *, cudaStream_t);

}  // namespace pic
