// Field probes and output-port signals recorded on the device, without a host round trip
// per sample, by extra blocks of the edge-residual kernel, one per probe group and port.
// Every `every` steps the sums of all groups (ports) are appended to a device buffer; the
// last block to finish advances the step phase and the record count (device counters, so
// a recorded CUDA graph replays correctly).
//
// Probe: group g sums w_k B_f^p_g over its entries (faces f_k, weights w_k, power p_g in
// {1, 2}).  Port (Secs. 5.1, 5.1.1): the Poynting flux through a plane z = const,
// P = (2 pi / mu0) int E_rho B_phi rho drho, as a quadrature over the triangles the plane
// crosses (the host tabulates points and weights; E_rho and rho are linear along a
// triangle's chord and B_phi constant in it, so two Gauss points per chord are exact).
// E_rho(lambda) = sum_k lambda_k c_k,rho and B_phi come from the triangle records the face
// kernel of this step wrote: E^n and (B^{n+1/2} + B^{n-1/2}) / (2A).  Neither B nor the
// records change between the face kernel and the next step's, so the sums can wait for the
// residual kernel: launches of their own cost a step of eight sweep instances 2.8 us each.
#pragma once

#include "pic_internal.h"

namespace pic {

namespace {

// Block g of a recorder's n groups: term(k) summed over the group's entries when due.  The
// sum is that of PARTS strided parts, folded the same way whatever the block's size (a
// multiple of 32): what is recorded does not depend on the launch shape that a tuner picks.
constexpr int PARTS = 256;

template <class Term>
__device__ __forceinline__ void record_block(int g, int n, const int64_t *ptr, long long *state,
                                             unsigned *done, int every, long long capacity, double *buf,
                                             Term term) {
    __shared__ double part[PARTS / 32];
    __shared__ long long s_step, s_rec;
    if (threadIdx.x == 0) {
        s_step = state[0];
        s_rec = state[1];
    }
    __syncthreads();
    const bool take = s_step % every == 0;
    if (take) {
        for (int v = threadIdx.x; v < PARTS; v += blockDim.x) {   // whole warps
            double s = 0.0;
            for (long long k = ptr[g] + v; k < ptr[g + 1]; k += PARTS) s += term(k);
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if ((v & 31) == 0) part[v >> 5] = s;
        }
        __syncthreads();
    }
    // every block has read the counters before it takes its ticket; the last one advances
    // them
    if (threadIdx.x == 0) {
        if (take && s_rec < capacity) {
            double t = 0.0;
            for (int w = 0; w < PARTS / 32; w++) t += part[w];
            buf[s_rec * n + g] = t;
        }
        __threadfence();
        if (atomicAdd(done, 1u) == (unsigned)(n - 1)) {
            state[0] = s_step + 1;
            if (take) {
                if (s_rec < capacity) state[1] = s_rec + 1;
                else state[2] += 1;   // records that did not fit
            }
            *done = 0;
            __threadfence();
        }
    }
}

template <class P>
__device__ __forceinline__ void probe_block(const ProbeArgs<P> &a, int g) {
    const bool quad = a.power[g] == 2;
    record_block(g, a.n_groups, a.ptr, a.state, a.done, a.every, a.capacity, a.buf, [&](long long k) {
        const double b = (double)a.B[a.face[k]];
        return a.weight[k] * (quad ? b * b : b);
    });
}

template <class P>
__device__ __forceinline__ void port_block(const PortArgs<P> &a, int g) {
    record_block(g, a.n_ports, a.ptr, a.state, a.done, a.every, a.capacity, a.buf, [&](long long k) {
        const TriRec<typename P::R> &r = a.rec[a.tri[k]];
        const double *l = a.lam + 3 * k;
        const double er = l[0] * (double)r.c[1] + l[1] * (double)r.c[3] + l[2] * (double)r.c[5];
        return a.weight[k] * er * (double)r.bphi;
    });
}

}  // namespace

}  // namespace pic
