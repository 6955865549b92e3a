// Kernels of the adjoint sweep for ADAPT-VQE with re-optimised angles (a
// standard extension of the paper's loop, Sec. III-D, which updates only the
// newest angle).  The ansatz is the product of the Taylor-5 factors of
// Eqs. (6)-(8); its energy gradient needs, per factor,
//   <chi | U'(theta) phi>,  U'(theta) = A sum_{m<=4} (theta A)^m / m!,
// and every pool generator has A^2 = -P (P: the rows A does not
// annihilate), so U'(theta) = c4 A - s4 P with c4 = 1 - theta^2/2 +
// theta^4/24 and s4 = theta - theta^3/6.
#include "dev.cuh"
#include "grad.cuh"
#include "pair.cuh"

#include <cooperative_groups.h>

#include <algorithm>

namespace cg = cooperative_groups;

namespace tq {

namespace {

__device__ __forceinline__ bool last_block_vqe(unsigned* ticket, unsigned nblocks) {
    __shared__ bool is_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        is_last = atomicAdd(ticket, 1u) == nblocks - 1;
    }
    __syncthreads();
    return is_last;
}

template <typename T>
__device__ __forceinline__ double cdot_re(typename C2<T>::type a, typename C2<T>::type b) {
    return (double)a.x * (double)b.x + (double)a.y * (double)b.y;
}

// Re<chi | (c4 A - s4 P) phi> over all rows, float64 sums in a fixed order
// (per block, then the last block over the block partials); writes
// 2 * sum / e_den.  Full-space pools read A's entries from the factored sign
// form, sector pools from their (column, sign) tables.
template <typename T>
__global__ void __launch_bounds__(256)
k_ansatz_dot(PoolView p, int k, double c4, double s4, const typename C2<T>::type* __restrict__ chi,
             const typename C2<T>::type* __restrict__ phi, long long D, double* partials, unsigned* ticket,
             const DevStep* step, double* out) {
    __shared__ double sh[8];
    double acc = 0.0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < D; r += stride) {
        long long c;
        double a;
        if (p.sdim) {
            a = (double)p.ssgn[(long long)k * p.sdim + r];
            c = p.scol[(long long)k * p.sdim + r];
        } else {
            c = r ^ (long long)p.x[k];
            a = op_value<double>(p, k, (uint32_t)c);
        }
        if (a != 0.0) acc += c4 * a * cdot_re<T>(chi[r], phi[c]) - s4 * cdot_re<T>(chi[r], phi[r]);
    }
    double v[1] = {acc};
    block_sum<1>(v, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = v[0];
    if (last_block_vqe(ticket, gridDim.x)) {
        double t = 0.0;
        for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) t += __ldcg(partials + i);
        double u[1] = {t};
        block_sum<1>(u, sh);
        if (threadIdx.x == 0) {
            *out = 2.0 * u[0] / step->e_den;
            *ticket = 0u;
        }
    }
}

// chi = w - E psi (E from the step record), in the state's precision.
template <typename T>
__global__ void k_residual(const double2* __restrict__ w, const typename C2<T>::type* __restrict__ psi,
                           typename C2<T>::type* __restrict__ chi, long long D, const DevStep* step) {
    const double E = step->energy;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < D; r += stride) {
        const double2 wr = w[r];
        const typename C2<T>::type pr = psi[r];
        chi[r] = {(T)(wr.x - E * (double)pr.x), (T)(wr.y - E * (double)pr.y)};
    }
}


// ------------------------------------------------- whole sweeps in one launch
//
// Forward and adjoint sweep of an ansatz whose state fits the shared memory
// of one thread-block cluster (each CTA holds a contiguous slice): one
// launch per sweep instead of a copy, an update and (backwards) a dot per
// factor.  A factor touches its generator's support only, as pairs {r, r^x};
// one thread owns a pair, reads and writes both amplitudes through
// distributed shared memory, and a cluster barrier separates factors.  The
// update is the pair update's own arithmetic (chain_pair for complex64, the
// closed form for complex128), so the states are bit for bit those of the
// per-factor launches.  The forward sweep stores each factor's input pairs
// in pair order for the adjoint sweep, which turns them into
//   X = sum_S Re<chi_r|A phi_r>,  Y = sum_S Re<chi_r|phi_r>,  grad = 2 (c4 X - s4 Y) / <psi|psi>,
// with complex64 products and sums carried in float32 pairs (about 48 bits):
// a float64 product per amplitude would hold the float64 pipe of the
// cluster's 16 SMs longer than everything else.
//
// What bounds it: the latency of a factor (barrier, distributed shared
// memory round trip, pair arithmetic).  20 factors at 14 qubits, complex64,
// energy and read-back included: 588 us as 40 update and 20 dot launches
// with their copies, 112 us here (forward 33, energy 18, adjoint 35 us, the
// rest launches and read-back).
template <typename T>
struct SweepOp {
    RowExp rx;
    uint32_t x, z0;
    int neg;               // entries of A are (-1)^{parity(col & z0)} (-1)^neg
    uint32_t pairs;
    T cf[6];
    double c5, s5;         // closed form (complex128)
    double c4, s4;         // derivative (adjoint sweep)
};

template <typename T>
__device__ __forceinline__ void sweep_prepare(const PoolView& p, const SweepOps& ops, int n, bool adjoint,
                                              SweepOp<T>* out) {
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int k = ops.k[j];
        const double t = ops.theta[j];
        SweepOp<T>& o = out[j];
        const SuppRec s = load_supp(p, k);
        o.rx = make_rowexp(s, p.supp[k].z);
        o.x = s.x;
        o.z0 = s.z0;
        o.neg = p.fc0f[k] < 0.0f;
        o.pairs = (uint32_t)((1ll << p.nq) >> (s.m + 1));
        taylor_coefs_fast<T>(adjoint ? -t : t, o.cf);
        if constexpr (sizeof(T) == 8) closed_coefs(o.cf, o.c5, o.s5);
        const double t2 = t * t;
        o.c4 = 1.0 - t2 / 2.0 + t2 * t2 / 24.0;
        o.s4 = t * (1.0 - t2 / 6.0);
    }
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// The update of one pair; neg_r: A[r][q] = -1 (then A[q][r] = +1).
__device__ __forceinline__ void sweep_pair(const SweepOp<float>& o, bool neg_r, float2& a, float2& b) {
    chain_pair(neg_r ? -1.f : 1.f, neg_r ? 1.f : -1.f, o.cf, a, b);
}
__device__ __forceinline__ void sweep_pair(const SweepOp<double>& o, bool neg_r, double2& a, double2& b) {
    closed_pair_sign(neg_r ? -1 : 1, neg_r ? 1 : -1, o.cf, o.c5, o.s5, a, b);
}

// The dots X and Y of a factor: float64 sums, or float32 (hi, lo) pairs with
// exact products.  A warp leaves its sums in a 16-byte slot; they are turned
// into float64 gradients after the last factor (a float64 instruction per
// warp and factor would sit on every factor's critical path).
template <typename T> struct SweepDot;
template <> struct SweepDot<double> {
    double x = 0.0, y = 0.0;
    __device__ __forceinline__ void add_x(double a, double b) { x = fma(a, b, x); }
    __device__ __forceinline__ void add_y(double a, double b) { y = fma(a, b, y); }
    __device__ __forceinline__ void leave(double2* slot) {
        const int lane = threadIdx.x & 31;
        const bool up = lane & 16;
        double v = (up ? y : x) + __shfl_xor_sync(0xffffffffu, up ? x : y, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane % 16 == 0) reinterpret_cast<double*>(slot)[lane / 16] = v;
    }
    static __device__ __forceinline__ double grad(const double2& s, double c4, double s4) { return c4 * s.x - s4 * s.y; }
};
template <> struct SweepDot<float> {
    float xh = 0.f, xl = 0.f, yh = 0.f, yl = 0.f;
    static __device__ __forceinline__ void add(float& hi, float& lo, float a, float b) {
        const float p = __fmul_rn(a, b), e = __fmaf_rn(a, b, -p);
        float s, r;
        two_sum(hi, p, s, r);
        hi = s;
        lo += r + e;
    }
    __device__ __forceinline__ void add_x(float a, float b) { add(xh, xl, a, b); }
    __device__ __forceinline__ void add_y(float a, float b) { add(yh, yl, a, b); }
    __device__ __forceinline__ void leave(double2* slot) {
        // X in the lower half, Y in the upper after the first step
        const int lane = threadIdx.x & 31;
        const bool up = lane & 16;
        float hi = up ? yh : xh, lo = up ? yl : xl;
        float oh = __shfl_xor_sync(0xffffffffu, up ? xh : yh, 16), ol = __shfl_xor_sync(0xffffffffu, up ? xl : yl, 16);
        float s, r;
        two_sum(hi, oh, s, r);
        hi = s;
        lo += ol + r;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            oh = __shfl_xor_sync(0xffffffffu, hi, o);
            ol = __shfl_xor_sync(0xffffffffu, lo, o);
            two_sum(hi, oh, s, r);
            hi = s;
            lo += ol + r;
        }
        if (lane % 16 == 0) reinterpret_cast<float2*>(slot)[lane / 16] = make_float2(hi, lo);
    }
    static __device__ __forceinline__ double grad(const double2& v, double c4, double s4) {
        const float2* f = reinterpret_cast<const float2*>(&v);
        return c4 * ((double)f[0].x + (double)f[0].y) - s4 * ((double)f[1].x + (double)f[1].y);
    }
};

// A thread's pair u of a factor: rows and the sign of A[r][q].
struct SweepPair {
    uint32_t r, q;
    bool on, neg;      // on: the thread has this pair; neg: A[r][q] = -1
};
template <typename T>
__device__ __forceinline__ SweepPair sweep_rows(const SweepOp<T>& o, uint32_t u) {
    SweepPair s;
    s.on = u < o.pairs;
    s.r = expand_row(o.rx, u);
    s.q = s.r ^ o.x;
    s.neg = (parity32(s.q & o.z0) ^ o.neg) != 0;
    return s;
}

template <typename T>
__global__ void __launch_bounds__(SWEEP_MAX_TPB)
k_ansatz_forward(PoolView p, const __grid_constant__ SweepOps ops, int n, int slice_log,
                 const typename C2<T>::type* psi0, typename C2<T>::type* psi_end,
                 typename C2<T>::type* __restrict__ pairs_out, long long stride) {
    using V = typename C2<T>::type;
    extern __shared__ __align__(16) unsigned char sw_raw[];
    cg::cluster_group cl = cg::this_cluster();
    SweepOp<T>* op = reinterpret_cast<SweepOp<T>*>(sw_raw);
    V* st = reinterpret_cast<V*>(sw_raw + SWEEP_OPS * sizeof(SweepOp<T>));
    const uint32_t per = 1u << slice_log, lo = per - 1u, rank = cl.block_rank();
    for (uint32_t i = threadIdx.x; i < per; i += blockDim.x) st[i] = psi0[((size_t)rank << slice_log) + i];
    sweep_prepare<T>(p, ops, n, false, op);
    __syncthreads();
    cluster_arrive();
    const uint32_t t0 = rank * blockDim.x + threadIdx.x, step = cl.num_blocks() * blockDim.x;
    SweepPair next = sweep_rows(op[0], t0);
    cluster_wait();                       // every slice is loaded
    for (int j = 0; j < n; ++j) {
        const SweepOp<T>& o = op[j];
        SweepPair s = next;
        for (uint32_t u = t0; s.on;) {
            V* pr = cl.map_shared_rank(st + (s.r & lo), s.r >> slice_log);
            V* pq = cl.map_shared_rank(st + (s.q & lo), s.q >> slice_log);
            V a = *pr, b = *pq;
            if (pairs_out) store2(pairs_out + (size_t)j * stride, 2 * u, a, b);
            sweep_pair(o, s.neg, a, b);
            *pr = a;
            *pq = b;
            u += step;
            if (u >= o.pairs) break;
            s = sweep_rows(o, u);
        }
        cluster_arrive();
        if (j + 1 < n) next = sweep_rows(op[j + 1], t0);      // while the others arrive
        cluster_wait();                   // the factor is applied, and no peer reads this slice any more
    }
    for (uint32_t i = threadIdx.x; i < per; i += blockDim.x) psi_end[((size_t)rank << slice_log) + i] = st[i];
}

// complex64 carries chi divided by 4^k, about <psi|psi>: the dots' float32
// products of chi and phi are then near 1 whatever the state's norm (at norm
// 1e-18 they fell below float32's range), and every other step is linear in
// chi, so the scaling changes no bit.  Returns k (0 for complex128).
template <typename T>
__device__ __forceinline__ int sweep_scale(double den) {
    const int e = ((__double2hiint(den) >> 20) & 0x7ff) - 1023;
    return sizeof(T) == 8 || e < -250 || e > 250 ? 0 : e >> 1;
}

// chi_in null: chi = (w - E psi) / 4^k at the end of the ansatz (the first
// launch of the sweep), else the chi an earlier launch left.  part:
// [SWEEP_OPS][CTAs].
template <typename T>
__global__ void __launch_bounds__(SWEEP_MAX_TPB)
k_ansatz_adjoint(PoolView p, const __grid_constant__ SweepOps ops, int n, int slice_log,
                 const double2* __restrict__ w, const typename C2<T>::type* __restrict__ psi, const DevStep* step,
                 const typename C2<T>::type* chi_in, typename C2<T>::type* chi_out,
                 const typename C2<T>::type* __restrict__ pairs_in, long long stride, double* part, double* grad) {
    using V = typename C2<T>::type;
    extern __shared__ __align__(16) unsigned char sw_raw[];
    cg::cluster_group cl = cg::this_cluster();
    SweepOp<T>* op = reinterpret_cast<SweepOp<T>*>(sw_raw);
    const int nw = blockDim.x >> 5, wid = threadIdx.x >> 5;
    double2* wsum = reinterpret_cast<double2*>(sw_raw + SWEEP_OPS * sizeof(SweepOp<T>));   // [n][nw]
    V* st = reinterpret_cast<V*>(wsum + (size_t)SWEEP_OPS * nw);
    const uint32_t per = 1u << slice_log, lo = per - 1u, rank = cl.block_rank();
    const double E = step->energy;
    const int k = sweep_scale<T>(step->e_den);
    const T sc = (T)__int_as_float((127 - k) << 23);             // 2^-k, applied twice: 4^-k may leave the range
    for (uint32_t i = threadIdx.x; i < per; i += blockDim.x) {
        const size_t r = ((size_t)rank << slice_log) + i;
        if (chi_in) {
            st[i] = chi_in[r];
        } else {
            const double2 wr = w[r];
            const V pr = psi[r];
            st[i] = {(T)(wr.x - E * (double)pr.x), (T)(wr.y - E * (double)pr.y)};
            if (sizeof(T) == 4) st[i] = {st[i].x * sc * sc, st[i].y * sc * sc};
        }
    }
    sweep_prepare<T>(p, ops, n, true, op);
    __syncthreads();
    cluster_arrive();
    const uint32_t t0 = rank * blockDim.x + threadIdx.x, step_u = cl.num_blocks() * blockDim.x;
    // the next factor's rows and forward pair load while the others arrive
    SweepPair next = sweep_rows(op[n - 1], t0);
    V nr = V{}, nq = V{};
    if (next.on) load2(pairs_in + (size_t)(n - 1) * stride, 2 * t0, nr, nq);
    cluster_wait();
    for (int j = n - 1; j >= 0; --j) {
        const SweepOp<T>& o = op[j];
        SweepDot<T> dot;
        SweepPair s = next;
        V fr = nr, fq = nq;
        for (uint32_t u = t0; s.on;) {
            V* pr = cl.map_shared_rank(st + (s.r & lo), s.r >> slice_log);
            V* pq = cl.map_shared_rank(st + (s.q & lo), s.q >> slice_log);
            V a = *pr, b = *pq;
            const V a0 = a, b0 = b;
            sweep_pair(o, s.neg, a, b);
            *pr = a;
            *pq = b;
            const T sg = s.neg ? T(-1) : T(1);       // A[r][q]; A[q][r] is its negative
            dot.add_x(sg * a0.x, fq.x);
            dot.add_x(sg * a0.y, fq.y);
            dot.add_x(-sg * b0.x, fr.x);
            dot.add_x(-sg * b0.y, fr.y);
            dot.add_y(a0.x, fr.x);
            dot.add_y(a0.y, fr.y);
            dot.add_y(b0.x, fq.x);
            dot.add_y(b0.y, fq.y);
            u += step_u;
            if (u >= o.pairs) break;
            load2(pairs_in + (size_t)j * stride, 2 * u, fr, fq);
            s = sweep_rows(o, u);
        }
        cluster_arrive();
        if (j > 0) {
            next = sweep_rows(op[j - 1], t0);
            if (next.on) load2(pairs_in + (size_t)(j - 1) * stride, 2 * t0, nr, nq);
        }
        dot.leave(wsum + j * nw + wid);
        cluster_wait();
    }
    for (uint32_t i = threadIdx.x; chi_out && i < per; i += blockDim.x) chi_out[((size_t)rank << slice_log) + i] = st[i];
    // this CTA's sums in warp order, then the CTAs' in rank order
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        double v = 0.0;
        for (int i = 0; i < nw; ++i) v += SweepDot<T>::grad(wsum[j * nw + i], op[j].c4, op[j].s4);
        part[(size_t)j * SWEEP_MAX_CLUSTER + rank] = v;
    }
    __threadfence();
    cluster_arrive();
    cluster_wait();
    if (rank == 0)
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
            double v = 0.0;
            for (unsigned i = 0; i < cl.num_blocks(); ++i) v += __ldcg(part + (size_t)j * SWEEP_MAX_CLUSTER + i);
            grad[j] = 2.0 * v / (step->e_den * __hiloint2double((1023 - 2 * k) << 20, 0));
        }
}

int small_grid(long long D, int sms) {
    long long g = (D + 255) / 256;
    if (g > (long long)sms * 4) g = (long long)sms * 4;
    return (int)(g < 1 ? 1 : g);
}

template <typename T>
size_t sweep_smem(bool adjoint, int slice_log, int tpb) {
    return SWEEP_OPS * sizeof(SweepOp<T>) + (adjoint ? (size_t)SWEEP_OPS * (tpb / 32) * sizeof(double2) : 0) +
           ((size_t)1 << slice_log) * 2 * sizeof(T);
}

// CTAs and threads per CTA for 2^nq amplitudes; a single excitation has D/4
// pairs.  64 pairs per CTA up to 16 CTAs, then 256 threads with several pairs
// each (more threads make the barriers longer: 20 factors at 16 qubits,
// complex64, forward + adjoint: 97 us with 256 threads, 132 with 1024; 12
// qubits: 61 us on 16 CTAs, 74 on 4), and 1024 threads only where a CTA has
// more than 1024 pairs (18 qubits: 184 us against 248).
void sweep_shape(int nq, int* cs, int* tpb) {
    const long long pairs = std::max(1ll, (1ll << nq) >> 2);
    const long long c = std::min<long long>(SWEEP_MAX_CLUSTER, std::max(1ll, pairs / 64));
    *cs = (int)c;
    const long long per = pairs / c;
    *tpb = (int)std::min<long long>(per > 1024 ? SWEEP_MAX_TPB : 256, std::max(32ll, per));
}

template <typename K>
cudaError_t sweep_config(K kern, int cs, int tpb, size_t smem, cudaStream_t s, cudaLaunchConfig_t* cfg,
                         cudaLaunchAttribute* attr) {
    cudaError_t e = allow_smem(kern);
    if (e == cudaSuccess && cs > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3(cs);
    cfg->blockDim = dim3(tpb);
    cfg->dynamicSmemBytes = smem;
    cfg->stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = cs;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
    return e;
}

template <typename T>
bool sweep_fits(int nq) {
    int cs, tpb;
    sweep_shape(nq, &cs, &tpb);
    int lg = nq;
    while (cs >> (nq - lg + 1)) --lg;          // slice of D / cs amplitudes
    const size_t smem = sweep_smem<T>(true, lg, tpb);
    if (smem > 220 * 1024) return false;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    int n = 0;
    cudaError_t e = sweep_config(k_ansatz_adjoint<T>, cs, tpb, smem, 0, &cfg, &attr);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k_ansatz_adjoint<T>, &cfg);
    if (e == cudaSuccess && n >= 1) {
        e = sweep_config(k_ansatz_forward<T>, cs, tpb, sweep_smem<T>(false, lg, tpb), 0, &cfg, &attr);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k_ansatz_forward<T>, &cfg);
    }
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e == cudaSuccess && n >= 1;
}

}  // namespace

// Asked once per call: a few microseconds of host queries beside the sweep.
bool ansatz_sweep_ready(int nq, int prec) {
    if (nq < 2 || nq >= 32) return false;
    return prec == TQ_C128 ? sweep_fits<double>(nq) : sweep_fits<float>(nq);
}

template <typename T>
static int forward_t(const PoolView& p, const SweepOps& ops, int n, const void* psi0, void* psi_end,
                     void* pairs, cudaStream_t s) {
    using V = typename C2<T>::type;
    int cs, tpb, lg = p.nq;
    sweep_shape(p.nq, &cs, &tpb);
    while (cs >> (p.nq - lg + 1)) --lg;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    cudaError_t e = sweep_config(k_ansatz_forward<T>, cs, tpb, sweep_smem<T>(false, lg, tpb), s, &cfg, &attr);
    if (e == cudaSuccess)
        e = cudaLaunchKernelEx(&cfg, k_ansatz_forward<T>, p, ops, n, lg, static_cast<const V*>(psi0),
                               static_cast<V*>(psi_end), static_cast<V*>(pairs), (1ll << p.nq) / 2);
    return e == cudaSuccess ? 1 : -1;
}

template <typename T>
static int adjoint_t(const PoolView& p, const SweepOps& ops, int n, const double2* w, const void* psi,
                     const DevStep* step, const void* chi_in, void* chi_out, const void* pairs, double* part,
                     double* grad, cudaStream_t s) {
    using V = typename C2<T>::type;
    int cs, tpb, lg = p.nq;
    sweep_shape(p.nq, &cs, &tpb);
    while (cs >> (p.nq - lg + 1)) --lg;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    cudaError_t e = sweep_config(k_ansatz_adjoint<T>, cs, tpb, sweep_smem<T>(true, lg, tpb), s, &cfg, &attr);
    if (e == cudaSuccess)
        e = cudaLaunchKernelEx(&cfg, k_ansatz_adjoint<T>, p, ops, n, lg, w, static_cast<const V*>(psi), step,
                               static_cast<const V*>(chi_in), static_cast<V*>(chi_out), static_cast<const V*>(pairs),
                               (1ll << p.nq) / 2, part, grad);
    return e == cudaSuccess ? 1 : -1;
}

int launch_ansatz_forward(const PoolView& p, const SweepOps& ops, int n, int prec, const void* psi0, void* psi_end,
                          void* pairs, cudaStream_t s) {
    return prec == TQ_C128 ? forward_t<double>(p, ops, n, psi0, psi_end, pairs, s)
                           : forward_t<float>(p, ops, n, psi0, psi_end, pairs, s);
}

int launch_ansatz_adjoint(const PoolView& p, const SweepOps& ops, int n, int prec, const double2* w, const void* psi,
                          const DevStep* step, const void* chi_in, void* chi_out, const void* pairs, double* part,
                          double* grad, cudaStream_t s) {
    return prec == TQ_C128
               ? adjoint_t<double>(p, ops, n, w, psi, step, chi_in, chi_out, pairs, part, grad, s)
               : adjoint_t<float>(p, ops, n, w, psi, step, chi_in, chi_out, pairs, part, grad, s);
}

int launch_ansatz_dot(const PoolView& p, int k, double c4, double s4, const void* chi, const void* phi, int prec,
                      long long D, double* partials, unsigned* ticket, const DevStep* step, double* grad_out,
                      int sms, cudaStream_t s) {
    const int grid = small_grid(D, sms);
    if (prec == TQ_C128)
        k_ansatz_dot<double><<<grid, 256, 0, s>>>(p, k, c4, s4, static_cast<const double2*>(chi),
                                                  static_cast<const double2*>(phi), D, partials, ticket, step, grad_out);
    else
        k_ansatz_dot<float><<<grid, 256, 0, s>>>(p, k, c4, s4, static_cast<const float2*>(chi),
                                                 static_cast<const float2*>(phi), D, partials, ticket, step, grad_out);
    return 1;
}

int launch_residual(const double2* w, const void* psi, void* chi, int prec, long long D, const DevStep* step,
                    cudaStream_t s) {
    const int grid = (int)((D + 255) / 256 < 2048 ? (D + 255) / 256 : 2048);
    if (prec == TQ_C128)
        k_residual<double><<<grid, 256, 0, s>>>(w, static_cast<const double2*>(psi), static_cast<double2*>(chi), D, step);
    else
        k_residual<float><<<grid, 256, 0, s>>>(w, static_cast<const float2*>(psi), static_cast<float2*>(chi), D, step);
    return 1;
}

}  // namespace tq
