// Conservation checks of the FETD-PIC step (run every check_interval steps):
//   - nodal charge q_i = sum_p Q lambda_i(r_p) (Eq. (scatter.charge.assign)) in
//     the same 64-bit fixed point as the current, so the discrete continuity
//     residual (q^{n+1} - q^n)/dt + S~ i^{n+1/2} (Eq. (full.dis.cont)) is an
//     exact integer sum of rounding errors;
//   - discrete Gauss law S~ d^n - q^n against its initial value (Eq.
//     (semi.dis.div.2) in the dual-flux form d^{n+1} = d^n + dt (C^T H b - i));
//   - field energy e.[*eps].e/2 + b.[*mu^-1].b/2.
// Node sums gather over a node -> edge incidence list in a fixed order, and
// the energy uses a two-pass reduction, so every check value is deterministic.
#include <algorithm>

#include <cuda_runtime.h>

#include "fetdpic_internal.h"
#include "fp64_int.h"

namespace fetdpic {

// Sum of v[0..2] over runs of equal key across the warp (sorted particles of one
// triangle are neighbours), complete on a run's first lane; returns whether this
// lane is one.  T: 32-bit sums for the FP32 path, 64-bit for the FP64 one.
template <typename T>
__device__ __forceinline__ bool run_sum(int key, T *v, int lane)
{
    const unsigned full = 0xffffffffu;
    const int kn = __shfl_down_sync(full, key, 1);
    const unsigned tails = __ballot_sync(full, (lane == 31) || (kn != key));
    const int seg_end = lane + __ffs(tails >> lane) - 1;
    const int kp = __shfl_up_sync(full, key, 1);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        if (!__any_sync(full, seg_end - lane >= off)) break;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const T o = __shfl_down_sync(full, v[m], off);
            if (lane + off <= seg_end) v[m] += o;
        }
    }
    return lane == 0 || kp != key;
}

// q_fix[node] += round(w lambda_i 2^shift).  Three 64-bit atomics per run of
// particles of one triangle, not per particle: 800k particles at 20 to a triangle
// and species 30.5 -> 16.3 us right after a sort, 36.8 -> 31.1 after 15 steps of
// drift (FP32), when the runs are short again.
// FP64 path from global coordinates.
__global__ void __launch_bounds__(256) k_charge64(long long nchunks, const int *__restrict__ cell,
                                                  const short *__restrict__ chunk_sp, const Species *__restrict__ sp,
                                                  const Geo64 *__restrict__ geo, const Topo *__restrict__ topo,
                                                  const double *__restrict__ x, const double *__restrict__ y,
                                                  unsigned long long *__restrict__ q)
{
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const long long ch = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (ch >= nchunks) return;
    const long long p = ch * 32 + lane;
    const int f = cell[p];
    long long v[3] = {0, 0, 0};
    if (f >= 0) {
        const double w = sp[chunk_sp[ch]].qfix;
        const Geo64 &G = geo[f];
        const double px = x[p], py = y[p];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const int a = (m + 1) % 3;
            const double l = G.gx[m] * (px - G.X[a]) + G.gy[m] * (py - G.Y[a]);
            v[m] = __double2ll_rn(l * w);
        }
    }
    if (run_sum(f, v, lane) && f >= 0) {
#pragma unroll
        for (int m = 0; m < 3; ++m)
            if (v[m]) atomicAdd(q + topo[f].node[m], (unsigned long long)v[m]);
    }
}

// FP32 path: lambda = (l0, l1, 1 - l0 - l1) exactly as the particle kernel forms
// it.  round((double)lambda w) in integer arithmetic but for one addition (the
// FP64 pipe passes 2 lanes per SM and clock).  Each warp takes CH_CHUNKS chunks,
// their state loaded before any of it is used.
constexpr int CH_CHUNKS = 4;

__global__ void __launch_bounds__(256) k_charge32(long long nchunks, const int *__restrict__ cell,
                                                  const short *__restrict__ chunk_sp, const Species *__restrict__ sp,
                                                  const Topo *__restrict__ topo, const float *__restrict__ l0,
                                                  const float *__restrict__ l1, unsigned long long *__restrict__ q)
{
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const long long c0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * CH_CHUNKS;
    int f[CH_CHUNKS];
    float a[CH_CHUNKS], b[CH_CHUNKS];
#pragma unroll
    for (int k = 0; k < CH_CHUNKS; ++k) {
        const long long p = (c0 + k) * 32 + lane;
        f[k] = -1; a[k] = 0.f; b[k] = 0.f;
        if (c0 + k < nchunks) { f[k] = cell[p]; a[k] = l0[p]; b[k] = l1[p]; }
    }
#pragma unroll
    for (int k = 0; k < CH_CHUNKS; ++k) {
        if (c0 + k >= nchunks) break;                                  // warp-uniform
        const double w = sp[chunk_sp[c0 + k]].qfix;
        const float l[3] = {a[k], b[k], 1.f - a[k] - b[k]};
        // inside its triangle (a stored particle is, but for round-off) |v| < 1.5 2^25, and 32 of
        // them fit 32 bits; a particle written outside the triangle it names adds by itself
        const bool in = fabsf(l[0] - 0.5f) <= 1.f && fabsf(l[1] - 0.5f) <= 1.f && fabsf(l[2] - 0.5f) <= 1.f;
        int v[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const double d = mul_i(to_f64(l[m]), w) + 0x1.8p52;
            v[m] = f[k] >= 0 && in ? __double2loint(d) : 0;
        }
        if (f[k] >= 0 && !in) {
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const long long s = __double2ll_rn((double)l[m] * w);
                if (s) atomicAdd(q + topo[f[k]].node[m], (unsigned long long)s);
            }
        }
        if (run_sum(f[k], v, lane) && f[k] >= 0) {
#pragma unroll
            for (int m = 0; m < 3; ++m)
                if (v[m]) atomicAdd(q + topo[f[k]].node[m], (unsigned long long)(long long)v[m]);
        }
    }
}

__device__ __forceinline__ void atomic_max_pos(double *addr, double v)
{
    // non-negative doubles order like their bit patterns
    atomicMax(reinterpret_cast<unsigned long long *>(addr), (unsigned long long)__double_as_longlong(v));
}

// The largest of the lanes' non-negative values into out[3 in + slot]: one atomic
// per warp where all its nodes belong to one instance (10k nodes on one address
// took 11 us).
__device__ __forceinline__ void warp_max_pos(double *out, int slot, int in, double v, bool live)
{
    const unsigned full = 0xffffffffu;
    unsigned long long b = live ? (unsigned long long)__double_as_longlong(v) : 0ull;
    const int in0 = __shfl_sync(full, in, 0);
    if (__all_sync(full, !live || in == in0)) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long o = __shfl_xor_sync(full, b, off);
            if (o > b) b = o;
        }
        if ((threadIdx.x & 31) == 0 && live && b) atomic_max_pos(out + 3 * in0 + slot, __longlong_as_double((long long)b));
    } else if (live) {
        atomic_max_pos(out + 3 * in + slot, v);
    }
}

// Edges of a node whose values are loaded before any is summed (in order).
constexpr int NB = 8;

// One instance's energy: a warp sums the block partials, in an order that depends on their number only.
__device__ __forceinline__ void energy_sum(long long nblocks, int ninst, const double *part, int in, int lane, double *out)
{
    double s = 0.0;
    for (long long k = lane; k < nblocks; k += 32) s += __ldcg(part + k * ninst + in);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) out[3 * in + 2] = s;
}

// Node k's sums over its edges: Gauss sum_e o(k,e) d_e and sum_e |d_e|.
__device__ __forceinline__ void node_flux(const int *__restrict__ nrp, const int *__restrict__ nedge,
                                          const double *__restrict__ d, int k, double &s, double &sa)
{
    s = 0.0; sa = 0.0;
    for (int r = nrp[k], r1 = nrp[k + 1]; r < r1; r += NB) {
        int w[NB];
        double v[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) w[i] = r + i < r1 ? nedge[r + i] : 0;
#pragma unroll
        for (int i = 0; i < NB; ++i) v[i] = r + i < r1 ? d[w[i] >> 1] : 0.0;
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (r + i < r1) {
                s += (w[i] & 1) ? -v[i] : v[i];
                sa += fabs(v[i]);
            }
    }
}

// The Gauss-law reference g0 = sum_e o(k,e) d_e - q (physical units).
__global__ void __launch_bounds__(256) k_gauss_reference(int N, const int *__restrict__ nrp,
                                                         const int *__restrict__ nedge, const int *__restrict__ ninst,
                                                         const double *__restrict__ qunit, const double *__restrict__ d,
                                                         const unsigned long long *__restrict__ q, double *__restrict__ g0)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N) return;
    double s, sa;
    node_flux(nrp, nedge, d, k, s, sa);
    const double qk = (double)(long long)q[k] * qunit[ninst[k]];
    g0[k] = s - qk;
}

// The checks of a step in one launch (they were four, each a short wave with a
// gap before it), thread i for node i, edge i and face i:
//   - continuity residual of node i: res = (q1 - q0) + sum_e o(k,e) i_e, exactly
//     in integers, over sum_e |i_e| + |q1 - q0| (at least one unit), the largest
//     per instance;
//   - Gauss residual |g - g0| / (sum |d_e| + |q| + |g0|) with g = sum_e o(k,e)
//     d_e - q, the largest per instance;
//   - energy: per block and instance the sum of e_k ([*eps] e)_k / 2 over its
//     edges and b_f^2 / (2 mu0 A_f) over its faces, in `part`, summed by the
//     last block (`ticket`; few partials) or by k_energy_final.
// q0, the charge before the step, is not needed any more: it is cleared for the
// next charge.
__global__ void __launch_bounds__(256) k_checks(CheckArgs a)
{
    pdl_begin();
    __shared__ double sh[256];
    __shared__ int lo_s, hi_s, last_s;
    const int tid = threadIdx.x, i = blockIdx.x * 256 + tid;
    {
        const bool live = i < a.N;
        long long flux = 0;
        double absf = 0.0, s = 0.0, sa = 0.0;
        if (live) {
            for (int r = a.nrp[i], r1 = a.nrp[i + 1]; r < r1; r += NB) {
                int w[NB];
                long long iv[NB];
#pragma unroll
                for (int k = 0; k < NB; ++k) w[k] = r + k < r1 ? a.nedge[r + k] : 0;
#pragma unroll
                for (int k = 0; k < NB; ++k) iv[k] = r + k < r1 ? (long long)a.ifix[w[k] >> 1] : 0;
#pragma unroll
                for (int k = 0; k < NB; ++k)
                    if (r + k < r1) {
                        flux += (w[k] & 1) ? -iv[k] : iv[k];
                        absf += fabs((double)iv[k]);
                    }
            }
            node_flux(a.nrp, a.nedge, a.d, i, s, sa);
        }
        const int in = live ? a.ninst[i] : 0;
        const long long q1 = live ? (long long)a.q1[i] : 0, dq = live ? q1 - (long long)a.q0[i] : 0;
        if (live) a.q0[i] = 0ull;
        const double scale = fmax(absf + fabs((double)dq), 1.0);
        warp_max_pos(a.out, 0, in, fabs((double)(dq + flux)) / scale, live);
        const double qk = live ? (double)q1 * a.qunit[in] : 0.0, ref = live ? a.g0[i] : 0.0;
        const double g = s - qk, gs = sa + fabs(qk) + fabs(ref);
        warp_max_pos(a.out, 1, in, gs > 0.0 ? fabs(g - ref) / gs : 0.0, live);
    }
    const bool edge = i < a.E, face = i < a.F;
    const int ie = edge ? a.einst[i] : -1, jf = face ? a.topo[i].inst : -1;
    double ve = 0.0, vf = 0.0;
    if (edge) {
        double s = 0.0;
        for (long long q = a.hrp[i]; q < a.hrp[i + 1]; ++q) s += a.hv[q] * a.e[a.hci[q]];
        ve = 0.5 * a.e[i] * s;
    }
    if (face) vf = 0.5 * a.b[i] * a.b[i] * a.geo[i].hb;
    // the instances this block holds part of: usually one
    if (tid == 0) { lo_s = a.ninst_n; hi_s = -1; }
    __syncthreads();
    if (edge) { atomicMin(&lo_s, ie); atomicMax(&hi_s, ie); }
    if (face) { atomicMin(&lo_s, jf); atomicMax(&hi_s, jf); }
    __syncthreads();
    const int lo = lo_s, hi = hi_s;
    double *out = a.part + (long long)blockIdx.x * a.ninst_n;
    for (int in = tid; in < a.ninst_n; in += 256)
        if (in < lo || in > hi) out[in] = 0.0;
    for (int in = lo; in <= hi; ++in) {
        double v = 0.0;
        if (ie == in) v += ve;
        if (jf == in) v += vf;
        sh[tid] = v;
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if (tid < o) sh[tid] += sh[tid + o];
            __syncthreads();
        }
        if (tid == 0) out[in] = sh[0];
        __syncthreads();
    }
    if (!a.ticket) return;
    __threadfence();
    __syncthreads();
    if (tid == 0) last_s = atomicAdd(a.ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last_s) return;
    if (tid == 0) *a.ticket = 0u;
    for (int in = tid >> 5; in < a.ninst_n; in += 8) energy_sum(gridDim.x, a.ninst_n, a.part, in, tid & 31, a.out);
}

// Energy, second pass for many partials: one warp per instance.
__global__ void k_energy_final(long long nblocks, int ninst, const double *__restrict__ part, double *__restrict__ out)
{
    const int in = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (in < ninst) energy_sum(nblocks, ninst, part, in, threadIdx.x & 31, out);
}

void launch_charge(cudaStream_t st, bool fp32, long long P, const int *cell, const short *chunk_sp, const Species *sp,
                   const Geo64 *geo, const Topo *topo, const void *f0, const void *f1, unsigned long long *q, int N,
                   bool clean, bool pdl)
{
    if (!clean) cudaMemsetAsync(q, 0, sizeof(unsigned long long) * (size_t)N, st);
    if (P <= 0) return;
    const long long nch = P / 32, warps = fp32 ? (nch + CH_CHUNKS - 1) / CH_CHUNKS : nch;
    const dim3 g((unsigned)((warps + 7) / 8));
    if (fp32) launch_k(pdl, k_charge32, g, dim3(256), st, nch, cell, chunk_sp, sp, topo, (const float *)f0, (const float *)f1, q);
    else launch_k(pdl, k_charge64, g, dim3(256), st, nch, cell, chunk_sp, sp, geo, topo, (const double *)f0, (const double *)f1, q);
}

void launch_gauss_reference(cudaStream_t st, int N, const int *nrp, const int *nedge, const int *ninst,
                            const double *qunit, const double *d, const unsigned long long *q, double *g0)
{
    if (N > 0) k_gauss_reference<<<(N + 255) / 256, 256, 0, st>>>(N, nrp, nedge, ninst, qunit, d, q, g0);
}

long long check_blocks(int N, int E, int F) { return ((long long)std::max(N, std::max(E, F)) + 255) / 256; }

int launch_checks(cudaStream_t st, const CheckArgs &a, bool pdl)
{
    const long long nb = check_blocks(a.N, a.E, a.F);
    if (nb <= 0) return 0;
    CheckArgs w = a;
    // one block sums the partials as fast as a launch would start; many are spread over more warps
    const bool own = nb * a.ninst_n <= 16384;
    if (!own) w.ticket = nullptr;
    launch_k(pdl, k_checks, dim3((unsigned)nb), dim3(256), st, w);
    if (!own) k_energy_final<<<(a.ninst_n + 7) / 8, 256, 0, st>>>(nb, a.ninst_n, a.part, a.out);
    return own ? 1 : 2;
}


// ------------------------------------------------------------- field probes
// One block: every thread reads the step counter before thread 0 advances it,
// so a captured graph writes consecutive ring rows on consecutive replays.
__global__ void __launch_bounds__(256) k_probe(long long n, const ProbeW *__restrict__ pw, const double *__restrict__ e,
                                               double2 *__restrict__ ring, long long cap,
                                               unsigned long long *count)
{
    const unsigned long long row = *count % (unsigned long long)cap;
    double2 *out = ring + (size_t)row * (size_t)n;
    for (long long p = threadIdx.x; p < n; p += blockDim.x) {
        const ProbeW w = pw[p];
        const double e0 = e[w.eg[0]], e1 = e[w.eg[1]], e2 = e[w.eg[2]];
        out[p] = make_double2(w.w[0] * e0 + w.w[2] * e1 + w.w[4] * e2, w.w[1] * e0 + w.w[3] * e1 + w.w[5] * e2);
    }
    __syncthreads();
    if (threadIdx.x == 0) *count += 1;
}

void launch_probe(cudaStream_t st, long long n, const ProbeW *pw, const double *e, double2 *ring, long long cap,
                  unsigned long long *count)
{
    if (n <= 0 || cap <= 0) return;
    k_probe<<<1, 256, 0, st>>>(n, pw, e, ring, cap, count);
}

}  // namespace fetdpic

// ------------------------------------------------- arithmetic-rate probe
// Measurement aid for the roofline of the arithmetic-bound FP64 particle path
// (no counterpart in the paper): eight independent FMA chains per thread,
// unrolled 16 deep, on a grid that fills every SM.
namespace fetdpic {

template <typename T>
__global__ void __launch_bounds__(256) k_fma_rate(int iters, T seed, T *out)
{
    T a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = seed + (T)(threadIdx.x + k);
    const T m = (T)0.9999999, c = (T)1e-7;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int u = 0; u < 16; ++u) {
#pragma unroll
            for (int k = 0; k < 8; ++k) a[k] = fma(a[k], m, c);
        }
    }
    T s = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += a[k];
    if (s == (T)-1) out[0] = s;                      // never true; keeps the chains live
}

}  // namespace fetdpic

extern "C" int fetdpic_fma_rate(int fp64, double *tflops)
{
    using namespace fetdpic;
    if (!tflops) return FETDPIC_EINVAL;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return FETDPIC_ECUDA;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return FETDPIC_ECUDA;
    cudaStream_t st = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    void *out = nullptr;
    int rc = FETDPIC_OK;
    if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess ||
        cudaMalloc(&out, 16) != cudaSuccess)
        rc = FETDPIC_ECUDA;
    const unsigned grid = (unsigned)sms * 8u;
    const double threads = (double)grid * 256.0;
    double best = 0.0;
    int iters = 64;
    for (int trial = 0; rc == FETDPIC_OK && trial < 12; ++trial) {
        cudaEventRecord(e0, st);
        if (fp64) k_fma_rate<double><<<grid, 256, 0, st>>>(iters, 1.0, (double *)out);
        else k_fma_rate<float><<<grid, 256, 0, st>>>(iters, 1.0f, (float *)out);
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess) { rc = FETDPIC_ECUDA; break; }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < 20.f) { iters = (int)std::min(1 << 22, iters * 2); continue; }   // grow to >= 20 ms
        best = std::max(best, 2.0 * 8 * 16 * (double)iters * threads / (ms * 1e-3) / 1e12);
    }
    if (rc == FETDPIC_OK && cudaGetLastError() != cudaSuccess) rc = FETDPIC_ECUDA;
    if (out) cudaFree(out);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (st) cudaStreamDestroy(st);
    *tflops = best;
    return rc;
}
