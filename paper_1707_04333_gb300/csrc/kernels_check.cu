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

// Continuity residual per node: res = (q1 - q0) + sum_e o(k,e) i_e, exactly in
// integers; normalised by sum_e |i_e| + |q1 - q0| (at least one unit).
__global__ void k_dce(int N, const int *__restrict__ nrp, const int *__restrict__ nedge,
                      const int *__restrict__ ninst, const unsigned long long *__restrict__ ifix,
                      const unsigned long long *__restrict__ q0, const unsigned long long *__restrict__ q1,
                      double *__restrict__ out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = k < N;
    long long flux = 0;
    double absf = 0.0;
    for (int r = live ? nrp[k] : 0, r1 = live ? nrp[k + 1] : 0; r < r1; r += NB) {
        int w[NB];
        long long iv[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) w[i] = r + i < r1 ? nedge[r + i] : 0;
#pragma unroll
        for (int i = 0; i < NB; ++i) iv[i] = r + i < r1 ? (long long)ifix[w[i] >> 1] : 0;
#pragma unroll
        for (int i = 0; i < NB; ++i)
            if (r + i < r1) {
                flux += (w[i] & 1) ? -iv[i] : iv[i];
                absf += fabs((double)iv[i]);
            }
    }
    const long long dq = live ? (long long)q1[k] - (long long)q0[k] : 0;
    const long long res = dq + flux;
    const double scale = fmax(absf + fabs((double)dq), 1.0);
    warp_max_pos(out, 0, live ? ninst[k] : 0, fabs((double)res) / scale, live);
}

// Gauss residual per node: g = sum_e o(k,e) d_e - q (physical units).  With
// init != 0 it stores g as the reference g0; otherwise it reports
// |g - g0| / (sum |d_e| + |q| + |g0|).
__global__ void k_dgl(int N, const int *__restrict__ nrp, const int *__restrict__ nedge,
                      const int *__restrict__ ninst, const double *__restrict__ qunit,
                      const double *__restrict__ d, const unsigned long long *__restrict__ q,
                      double *__restrict__ g0, int init, double *__restrict__ out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = k < N;
    double s = 0.0, sa = 0.0;
    for (int r = live ? nrp[k] : 0, r1 = live ? nrp[k + 1] : 0; r < r1; r += NB) {
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
    const int in = live ? ninst[k] : 0;
    const double qk = live ? (double)(long long)q[k] * qunit[in] : 0.0;
    const double g = s - qk;
    if (init) { if (live) g0[k] = g; return; }
    const double ref = live ? g0[k] : 0.0;
    const double scale = sa + fabs(qk) + fabs(ref);
    const double nr = scale > 0.0 ? fabs(g - ref) / scale : 0.0;
    warp_max_pos(out, 1, in, nr, live);
}

// Energy, first pass: per block, sum over its edges of e_k ([*eps] e)_k / 2 and
// over its faces of b_f^2 / (2 mu0 A_f), per instance; written to part[block].
__global__ void k_energy_part(int E, int F, const long long *__restrict__ hrp, const int *__restrict__ hci,
                              const double *__restrict__ hv, const double *__restrict__ e,
                              const int *__restrict__ einst, const double *__restrict__ b,
                              const Geo64 *__restrict__ geo, const Topo *__restrict__ topo,
                              int ninst, double *__restrict__ part)
{
    extern __shared__ double sh[];              // [blockDim.x]
    __shared__ int lo_s, hi_s;
    const int tid = threadIdx.x;
    const long long i = (long long)blockIdx.x * blockDim.x + tid;
    const bool edge = i < E, face = i < F;
    const int ie = edge ? einst[i] : -1, jf = face ? topo[i].inst : -1;
    double ve = 0.0, vf = 0.0;
    if (edge) {
        double s = 0.0;
        for (long long q = hrp[i]; q < hrp[i + 1]; ++q) s += hv[q] * e[hci[q]];
        ve = 0.5 * e[i] * s;
    }
    if (face) vf = 0.5 * b[i] * b[i] * geo[i].hb;
    // the instances this block holds part of: usually one
    if (tid == 0) { lo_s = ninst; hi_s = -1; }
    __syncthreads();
    if (edge) { atomicMin(&lo_s, ie); atomicMax(&hi_s, ie); }
    if (face) { atomicMin(&lo_s, jf); atomicMax(&hi_s, jf); }
    __syncthreads();
    const int lo = lo_s, hi = hi_s;
    double *out = part + (long long)blockIdx.x * ninst;
    for (int in = tid; in < ninst; in += blockDim.x)
        if (in < lo || in > hi) out[in] = 0.0;
    for (int in = lo; in <= hi; ++in) {
        double v = 0.0;
        if (ie == in) v += ve;
        if (jf == in) v += vf;
        sh[tid] = v;
        __syncthreads();
        for (int o = blockDim.x / 2; o > 0; o >>= 1) {
            if (tid < o) sh[tid] += sh[tid + o];
            __syncthreads();
        }
        if (tid == 0) out[in] = sh[0];
        __syncthreads();
    }
}

// Energy, second pass: one warp per instance sums the block partials, in an order
// that depends on their number only.
__global__ void k_energy_final(long long nblocks, int ninst, const double *__restrict__ part, double *__restrict__ out)
{
    const int in = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (in >= ninst) return;
    double s = 0.0;
    for (long long k = lane; k < nblocks; k += 32) s += part[k * ninst + in];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) out[3 * in + 2] = s;
}

void launch_charge(cudaStream_t st, bool fp32, long long P, const int *cell, const short *chunk_sp, const Species *sp,
                   const Geo64 *geo, const Topo *topo, const void *f0, const void *f1, unsigned long long *q, int N)
{
    cudaMemsetAsync(q, 0, sizeof(unsigned long long) * (size_t)N, st);
    if (P <= 0) return;
    const long long nch = P / 32, warps = fp32 ? (nch + CH_CHUNKS - 1) / CH_CHUNKS : nch;
    const unsigned g = (unsigned)((warps + 7) / 8);
    if (fp32) k_charge32<<<g, 256, 0, st>>>(nch, cell, chunk_sp, sp, topo, (const float *)f0, (const float *)f1, q);
    else k_charge64<<<g, 256, 0, st>>>(nch, cell, chunk_sp, sp, geo, topo, (const double *)f0, (const double *)f1, q);
}

void launch_dce(cudaStream_t st, int N, const int *nrp, const int *nedge, const int *ninst,
                const unsigned long long *ifix, const unsigned long long *q0, const unsigned long long *q1, double *out)
{
    if (N <= 0) return;
    k_dce<<<(N + 255) / 256, 256, 0, st>>>(N, nrp, nedge, ninst, ifix, q0, q1, out);
}

void launch_dgl(cudaStream_t st, int N, const int *nrp, const int *nedge, const int *ninst, const double *qunit,
                const double *d, const unsigned long long *q, double *g0, int init, double *out)
{
    if (N <= 0) return;
    k_dgl<<<(N + 255) / 256, 256, 0, st>>>(N, nrp, nedge, ninst, qunit, d, q, g0, init, out);
}

long long energy_blocks(int E, int F) { return ((long long)(E > F ? E : F) + 255) / 256; }

void launch_energy(cudaStream_t st, int E, int F, const long long *hrp, const int *hci, const double *hv,
                   const double *e, const int *einst, const double *b, const Geo64 *geo, const Topo *topo,
                   int ninst, double *part, double *out)
{
    const long long nb = energy_blocks(E, F);
    if (nb <= 0) return;
    k_energy_part<<<(unsigned)nb, 256, 256 * sizeof(double), st>>>(E, F, hrp, hci, hv, e, einst, b, geo, topo, ninst,
                                                                    part);
    k_energy_final<<<(ninst + 7) / 8, 256, 0, st>>>(nb, ninst, part, out);
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
