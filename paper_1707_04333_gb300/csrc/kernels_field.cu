// The field update by patches: Ampere's law, and with it the Faraday update of
// the next step, in one launch of one block per patch of triangles
// (field_patches.cpp).
//
// A step's field update was three dependent kernels (curl and current, SPAI
// product, Faraday), each a single wave of short threads bound by the latency
// of dependent loads and the gaps between launches.  A patch recomputes the
// curl on the edges around it (about a third more) instead of waiting for
// another block's, so the three run behind one another in shared memory, the
// SPAI's columns shrink to 16-bit numbers inside the patch, and r never goes
// to memory.  Same operations per edge, row and triangle, in the same order,
// as the separate kernels: the same bits.
//
// Measured (device time of a step, graph replay, with the particles): 2,048
// triangles and 64 electrons 9.8 -> 6.6 us, 8,192 triangles and 328k particles
// 19.0 -> 15.6, 320k triangles and 640k particles 52.7 -> 42.8, 201k triangles
// and 8 M particles 134.8 -> 128.9.  Bound by the FP64 pipe (2 lanes per SM and
// clock, 53 % busy; conversions to and from FP32 run in integer arithmetic beside
// it) and by the latency of the loads between its phases (320k triangles: 26 of
// a warp's 36 cycles per issue wait for memory or a barrier, issue 27 %, DRAM 37 %).
#include <cuda_runtime.h>

#include "fetdpic_internal.h"
#include "field_device.cuh"

namespace fetdpic {

namespace {

constexpr int RB = 2;                       // edges of the curl phase a thread has in flight
// Threads of a block: 512, three blocks per SM, for patches of more than 128
// triangles; 256 for the small meshes, whose rows are loaded whole (seven
// pairs at a time): only latency counts there.
constexpr int NT_LARGE = 512, NT_SMALL = 256, PER_SM = FIELD_PER_SM;
template <typename V> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };

// FAR: 0 = Ampere only, 1 = the FP32 Faraday update with it, 2 = the FP64 one.
template <typename V, int FAR, bool EXT, int NT>
__global__ void __launch_bounds__(NT, NT == NT_LARGE ? PER_SM : 4) k_field(FieldArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    double *hs = reinterpret_cast<double *>(sm);                       // C^T [*mu^-1] b; then, in FP64, r
    double *es = hs + a.max_r;                                         // e^{n+1} on the patch's edges and the ring
    V *rs = sizeof(V) == 8 ? reinterpret_cast<V *>(hs) : reinterpret_cast<V *>(es + a.max_e);
    const int tid = threadIdx.x;
    const unsigned long long keep = l2_keep();
    const FieldPatch P = a.patch[blockIdx.x];
    const int nr = P.ne + P.nx;
    if (!a.early) pdl_begin();
    // the curl part needs b only, which is older than the kernel before this one
    for (int k0 = tid; k0 < nr; k0 += RB * NT) {
        int2 fa[RB];
        double2 cf[RB];
        double b0[RB], b1[RB];
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int k = k0 + i * NT;
            if (k >= nr) continue;
            const int g = k < P.ne ? P.e0 + k : __ldg(a.xlist + P.x0 + (k - P.ne));
            fa[i] = ld_keep(a.efac + g, keep);
            cf[i] = ld_keep(a.ecoef + g, keep);
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            if (k0 + i * NT >= nr) continue;
            b0[i] = __ldcg(a.b + fa[i].x);
            b1[i] = fa[i].y >= 0 ? __ldcg(a.b + fa[i].y) : 0.0;
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int k = k0 + i * NT;
            if (k >= nr) continue;
            double h = b0[i] * cf[i].x;
            if (fa[i].y >= 0) h += b1[i] * cf[i].y;
            hs[k] = h;
        }
    }
    if (FAR)
        for (int k = tid; k < P.ne + P.nring; k += NT) es[k] = 0.0;     // PEC edges stay 0
    if (a.early) pdl_begin();
    // r = C^T [*mu^-1] b^{n+1/2} - i^{n+1/2}
    for (int k0 = tid; k0 < nr; k0 += RB * NT) {
        long long iv[RB];
        int in[RB], g[RB];
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int k = k0 + i * NT;
            if (k >= nr) continue;
            g[i] = k < P.ne ? P.e0 + k : __ldg(a.xlist + P.x0 + (k - P.ne));
            iv[i] = (long long)a.ifix[g[i]];
            in[i] = a.one_inst ? 0 : ld_keep(a.einst + g[i], keep);
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int k = k0 + i * NT;
            if (k >= nr) continue;
            const double h = hs[k];
            const double cur = (double)iv[i] * a.inst_unit[in[i]];
            const double rv = h - cur;
            if constexpr (sizeof(V) == 4) rs[k] = to_f32(rv);
            else rs[k] = rv;
            if (k < P.ne) {
                a.j[g[i]] = cur;
                if (a.d) a.d[g[i]] += a.inst_dt[in[i]] * rv;
                if (FAR) a.ifix_next[g[i]] = 0ull;
            }
        }
    }
    __syncthreads();
    // e += (dt M) r on the patch's rows, and on the ring's when its triangles go on to Faraday; a
    // row's entries are loaded RP pairs at a time
    {
        using V2 = typename Pair<V>::type;
        constexpr int RP = NT == NT_SMALL ? 7 : 4;
        const V2 *__restrict__ val;
        if constexpr (sizeof(V) == 4) val = reinterpret_cast<const V2 *>(a.v32);
        else val = reinterpret_cast<const V2 *>(a.v64);
        const int lane = tid & 31, no = (P.nown + 31) >> 5, ns = no + (FAR ? (P.nringrow + 31) >> 5 : 0);
        for (int sl = tid >> 5; sl < ns; sl += NT / 32) {
            const int loc = __ldg(a.row_loc + P.row0 + sl * 32 + lane);
            const bool valid = sl < no ? sl * 32 + lane < P.nown : (sl - no) * 32 + lane < P.nringrow;
            const int g = loc < P.ne ? P.e0 + loc : __ldg(a.xlist + P.x0 + (loc - P.ne));
            const double eo = a.e[g];
            const long long o0 = __ldg(a.soff + P.slice0 + sl);
            const int n = (int)(__ldg(a.soff + P.slice0 + sl + 1) - o0);        // 32 x pairs
            const V2 *vp = val + o0 + lane;
            const unsigned *cp = a.col + o0 + lane;
            V s0 = V(0), s1 = V(0);
            for (int q = 0; q < n; q += 32 * RP) {
                V2 v[RP];
                unsigned c[RP];
#pragma unroll
                for (int i = 0; i < RP; ++i) {
                    if (q + 32 * i < n) { v[i] = ld_keep(vp + q + 32 * i, keep); c[i] = ld_keep(cp + q + 32 * i, keep); }
                }
#pragma unroll
                for (int i = 0; i < RP; ++i) {
                    if (q + 32 * i < n) {
                        s0 += v[i].x * rs[c[i] & 0xffffu];
                        s1 += v[i].y * rs[c[i] >> 16];
                    }
                }
            }
            if (valid) {
                double en;
                if constexpr (sizeof(V) == 4) en = eo + to_f64(s0 + s1);
                else en = eo + (s0 + s1);
                if (FAR) es[loc] = en;
                if (sl < no) a.e_next[g] = en;
            }
        }
    }
    if constexpr (FAR != 0) {
        __syncthreads();
        for (int k = tid; k < P.nt; k += NT) {
            const int f = P.t0 + k;
            const ushort4 l = __ldg(a.tloc + f);
            double se[3] = {es[l.x], es[l.y], es[l.z]};
            const double bo = a.b[f];
            if constexpr (FAR == 1) {
                const float4 *cp = reinterpret_cast<const float4 *>(a.csta + f);
                const float4 c0 = __ldg(cp), c1 = __ldg(cp + 1);
                const int ew0 = __ldg(&a.cstb[f].ew0);
                if (ew0 & 1) se[0] = -se[0];
                if (__float_as_int(c1.x) & 1) se[1] = -se[1];
                if (__float_as_int(c1.y) & 1) se[2] = -se[2];
                a.b_next[f] = faraday32_rec(f, se, bo, a.dtinv[f], c0, c1, ew0, a.rec32, a.inv2c2, a.ext, EXT);
            } else {
                // every operation rounded as written (k_faraday64)
                const Topo *T = a.topo + f;
                if (__ldg(&T->ew[0]) & 1) se[0] = -se[0];
                if (__ldg(&T->ew[1]) & 1) se[1] = -se[1];
                if (__ldg(&T->ew[2]) & 1) se[2] = -se[2];
                const double ce = __dadd_rn(__dadd_rn(__dadd_rn(0.0, se[0]), se[1]), se[2]);
                const double bn = __dsub_rn(bo, __dmul_rn(a.geo[f].dt, ce));
                a.b_next[f] = bn;
                Rec64 r;
                r.se[0] = se[0]; r.se[1] = se[1]; r.se[2] = se[2];
                r.bz = __dmul_rn(__dadd_rn(bn, bo), a.geo[f].inv2A);
                a.rec64[f] = r;
            }
        }
    }
}

// The limit belongs to the kernel, for every context of the process: always the same value, since one
// context's smaller need would take from another's.
template <typename V, int FAR, bool EXT>
cudaError_t setup()
{
    constexpr cudaFuncAttribute limit = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_field<V, FAR, EXT, NT_SMALL>, limit, (int)FIELD_SMEM_MAX);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_field<V, FAR, EXT, NT_LARGE>, limit, (int)FIELD_SMEM_MAX);
    return e;
}

template <typename V, int FAR, bool EXT>
void go(cudaStream_t st, const FieldArgs &a)
{
    const size_t smem = field_smem(sizeof(V) == 4, a.max_r, a.max_e);
    if (a.T > 128) launch_ks(a.pdl, k_field<V, FAR, EXT, NT_LARGE>, dim3(a.npatch), dim3(NT_LARGE), smem, st, a);
    else launch_ks(a.pdl, k_field<V, FAR, EXT, NT_SMALL>, dim3(a.npatch), dim3(NT_SMALL), smem, st, a);
}

}  // namespace

cudaError_t field_setup(size_t smem)
{
    if (smem <= 48 * 1024) return cudaSuccess;         // what every kernel may use
    cudaError_t e = setup<float, 0, false>();
    if (e == cudaSuccess) e = setup<float, 1, false>();
    if (e == cudaSuccess) e = setup<float, 1, true>();
    if (e == cudaSuccess) e = setup<double, 0, false>();
    if (e == cudaSuccess) e = setup<double, 2, false>();
    return e;
}

void launch_field(cudaStream_t st, const FieldArgs &a)
{
    if (a.npatch <= 0) return;
    if (a.v32) {
        if (!a.faraday) go<float, 0, false>(st, a);
        else if (a.ext.ext) go<float, 1, true>(st, a);
        else go<float, 1, false>(st, a);
    } else {
        if (!a.faraday) go<double, 0, false>(st, a);
        else go<double, 2, false>(st, a);
    }
}

}  // namespace fetdpic
