// The C ABI of include/fetdpic.h: context, device memory, launch sequence.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "fetdpic_internal.h"

using namespace fetdpic;

namespace {

constexpr double CODATA_EPS0 = 8.8541878128e-12;
constexpr double CODATA_MU0 = 1.25663706212e-6;
constexpr double CODATA_C = 299792458.0;
constexpr long long SPECIES_ALIGN = 1024;   // species storage ranges start on this multiple
// FP32-path current quantum 1/(2^25 - 64) of q_ref/dt: a per-particle contribution is at
// most 2^25 - 60 in magnitude, so a warp's 64-particle run sum stays below 2^31.
constexpr double FP32_SCALE = 33554368.0;

struct StagedSpecies {
    int inst;
    double q, m;
    std::vector<int> cell;                   // instance-local
    std::vector<double> x, y, ux, uy;
};

}  // namespace

struct fetdpic_ctx {
    fetdpic_params p{};
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    // a stream of the context's own on which the particle sort runs beside the
    // Ampere update (both only read what the particle kernel wrote), forked
    // from and joined back into `stream` by the two events
    cudaStream_t side = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    std::string err;

    std::vector<HostMesh> mesh;
    std::vector<fetdpic_instance> inst;
    std::vector<int> cell_off, edge_off, node_off;
    int F = 0, E = 0, N = 0;
    long long nfree = 0;

    // device: mesh and fields
    Geo64 *geo64 = nullptr; double2 *dtinv = nullptr; Topo *topo = nullptr;
    CstA *csta = nullptr; CstB *cstb = nullptr;
    Rec64 *rec64 = nullptr; Rec32 *rec32 = nullptr;
    double *e = nullptr, *b = nullptr, *d = nullptr, *r = nullptr, *j = nullptr;
    unsigned long long *ifix = nullptr;
    // field update by patches (kernels_field.cu): its tables, and the second buffers that e, b and
    // the current accumulator go to and from when it carries the next step's Faraday update
    bool patches = false;
    FieldArgs field{};
    double *e_alt = nullptr, *b_alt = nullptr, *e_a = nullptr;     // e_a: the first buffer (parity reference)
    unsigned long long *ifix_alt = nullptr;
    int2 *efac = nullptr; double2 *ecoef = nullptr; int *einst = nullptr;
    double *inst_unit = nullptr, *inst_dt = nullptr;
    int *edge_off_dev = nullptr;
    long long *m_soff = nullptr; int *m_row = nullptr, *m_ci = nullptr; double *m_v = nullptr;
    long long m_entries = 0;                  // stored SPAI entries (sliced ELL, padding included)
    float *m_v32 = nullptr, *r32 = nullptr;
    unsigned *status = nullptr;
    unsigned *gbar = nullptr;                // grid-barrier state of the fused Ampere launch (GBAR_WORDS)
    std::vector<double> unit_host;           // per instance (q_ref/dt) / scale
    std::vector<double> fixscale;            // per instance fixed-point scale (2^shift in FP64)
    std::vector<double> qunit_host;          // per instance charge of one fixed-point unit: q_ref / scale
    unsigned long long *qread = nullptr;     // nodal charge for fetdpic_read_charge (allocated on first use)

    // particles
    std::vector<StagedSpecies> staged;
    bool finalized = false;
    std::vector<Species> sp;
    Species *sp_dev = nullptr;
    Sp32 *sp32_dev = nullptr;
    int sms = 0;                             // of the device
    bool soft64 = false;                     // FP64 constants within the integer arithmetic's range
    double density = 0.0;                    // particles per triangle where the particles are
    long long P = 0, nblocks = 0;
    int block = 256;
    int *cell = nullptr, *cell_tmp = nullptr, *id = nullptr, *id_tmp = nullptr;
    void *f[4] = {nullptr, nullptr, nullptr, nullptr}, *f_tmp[4] = {nullptr, nullptr, nullptr, nullptr};
    short *chunk_sp = nullptr;               // species of each 32-particle chunk
    signed char *tshift = nullptr;           // periodic shift codes (FP64 walk), NULL without periodic walls
    double2 *period = nullptr;               // per instance
    // applied fields: per-instance (E_x, E_y, B_z, 0) and amplitude of E, per-triangle weights
    ExtField *ext_dev = nullptr;
    double *ext_amp = nullptr;
    double2 *extw = nullptr;                 // NULL until a profile is set
    int *face_inst = nullptr;                // FP32: instance of each triangle
    int *tri_c2i = nullptr;                  // [cell_off + caller index] -> stored instance-local index
    int *edge_c2i = nullptr;                  // [edge_off + caller index] -> stored instance-local index
    double *field_out = nullptr;              // one instance's e, b, j in the caller's order (reads)
    int *tri_i2c = nullptr;                  // [stored global index] -> caller's instance-local index
    bool ext_on = false;                     // FP32: fold applied fields into the field record
    int *hist = nullptr, *hoff = nullptr, *scan_tmp = nullptr; long long hist_n = 0;
    int *rec_cnt = nullptr, *rec = nullptr;

    long long steps_done = 0;
    long long launches_acc = 0;
    std::vector<cudaEvent_t> ev;             // event pool, grown on demand
    std::vector<int> ev_stage;               // stage closed by each recorded event (-1 = start of a step)
    int ev_used = 0;
    double stage_ms[6] = {0, 0, 0, 0, 0, 0};
    // checks: node -> edge incidence (edge << 1 | enters-node), node instance,
    // charge in fixed point (q0 before / q1 after the particle kernel), Gauss
    // reference g0, full [*eps] for the energy, results per instance
    int *nrp = nullptr, *nedge = nullptr, *ninst = nullptr;
    unsigned long long *q0 = nullptr, *q1 = nullptr;
    double *g0 = nullptr, *qunit = nullptr, *chk_out = nullptr, *eng_part = nullptr;
    long long *h_rp = nullptr; int *h_ci = nullptr; double *h_v = nullptr;
    unsigned *chk_ticket = nullptr;           // blocks of the check kernel that are done
    bool q1_clean = false;                    // q1 is zero (cleared by the last check)
    bool q_prev_valid = false;                // q0 holds the charge of the current particle state
    bool g0_ready = false;
    std::vector<char> gauss_abs;              // per instance: Gauss law checked absolutely (after the solve)
    std::vector<std::vector<char>> abs_nodes; // per instance: nodes off the PEC walls (absolute reference 0)
    // reusable device scratch for host <-> device transfers of particle state
    void *xfer = nullptr; size_t xfer_bytes = 0;
    // page-locked host memory: small reads come back in one copy each, with the status word behind
    // them, and one wait (SMALL_READ bytes for them, then the status)
    char *pin = nullptr, *pin_locked = nullptr;
    std::vector<char> pin_plain;              // in its place where the host has none to lock
    // asynchronous particle reads: staging of their own (one region per species), copied to the
    // host on the io stream while the context stream goes on; set up by the first such read
    cudaStream_t io = nullptr;
    cudaEvent_t ev_rd = nullptr;              // load-order copy done on the context stream
    std::vector<cudaEvent_t> ev_rd_done;      // per species: its last host copy finished (io stream)
    std::vector<char> rd_pending;             // per species: ev_rd_done has been recorded
    char *rd_buf = nullptr;
    std::vector<size_t> rd_off;

    // captured one-step graphs: [pusher][particle-buffer parity][step sorts][late hybrid step]
    // [field-buffer parity]
    cudaGraphExec_t graph[4][2][2][2][2] = {};
    long long graph_launches[4][2][2][2][2] = {};
    // captured sort cycles (sort_interval steps, the last of which sorts): [pusher][particle-buffer
    // parity at the start][field-buffer parity]
    cudaGraphExec_t cycle[4][2][2] = {};
    long long cycle_launches[4][2][2] = {};
    int *cell_a = nullptr;                    // the first particle buffer (parity reference)

    std::vector<void *> allocs;

    // field probes (diagnostic): weights, ring of E samples, device step counter
    long long probe_n = 0, probe_cap = 0;
    ProbeW *probe_w = nullptr;
    double2 *probe_ring = nullptr;
    unsigned long long *probe_count = nullptr;

    ~fetdpic_ctx()
    {
        cudaSetDevice(device);
        // every stream of the context is idle before its memory goes back
        if (stream) cudaStreamSynchronize(stream);
        if (side) cudaStreamSynchronize(side);
        if (io) cudaStreamSynchronize(io);
        for (auto &a : graph) for (auto &b : a) for (auto &c : b) for (auto &d : c) for (auto &g : d)
            if (g) cudaGraphExecDestroy(g);
        for (auto &a : cycle) for (auto &b : a) for (auto &g : b) if (g) cudaGraphExecDestroy(g);
        for (void *q : allocs) {
            if (p.dev_free) p.dev_free(q, p.alloc_user);
            else cudaFree(q);
        }
        if (pin_locked) cudaFreeHost(pin_locked);
        for (auto &x : ev) cudaEventDestroy(x);
        for (auto &x : ev_rd_done) if (x) cudaEventDestroy(x);
        if (ev_rd) cudaEventDestroy(ev_rd);
        if (io) cudaStreamDestroy(io);
        if (ev_fork) cudaEventDestroy(ev_fork);
        if (ev_join) cudaEventDestroy(ev_join);
        if (side) cudaStreamDestroy(side);
        if (own_stream && stream) cudaStreamDestroy(stream);
    }

    template <typename T>
    T *alloc(size_t count)
    {
        size_t bytes = std::max<size_t>(count * sizeof(T), 16);
        void *q = nullptr;
        if (p.dev_alloc) q = p.dev_alloc(bytes, p.alloc_user);
        else if (cudaMalloc(&q, bytes) != cudaSuccess) q = nullptr;
        if (!q) throw std::bad_alloc();
        allocs.push_back(q);
        return (T *)q;
    }

    // Frees one allocation made by alloc().
    void release(void *q)
    {
        if (!q) return;
        for (size_t k = 0; k < allocs.size(); ++k)
            if (allocs[k] == q) { allocs.erase(allocs.begin() + k); break; }
        if (p.dev_free) p.dev_free(q, p.alloc_user);
        else cudaFree(q);
    }

    int fail(int code, const std::string &m)
    {
        err = m;
        return code;
    }

    int cuda_fail(cudaError_t e, const char *where)
    {
        err = std::string(where) + ": " + cudaGetErrorString(e);
        return FETDPIC_ECUDA;
    }
};

// Reads of up to this many bytes go through the context's page-locked buffer (one copy and one wait:
// a particle read took three pageable copies, each a wait of its own, and a fourth for the status).  A
// field read of 160 KB takes 37 us so against 55 in pageable copies, of 315 KB 49 against 61; of 640 KB, 78
// against 68: there the host's own copy out of the buffer costs more than the waits.
constexpr size_t SMALL_READ = 384 * 1024;

#define CK(call)                                                                     \
    do {                                                                             \
        cudaError_t _e = (call);                                                     \
        if (_e != cudaSuccess) return ctx->cuda_fail(_e, #call);                     \
    } while (0)

template <typename T>
static int upload(fetdpic_ctx *ctx, T *dst, const T *src, size_t n)
{
    if (n == 0) return FETDPIC_OK;
    CK(cudaMemcpyAsync(dst, src, n * sizeof(T), cudaMemcpyHostToDevice, ctx->stream));
    return FETDPIC_OK;
}

static int map_status(fetdpic_ctx *ctx, unsigned st)
{
    if (st & ST_WALK) return ctx->fail(FETDPIC_EWALK, "a particle crossed more than max_crossings edges in one step");
    if (st & ST_NONFINITE) return ctx->fail(FETDPIC_ENONFINITE, "non-finite momentum or Lorentz factor");
    if (st & ST_TIMEOUT) return ctx->fail(FETDPIC_ETIMEOUT, "a bounded wait for staged particle data gave up");
    if (st & ST_BADCELL)
        return ctx->fail(FETDPIC_EINVAL, "fetdpic_write_particles was given a triangle outside the mesh; "
                                         "those particles were dropped");
    if (st) return ctx->fail(FETDPIC_EMESH, "device status " + std::to_string(st));
    return FETDPIC_OK;
}

// Waits for the context stream with the device status word behind its work, and clears the word when
// set, so a latched fault is reported once; returns the mapped status.
static int take_status(fetdpic_ctx *ctx)
{
    unsigned *st = reinterpret_cast<unsigned *>(ctx->pin + SMALL_READ);
    CK(cudaMemcpyAsync(st, ctx->status, sizeof(unsigned), cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    const unsigned s = *st;
    if (s) CK(cudaSetDevice(ctx->device));      // a clear needs the stream's device
    if (s) CK(cudaMemsetAsync(ctx->status, 0, sizeof(unsigned), ctx->stream));
    // a step that timed out is incomplete: drop the current it deposited, and the counts a grid
    // barrier that gave up left behind
    if (s & ST_TIMEOUT) {
        if (ctx->gbar) CK(cudaMemsetAsync(ctx->gbar, 0, sizeof(unsigned) * GBAR_WORDS, ctx->stream));
        if (ctx->ifix) CK(cudaMemsetAsync(ctx->ifix, 0, sizeof(unsigned long long) * ctx->E, ctx->stream));
    }
    return map_status(ctx, s);
}

extern "C" int fetdpic_create(fetdpic_ctx **out, const fetdpic_params *prm, int n_inst, const fetdpic_instance *inst)
{
    if (!out) return FETDPIC_EINVAL;
    *out = nullptr;
    if (!prm || n_inst <= 0 || !inst) return FETDPIC_EINVAL;
    std::unique_ptr<fetdpic_ctx> holder;
    try { holder.reset(new fetdpic_ctx()); } catch (...) { return FETDPIC_ENOMEM; }
    fetdpic_ctx *ctx = holder.get();
    ctx->p = *prm;
    auto &P = ctx->p;
    if (P.eps0 == 0) P.eps0 = CODATA_EPS0;
    if (P.mu0 == 0) P.mu0 = CODATA_MU0;
    if (P.c == 0) P.c = CODATA_C;
    if (P.precision != FETDPIC_FP64 && P.precision != FETDPIC_FP32) return FETDPIC_EINVAL;
    if (P.sort_interval == 0) P.sort_interval = 16;
    if (P.max_crossings <= 0) P.max_crossings = 64;
    if (P.block_size == 0) P.block_size = 256;
    if (P.block_size < 32 || P.block_size > 256 || (P.block_size & 31) || (SPECIES_ALIGN % P.block_size))
        return FETDPIC_EINVAL;
    if (P.record_walk < 0) return FETDPIC_EINVAL;
    if (P.kernel_variant < 0 || P.kernel_variant == 1 || P.kernel_variant > 22) return FETDPIC_EINVAL;
    ctx->block = P.block_size;
    CK(cudaGetDevice(&ctx->device));
    CK(cudaDeviceGetAttribute(&ctx->sms, cudaDevAttrMultiProcessorCount, ctx->device));
    if (P.cuda_stream) ctx->stream = (cudaStream_t)P.cuda_stream;
    else { CK(cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking)); ctx->own_stream = true; }
    CK(cudaStreamCreateWithFlags(&ctx->side, cudaStreamNonBlocking));
    CK(cudaEventCreateWithFlags(&ctx->ev_fork, cudaEventDisableTiming));
    CK(cudaEventCreateWithFlags(&ctx->ev_join, cudaEventDisableTiming));

    if (cudaHostAlloc((void **)&ctx->pin_locked, SMALL_READ + 256, cudaHostAllocDefault) != cudaSuccess) {
        // no page-locked memory to be had: reads go through ordinary memory, slower
        ctx->pin_locked = nullptr;
        cudaGetLastError();
        try { ctx->pin_plain.resize(SMALL_READ + 256); } catch (const std::bad_alloc &) { return FETDPIC_ENOMEM; }
    }
    ctx->pin = ctx->pin_locked ? ctx->pin_locked : ctx->pin_plain.data();

    // ---- host setup per instance
    ctx->mesh.resize(n_inst);
    ctx->gauss_abs.assign(n_inst, 0);
    ctx->abs_nodes.assign(n_inst, {});
    ctx->inst.assign(inst, inst + n_inst);
    ctx->cell_off.assign(n_inst + 1, 0);
    ctx->edge_off.assign(n_inst + 1, 0);
    ctx->node_off.assign(n_inst + 1, 0);
    for (int k = 0; k < n_inst; ++k) {
        const fetdpic_instance &I = inst[k];
        if (!(I.dt > 0)) return ctx->fail(FETDPIC_EINVAL, "dt must be > 0"), FETDPIC_EINVAL;
        std::string msg;
        int rc = build_mesh(ctx->mesh[k], I.n_nodes, I.nodes_xy, I.n_tri, I.triangles,
                            I.edges ? I.n_edges : 0, I.edges, I.edge_tags,
                            I.n_periodic, I.periodic_nodes, I.period_x, I.period_y, msg);
        if (rc == FETDPIC_OK) rc = build_hodge(ctx->mesh[k], P.eps0, msg);
        if (rc == FETDPIC_OK) rc = build_spai(ctx->mesh[k], P.spai_level, msg);
        if (rc != FETDPIC_OK) {
            fprintf(stderr, "fetdpic_create: instance %d: %s\n", k, msg.c_str());
            return rc;
        }
        ctx->cell_off[k + 1] = ctx->cell_off[k] + ctx->mesh[k].nf;
        ctx->edge_off[k + 1] = ctx->edge_off[k] + ctx->mesh[k].ne;
        ctx->node_off[k + 1] = ctx->node_off[k] + ctx->mesh[k].nn;
    }
    ctx->F = ctx->cell_off[n_inst];
    ctx->E = ctx->edge_off[n_inst];
    ctx->N = ctx->node_off[n_inst];
    if ((long long)ctx->F * 4 >= (1LL << 31) || (long long)ctx->E * 2 >= (1LL << 31))
        return FETDPIC_EINVAL;

    // ---- host images of the device tables
    std::vector<Geo64> g64(ctx->F);
    std::vector<CstA> g32(P.precision == FETDPIC_FP32 ? ctx->F : 0);
    std::vector<CstB> g32b(g32.size());
    std::vector<double2> dti(P.precision == FETDPIC_FP32 ? ctx->F : 0);
    std::vector<Topo> tp(ctx->F);
    std::vector<double> e0(ctx->E, 0.0), b0(ctx->F, 0.0), d0(ctx->E, 0.0);
    std::vector<int2> efac(ctx->E);
    std::vector<double2> ecoef(ctx->E);
    std::vector<int> einst(ctx->E);
    std::vector<long long> mrp(1, 0);
    std::vector<int> mrow, mci;
    std::vector<double> mv;
    std::vector<double> idt(n_inst);
    for (int k = 0; k < n_inst; ++k) {
        const HostMesh &M = ctx->mesh[k];
        const fetdpic_instance &I = inst[k];
        const int co = ctx->cell_off[k], eo = ctx->edge_off[k], no = ctx->node_off[k];
        idt[k] = I.dt;
        for (int f = 0; f < M.nf; ++f) {
            Geo64 &G = g64[co + f];
            for (int m = 0; m < 3; ++m) {
                G.gx[m] = M.gx[3 * f + m]; G.gy[m] = M.gy[3 * f + m];
                G.X[m] = M.X[3 * f + m]; G.Y[m] = M.Y[3 * f + m];
            }
            G.inv2A = M.inv2A[f];
            G.dt = I.dt;
            G.hb = 1.0 / (P.mu0 * (0.5 * M.d2A[f]));
            G.pad = 0;
            Topo &T = tp[co + f];
            for (int m = 0; m < 3; ++m) {
                const int eg = eo + M.einv[M.tedge[3 * f + m]];
                T.ew[m] = (eg << 1) | (M.tsign[3 * f + m] < 0 ? 1 : 0);
                T.nb[m] = M.tnb[3 * f + m] < 0 ? -1 : (((co + M.tnb[3 * f + m]) << 2) | M.tnbm[3 * f + m]);
                T.node[m] = no + M.rep[M.tri[3 * f + m]];
            }
            T.inst = k;
            b0[co + f] = I.b0 * (0.5 * M.d2A[f]);          // b_f = B0 A_f
            if (!g32.empty()) {
                CstA &H = g32[co + f];
                for (int m = 0; m < 2; ++m) {
                    H.G[2 * m] = (float)(P.c * I.dt * M.gx[3 * f + m]);
                    H.G[2 * m + 1] = (float)(P.c * I.dt * M.gy[3 * f + m]);
                }
                H.ew1 = T.ew[1]; H.ew2 = T.ew[2];
                H.nb0 = T.nb[0]; H.nb1 = T.nb[1];
                g32b[co + f] = CstB{T.ew[0], T.nb[2]};
                dti[co + f] = make_double2(I.dt, M.inv2A[f]);
            }
        }
        for (int e = 0; e < M.ne; ++e) {
            const int i = eo + M.einv[e];
            if (!M.pec[e]) e0[i] = I.e0x * M.evec[2 * e] + I.e0y * M.evec[2 * e + 1];
            efac[i] = make_int2(co + M.efac[2 * e], M.efac[2 * e + 1] < 0 ? -1 : co + M.efac[2 * e + 1]);
            const double h0 = 1.0 / (P.mu0 * (0.5 * M.d2A[M.efac[2 * e]]));
            const double h1 = M.efac[2 * e + 1] < 0 ? 0.0 : 1.0 / (P.mu0 * (0.5 * M.d2A[M.efac[2 * e + 1]]));
            ecoef[i] = make_double2(M.efsign[2 * e] * h0, M.efsign[2 * e + 1] * h1);
            einst[i] = k;
        }
        // d^0 = [*eps] e^0 over all edges
        for (int e = 0; e < M.ne; ++e) {
            double s = 0.0;
            for (long long q = M.h_rp[e]; q < M.h_rp[e + 1]; ++q) s += M.h_v[q] * e0[eo + M.einv[M.h_ci[q]]];
            d0[eo + M.einv[e]] = s;
        }
        // rows in stored edge order, a row's entries in the caller's (the order of its sum)
        std::vector<int> fidx(M.ne, -1);
        for (size_t a = 0; a < M.free_edges.size(); ++a) fidx[M.free_edges[a]] = (int)a;
        for (int i = 0; i < M.ne; ++i) {
            const int a = fidx[M.eperm[i]];
            if (a < 0) continue;
            mrow.push_back(eo + i);
            for (long long q = M.m_rp[a]; q < M.m_rp[a + 1]; ++q) {
                mci.push_back(eo + M.einv[M.m_ci[q]]);
                mv.push_back(I.dt * M.m_v[q]);
            }
            mrp.push_back((long long)mci.size());
        }
    }
    // periodic walls: shift codes of every (triangle, local edge) and the period of each instance
    bool any_periodic = false;
    for (int k = 0; k < n_inst; ++k) any_periodic = any_periodic || ctx->mesh[k].periodic;
    std::vector<signed char> tsh(any_periodic ? 3 * (size_t)ctx->F : 0, 0);
    std::vector<double2> per(any_periodic ? n_inst : 0);
    if (any_periodic)
        for (int k = 0; k < n_inst; ++k) {
            const HostMesh &M = ctx->mesh[k];
            per[k] = make_double2(M.tx, M.ty);
            if (M.periodic)
                std::copy(M.tshift.begin(), M.tshift.end(), tsh.begin() + 3 * (size_t)ctx->cell_off[k]);
        }
    ctx->nfree = (long long)mrow.size();
    const bool f32 = P.precision == FETDPIC_FP32;
    // the field update by patches, unless the cooperative form is asked for, a patch's edges do not fit
    // its block (a dense inverse) or the patches would compute too much twice.  Beyond patch_max
    // triangles the update is bound by memory bandwidth, of which the three kernels need less.  Us a step
    // by patches and without, FP32: 0.98 M triangles 98.6 and 99.3, 1.45 M 138.4 and 140.2 (with 2.9 M
    // particles 181.7 and 184.0), 1.69 M 162.8 and 161.5 (219.4 and 218.3), 2 M 194.7 and 188.4; FP64:
    // 0.64 M 127.1 and 130.1, 0.82 M 153.0 and 152.5, 0.98 M 180.6 and 178.7, 1.69 M 284.8 and 277.4.
    const int patch_max = f32 ? 1550000 : 750000;
    PatchSet ps;
    if (!P.fuse_field_update && P.spai_level >= 0 && ctx->F <= patch_max) {
        std::vector<int> te(3 * (size_t)ctx->F), row(ctx->E, -1);
        for (int f = 0; f < ctx->F; ++f)
            for (int m = 0; m < 3; ++m) te[3 * (size_t)f + m] = tp[f].ew[m] >> 1;
        for (size_t r = 0; r < mrow.size(); ++r) row[mrow[r]] = (int)r;
        try {
            ps = build_patches(PatchInput{ctx->F, te.data(), row.data(), mrp.data(), mci.data(), mv.data()},
                               field_patch_size(ctx->F, ctx->sms));
        } catch (const std::bad_alloc &) {
            return FETDPIC_ENOMEM;
        }
        ctx->patches = ps.ok && field_smem(f32, ps.max_r, ps.max_e) <= FIELD_SMEM_MAX &&
                       patches_pay(ps, ctx->E, (long long)mci.size());
    }
    // else sliced ELL over all rows (32 rows per slice, column-major inside a slice)
    std::vector<long long> soff(1, 0);
    std::vector<int> sci;
    std::vector<double> sv;
    if (!ctx->patches) {
        const long long nr = ctx->nfree;
        for (long long s0 = 0; s0 < nr; s0 += 32) {
            long long wmax = 0;
            for (long long r = s0; r < std::min(nr, s0 + 32); ++r) wmax = std::max(wmax, mrp[r + 1] - mrp[r]);
            const long long base = soff.back();
            sci.resize(base + 32 * wmax);
            sv.resize(base + 32 * wmax);
            for (int l = 0; l < 32; ++l) {
                const long long r = s0 + l;
                const int pad_col = r < nr ? mrow[r] : (nr > 0 ? mrow[0] : 0);
                for (long long k = 0; k < wmax; ++k) {
                    const long long q = base + k * 32 + l;
                    if (r < nr && k < mrp[r + 1] - mrp[r]) { sci[q] = mci[mrp[r] + k]; sv[q] = mv[mrp[r] + k]; }
                    else { sci[q] = pad_col; sv[q] = 0.0; }
                }
            }
            soff.push_back(base + 32 * wmax);
        }
    }
    // the patches' tables one after another, each on a 256-byte boundary
    std::vector<char> tables;
    std::vector<size_t> at;
    if (ctx->patches) {
        auto put = [&](const void *p, size_t bytes) {
            at.push_back((tables.size() + 255) / 256 * 256);
            tables.resize(at.back() + bytes);
            std::memcpy(tables.data() + at.back(), p, bytes);
        };
        tables.reserve(ps.patch.size() * sizeof(FieldPatch) + 4 * ps.xlist.size() + 2 * ps.tloc.size() +
                       2 * ps.row_loc.size() + 2 * ps.col.size() + 8 * ps.soff.size() + 6 * 256);
        put(ps.patch.data(), ps.patch.size() * sizeof(FieldPatch));
        put(ps.xlist.data(), ps.xlist.size() * sizeof(int));
        put(ps.tloc.data(), ps.tloc.size() * sizeof(unsigned short));
        put(ps.row_loc.data(), ps.row_loc.size() * sizeof(unsigned short));
        put(ps.col.data(), ps.col.size() * sizeof(unsigned short));
        put(ps.soff.data(), ps.soff.size() * sizeof(long long));
    }
    const std::vector<double> &mat = ctx->patches ? ps.val : sv;
    std::vector<float> sv32;
    if (f32) sv32.assign(mat.begin(), mat.end());
    // node -> edge incidence (fixed order: ascending edge id per node) and the full [*eps]
    std::vector<int> nrp, nedge, ninst(ctx->N);
    std::vector<long long> hrp(1, 0);
    std::vector<int> hci;
    std::vector<double> hv;
    if (P.check_interval > 0) {
        std::vector<int> deg(ctx->N + 1, 0);
        for (int k = 0; k < n_inst; ++k) {
            const HostMesh &M = ctx->mesh[k];
            for (int e = 0; e < M.ne; ++e) {
                ++deg[ctx->node_off[k] + M.edge[2 * e]];
                ++deg[ctx->node_off[k] + M.edge[2 * e + 1]];
            }
            for (int n = 0; n < M.nn; ++n) ninst[ctx->node_off[k] + n] = k;
        }
        nrp.assign(ctx->N + 1, 0);
        for (int n = 0; n < ctx->N; ++n) nrp[n + 1] = nrp[n] + deg[n];
        nedge.assign(nrp[ctx->N], 0);
        std::vector<int> fill(nrp.begin(), nrp.end() - 1);
        for (int k = 0; k < n_inst; ++k) {
            const HostMesh &M = ctx->mesh[k];
            for (int e = 0; e < M.ne; ++e) {
                const int eg = ctx->edge_off[k] + M.einv[e];
                nedge[fill[ctx->node_off[k] + M.edge[2 * e]]++] = eg << 1;            // leaves the node: +1
                nedge[fill[ctx->node_off[k] + M.edge[2 * e + 1]]++] = (eg << 1) | 1;  // enters the node: -1
            }
        }
        for (int k = 0; k < n_inst; ++k) {
            const HostMesh &M = ctx->mesh[k];
            const int eo = ctx->edge_off[k];
            for (int e : M.eperm) {
                for (long long q = M.h_rp[e]; q < M.h_rp[e + 1]; ++q) { hci.push_back(eo + M.einv[M.h_ci[q]]); hv.push_back(M.h_v[q]); }
                hrp.push_back((long long)hci.size());
            }
        }
    }
    try {
        ctx->geo64 = ctx->alloc<Geo64>(ctx->F);
        if (P.precision == FETDPIC_FP32) {
            ctx->csta = ctx->alloc<CstA>(ctx->F);
            ctx->cstb = ctx->alloc<CstB>(ctx->F);
            ctx->dtinv = ctx->alloc<double2>(ctx->F);
            ctx->rec32 = ctx->alloc<Rec32>(ctx->F);
        } else {
            ctx->rec64 = ctx->alloc<Rec64>(ctx->F);
        }
        ctx->topo = ctx->alloc<Topo>(ctx->F);
        ctx->e = ctx->alloc<double>(ctx->E);
        ctx->b = ctx->alloc<double>(ctx->F);
        ctx->d = ctx->alloc<double>(ctx->E);
        ctx->j = ctx->alloc<double>(ctx->E);
        ctx->ifix = ctx->alloc<unsigned long long>(ctx->E);
        ctx->efac = ctx->alloc<int2>(ctx->E);
        ctx->ecoef = ctx->alloc<double2>(ctx->E);
        ctx->einst = ctx->alloc<int>(ctx->E);
        ctx->inst_unit = ctx->alloc<double>(n_inst);
        ctx->inst_dt = ctx->alloc<double>(n_inst);
        ctx->edge_off_dev = ctx->alloc<int>(n_inst + 1);
        if (any_periodic) {
            ctx->tshift = ctx->alloc<signed char>(3 * (size_t)ctx->F);
            ctx->period = ctx->alloc<double2>(n_inst);
        }
        ctx->tri_c2i = ctx->alloc<int>(ctx->F);
        ctx->tri_i2c = ctx->alloc<int>(ctx->F);
        ctx->edge_c2i = ctx->alloc<int>(ctx->E);
        size_t most = 0;
        for (const HostMesh &M : ctx->mesh) most = std::max(most, 2 * (size_t)M.ne + M.nf);
        ctx->field_out = ctx->alloc<double>(most);
        ctx->ext_dev = ctx->alloc<ExtField>(n_inst);
        ctx->ext_amp = ctx->alloc<double>(n_inst);
        if (P.precision == FETDPIC_FP32) ctx->face_inst = ctx->alloc<int>(ctx->F);
        if (f32) ctx->m_v32 = ctx->alloc<float>(mat.size());
        else ctx->m_v = ctx->alloc<double>(mat.size());
        if (ctx->patches) {
            FieldArgs &A = ctx->field;
            // the tables in one piece, the second buffers in another (cleared: PEC edges are 0 in both)
            char *tab = ctx->alloc<char>(tables.size());
            A.patch = (const FieldPatch *)(tab + at[0]);
            A.xlist = (const int *)(tab + at[1]);
            A.tloc = (const ushort4 *)(tab + at[2]);
            A.row_loc = (const unsigned short *)(tab + at[3]);
            A.col = (const unsigned *)(tab + at[4]);
            A.soff = (const long long *)(tab + at[5]);
            const size_t be = ((size_t)ctx->E * 8 + 255) / 256 * 256, bf = ((size_t)ctx->F * 8 + 255) / 256 * 256;
            char *alt = ctx->alloc<char>(2 * be + bf);
            CK(cudaMemsetAsync(alt, 0, 2 * be + bf, ctx->stream));
            ctx->e_alt = (double *)alt;
            ctx->ifix_alt = (unsigned long long *)(alt + be);
            ctx->b_alt = (double *)(alt + 2 * be);
            A.npatch = (int)ps.patch.size();
            A.max_r = ps.max_r; A.max_e = ps.max_e; A.T = ps.T;
            CK(field_setup(field_smem(f32, ps.max_r, ps.max_e)));
        } else {
            ctx->m_soff = ctx->alloc<long long>(soff.size());
            ctx->m_row = ctx->alloc<int>(mrow.size());
            ctx->m_ci = ctx->alloc<int>(sci.size());
            ctx->r = ctx->alloc<double>(ctx->E);
            CK(cudaMemsetAsync(ctx->r, 0, sizeof(double) * ctx->E, ctx->stream));
            if (f32) {
                ctx->r32 = ctx->alloc<float>(ctx->E);
                CK(cudaMemsetAsync(ctx->r32, 0, sizeof(float) * ctx->E, ctx->stream));     // read by the SPAI product
            }
        }
        ctx->e_a = ctx->e;
        ctx->status = ctx->alloc<unsigned>(1);
        ctx->gbar = ctx->alloc<unsigned>(GBAR_WORDS);
        if (ctx->gbar) CK(cudaMemsetAsync(ctx->gbar, 0, sizeof(unsigned) * GBAR_WORDS, ctx->stream));
        if (P.check_interval > 0) {
            ctx->nrp = ctx->alloc<int>(nrp.size());
            ctx->nedge = ctx->alloc<int>(nedge.size());
            ctx->ninst = ctx->alloc<int>(ninst.size());
            ctx->q0 = ctx->alloc<unsigned long long>(ctx->N);
            ctx->q1 = ctx->alloc<unsigned long long>(ctx->N);
            ctx->g0 = ctx->alloc<double>(ctx->N);
            ctx->qunit = ctx->alloc<double>(n_inst);
            ctx->chk_out = ctx->alloc<double>(3 * (size_t)n_inst);
            ctx->eng_part = ctx->alloc<double>((size_t)check_blocks(ctx->N, ctx->E, ctx->F) * n_inst);
            ctx->chk_ticket = ctx->alloc<unsigned>(1);
            ctx->h_rp = ctx->alloc<long long>(hrp.size());
            ctx->h_ci = ctx->alloc<int>(hci.size());
            ctx->h_v = ctx->alloc<double>(hv.size());
        }
    } catch (const std::bad_alloc &) {
        return FETDPIC_ENOMEM;
    }
    int rc = FETDPIC_OK;
    if (P.check_interval > 0) {
        rc = rc ? rc : upload(ctx, ctx->nrp, nrp.data(), nrp.size());
        rc = rc ? rc : upload(ctx, ctx->nedge, nedge.data(), nedge.size());
        rc = rc ? rc : upload(ctx, ctx->ninst, ninst.data(), ninst.size());
        rc = rc ? rc : upload(ctx, ctx->h_rp, hrp.data(), hrp.size());
        rc = rc ? rc : upload(ctx, ctx->h_ci, hci.data(), hci.size());
        rc = rc ? rc : upload(ctx, ctx->h_v, hv.data(), hv.size());
        if (rc) return rc;
        CK(cudaMemsetAsync(ctx->chk_out, 0, sizeof(double) * 3 * n_inst, ctx->stream));
        CK(cudaMemsetAsync(ctx->chk_ticket, 0, sizeof(unsigned), ctx->stream));
    }
    rc = rc ? rc : upload(ctx, ctx->geo64, g64.data(), g64.size());
    if (!g32.empty()) rc = rc ? rc : upload(ctx, ctx->csta, g32.data(), g32.size());
    if (!g32b.empty()) rc = rc ? rc : upload(ctx, ctx->cstb, g32b.data(), g32b.size());
    if (!dti.empty()) rc = rc ? rc : upload(ctx, ctx->dtinv, dti.data(), dti.size());
    rc = rc ? rc : upload(ctx, ctx->topo, tp.data(), tp.size());
    rc = rc ? rc : upload(ctx, ctx->e, e0.data(), e0.size());
    rc = rc ? rc : upload(ctx, ctx->b, b0.data(), b0.size());
    rc = rc ? rc : upload(ctx, ctx->d, d0.data(), d0.size());
    rc = rc ? rc : upload(ctx, ctx->efac, efac.data(), efac.size());
    rc = rc ? rc : upload(ctx, ctx->ecoef, ecoef.data(), ecoef.size());
    rc = rc ? rc : upload(ctx, ctx->einst, einst.data(), einst.size());
    rc = rc ? rc : upload(ctx, ctx->inst_dt, idt.data(), idt.size());
    rc = rc ? rc : upload(ctx, ctx->edge_off_dev, ctx->edge_off.data(), ctx->edge_off.size());
    if (any_periodic) {
        rc = rc ? rc : upload(ctx, ctx->tshift, tsh.data(), tsh.size());
        rc = rc ? rc : upload(ctx, ctx->period, per.data(), per.size());
    }
    {
        std::vector<ExtField> ex(n_inst);
        std::vector<double> amp(n_inst, 1.0);
        for (int k = 0; k < n_inst; ++k) {
            ex[k] = ExtField{inst[k].ext_ex, inst[k].ext_ey, inst[k].ext_bz, 0.0};
            ctx->ext_on = ctx->ext_on || inst[k].ext_ex != 0.0 || inst[k].ext_ey != 0.0 || inst[k].ext_bz != 0.0;
        }
        rc = rc ? rc : upload(ctx, ctx->ext_dev, ex.data(), ex.size());
        rc = rc ? rc : upload(ctx, ctx->ext_amp, amp.data(), amp.size());
        if (ctx->face_inst) {
            std::vector<int> fi(ctx->F);
            for (int k = 0; k < n_inst; ++k)
                for (int f = ctx->cell_off[k]; f < ctx->cell_off[k + 1]; ++f) fi[f] = k;
            rc = rc ? rc : upload(ctx, ctx->face_inst, fi.data(), fi.size());
        }
    }
    {
        std::vector<int> c2i(ctx->F), i2c(ctx->F), ec2i(ctx->E);
        for (int k = 0; k < n_inst; ++k) {
            const HostMesh &M = ctx->mesh[k];
            for (int f = 0; f < M.nf; ++f) {
                c2i[ctx->cell_off[k] + f] = M.inv[f];
                i2c[ctx->cell_off[k] + f] = M.perm[f];
            }
            std::copy(M.einv.begin(), M.einv.end(), ec2i.begin() + ctx->edge_off[k]);
        }
        rc = rc ? rc : upload(ctx, ctx->tri_c2i, c2i.data(), c2i.size());
        rc = rc ? rc : upload(ctx, ctx->tri_i2c, i2c.data(), i2c.size());
        rc = rc ? rc : upload(ctx, ctx->edge_c2i, ec2i.data(), ec2i.size());
    }
    if (ctx->patches) {
        rc = rc ? rc : upload(ctx, (char *)ctx->field.patch, tables.data(), tables.size());
    } else {
        rc = rc ? rc : upload(ctx, ctx->m_soff, soff.data(), soff.size());
        ctx->m_entries = soff.back();
        rc = rc ? rc : upload(ctx, ctx->m_row, mrow.data(), mrow.size());
        rc = rc ? rc : upload(ctx, ctx->m_ci, sci.data(), sci.size());
    }
    if (f32) rc = rc ? rc : upload(ctx, ctx->m_v32, sv32.data(), sv32.size());
    else rc = rc ? rc : upload(ctx, ctx->m_v, mat.data(), mat.size());
    if (rc) return rc;
    CK(cudaMemsetAsync(ctx->ifix, 0, sizeof(unsigned long long) * ctx->E, ctx->stream));
    CK(cudaMemsetAsync(ctx->j, 0, sizeof(double) * ctx->E, ctx->stream));
    CK(cudaMemsetAsync(ctx->status, 0, sizeof(unsigned), ctx->stream));
    ctx->unit_host.assign(n_inst, 0.0);
    ctx->fixscale.assign(n_inst, 1.0);
    ctx->qunit_host.assign(n_inst, 0.0);
    CK(cudaStreamSynchronize(ctx->stream));
    *out = holder.release();
    return FETDPIC_OK;
}

extern "C" int fetdpic_load_particles(fetdpic_ctx *ctx, int inst, double q, double m, long long n,
                                      const double *x, const double *u, const int *cell_hint)
{
    if (!ctx) return FETDPIC_EINVAL;
    if (ctx->finalized) return ctx->fail(FETDPIC_ESTATE, "particles must be loaded before the first step");
    if (inst < 0 || inst >= (int)ctx->mesh.size() || n < 0 || (n > 0 && (!x || !u)) || !(m > 0))
        return ctx->fail(FETDPIC_EINVAL, "bad load arguments");
    if (ctx->staged.size() >= 32767) return ctx->fail(FETDPIC_EINVAL, "too many species");
    const HostMesh &M = ctx->mesh[inst];
    StagedSpecies s;
    s.inst = inst; s.q = q; s.m = m;
    s.cell.resize(n); s.x.resize(n); s.y.resize(n); s.ux.resize(n); s.uy.resize(n);
    for (long long k = 0; k < n; ++k) {
        const int c = host_locate(M, x[2 * k], x[2 * k + 1], cell_hint ? cell_hint[k] : -1);
        if (c < 0) return ctx->fail(FETDPIC_EOUTSIDE, "particle " + std::to_string(k) + " lies in no triangle");
        if (!std::isfinite(u[2 * k]) || !std::isfinite(u[2 * k + 1]))
            return ctx->fail(FETDPIC_ENONFINITE, "non-finite momentum at load");
        s.cell[k] = c;
        s.x[k] = x[2 * k]; s.y[k] = x[2 * k + 1];
        s.ux[k] = u[2 * k]; s.uy[k] = u[2 * k + 1];
    }
    ctx->staged.push_back(std::move(s));
    return (int)ctx->staged.size() - 1;
}

// Charge of the current particle state into q (fixed point).
static void charge_now(fetdpic_ctx *ctx, unsigned long long *q, bool clean = false, bool pdl = false)
{
    launch_charge(ctx->stream, ctx->p.precision == FETDPIC_FP32, ctx->P, ctx->cell, ctx->chunk_sp, ctx->sp_dev,
                  ctx->geo64, ctx->topo, ctx->f[0], ctx->f[1], q, ctx->N, clean, pdl);
}

// The Gauss-law check compares S~ d - q with its value at this point (after
// load, or after a state is written from the host).
static void reset_gauss_reference(fetdpic_ctx *ctx)
{
    if (!ctx->g0 || !ctx->finalized) { ctx->q_prev_valid = false; return; }
    charge_now(ctx, ctx->q0);
    launch_gauss_reference(ctx->stream, ctx->N, ctx->nrp, ctx->nedge, ctx->ninst, ctx->qunit, ctx->d, ctx->q0, ctx->g0);
    // after the electrostatic solve the reference is zero off the PEC walls: S~ d^n = q^n itself is
    // checked there; on wall nodes S~ d - q is the conductor's induced charge and stays relative
    for (size_t k = 0; k < ctx->gauss_abs.size(); ++k) {
        if (!ctx->gauss_abs[k]) continue;
        const int nn = ctx->mesh[k].nn;
        std::vector<double> g(nn);
        if (cudaMemcpyAsync(g.data(), ctx->g0 + ctx->node_off[k], sizeof(double) * nn, cudaMemcpyDeviceToHost,
                            ctx->stream) != cudaSuccess || cudaStreamSynchronize(ctx->stream) != cudaSuccess)
            continue;
        for (int n = 0; n < nn; ++n) if (ctx->abs_nodes[k][n]) g[n] = 0.0;
        cudaMemcpyAsync(ctx->g0 + ctx->node_off[k], g.data(), sizeof(double) * nn, cudaMemcpyHostToDevice, ctx->stream);
        cudaStreamSynchronize(ctx->stream);
    }
    ctx->q_prev_valid = true;
    ctx->g0_ready = true;
}

// Whether the FP64 particle kernel may form products and quotients with `v` in
// integer arithmetic (fp64_int.h): zero, or a magnitude that leaves chains of
// them normal.
static bool soft_constant(double v)
{
    const double m = std::fabs(v);
    return (m == 0.0) | ((m >= 0x1p-100) & (m < 0x1p64));
}

// Move the staged species to the device: padded species ranges, block ->
// species table, fixed-point scale of the current per instance.
static int finalize(fetdpic_ctx *ctx)
{
    if (ctx->finalized) return FETDPIC_OK;
    const auto &P = ctx->p;
    const int ni = (int)ctx->mesh.size();
    const int ns = (int)ctx->staged.size();
    // q_ref and the fixed-point shift per instance: the largest per-triangle
    // charge weight sets the head room (x16 for clumping, crossings and the
    // two triangles of an edge); shift <= 52 keeps the quantum at FP64 epsilon
    // of one unit contribution.
    std::vector<double> qref(ni, 0.0);
    for (auto &s : ctx->staged) qref[s.inst] = std::max(qref[s.inst], std::fabs(s.q));
    std::vector<std::vector<double>> wcell(ni);
    for (int k = 0; k < ni; ++k) wcell[k].assign(ctx->mesh[k].nf, 0.0);
    for (auto &s : ctx->staged) {
        const double w = qref[s.inst] > 0 ? std::fabs(s.q) / qref[s.inst] : 0.0;
        for (int c : s.cell) wcell[s.inst][c] += w;
    }
    for (int k = 0; k < ni; ++k) {
        double wmax = 1.0;
        for (double w : wcell[k]) wmax = std::max(wmax, w);
        int sh = 62 - (int)std::ceil(std::log2(16.0 * wmax + 1.0));
        sh = std::max(20, std::min(52, sh));
        // FP32 path: per-particle contributions are summed across a warp in 32-bit integers
        ctx->fixscale[k] = P.precision == FETDPIC_FP32 ? FP32_SCALE : std::ldexp(1.0, sh);
        const double qr = qref[k] > 0 ? qref[k] : 1.0;
        ctx->unit_host[k] = (qr / ctx->inst[k].dt) / ctx->fixscale[k];
        ctx->qunit_host[k] = qr / ctx->fixscale[k];
    }
    ctx->sp.resize(ns);
    long long off = 0, hist_n = 0;
    std::vector<int> hoff(ns);
    for (int s = 0; s < ns; ++s) {
        const StagedSpecies &S = ctx->staged[s];
        Species &D = ctx->sp[s];
        std::memset(&D, 0, sizeof(D));
        const fetdpic_instance &I = ctx->inst[S.inst];
        const double dt = I.dt;
        D.alpha = S.q * dt / (2.0 * S.m);
        const double qr = qref[S.inst] > 0 ? qref[S.inst] : 1.0;
        D.wfix = (S.q / qr) * ctx->fixscale[S.inst];
        // (below 1e-250 of a unit every particle's charge rounds to 0; k_charge32's integer product needs the
        // factor to leave it in range)
        D.qfix = std::fabs(D.wfix) < 1e-250 ? 0.0 : D.wfix;
        D.wfix32 = (float)D.wfix;
        D.dt = dt; D.c = P.c; D.ic2 = 1.0 / (P.c * P.c);
        D.ext_ex = I.ext_ex; D.ext_ey = I.ext_ey; D.ext_bz = I.ext_bz;
        D.kappa = (float)(S.q / S.m);
        D.xe_x = (float)(S.q / S.m * dt / (2.0 * P.c) * I.ext_ex);
        D.xe_y = (float)(S.q / S.m * dt / (2.0 * P.c) * I.ext_ey);
        D.xb = (float)(S.q / S.m * dt / 2.0 * I.ext_bz);
        D.inst = S.inst;
        D.n = (long long)S.cell.size();
        D.cap = ((D.n + SPECIES_ALIGN - 1) / SPECIES_ALIGN) * SPECIES_ALIGN;
        D.off = off;
        D.cell_off = ctx->cell_off[S.inst];
        D.nf = ctx->mesh[S.inst].nf;
        hoff[s] = (int)hist_n;
        hist_n += D.nf + 1;                  // the species' triangles, then its padding bin
        off += D.cap;
    }
    {
        std::vector<double> n(ni, 0.0);
        for (const Species &D : ctx->sp) n[D.inst] += (double)D.n;
        double all = 0.0, sum = 0.0;
        for (int k = 0; k < ni; ++k) { all += n[k]; sum += n[k] * (n[k] / ctx->mesh[k].nf); }
        ctx->density = all > 0.0 ? sum / all : 0.0;
    }
    if (P.precision == FETDPIC_FP64) {           // the FP32 path does not ask
        bool soft = true;
        for (const Species &D : ctx->sp)
            soft = soft && soft_constant(D.alpha) && soft_constant(D.ic2) && soft_constant(D.dt) && soft_constant(D.wfix);
        for (const HostMesh &M : ctx->mesh)
            for (const std::vector<double> *g : {&M.gx, &M.gy, &M.X, &M.Y})
                for (const double v : *g) soft &= soft_constant(v);
        ctx->soft64 = soft;
    }
    ctx->P = off;
    ctx->nblocks = off / ctx->block;
    if (off >= (1ll << 31))      // particle slots and load indices are 32-bit
        return ctx->fail(FETDPIC_EINVAL, "more than 2^31 - 1 particle slots (species padded to 1024)");
    ctx->hist_n = hist_n;
    const bool f32 = P.precision == FETDPIC_FP32;
    const size_t fb = f32 ? 4 : 8;
    std::vector<Sp32> s32(std::max(ns, 1));
    for (int s = 0; s < ns; ++s) {
        const Species &D = ctx->sp[s];
        Sp32 &T = s32[s];
        // the FP32 path takes the applied fields from the per-triangle field record
        T = Sp32{};
        T.kappa = D.kappa;
        T.wfix = (float)D.wfix;
        T.inst = D.inst; T.edge_off = ctx->edge_off[D.inst]; T.off = (int)D.off;
    }
    try {
        ctx->sp32_dev = ctx->alloc<Sp32>(s32.size());
        ctx->sp_dev = ctx->alloc<Species>(std::max(ns, 1));
        ctx->cell = ctx->alloc<int>(ctx->P);
        ctx->cell_a = ctx->cell;
        ctx->cell_tmp = ctx->alloc<int>(ctx->P);
        ctx->id = ctx->alloc<int>(ctx->P);
        ctx->id_tmp = ctx->alloc<int>(ctx->P);
        for (int k = 0; k < 4; ++k) {
            ctx->f[k] = ctx->alloc<char>(fb * ctx->P);
            ctx->f_tmp[k] = ctx->alloc<char>(fb * ctx->P);
        }
        ctx->chunk_sp = ctx->alloc<short>(std::max<long long>(ctx->P / 32, 1));
        ctx->hist = ctx->alloc<int>(std::max<long long>(hist_n, 1));
        ctx->hoff = ctx->alloc<int>(std::max(ns, 1));
        ctx->scan_tmp = ctx->alloc<int>(scan_tmp_ints(std::max<long long>(hist_n, 1)));
        if (P.record_walk > 0) {
            ctx->rec_cnt = ctx->alloc<int>(ctx->P);
            ctx->rec = ctx->alloc<int>((size_t)ctx->P * P.record_walk);
        }
    } catch (const std::bad_alloc &) {
        return FETDPIC_ENOMEM;
    }
    // host images
    std::vector<int> cell(ctx->P, -1), id(ctx->P, -1);       // padding: no triangle, no load index
    std::vector<char> fh[4];
    for (int k = 0; k < 4; ++k) fh[k].assign(fb * ctx->P, 0);
    std::vector<short> chk(ctx->P / 32);
    for (int s = 0; s < ns; ++s) {
        const StagedSpecies &S = ctx->staged[s];
        const Species &D = ctx->sp[s];
        const HostMesh &M = ctx->mesh[S.inst];
        for (long long b = D.off / 32; b < (D.off + D.cap) / 32; ++b) chk[b] = (short)s;
        // storage in stored-triangle order from the start (a counting sort; load order in id)
        std::vector<long long> start(M.nf + 1, 0), order(D.n);
        for (long long k = 0; k < D.n; ++k) ++start[S.cell[k] + 1];
        for (int f = 0; f < M.nf; ++f) start[f + 1] += start[f];
        for (long long k = 0; k < D.n; ++k) order[start[S.cell[k]]++] = k;
        for (long long r = 0; r < D.n; ++r) {
            const long long k = order[r];
            const long long q = D.off + r;
            cell[q] = D.cell_off + S.cell[k];
            id[q] = (int)k;
            if (f32) {
                double l[3];
                host_lambdas(M, S.cell[k], S.x[k], S.y[k], l);
                ((float *)fh[0].data())[q] = (float)l[0];
                ((float *)fh[1].data())[q] = (float)l[1];
                ((float *)fh[2].data())[q] = (float)(S.ux[k] / P.c);
                ((float *)fh[3].data())[q] = (float)(S.uy[k] / P.c);
            } else {
                ((double *)fh[0].data())[q] = S.x[k];
                ((double *)fh[1].data())[q] = S.y[k];
                ((double *)fh[2].data())[q] = S.ux[k];
                ((double *)fh[3].data())[q] = S.uy[k];
            }
        }
    }
    int rc = FETDPIC_OK;
    rc = rc ? rc : upload(ctx, ctx->sp_dev, ctx->sp.data(), ctx->sp.size());
    rc = rc ? rc : upload(ctx, ctx->sp32_dev, s32.data(), s32.size());
    rc = rc ? rc : upload(ctx, ctx->cell, cell.data(), cell.size());
    rc = rc ? rc : upload(ctx, ctx->cell_tmp, cell.data(), cell.size());   // padding stays -1 in both buffers
    rc = rc ? rc : upload(ctx, ctx->id, id.data(), id.size());
    for (int k = 0; k < 4; ++k) rc = rc ? rc : upload(ctx, (char *)ctx->f[k], fh[k].data(), fh[k].size());
    rc = rc ? rc : upload(ctx, ctx->chunk_sp, chk.data(), chk.size());
    rc = rc ? rc : upload(ctx, ctx->hoff, hoff.data(), hoff.size());
    rc = rc ? rc : upload(ctx, ctx->inst_unit, ctx->unit_host.data(), ctx->unit_host.size());
    if (ctx->qunit) {
        rc = rc ? rc : upload(ctx, ctx->qunit, ctx->qunit_host.data(), ctx->qunit_host.size());
    }
    if (rc) return rc;
    if (ctx->rec_cnt) CK(cudaMemsetAsync(ctx->rec_cnt, 0, sizeof(int) * ctx->P, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    ctx->finalized = true;
    reset_gauss_reference(ctx);
    CK(cudaStreamSynchronize(ctx->stream));
    return FETDPIC_OK;
}

// Polls per bounded wait inside a kernel: 0 = 2^20; negative = none (the wait gives up at once).
static unsigned wait_polls(const fetdpic_ctx *ctx)
{
    const long long lim = ctx->p.wait_spin_limit;
    return lim > 0 ? (unsigned)std::min<long long>(lim, 1ll << 30) : (lim < 0 ? 0u : (1u << 20));
}

static StepArgs64 args64(fetdpic_ctx *ctx)
{
    StepArgs64 a{};
    a.geo = ctx->geo64; a.topo = ctx->topo; a.rec = ctx->rec64;
    a.sp = ctx->sp_dev; a.chunk_sp = ctx->chunk_sp; a.nchunks = ctx->P / 32;
    a.soft = ctx->soft64; a.ext_on = ctx->ext_on;
    a.x = (double *)ctx->f[0]; a.y = (double *)ctx->f[1]; a.ux = (double *)ctx->f[2]; a.uy = (double *)ctx->f[3];
    a.cell = ctx->cell;
    a.ifix = ctx->ifix; a.status = ctx->status;
    a.max_cross = ctx->p.max_crossings;
    a.rec_cap = ctx->p.record_walk; a.rec_cnt = ctx->rec_cnt; a.wrec = ctx->rec; a.id = ctx->id;
    a.edge_off = ctx->edge_off_dev;
    a.block = ctx->block;
    a.tshift = ctx->tshift; a.period = ctx->period;
    a.extw = ctx->extw; a.ext_amp = ctx->ext_amp;
    return a;
}

// Hybrid FP32 variants: (variant, early kernel variant, late kernel variant,
// steps after a sort that run the early one).  While runs of equal triangle
// are long (just after a sort) the early kernel runs; once the particles have
// drifted, the late one with the deposit window.  All variants give identical
// results.
struct Hybrid { int v, early, late, steps; };
static constexpr Hybrid HYBRIDS[] = {{17, 12, 14, 6}, {18, 12, 14, 4}, {21, 19, 14, 6}, {22, 19, 20, 6}};

// The FP32 kernels a context runs, by its variant; one kernel throughout where early and late agree.
// Variant 0, nothing chosen by the caller (device us a step, a sort every 16 steps):
//   - up to one 64-particle chunk per SM: the kernel with one particle per lane is through it soonest
//     (64 particles: 6.15 against 6.7 with variant 22; 4,000: 7.0 against 7.6; with two chunks per
//     SM variant 12 is ahead, 8.72 against 8.93);
//   - fewer than twenty particles per triangle: runs are short and the window's flush does not pay.
//     Variant 12 against window kernels (Vay): 8,192 triangles, 4 to 30 a triangle, 1.5 to 6 % ahead
//     throughout; 20,000 2 to 12 % ahead but at 12 and 24 a triangle (2 to 3 % behind); 51,200, 4 a
//     triangle 14.3 and 15.8, 8 16.5 and 17.9, 10 18.6 and 18.0, 12 18.8 and 20.1, 14 21.0 and 20.2, 16 21.5
//     and 22.5, 20 23.8 and 24.0; 180,000, 10 a triangle 42.2 and 43.8, 16 57.2 and 57.4, 20 65.8 and 66.6;
//     201k, 40 a triangle 131.6 and 128.9.  Counted where the particles are, since a batch may be uneven
//     (16 instances with 2 to 96 per triangle, 6.8 in all but 30 around the mean particle: 53.9 with the
//     window kernels, 56.6 without);
//   - else an early and a late kernel.  Early, 28 warps per SM for the Vay pusher, 24 for the others, whose
//     28-warp kernels spill: 6.25 M particles above gamma = 10 161.6 against 168.7 (Higuera-Cary) and 152.6
//     against 159.3 (Boris), 8 M thermal ones 130.9 against 129.9 and 129.4 against 128.3.  Late, the 20-warp
//     window kernel up to 2 M particles (1.1 M in 16 instances: 53.8 against 55.6), the 24-warp one above:
//     they are within 1.3 % of one another from 0.8 to 3.9 M, 5.8 M take 89.2 with the 24-warp one and 109.8
//     with the other.
static Hybrid kernels_of(const fetdpic_ctx *ctx, int pusher)
{
    const int v = ctx->p.kernel_variant;
    for (const Hybrid &h : HYBRIDS)
        if (h.v == v) return h;
    if (v != 0) return Hybrid{v, v, v, 0};
    const long long n64 = ctx->P / 64;
    if (n64 <= ctx->sms) return Hybrid{0, 4, 4, 0};
    if (ctx->density < 20.0) return Hybrid{0, 12, 12, 0};
    return Hybrid{0, pusher == FETDPIC_VAY ? 19 : 12, n64 < 32768 ? 14 : 20, 6};
}

// Whether the coming step runs the late kernel.
static bool late_step(const fetdpic_ctx *ctx, const Hybrid &h)
{
    const long long since = ctx->p.sort_interval > 0 ? ctx->steps_done % ctx->p.sort_interval : ctx->steps_done;
    return since >= h.steps;
}

static StepArgs32 args32(fetdpic_ctx *ctx, int pusher)
{
    StepArgs32 a{};
    const Hybrid h = kernels_of(ctx, pusher);
    a.csta = ctx->csta; a.cstb = ctx->cstb; a.rec = ctx->rec32;
    a.sp = ctx->sp32_dev; a.chunk_sp = ctx->chunk_sp; a.nchunks = ctx->P / 32;
    a.variant = late_step(ctx, h) ? h.late : h.early;
    a.l0 = (float *)ctx->f[0]; a.l1 = (float *)ctx->f[1]; a.ux = (float *)ctx->f[2]; a.uy = (float *)ctx->f[3];
    a.cell = ctx->cell;
    a.ifix = ctx->ifix; a.status = ctx->status;
    a.max_cross = ctx->p.max_crossings;
    a.rec_cap = ctx->p.record_walk; a.rec_cnt = ctx->rec_cnt; a.wrec = ctx->rec; a.id = ctx->id;
    a.edge_off = ctx->edge_off_dev;
    a.nblocks = ctx->nblocks; a.block = ctx->block;
    a.spin = wait_polls(ctx);
    return a;
}

static void mark(fetdpic_ctx *ctx, int stage)
{
    if (ctx->ev_used == (int)ctx->ev.size()) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) return;
        ctx->ev.push_back(e);
        ctx->ev_stage.push_back(0);
    }
    cudaEventRecord(ctx->ev[ctx->ev_used], ctx->stream);
    ctx->ev_stage[ctx->ev_used] = stage;
    ++ctx->ev_used;
}

// Fold the recorded events into the per-stage sums (stream must be idle).
static void collect_events(fetdpic_ctx *ctx)
{
    for (int k = 1; k < ctx->ev_used; ++k) {
        const int sg = ctx->ev_stage[k];
        if (sg < 0) continue;
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, ctx->ev[k - 1], ctx->ev[k]) == cudaSuccess) {
            if (sg == 3) { ctx->stage_ms[2] += ms; ctx->stage_ms[3] += 1.0; }
            else if (sg < 6) ctx->stage_ms[sg] += ms;
        }
    }
    ctx->ev_used = 0;
}

static void swap_particles(fetdpic_ctx *ctx)
{
    std::swap(ctx->cell, ctx->cell_tmp);
    std::swap(ctx->id, ctx->id_tmp);
    for (int k = 0; k < 4; ++k) std::swap(ctx->f[k], ctx->f_tmp[k]);
}

// Up to this many slots are not sorted: no result depends on the order, a few warps gain nothing from it,
// and its four launches and their join take 0.6 us of a step (us a step with a sort every 16 and without,
// 2,048 triangles: 64 particles 6.07 and 5.50, 1,024 6.87 and 6.28, 2,048 7.06 and 6.41).  At 4,096 particles
// the two are even (7.26 and 7.19); at 8,192 scattered ones lose (7.33 and 8.66).
constexpr long long SORT_MIN_SLOTS = 2048;

// Whether step `step` (from 1) ends with a sort.
static bool sorts_at(const fetdpic_ctx *ctx, long long step)
{
    return ctx->p.sort_interval > 0 && ctx->P > SORT_MIN_SLOTS && step % ctx->p.sort_interval == 0;
}

static void do_sort(fetdpic_ctx *ctx, cudaStream_t st)
{
    SortArgs s{};
    s.nsp = (int)ctx->sp.size(); s.sp_dev = ctx->sp_dev; s.sp_host = ctx->sp.data();
    s.P = ctx->P;
    s.cell = ctx->cell; s.cell_tmp = ctx->cell_tmp; s.id = ctx->id; s.id_tmp = ctx->id_tmp;
    for (int k = 0; k < 4; ++k) { s.f[k] = ctx->f[k]; s.f_tmp[k] = ctx->f_tmp[k]; }
    s.fbytes = ctx->p.precision == FETDPIC_FP32 ? 4 : 8;
    s.hist = ctx->hist; s.hoff = ctx->hoff; s.hist_n = ctx->hist_n; s.scan_tmp = ctx->scan_tmp;
    s.chunk_sp = ctx->chunk_sp;
    launch_sort(st, s);
    swap_particles(ctx);
}

// The buffers of e, b and the current accumulator change places (a field update
// that carried the next step's Faraday).
static void swap_fields(fetdpic_ctx *ctx)
{
    std::swap(ctx->e, ctx->e_alt);
    std::swap(ctx->b, ctx->b_alt);
    std::swap(ctx->ifix, ctx->ifix_alt);
}

// Whether a step computes the conservation checks.
static bool checks_at(const fetdpic_ctx *ctx, long long step)
{
    return ctx->p.check_interval > 0 && ctx->g0 && step % ctx->p.check_interval == 0;
}
// Whether the step that `after` more steps follow may share its field update with
// the next: Ampere's of one step with Faraday's of the next (not with stage events,
// whose stages are separate).
static bool can_merge(const fetdpic_ctx *ctx, long long after)
{
    return after > 0 && ctx->patches && ctx->p.time_stages == 0;
}

// One time step: Faraday (+ field record), particles, Ampere, periodic sort.
// `timed`: record stage events (time_stages = 1).  `begun`: the previous step's
// field update carried this step's Faraday; `more`: this step's carries the next's.
static long long enqueue_step(fetdpic_ctx *ctx, int pusher, bool timed, bool begun = false, bool more = false)
{
    long long launches = 0;
    const bool f32 = ctx->p.precision == FETDPIC_FP32;
    const bool check = checks_at(ctx, ctx->steps_done + 1);
    Ext32 x{};
    if (f32 && ctx->ext_on) {
        x.finst = ctx->face_inst; x.ext = ctx->ext_dev; x.amp = ctx->ext_amp; x.extw = ctx->extw;
        x.half_over_c = 0.5 / ctx->p.c;
    }
    AmpereArgs A{};
    A.E = ctx->E; A.efac = ctx->efac; A.ecoef = ctx->ecoef; A.einst = ctx->einst;
    A.inst_unit = ctx->inst_unit; A.inst_dt = ctx->inst_dt; A.b = ctx->b; A.ifix = ctx->ifix;
    // FP32 mode reads r32 only; without checks nothing reads the dual flux d
    A.r = f32 ? nullptr : ctx->r; A.d = ctx->p.check_interval > 0 ? ctx->d : nullptr;
    A.j = ctx->j; A.r32 = ctx->r32;
    A.nfree = ctx->nfree; A.m_soff = ctx->m_soff; A.m_row = ctx->m_row; A.m_ci = ctx->m_ci; A.m_v = ctx->m_v;
    A.m_entries = ctx->m_entries;
    A.m_v32 = ctx->m_v32;
    A.e = ctx->e;
    A.fused = ctx->p.fuse_field_update != 0;
    A.gbar = ctx->gbar; A.spin = wait_polls(ctx); A.status = ctx->status;
    // stage events need each stage to start after the previous one: no early launch when timed
    A.pdl = !timed;
    if (timed) mark(ctx, -1);
    const float inv2c2 = (float)(0.5 / (ctx->p.c * ctx->p.c));
    if (begun) {}
    else if (f32)
        launch_faraday32(ctx->stream, ctx->F, ctx->csta, ctx->cstb, ctx->dtinv, ctx->e, ctx->b, ctx->rec32, inv2c2, x,
                         ctx->E, ctx->ifix, !timed);
    else launch_faraday64(ctx->stream, ctx->F, ctx->geo64, ctx->topo, ctx->e, ctx->b, ctx->rec64, ctx->E, ctx->ifix,
                          !timed);
    launches += ctx->F > 0 && !begun;
    if (timed) mark(ctx, 0);
    if (check && !ctx->q_prev_valid) { charge_now(ctx, ctx->q0, false, !timed); launches += 1; }
    if (ctx->nblocks > 0) {
        if (f32) {
            StepArgs32 a = args32(ctx, pusher);
            a.pdl = !timed;
            launch_particles32(ctx->stream, pusher, a);
        }
        else {
            StepArgs64 a = args64(ctx);
            a.pdl = !timed;
            launch_particles64(ctx->stream, pusher, a);
        }
        ++launches;
    }
    if (timed) mark(ctx, 1);
    if (check) {
        charge_now(ctx, ctx->q1, ctx->q1_clean, !timed);
        ++launches;
    }
    // the sort of this step's end reads only the particle state, which the field update and the
    // checks after the charge do not touch: without stage events it runs on the side stream meanwhile
    // (a check every fourth step, 20k triangles: 37.8 us a step against 39.0 with the sort behind it).
    // The particle kernel reads the sorted state before its own wait, so it has to follow a join by an event.
    const bool sorts = sorts_at(ctx, ctx->steps_done + 1);
    const bool side_sort = sorts && !timed;
    if (side_sort) {
        cudaEventRecord(ctx->ev_fork, ctx->stream);       // errors surface through cudaGetLastError
        cudaStreamWaitEvent(ctx->side, ctx->ev_fork, 0);
        do_sort(ctx, ctx->side);
        launches += 4;
        cudaEventRecord(ctx->ev_join, ctx->side);
    }
    if (ctx->patches) {
        FieldArgs W = ctx->field;
        W.v32 = ctx->m_v32; W.v64 = ctx->m_v;
        W.efac = ctx->efac; W.ecoef = ctx->ecoef; W.einst = ctx->einst;
        W.inst_unit = ctx->inst_unit; W.inst_dt = ctx->inst_dt;
        W.b = ctx->b; W.ifix = ctx->ifix; W.j = ctx->j; W.d = A.d;
        W.e = ctx->e; W.e_next = more ? ctx->e_alt : ctx->e;
        W.one_inst = ctx->mesh.size() == 1;
        W.early = ctx->nblocks > 0;
        W.pdl = !timed;
        W.faraday = more;
        W.b_next = ctx->b_alt; W.ifix_next = ctx->ifix_alt;
        W.csta = ctx->csta; W.cstb = ctx->cstb; W.dtinv = ctx->dtinv; W.rec32 = ctx->rec32; W.inv2c2 = inv2c2; W.ext = x;
        W.geo = ctx->geo64; W.topo = ctx->topo; W.rec64 = ctx->rec64;
        launch_field(ctx->stream, W);
        ++launches;
        if (more) swap_fields(ctx);
    } else {
        launch_ampere(ctx->stream, A);
        launches += A.fused ? (ctx->E > 0 || ctx->nfree > 0) : (ctx->E > 0) + (ctx->nfree > 0);
    }
    if (ctx->probe_n > 0) {
        launch_probe(ctx->stream, ctx->probe_n, ctx->probe_w, ctx->e, ctx->probe_ring, ctx->probe_cap,
                     ctx->probe_count);
        ++launches;
    }
    if (timed) mark(ctx, 3);
    if (check) {
        CheckArgs C{};
        C.N = ctx->N; C.E = ctx->E; C.F = ctx->F; C.ninst_n = (int)ctx->mesh.size();
        C.nrp = ctx->nrp; C.nedge = ctx->nedge; C.ninst = ctx->ninst;
        // after a field update that carried the next Faraday, this step's current and b are in the
        // other buffers (and stay there until the next field update)
        C.ifix = more ? ctx->ifix_alt : ctx->ifix;
        C.b = more ? ctx->b_alt : ctx->b;
        C.q0 = ctx->q0; C.q1 = ctx->q1; C.qunit = ctx->qunit; C.d = ctx->d; C.g0 = ctx->g0;
        C.hrp = ctx->h_rp; C.hci = ctx->h_ci; C.hv = ctx->h_v;
        C.e = ctx->e; C.einst = ctx->einst; C.geo = ctx->geo64; C.topo = ctx->topo;
        C.part = ctx->eng_part; C.out = ctx->chk_out; C.ticket = ctx->chk_ticket;
        launches += launch_checks(ctx->stream, C, !timed);
        ctx->q1_clean = true;                 // q0, cleared, becomes q1
        std::swap(ctx->q0, ctx->q1);          // the charge after this step is the next step's q^n
        ctx->q_prev_valid = true;
        if (timed) mark(ctx, 5);
    } else {
        ctx->q_prev_valid = false;
    }
    ++ctx->steps_done;
    if (side_sort) {
        cudaStreamWaitEvent(ctx->stream, ctx->ev_join, 0);
    } else if (sorts) {
        do_sort(ctx, ctx->stream);
        launches += 4;
        if (timed) mark(ctx, 4);
    }
    return launches;
}

// Ends the capture begun on the context stream and makes `g` of it.  A launch refused meanwhile is not
// in the graph: then nothing is kept, and the error is reported.
static int end_capture(fetdpic_ctx *ctx, cudaGraphExec_t &g)
{
    cudaGraph_t graph = nullptr;
    const cudaError_t refused = cudaGetLastError();
    cudaError_t e = cudaStreamEndCapture(ctx->stream, &graph);
    if (e != cudaSuccess) return ctx->cuda_fail(e, "cudaStreamEndCapture");
    e = refused;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&g, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
        g = nullptr;
        return ctx->cuda_fail(e, refused != cudaSuccess ? "launch during capture" : "cudaGraphInstantiate");
    }
    return FETDPIC_OK;
}

// One step through a captured graph: the launch sequence of a step depends only
// on the pusher, which particle buffer is current and whether the step sorts,
// so each combination is captured once (capture enqueues nothing; the host-side
// bookkeeping of the step happens during capture) and replayed.
static int graph_step(fetdpic_ctx *ctx, int pusher, long long &launches)
{
    const bool sorts = sorts_at(ctx, ctx->steps_done + 1);
    const int parity = ctx->cell == ctx->cell_a ? 0 : 1;
    const int late = ctx->p.precision == FETDPIC_FP32 && late_step(ctx, kernels_of(ctx, pusher)) ? 1 : 0;
    const int fields = ctx->e == ctx->e_a ? 0 : 1;
    cudaGraphExec_t &g = ctx->graph[pusher][parity][sorts ? 1 : 0][late][fields];
    if (!g) {
        CK(cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal));
        const long long n = enqueue_step(ctx, pusher, false);
        const int rc = end_capture(ctx, g);
        if (rc) {                                 // no step was taken
            --ctx->steps_done;
            if (sorts) swap_particles(ctx);
            return rc;
        }
        ctx->graph_launches[pusher][parity][sorts ? 1 : 0][late][fields] = n;
        CK(cudaGraphLaunch(g, ctx->stream));
        launches += n;
        return FETDPIC_OK;
    }
    CK(cudaGraphLaunch(g, ctx->stream));
    launches += ctx->graph_launches[pusher][parity][sorts ? 1 : 0][late][fields];
    // host-side effects of the step the graph replays
    ++ctx->steps_done;
    ctx->q_prev_valid = false;
    if (sorts) swap_particles(ctx);
    return FETDPIC_OK;
}

// A whole sort cycle (sort_interval steps from just after a sort up to and
// including the next one) through one captured graph: inside it every kernel
// may launch early behind the previous one (programmatic dependent launch),
// across step boundaries too, and the cycle is one graph launch.  The graph
// depends on the pusher and on which particle buffer is current at its start.
static int cycle_step(fetdpic_ctx *ctx, int pusher, long long &launches)
{
    const int parity = ctx->cell == ctx->cell_a ? 0 : 1;
    const int L = ctx->p.sort_interval;
    const int fields = ctx->e == ctx->e_a ? 0 : 1;
    const bool merge = can_merge(ctx, L - 1);
    cudaGraphExec_t &g = ctx->cycle[pusher][parity][fields];
    if (!g) {
        CK(cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal));
        long long n = 0;
        for (int k = 0; k < L; ++k) n += enqueue_step(ctx, pusher, false, merge && k > 0, merge && k + 1 < L);
        const int rc = end_capture(ctx, g);
        if (rc) {                                 // no step was taken
            if (merge && ((L - 1) & 1)) swap_fields(ctx);
            if (sorts_at(ctx, ctx->steps_done)) swap_particles(ctx);
            ctx->steps_done -= L;
            return rc;
        }
        ctx->cycle_launches[pusher][parity][fields] = n;
        CK(cudaGraphLaunch(g, ctx->stream));
        launches += n;
        return FETDPIC_OK;
    }
    CK(cudaGraphLaunch(g, ctx->stream));
    launches += ctx->cycle_launches[pusher][parity][fields];
    // host-side effects of the replayed steps: one sort, at the end; L - 1 exchanges of the fields
    if (merge && ((L - 1) & 1)) swap_fields(ctx);
    ctx->steps_done += L;
    ctx->q_prev_valid = false;
    if (sorts_at(ctx, ctx->steps_done)) swap_particles(ctx);
    return FETDPIC_OK;
}

extern "C" int fetdpic_step(fetdpic_ctx *ctx, long long nsteps, int pusher)
{
    if (!ctx) return FETDPIC_EINVAL;
    if (nsteps < 0 || pusher < 0 || pusher > 3) return ctx->fail(FETDPIC_EINVAL, "bad step arguments");
    int rc = finalize(ctx);
    if (rc) return rc;
    CK(cudaSetDevice(ctx->device));
    // keep the event pool bounded: fold what an earlier call recorded first
    if (ctx->ev_used > 0 && ctx->ev_used + 8 * nsteps > 4096) {
        CK(cudaStreamSynchronize(ctx->stream));
        collect_events(ctx);
    }
    long long launches = 0;
    const bool timed = ctx->p.time_stages != 0;
    const bool graphs = ctx->p.use_graphs != 0 && !timed && ctx->p.check_interval <= 0;
    const int L = ctx->p.sort_interval;
    // a graph of the caller's own is replayed on the buffers it was captured on: there the fields stay in theirs
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CK(cudaStreamIsCapturing(ctx->stream, &cap));
    const bool in_place = cap != cudaStreamCaptureStatusNone;
    for (long long s = 0; s < nsteps;) {
        long long run = nsteps - s;              // steps up to the next whole cycle, or the rest
        if (graphs) {
            if (L > 1 && ctx->nblocks > 0 && ctx->steps_done % L == 0 && run >= L) {
                rc = cycle_step(ctx, pusher, launches);
                if (rc) return rc;
                s += L;
                continue;
            }
            if (L > 1 && ctx->nblocks > 0) run = std::min<long long>(run, L - ctx->steps_done % L);
            // a single step is one graph launch; of two or more the field updates are shared, which
            // plain launches do too (two a step, as fast as the kernels run on the smallest meshes:
            // 2,048 triangles 10.3 us a step as one-step graphs)
            if (run == 1) {
                rc = graph_step(ctx, pusher, launches);
                if (rc) return rc;
                ++s;
                continue;
            }
        }
        bool begun = false;                      // the previous step's field update carried this one's Faraday
        for (long long k = 0; k < run; ++k) {
            if (timed && ctx->ev_used > 4000) {
                CK(cudaStreamSynchronize(ctx->stream));
                collect_events(ctx);
            }
            const bool more = !in_place && can_merge(ctx, run - 1 - k);
            launches += enqueue_step(ctx, pusher, timed, begun, more);
            begun = more;
        }
        s += run;
    }
    ctx->launches_acc += launches;
    CK(cudaGetLastError());
    return FETDPIC_OK;
}

extern "C" int fetdpic_sync(fetdpic_ctx *ctx)
{
    if (!ctx) return FETDPIC_EINVAL;
    const int rc = take_status(ctx);                       // waits for the stream
    if (ctx->io) CK(cudaStreamSynchronize(ctx->io));      // host copies of asynchronous reads
    collect_events(ctx);
    return rc;
}

// Reusable device scratch for particle-state transfers (grown on demand).
static void *xfer_buf(fetdpic_ctx *ctx, size_t bytes)
{
    if (bytes <= ctx->xfer_bytes) return ctx->xfer;
    if (ctx->xfer) {
        // an asynchronous write may still be copying into the old buffer
        if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) return nullptr;
        for (size_t k = 0; k < ctx->allocs.size(); ++k)
            if (ctx->allocs[k] == ctx->xfer) { ctx->allocs.erase(ctx->allocs.begin() + k); break; }
        if (ctx->p.dev_free) ctx->p.dev_free(ctx->xfer, ctx->p.alloc_user);
        else cudaFree(ctx->xfer);
        ctx->xfer = nullptr; ctx->xfer_bytes = 0;
    }
    try { ctx->xfer = ctx->alloc<char>(bytes); } catch (const std::bad_alloc &) { return nullptr; }
    ctx->xfer_bytes = bytes;
    return ctx->xfer;
}

extern "C" int fetdpic_write_particles(fetdpic_ctx *ctx, int species, const double *x, const double *u, const int *cell)
{
    if (!ctx || species < 0) return FETDPIC_EINVAL;
    int rc = finalize(ctx);
    if (rc) return rc;
    if (species >= (int)ctx->sp.size() || (!x && ctx->sp[species].n) || (!u && ctx->sp[species].n))
        return ctx->fail(FETDPIC_EINVAL, "bad species or buffers");
    const Species &D = ctx->sp[species];
    const HostMesh &M = ctx->mesh[D.inst];
    if (D.n == 0) return FETDPIC_OK;
    std::vector<int> located;
    const int *cl = cell;
    if (!cl) {
        located.resize(D.n);
        for (long long k = 0; k < D.n; ++k) {
            const int f = host_locate(M, x[2 * k], x[2 * k + 1], -1);
            if (f < 0) return ctx->fail(FETDPIC_EOUTSIDE, "particle outside the mesh");
            located[k] = M.perm[f];                  // the caller's index, as a given cell would be
        }
        cl = located.data();
    }
    // caller-supplied triangles are range-checked by the ingest kernel (reported at the next sync)
    // staging: x [n][2], u [n][2] (FP64), cell [n]
    const size_t bx = sizeof(double) * 2 * D.n, bc = sizeof(int) * D.n;
    char *st = (char *)xfer_buf(ctx, 2 * bx + bc);
    if (!st) return FETDPIC_ENOMEM;
    CK(cudaMemcpyAsync(st, x, bx, cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaMemcpyAsync(st + bx, u, bx, cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaMemcpyAsync(st + 2 * bx, cl, bc, cudaMemcpyHostToDevice, ctx->stream));
    launch_ingest(ctx->stream, D.n, D.cap, D.off, D.cell_off, M.nf, ctx->p.precision == FETDPIC_FP32,
                  (const double *)st, (const double *)(st + bx), (const int *)(st + 2 * bx), ctx->tri_c2i, ctx->geo64,
                  1.0 / ctx->p.c, ctx->cell, ctx->id, ctx->f[0], ctx->f[1], ctx->f[2], ctx->f[3], ctx->status);
    CK(cudaGetLastError());
    if (!cell) CK(cudaStreamSynchronize(ctx->stream));   // `located` goes out of scope
    ctx->q_prev_valid = false;
    if (ctx->g0) reset_gauss_reference(ctx);
    return FETDPIC_OK;
}

// Edge unknowns of an instance (caller's order, 0 on PEC edges) to the device, with the dual flux
// restarted consistently: d = [*eps] e.  Waits for the copies.
static int upload_edges(fetdpic_ctx *ctx, int inst, const std::vector<double> &ev)
{
    const HostMesh &M = ctx->mesh[inst];
    std::vector<double> es(M.ne), ds(M.ne);
    for (int k = 0; k < M.ne; ++k) {
        double s = 0.0;
        for (long long q = M.h_rp[k]; q < M.h_rp[k + 1]; ++q) s += M.h_v[q] * ev[M.h_ci[q]];
        es[M.einv[k]] = ev[k];
        ds[M.einv[k]] = s;
    }
    int rc = upload(ctx, ctx->e + ctx->edge_off[inst], es.data(), es.size());
    rc = rc ? rc : upload(ctx, ctx->d + ctx->edge_off[inst], ds.data(), ds.size());
    if (rc) return rc;
    CK(cudaStreamSynchronize(ctx->stream));
    return FETDPIC_OK;
}

extern "C" int fetdpic_write_fields(fetdpic_ctx *ctx, int inst, const double *e, const double *b)
{
    if (!ctx || inst < 0 || inst >= (int)ctx->mesh.size()) return FETDPIC_EINVAL;
    const HostMesh &M = ctx->mesh[inst];
    if (e) {
        std::vector<double> ev(e, e + M.ne);
        for (int k = 0; k < M.ne; ++k) if (M.pec[k]) ev[k] = 0.0;
        int rc = upload_edges(ctx, inst, ev);
        if (rc) return rc;
    }
    if (b) {
        std::vector<double> bs(M.nf);                // stored triangle order
        for (int f = 0; f < M.nf; ++f) bs[f] = b[M.perm[f]];
        int rc = upload(ctx, ctx->b + ctx->cell_off[inst], bs.data(), bs.size());
        if (rc) return rc;
        CK(cudaStreamSynchronize(ctx->stream));
    }
    if (e) {
        ctx->gauss_abs[inst] = 0;              // a caller's field need not satisfy Gauss's law
        reset_gauss_reference(ctx);
    }
    return FETDPIC_OK;
}

extern "C" int fetdpic_solve_electrostatic(fetdpic_ctx *ctx, int inst, int *iterations, double *residual)
{
    if (!ctx || inst < 0 || inst >= (int)ctx->mesh.size()) return FETDPIC_EINVAL;
    if (ctx->steps_done > 0)
        return ctx->fail(FETDPIC_ESTATE, "the electrostatic solve uses the loaded particles: call it before the first step");
    const HostMesh &M = ctx->mesh[inst];
    // nodal charge of the loaded particles, Eq. (scatter.charge.assign): q_i += Q lambda_i(r_p)
    std::vector<double> q(M.nn, 0.0);
    for (const auto &S : ctx->staged) {
        if (S.inst != inst) continue;
        for (size_t k = 0; k < S.cell.size(); ++k) {
            double l[3];
            host_lambdas(M, S.cell[k], S.x[k], S.y[k], l);
            for (int m = 0; m < 3; ++m) q[M.rep[M.tri[3 * S.cell[k] + m]]] += S.q * l[m];
        }
    }
    std::vector<double> de;
    int it = 0;
    double res = 0.0;
    std::string msg;
    int rc = electrostatic_solve(M, q, de, it, res, msg);
    if (rc) return ctx->fail(rc, msg);
    CK(cudaSetDevice(ctx->device));
    CK(cudaStreamSynchronize(ctx->stream));
    std::vector<double> es(M.ne), ev(M.ne);
    CK(cudaMemcpy(es.data(), ctx->e + ctx->edge_off[inst], sizeof(double) * M.ne, cudaMemcpyDeviceToHost));
    for (int k = 0; k < M.ne; ++k) ev[k] = es[M.einv[k]] + de[k];
    rc = upload_edges(ctx, inst, ev);
    if (rc) return rc;
    ctx->gauss_abs[inst] = 1;
    auto &an = ctx->abs_nodes[inst];
    an.assign(M.nn, 0);
    {
        std::vector<char> pec_node(M.nn, 0), free_node(M.nn, 0);
        for (int k = 0; k < M.ne; ++k) {
            char *t = M.pec[k] ? pec_node.data() : free_node.data();
            t[M.edge[2 * k]] = t[M.edge[2 * k + 1]] = 1;
        }
        for (int n = 0; n < M.nn; ++n) an[n] = free_node[n] && !pec_node[n];
    }
    reset_gauss_reference(ctx);
    if (iterations) *iterations = it;
    if (residual) *residual = res;
    return FETDPIC_OK;
}

extern "C" int fetdpic_read(fetdpic_ctx *ctx, int inst, double *e, double *b, double *j,
                            int species, double *x, double *u, int *cell)
{
    if (!ctx || inst < 0 || inst >= (int)ctx->mesh.size()) return FETDPIC_EINVAL;
    const HostMesh &M = ctx->mesh[inst];
    CK(cudaSetDevice(ctx->device));
    {
        // to the caller's edge and triangle order on the device (in one launch: 2,000 to 30,000 triangles
        // 12-14 us less than with one for each array), then to the host
        const int eo = ctx->edge_off[inst], co = ctx->cell_off[inst];
        double *oe = ctx->field_out, *oj = oe + M.ne, *ob = oj + M.ne;
        if (e || b || j)
            launch_gather_fields(ctx->stream, GatherFields{M.ne, M.nf, eo, co, ctx->edge_c2i, ctx->tri_c2i, e ? ctx->e : nullptr,
                                                           j ? ctx->j : nullptr, b ? ctx->b : nullptr, oe});
        CK(cudaGetLastError());
        const size_t be = sizeof(double) * M.ne, bf = sizeof(double) * M.nf;
        if ((e || b || j) && 2 * be + bf <= SMALL_READ) {
            CK(cudaMemcpyAsync(ctx->pin, oe, 2 * be + bf, cudaMemcpyDeviceToHost, ctx->stream));
            if (x || u || cell) {                    // the buffer is used again below
                CK(cudaStreamSynchronize(ctx->stream));
            } else {
                const int rc = take_status(ctx);
                if (rc == FETDPIC_ECUDA) return rc;
                if (e) std::memcpy(e, ctx->pin, be);
                if (j) std::memcpy(j, ctx->pin + be, be);
                if (b) std::memcpy(b, ctx->pin + 2 * be, bf);
                return rc;
            }
            if (e) std::memcpy(e, ctx->pin, be);
            if (j) std::memcpy(j, ctx->pin + be, be);
            if (b) std::memcpy(b, ctx->pin + 2 * be, bf);
        } else {
            if (e) CK(cudaMemcpyAsync(e, oe, be, cudaMemcpyDeviceToHost, ctx->stream));
            if (b) CK(cudaMemcpyAsync(b, ob, bf, cudaMemcpyDeviceToHost, ctx->stream));
            if (j) CK(cudaMemcpyAsync(j, oj, be, cudaMemcpyDeviceToHost, ctx->stream));
        }
    }
    if (x || u || cell) {
        // an error below does not return before the field copies have reached the caller's memory
        int rc = finalize(ctx);
        if (rc == FETDPIC_OK && (species < 0 || species >= (int)ctx->sp.size()))
            rc = ctx->fail(FETDPIC_EINVAL, "bad species");
        if (rc) {
            CK(cudaStreamSynchronize(ctx->stream));
            return rc;
        }
        const Species &D = ctx->sp[species];
        if (D.n > 0) {
            const size_t bx = sizeof(double) * 2 * D.n, bc = sizeof(int) * D.n;
            char *st = (char *)xfer_buf(ctx, 2 * bx + bc);
            if (!st) {
                CK(cudaStreamSynchronize(ctx->stream));
                return FETDPIC_ENOMEM;
            }
            double *ox = (double *)st, *ou = (double *)(st + bx);
            int *oc = (int *)(st + 2 * bx);
            if (ctx->p.precision == FETDPIC_FP32)
                launch_unsort32(ctx->stream, D.n, ctx->cell, ctx->id, (float *)ctx->f[0], (float *)ctx->f[1],
                                (float *)ctx->f[2], (float *)ctx->f[3], ctx->geo64, ctx->p.c, D.off, D.cap,
                                ctx->tri_i2c, ox, ou, oc);
            else
                launch_unsort64(ctx->stream, D.n, ctx->cell, ctx->id, (double *)ctx->f[0], (double *)ctx->f[1],
                                (double *)ctx->f[2], (double *)ctx->f[3], D.off, D.cap, ctx->tri_i2c, ox, ou, oc);
            CK(cudaGetLastError());
            if (2 * bx + bc <= SMALL_READ) {
                CK(cudaMemcpyAsync(ctx->pin, st, 2 * bx + bc, cudaMemcpyDeviceToHost, ctx->stream));
                const int rc = take_status(ctx);
                if (rc == FETDPIC_ECUDA) return rc;
                if (x) std::memcpy(x, ctx->pin, bx);
                if (u) std::memcpy(u, ctx->pin + bx, bx);
                if (cell) std::memcpy(cell, ctx->pin + 2 * bx, bc);
                return rc;
            }
            if (x) CK(cudaMemcpyAsync(x, ox, bx, cudaMemcpyDeviceToHost, ctx->stream));
            if (u) CK(cudaMemcpyAsync(u, ou, bx, cudaMemcpyDeviceToHost, ctx->stream));
            if (cell) CK(cudaMemcpyAsync(cell, oc, bc, cudaMemcpyDeviceToHost, ctx->stream));
        }
    }
    return take_status(ctx);
}

// Stream, events and staging of the asynchronous particle reads (first use).
static int setup_async_reads(fetdpic_ctx *ctx)
{
    if (ctx->io) return FETDPIC_OK;
    const size_t ns = ctx->sp.size();
    size_t off = 0;
    ctx->rd_off.assign(ns, 0);
    for (size_t s = 0; s < ns; ++s) {
        ctx->rd_off[s] = off;
        off += ((36 * (size_t)ctx->sp[s].n + 255) / 256) * 256;      // x, u (FP64), cell per particle
    }
    try { ctx->rd_buf = ctx->alloc<char>(std::max<size_t>(off, 256)); } catch (const std::bad_alloc &) {
        return FETDPIC_ENOMEM;
    }
    ctx->ev_rd_done.assign(ns, nullptr);
    ctx->rd_pending.assign(ns, 0);
    CK(cudaEventCreateWithFlags(&ctx->ev_rd, cudaEventDisableTiming));
    for (auto &e : ctx->ev_rd_done) CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    CK(cudaStreamCreateWithFlags(&ctx->io, cudaStreamNonBlocking));
    return FETDPIC_OK;
}

extern "C" int fetdpic_read_particles_async(fetdpic_ctx *ctx, int species, double *x, double *u, int *cell)
{
    if (!ctx) return FETDPIC_EINVAL;
    int rc = finalize(ctx);
    if (rc) return rc;
    if (species < 0 || species >= (int)ctx->sp.size()) return ctx->fail(FETDPIC_EINVAL, "bad species");
    CK(cudaSetDevice(ctx->device));
    rc = setup_async_reads(ctx);
    if (rc) return rc;
    const Species &D = ctx->sp[species];
    if (D.n == 0 || (!x && !u && !cell)) return FETDPIC_OK;
    const size_t bx = sizeof(double) * 2 * D.n, bc = sizeof(int) * D.n;
    char *st = ctx->rd_buf + ctx->rd_off[species];
    double *ox = (double *)st, *ou = (double *)(st + bx);
    int *oc = (int *)(st + 2 * bx);
    // the previous asynchronous read of this species must have copied its staging out first
    if (ctx->rd_pending[species]) CK(cudaStreamWaitEvent(ctx->stream, ctx->ev_rd_done[species], 0));
    if (ctx->p.precision == FETDPIC_FP32)
        launch_unsort32(ctx->stream, D.n, ctx->cell, ctx->id, (float *)ctx->f[0], (float *)ctx->f[1],
                        (float *)ctx->f[2], (float *)ctx->f[3], ctx->geo64, ctx->p.c, D.off, D.cap, ctx->tri_i2c,
                        ox, ou, oc);
    else
        launch_unsort64(ctx->stream, D.n, ctx->cell, ctx->id, (double *)ctx->f[0], (double *)ctx->f[1],
                        (double *)ctx->f[2], (double *)ctx->f[3], D.off, D.cap, ctx->tri_i2c, ox, ou, oc);
    CK(cudaGetLastError());
    // the host copies run on the io stream: the context stream goes on with the next writes,
    // steps or reads meanwhile (the state they change has already been copied to the staging)
    CK(cudaEventRecord(ctx->ev_rd, ctx->stream));
    CK(cudaStreamWaitEvent(ctx->io, ctx->ev_rd, 0));
    if (x) CK(cudaMemcpyAsync(x, ox, bx, cudaMemcpyDeviceToHost, ctx->io));
    if (u) CK(cudaMemcpyAsync(u, ou, bx, cudaMemcpyDeviceToHost, ctx->io));
    if (cell) CK(cudaMemcpyAsync(cell, oc, bc, cudaMemcpyDeviceToHost, ctx->io));
    CK(cudaEventRecord(ctx->ev_rd_done[species], ctx->io));
    ctx->rd_pending[species] = 1;
    return FETDPIC_OK;
}

extern "C" int fetdpic_read_charge(fetdpic_ctx *ctx, int inst, double *q, double *quantum)
{
    if (!ctx || inst < 0 || inst >= (int)ctx->mesh.size()) return FETDPIC_EINVAL;
    int rc = finalize(ctx);
    if (rc) return rc;
    CK(cudaSetDevice(ctx->device));
    if (quantum) *quantum = ctx->qunit_host[inst];
    if (!q) return FETDPIC_OK;
    if (!ctx->qread) {
        try { ctx->qread = ctx->alloc<unsigned long long>(std::max(ctx->N, 1)); }
        catch (const std::bad_alloc &) { return FETDPIC_ENOMEM; }
    }
    charge_now(ctx, ctx->qread);
    CK(cudaGetLastError());
    const int nn = ctx->mesh[inst].nn;
    std::vector<unsigned long long> v(nn);
    CK(cudaMemcpyAsync(v.data(), ctx->qread + ctx->node_off[inst], sizeof(unsigned long long) * nn,
                       cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    const double qu = ctx->qunit_host[inst];
    for (int n = 0; n < nn; ++n) q[n] = (double)(long long)v[n] * qu;
    return FETDPIC_OK;
}

extern "C" int fetdpic_read_walk(fetdpic_ctx *ctx, int species, int *cnt, int *rec)
{
    if (!ctx || !cnt || !rec) return FETDPIC_EINVAL;
    if (ctx->p.record_walk <= 0) return ctx->fail(FETDPIC_ESTATE, "record_walk is off");
    int rc = finalize(ctx);
    if (rc) return rc;
    if (species < 0 || species >= (int)ctx->sp.size()) return FETDPIC_EINVAL;
    const Species &D = ctx->sp[species];
    if (D.n == 0) return FETDPIC_OK;
    // the kernels write the record at species storage offset + load index: already in load order
    const size_t rc_ = (size_t)ctx->p.record_walk;
    CK(cudaStreamSynchronize(ctx->stream));
    CK(cudaMemcpy(cnt, ctx->rec_cnt + D.off, sizeof(int) * D.n, cudaMemcpyDeviceToHost));
    CK(cudaMemcpy(rec, ctx->rec + D.off * rc_, sizeof(int) * D.n * rc_, cudaMemcpyDeviceToHost));
    // the kernels record stored edge ids; entries beyond a particle's count are not set
    const HostMesh &M = ctx->mesh[D.inst];
    for (long long k = 0; k < D.n; ++k)
        for (int c = 0; c < std::min<int>(cnt[k], (int)rc_); ++c) {
            int &v = rec[k * (long long)rc_ + c];
            v = v >= 0 ? M.eperm[v] : -(M.eperm[-v - 1] + 1);
        }
    return FETDPIC_OK;
}

extern "C" int fetdpic_check(fetdpic_ctx *ctx, int inst, double *dce_max, double *dgl_max, double *energy)
{
    if (!ctx || inst < 0 || inst >= (int)ctx->mesh.size()) return FETDPIC_EINVAL;
    if (!ctx->chk_out) return ctx->fail(FETDPIC_ESTATE, "check_interval is 0: no checks are computed");
    CK(cudaSetDevice(ctx->device));
    CK(cudaStreamSynchronize(ctx->stream));
    double v[3] = {0, 0, 0};
    CK(cudaMemcpy(v, ctx->chk_out + 3 * inst, sizeof(v), cudaMemcpyDeviceToHost));
    if (dce_max) *dce_max = v[0];
    if (dgl_max) *dgl_max = v[1];
    if (energy) *energy = v[2];
    CK(cudaMemsetAsync(ctx->chk_out + 3 * inst, 0, 2 * sizeof(double), ctx->stream));   // maxima restart; energy stays
    return take_status(ctx);
}

extern "C" int fetdpic_info(fetdpic_ctx *ctx, int inst, long long out[6])
{
    if (!ctx || !out || inst < 0 || inst >= (int)ctx->mesh.size()) return FETDPIC_EINVAL;
    const HostMesh &M = ctx->mesh[inst];
    out[0] = M.nn; out[1] = M.ne; out[2] = M.nf; out[3] = (long long)M.free_edges.size();
    out[4] = M.m_rp.empty() ? 0 : M.m_rp.back();
    long long np = 0;
    for (auto &s : ctx->staged) if (s.inst == inst) np += (long long)s.cell.size();
    out[5] = np;
    return FETDPIC_OK;
}

static void drop_graphs(fetdpic_ctx *ctx);

extern "C" int fetdpic_set_external_profile(fetdpic_ctx *ctx, int inst, const double *w)
{
    if (!ctx || inst < 0 || inst >= (int)ctx->mesh.size()) return FETDPIC_EINVAL;
    const int nf = ctx->mesh[inst].nf;
    std::vector<double2> wv(nf, make_double2(1.0, 1.0));
    if (w)
        for (int f = 0; f < nf; ++f) {
            if (!std::isfinite(w[2 * f]) || !std::isfinite(w[2 * f + 1]))
                return ctx->fail(FETDPIC_EINVAL, "non-finite applied-field weight");
            wv[ctx->mesh[inst].inv[f]] = make_double2(w[2 * f], w[2 * f + 1]);    // stored order
        }
    CK(cudaSetDevice(ctx->device));
    CK(cudaStreamSynchronize(ctx->stream));
    if (!ctx->extw) {
        try { ctx->extw = ctx->alloc<double2>(ctx->F); } catch (const std::bad_alloc &) { return FETDPIC_ENOMEM; }
        std::vector<double2> ones(ctx->F, make_double2(1.0, 1.0));
        int rc = upload(ctx, ctx->extw, ones.data(), ones.size());
        if (rc) return rc;
        drop_graphs(ctx);                      // captured steps hold no weights
    }
    int rc = upload(ctx, ctx->extw + ctx->cell_off[inst], wv.data(), wv.size());
    if (rc) return rc;
    if (!ctx->ext_on) { ctx->ext_on = true; drop_graphs(ctx); }
    CK(cudaStreamSynchronize(ctx->stream));
    return FETDPIC_OK;
}

extern "C" int fetdpic_set_external_amplitude(fetdpic_ctx *ctx, int inst, double amplitude)
{
    if (!ctx || inst < 0 || inst >= (int)ctx->mesh.size()) return FETDPIC_EINVAL;
    if (!std::isfinite(amplitude)) return ctx->fail(FETDPIC_EINVAL, "non-finite amplitude");
    CK(cudaSetDevice(ctx->device));
    // a captured launch would set this amplitude again at every replay
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CK(cudaStreamIsCapturing(ctx->stream, &cap));
    if (cap != cudaStreamCaptureStatusNone)
        return ctx->fail(FETDPIC_ECUDA, "fetdpic_set_external_amplitude: the stream is being captured");
    // stream-ordered: steps enqueued before see the old value, later ones the new
    launch_set_value(ctx->stream, ctx->ext_amp + inst, amplitude);
    CK(cudaGetLastError());
    return FETDPIC_OK;
}

extern "C" int fetdpic_set_probes(fetdpic_ctx *ctx, long long n, const int *inst, const double *xy,
                                  long long capacity)
{
    if (!ctx) return FETDPIC_EINVAL;
    if (n < 0 || (n > 0 && (!inst || !xy || capacity <= 0)) || n > (1ll << 24) ||
        (n > 0 && (double)n * (double)capacity > 1e10))
        return ctx->fail(FETDPIC_EINVAL, "bad probe arguments (n <= 2^24, n * capacity <= 1e10 samples)");
    std::vector<ProbeW> w((size_t)n);
    for (long long p = 0; p < n; ++p) {
        const int k = inst[p];
        if (k < 0 || k >= (int)ctx->mesh.size()) return ctx->fail(FETDPIC_EINVAL, "probe instance out of range");
        const HostMesh &M = ctx->mesh[k];
        const double x = xy[2 * p], y = xy[2 * p + 1];
        const int f = host_locate(M, x, y, -1);
        if (f < 0) return ctx->fail(FETDPIC_EOUTSIDE, "probe " + std::to_string(p) + " lies in no triangle");
        double l[3];
        host_lambdas(M, f, x, y, l);
        ProbeW &W = w[(size_t)p];
        for (int m = 0; m < 3; ++m) {
            const int a = (m + 1) % 3, b = (m + 2) % 3;
            const double sg = M.tsign[3 * f + m];
            W.w[2 * m] = sg * (l[a] * M.gx[3 * f + b] - l[b] * M.gx[3 * f + a]);
            W.w[2 * m + 1] = sg * (l[a] * M.gy[3 * f + b] - l[b] * M.gy[3 * f + a]);
            W.eg[m] = ctx->edge_off[k] + M.einv[M.tedge[3 * f + m]];
        }
        W.pad = 0;
    }
    CK(cudaSetDevice(ctx->device));
    CK(cudaStreamSynchronize(ctx->stream));
    ctx->release(ctx->probe_w); ctx->release(ctx->probe_ring); ctx->release(ctx->probe_count);
    ctx->probe_w = nullptr; ctx->probe_ring = nullptr; ctx->probe_count = nullptr;
    ctx->probe_n = 0; ctx->probe_cap = 0;
    drop_graphs(ctx);                          // the step's launch sequence changes
    if (n == 0) return FETDPIC_OK;
    try {
        ctx->probe_w = ctx->alloc<ProbeW>((size_t)n);
        ctx->probe_ring = ctx->alloc<double2>((size_t)n * (size_t)capacity);
        ctx->probe_count = ctx->alloc<unsigned long long>(1);
    } catch (const std::bad_alloc &) {
        return ctx->fail(FETDPIC_ENOMEM, "probe buffers");
    }
    CK(cudaMemcpyAsync(ctx->probe_w, w.data(), sizeof(ProbeW) * (size_t)n, cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaMemsetAsync(ctx->probe_count, 0, sizeof(unsigned long long), ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    ctx->probe_n = n;
    ctx->probe_cap = capacity;
    return FETDPIC_OK;
}

extern "C" int fetdpic_read_probes(fetdpic_ctx *ctx, double *exy, long long max_rows, long long *rows,
                                   long long *total)
{
    if (!ctx) return FETDPIC_EINVAL;
    if (max_rows < 0 || (max_rows > 0 && !exy)) return ctx->fail(FETDPIC_EINVAL, "bad probe read arguments");
    if (ctx->probe_n == 0) return ctx->fail(FETDPIC_ESTATE, "no probes set");
    CK(cudaSetDevice(ctx->device));
    CK(cudaStreamSynchronize(ctx->stream));
    unsigned long long cnt = 0;
    CK(cudaMemcpy(&cnt, ctx->probe_count, sizeof(cnt), cudaMemcpyDeviceToHost));
    const long long have = std::min<long long>((long long)cnt, ctx->probe_cap);
    const long long take = std::min(have, max_rows);
    // the last `take` rows, oldest first: one piece of the ring, or two where it wraps
    const size_t row_bytes = sizeof(double2) * (size_t)ctx->probe_n;
    const long long first = take > 0 ? (long long)((cnt - (unsigned long long)take) % (unsigned long long)ctx->probe_cap) : 0;
    const long long run = std::min(take, ctx->probe_cap - first);
    if (run > 0)
        CK(cudaMemcpyAsync(exy, ctx->probe_ring + (size_t)first * ctx->probe_n, row_bytes * run, cudaMemcpyDeviceToHost,
                           ctx->stream));
    if (take > run)
        CK(cudaMemcpyAsync(exy + (size_t)run * 2 * (size_t)ctx->probe_n, ctx->probe_ring, row_bytes * (take - run),
                           cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    if (rows) *rows = take;
    if (total) *total = (long long)cnt;
    return FETDPIC_OK;
}

extern "C" int fetdpic_read_edges(fetdpic_ctx *ctx, int inst, int *edges)
{
    if (!ctx || !edges || inst < 0 || inst >= (int)ctx->mesh.size()) return FETDPIC_EINVAL;
    const HostMesh &M = ctx->mesh[inst];
    std::memcpy(edges, M.edge.data(), sizeof(int) * M.edge.size());
    return FETDPIC_OK;
}

extern "C" int fetdpic_read_spai(fetdpic_ctx *ctx, int inst, long long *rowptr, int *row_edge, int *col, double *val)
{
    if (!ctx || inst < 0 || inst >= (int)ctx->mesh.size()) return FETDPIC_EINVAL;
    const HostMesh &M = ctx->mesh[inst];
    if (rowptr) std::memcpy(rowptr, M.m_rp.data(), sizeof(long long) * M.m_rp.size());
    if (row_edge) std::memcpy(row_edge, M.free_edges.data(), sizeof(int) * M.free_edges.size());
    if (col) std::memcpy(col, M.m_ci.data(), sizeof(int) * M.m_ci.size());
    if (val) std::memcpy(val, M.m_v.data(), sizeof(double) * M.m_v.size());
    return FETDPIC_OK;
}

// ------------------------------------------------------------ autotuning

static void drop_graphs(fetdpic_ctx *ctx)
{
    for (auto &a : ctx->graph) for (auto &b : a) for (auto &c : b) for (auto &d : c) for (auto &g : d)
        if (g) { cudaGraphExecDestroy(g); g = nullptr; }
    for (auto &a : ctx->cycle) for (auto &b : a) for (auto &g : b)
        if (g) { cudaGraphExecDestroy(g); g = nullptr; }
}

extern "C" int fetdpic_set_wait_limit(fetdpic_ctx *ctx, long long wait_spin_limit)
{
    if (!ctx) return FETDPIC_EINVAL;
    CK(cudaStreamSynchronize(ctx->stream));
    ctx->p.wait_spin_limit = wait_spin_limit;
    drop_graphs(ctx);                          // captured steps hold the old limit
    return FETDPIC_OK;
}

extern "C" int fetdpic_set_tuning(fetdpic_ctx *ctx, int variant, int sort_interval)
{
    if (!ctx) return FETDPIC_EINVAL;
    if (variant < 0 || variant > 22 || variant == 1 || sort_interval == 0) return ctx->fail(FETDPIC_EINVAL, "bad tuning");
    CK(cudaStreamSynchronize(ctx->stream));
    ctx->p.kernel_variant = variant;              // 0 = the untuned default
    ctx->p.sort_interval = sort_interval;
    drop_graphs(ctx);
    return FETDPIC_OK;
}

extern "C" int fetdpic_autotune(fetdpic_ctx *ctx, int pusher, int trial_steps, int *variant, int *sort_interval)
{
    if (!ctx || pusher < 0 || pusher > 3) return FETDPIC_EINVAL;
    int rc = finalize(ctx);
    if (rc) return rc;
    if (trial_steps <= 0) trial_steps = 32;
    CK(cudaStreamSynchronize(ctx->stream));
    // save the state the trials disturb
    const size_t fb = ctx->p.precision == FETDPIC_FP32 ? 4 : 8;
    const size_t pbytes = (size_t)ctx->P * (8 + 4 * fb);
    const size_t fbytes = sizeof(double) * (2 * (size_t)ctx->E + ctx->F);
    char *save = nullptr;
    try { save = ctx->alloc<char>(pbytes + fbytes); } catch (const std::bad_alloc &) { return FETDPIC_ENOMEM; }
    auto copy_state = [&](bool to_save) -> int {
        char *q = save;
        void *dst[8], *src[8];
        size_t n[8];
        int k = 0;
        dst[k] = ctx->cell; n[k++] = sizeof(int) * ctx->P;
        dst[k] = ctx->id; n[k++] = sizeof(int) * ctx->P;
        for (int a = 0; a < 4; ++a) { dst[k] = ctx->f[a]; n[k++] = fb * ctx->P; }
        dst[k] = ctx->e; n[k++] = sizeof(double) * ctx->E;
        dst[k] = ctx->d; n[k++] = sizeof(double) * ctx->E;
        for (int a = 0; a < k; ++a) { src[a] = q; q += n[a]; }
        for (int a = 0; a < k; ++a) {
            if (to_save) CK(cudaMemcpyAsync(src[a], dst[a], n[a], cudaMemcpyDeviceToDevice, ctx->stream));
            else CK(cudaMemcpyAsync(dst[a], src[a], n[a], cudaMemcpyDeviceToDevice, ctx->stream));
        }
        if (to_save) CK(cudaMemcpyAsync(q, ctx->b, sizeof(double) * ctx->F, cudaMemcpyDeviceToDevice, ctx->stream));
        else CK(cudaMemcpyAsync(ctx->b, q, sizeof(double) * ctx->F, cudaMemcpyDeviceToDevice, ctx->stream));
        return FETDPIC_OK;
    };
    const int keep_variant = ctx->p.kernel_variant, keep_sort = ctx->p.sort_interval;
    const bool keep_timed = ctx->p.time_stages != 0;
    const int keep_check = ctx->p.check_interval;
    const long long keep_steps = ctx->steps_done;
    const long long keep_probes = ctx->probe_n;        // trial steps record no probe rows
    unsigned keep_status = 0;                          // errors the caller has not read yet survive
    CK(cudaMemcpy(&keep_status, ctx->status, sizeof(unsigned), cudaMemcpyDeviceToHost));
    ctx->p.time_stages = 0;
    ctx->p.check_interval = 0;
    ctx->probe_n = 0;
    rc = copy_state(true);
    std::vector<int> variants = ctx->p.precision == FETDPIC_FP32 ? std::vector<int>{2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 14, 17, 18, 19, 20, 21, 22}
                                                          : std::vector<int>{3};
    // the default where it is none of them (above 2 M particles with 20 or more per triangle, the pushers
    // other than Vay: variant 12, then 20)
    if (ctx->p.precision == FETDPIC_FP32) {
        ctx->p.kernel_variant = 0;
        const Hybrid d = kernels_of(ctx, pusher);
        bool listed = d.early == d.late;
        for (const Hybrid &h : HYBRIDS) listed = listed || (h.early == d.early && h.late == d.late && h.steps == d.steps);
        if (!listed) variants.push_back(0);
    }
    std::vector<int> sorts = keep_sort < 0 ? std::vector<int>{-1} : std::vector<int>{8, 12, 16, 32};
    double best = 1e300;
    int bv = keep_variant, bs = keep_sort;
    cudaEvent_t t0, t1;
    CK(cudaEventCreate(&t0));
    CK(cudaEventCreate(&t1));
    for (int v : variants)
        for (int si : sorts) {
            if (rc) break;
            rc = copy_state(false);
            if (rc) break;
            ctx->p.kernel_variant = v;
            ctx->p.sort_interval = si;
            ctx->steps_done = 0;
            const int n = si > 0 ? std::max(trial_steps, si) / si * si : trial_steps;
            enqueue_step(ctx, pusher, false);                           // warm-up
            CK(cudaEventRecord(t0, ctx->stream));
            for (int k = 0; k < n; ++k)
                enqueue_step(ctx, pusher, false, k > 0 && can_merge(ctx, 1), can_merge(ctx, n - 1 - k));
            CK(cudaEventRecord(t1, ctx->stream));
            CK(cudaEventSynchronize(t1));
            float ms = 0.f;
            CK(cudaEventElapsedTime(&ms, t0, t1));
            if (ms / n < best) { best = ms / n; bv = v; bs = si; }
        }
    cudaEventDestroy(t0);
    cudaEventDestroy(t1);
    // back to the saved state; the trials' currents are discarded
    if (!rc) rc = copy_state(false);
    CK(cudaMemsetAsync(ctx->ifix, 0, sizeof(unsigned long long) * ctx->E, ctx->stream));
    CK(cudaMemcpyAsync(ctx->status, &keep_status, sizeof(unsigned), cudaMemcpyHostToDevice, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    ctx->probe_n = keep_probes;
    for (size_t k = 0; k < ctx->allocs.size(); ++k)
        if (ctx->allocs[k] == save) { ctx->allocs.erase(ctx->allocs.begin() + k); break; }
    if (ctx->p.dev_free) ctx->p.dev_free(save, ctx->p.alloc_user);
    else cudaFree(save);
    ctx->p.time_stages = keep_timed ? 1 : 0;
    ctx->p.check_interval = keep_check;
    ctx->steps_done = keep_steps;
    ctx->q_prev_valid = false;
    if (rc) { ctx->p.kernel_variant = keep_variant; ctx->p.sort_interval = keep_sort; return rc; }
    ctx->p.kernel_variant = bv;
    ctx->p.sort_interval = bs;
    drop_graphs(ctx);
    if (variant) *variant = bv;
    if (sort_interval) *sort_interval = bs;
    return FETDPIC_OK;
}

extern "C" int fetdpic_stage_times(fetdpic_ctx *ctx, double out[6], long long *launches)
{
    if (!ctx || !out) return FETDPIC_EINVAL;
    CK(cudaStreamSynchronize(ctx->stream));
    collect_events(ctx);
    for (int k = 0; k < 6; ++k) { out[k] = ctx->stage_ms[k]; ctx->stage_ms[k] = 0.0; }
    if (launches) *launches = ctx->launches_acc;
    ctx->launches_acc = 0;
    return FETDPIC_OK;
}

extern "C" int fetdpic_particle_bytes(fetdpic_ctx *ctx, double *bytes, long long *n_particles)
{
    if (!ctx) return FETDPIC_EINVAL;
    long long n = 0;
    for (auto &s : ctx->sp) n += s.n;
    if (!ctx->finalized) for (auto &s : ctx->staged) n += (long long)s.cell.size();
    // per particle-step: state in + out (cell 4 B + 4 values); see the design notes
    const double per = ctx->p.precision == FETDPIC_FP32 ? 2.0 * (4 + 4 * 4) : 2.0 * (4 + 4 * 8);
    if (bytes) *bytes = per * (double)n;
    if (n_particles) *n_particles = n;
    return FETDPIC_OK;
}

extern "C" const char *fetdpic_last_error(const fetdpic_ctx *ctx)
{
    return ctx ? ctx->err.c_str() : "null context";
}

extern "C" void fetdpic_destroy(fetdpic_ctx *ctx)
{
    delete ctx;
}

// ---------------------------------------------------------------------------
// Particle read-back that allocates nothing.
//
// fetdpic_read stages the load-ordered particle state in device memory that
// it allocates (cudaMalloc, or the caller's allocator callback) the first
// time it runs.  Some callers cannot allocate at that point: real-time loops
// that forbid allocator latency, or plug-ins whose host framework owns all
// device memory and gives none out.  This variant stages through a fixed
// file-scope device array instead.  The array is part of the library image:
// every GPU that loads the library holds it until the process exits.
namespace {

constexpr long long STATIC_READ_MAX = 262144;                    // particles per call
constexpr size_t STATIC_READ_BYTES = (size_t)STATIC_READ_MAX * 36; // x, u (FP64) + cell (int32)

static __device__ __align__(256) unsigned char g_static_read[STATIC_READ_BYTES];

// Device address of g_static_read, looked up once per device with that device
// current (the host-side symbol is only a stand-in, never a device address).
struct StaticReadSlot { bool ready = false; void *ptr = nullptr; };
static StaticReadSlot g_static_slots[64];
static std::mutex g_static_mu;

}  // namespace

extern "C" int fetdpic_read_particles_static(fetdpic_ctx *ctx, int species, double *x, double *u, int *cell)
{
    if (!ctx) return FETDPIC_EINVAL;
    if (!ctx->finalized)
        return ctx->fail(FETDPIC_ESTATE, "the particles are not on the device yet: call fetdpic_step, "
                                         "fetdpic_write_particles or fetdpic_read with a particle buffer first");
    if (species < 0 || species >= (int)ctx->sp.size()) return ctx->fail(FETDPIC_EINVAL, "bad species");
    const Species &D = ctx->sp[species];
    if (D.n > STATIC_READ_MAX)
        return ctx->fail(FETDPIC_EINVAL, "species has " + std::to_string(D.n) + " particles; the static read takes at most "
                                             + std::to_string(STATIC_READ_MAX));
    if (ctx->device < 0 || ctx->device >= 64) return ctx->fail(FETDPIC_EINVAL, "device ordinal out of range");
    void *base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_static_mu);
        StaticReadSlot &s = g_static_slots[ctx->device];
        if (!s.ready) {
            int cur = -1;
            CK(cudaGetDevice(&cur));
            CK(cudaSetDevice(ctx->device));
            cudaError_t e = cudaGetSymbolAddress(&s.ptr, g_static_read);
            cudaSetDevice(cur);
            if (e != cudaSuccess) return ctx->cuda_fail(e, "cudaGetSymbolAddress(g_static_read)");
            s.ready = true;
        }
        base = s.ptr;
    }
    if (D.n == 0) {
        CK(cudaStreamSynchronize(ctx->stream));
        return take_status(ctx);
    }
    const size_t bx = sizeof(double) * 2 * D.n, bc = sizeof(int) * D.n;
    char *st = (char *)base;
    // every live particle writes its slot; a particle dropped by fetdpic_write_particles (a
    // triangle outside the mesh) writes none, so the slots are first set to all-one bytes: NaN
    // positions and momenta, triangle -1, instead of what an earlier call left there
    CK(cudaMemsetAsync(st, 0xFF, 2 * bx + bc, ctx->stream));
    double *ox = (double *)st, *ou = (double *)(st + bx);
    int *oc = (int *)(st + 2 * bx);
    if (ctx->p.precision == FETDPIC_FP32)
        launch_unsort32(ctx->stream, D.n, ctx->cell, ctx->id, (float *)ctx->f[0], (float *)ctx->f[1],
                        (float *)ctx->f[2], (float *)ctx->f[3], ctx->geo64, ctx->p.c, D.off, D.cap, ctx->tri_i2c,
                        ox, ou, oc);
    else
        launch_unsort64(ctx->stream, D.n, ctx->cell, ctx->id, (double *)ctx->f[0], (double *)ctx->f[1],
                        (double *)ctx->f[2], (double *)ctx->f[3], D.off, D.cap, ctx->tri_i2c, ox, ou, oc);
    CK(cudaGetLastError());
    if (x) CK(cudaMemcpyAsync(x, ox, bx, cudaMemcpyDeviceToHost, ctx->stream));
    if (u) CK(cudaMemcpyAsync(u, ou, bx, cudaMemcpyDeviceToHost, ctx->stream));
    if (cell) CK(cudaMemcpyAsync(cell, oc, bc, cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    return take_status(ctx);
}
