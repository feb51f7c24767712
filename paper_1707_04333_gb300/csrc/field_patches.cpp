// Partition of the field update into patches of consecutive stored triangles
// (a compact piece of the Hilbert curve), one thread block each
// (kernels_field.cu): the edges a patch owns, the further edges whose curl it
// recomputes, and its rows of the sparse approximate inverse with columns
// numbered inside the patch.
#include <algorithm>
#include <exception>
#include <thread>
#include <vector>

#include "fetdpic_internal.h"

namespace fetdpic {

namespace {

// Patches [p0, p1) into S, offsets relative to S.
void build_range(PatchSet &S, const PatchInput &in, const std::vector<int> &own, int T, int p0, int p1)
{
    std::vector<int> ring, ext, other, edge;
    for (int p = p0; p < p1; ++p) {
        FieldPatch P{};
        P.t0 = p * T;
        P.nt = std::min(T, in.F - P.t0);
        P.e0 = own[p];
        P.ne = own[p + 1] - own[p];
        const int e1 = P.e0 + P.ne;
        // edges of the patch's triangles that an earlier patch owns
        ring.clear();
        for (int k = 3 * P.t0; k < 3 * (P.t0 + P.nt); ++k) {
            const int e = in.tedge[k];
            if (e < P.e0 || e >= e1) ring.push_back(e);
        }
        std::sort(ring.begin(), ring.end());
        ring.erase(std::unique(ring.begin(), ring.end()), ring.end());
        P.nring = (int)ring.size();
        // its rows (free edges: owned, then ring), and the other edges their columns name
        edge.clear();
        for (int e = P.e0; e < e1; ++e) if (in.row[e] >= 0) edge.push_back(e);
        P.nown = (int)edge.size();
        for (int e : ring) if (in.row[e] >= 0) edge.push_back(e);
        P.nringrow = (int)edge.size() - P.nown;
        ext.clear();
        for (int e : edge)
            for (long long q = in.mrp[in.row[e]]; q < in.mrp[in.row[e] + 1]; ++q)
                if (in.mci[q] < P.e0 || in.mci[q] >= e1) ext.push_back(in.mci[q]);
        std::sort(ext.begin(), ext.end());
        ext.erase(std::unique(ext.begin(), ext.end()), ext.end());
        other.clear();
        std::set_difference(ext.begin(), ext.end(), ring.begin(), ring.end(), std::back_inserter(other));
        P.x0 = (int)S.xlist.size();
        P.nx = P.nring + (int)other.size();
        S.xlist.insert(S.xlist.end(), ring.begin(), ring.end());
        S.xlist.insert(S.xlist.end(), other.begin(), other.end());
        auto local = [&](int e) {
            if (e >= P.e0 && e < e1) return e - P.e0;
            auto it = std::lower_bound(ring.begin(), ring.end(), e);
            if (it != ring.end() && *it == e) return P.ne + (int)(it - ring.begin());
            return P.ne + P.nring + (int)(std::lower_bound(other.begin(), other.end(), e) - other.begin());
        };
        S.max_r = std::max(S.max_r, P.ne + P.nx);
        S.max_e = std::max(S.max_e, P.ne + P.nring);
        for (int f = P.t0; f < P.t0 + P.nt; ++f)
            for (int m = 0; m < 4; ++m) S.tloc.push_back(m < 3 ? (unsigned short)local(in.tedge[3 * f + m]) : 0);
        // rows in slices of 32, pairs of entries column-major; owned rows and ring rows in slices of their own
        P.row0 = (int)S.row_loc.size();
        P.slice0 = (int)S.soff.size() - 1;
        for (int part = 0; part < 2; ++part) {
            const int r0 = part ? P.nown : 0, r1 = part ? P.nown + P.nringrow : P.nown;
            for (int s0 = r0; s0 < r1; s0 += 32) {
                long long w = 0;
                for (int r = s0; r < std::min(r1, s0 + 32); ++r)
                    w = std::max(w, in.mrp[in.row[edge[r]] + 1] - in.mrp[in.row[edge[r]]]);
                w += w & 1;                 // entries in pairs; the added ones are 0
                const size_t base = S.col.size();
                S.col.resize(base + 32 * w, 0);
                S.val.resize(base + 32 * w, 0.0);
                for (int l = 0; l < 32; ++l) {
                    const int r = s0 + l;
                    S.row_loc.push_back(r < r1 ? (unsigned short)local(edge[r]) : 0);
                    if (r >= r1) continue;
                    const long long q0 = in.mrp[in.row[edge[r]]], n = in.mrp[in.row[edge[r]] + 1] - q0;
                    // (padding names the row's own edge: 0 times another's NaN is not 0)
                    for (long long k = n; k < w; ++k)
                        S.col[base + 64 * (k / 2) + 2 * l + (k & 1)] = S.row_loc.back();
                    for (long long k = 0; k < n; ++k) {
                        const size_t q = base + 64 * (k / 2) + 2 * l + (k & 1);
                        S.col[q] = (unsigned short)local(in.mci[q0 + k]);
                        S.val[q] = in.mv[q0 + k];
                    }
                }
                S.soff.push_back((long long)S.col.size() / 2);          // in pairs
            }
        }
        S.patch.push_back(P);
    }
}

}  // namespace

// Whole waves of three blocks per SM: a second, nearly empty wave costs as much
// as the first (a fine mesh of 329,672 triangles, us a step with the particles:
// 44.6 in one wave, 49.8 in one and a half).  One wave as long as its patches
// are of at most 850 triangles, then two: 231,200 triangles 30.7 in one and 33.0
// in two, 312,050 42.4 and 45.8, 364,658 49.6 and 52.6, 387,200 (patches of 850)
// 51.8 and 54.0, 410,418 (901) 57.2 and 56.3, 428,738 (941) 68.1 and 58.7.  The
// turn lies in the overlap with the particle kernels around it, not in the
// kernel: alone and cold it takes 39.0 us in one wave there and 43.5 in two, and
// no setting of the SM's shared memory moves it.  Two and three waves differ
// alike (720,000 triangles 91.9 and 97.8; 768,800, patches of 843, 96.3 and
// 101.1).  At least 64 triangles: smaller patches gain nothing on 2,048 triangles
// (6.77 with 48, 6.71 with 64, 6.88 with 96).
int field_patch_size(int F, int sms)
{
    constexpr int most = 850, least = 64;
    const long long slots = (long long)(sms > 0 ? sms : 1) * FIELD_PER_SM;
    const long long waves = ((long long)F + slots * most - 1) / (slots * most);
    const long long room = slots * (waves > 0 ? waves : 1);
    const long long T = (F + room - 1) / room;
    return (int)(T < least ? least : T);
}

// The patches recompute the curl on the edges around them and the rows of the
// ring, and pad the rows in slices of their own.  On a mesh whose storage order
// is compact that is little (the weighted sum below stays under 0.7 of the
// bound, also with small patches and high levels of the inverse, and the patches
// win throughout: 28,800 triangles, level 6, 12.9 us a step against 19.7).  Where it
// is not (many triangles in one cell of the curve, in no order), the separate
// kernels win, the sooner the larger the mesh.  Patches and separate kernels, us
// a step, by the weighted sum over the bound: 8,192 triangles, 0.80: 10.4 and
// 11.3; 20,000, 0.98: 10.7 and 11.4, 1.66: 14.8 and 11.5; 51,200, 1.07: 14.5 and
// 15.6, 1.88: 18.1 and 16.0; 200,978, 0.61: 20.8 and 24.0, 1.47: 31.9 and 24.9.
bool patches_pay(const PatchSet &S, long long edges, long long entries)
{
    const double extra = 4.0 * (double)S.xlist.size() + (double)S.val.size() - (double)entries;
    return extra <= 9e5 + 0.85 * (double)(edges + entries);
}

size_t field_smem(bool f32, int max_r, int max_e)
{
    return sizeof(double) * ((size_t)max_r + max_e) + (f32 ? sizeof(float) * (size_t)max_r : 0);
}

PatchSet build_patches(const PatchInput &in, int T)
{
    const int np = in.F > 0 ? (in.F + T - 1) / T : 0;
    // first edge of each patch: edges are numbered in the order the triangles touch them
    std::vector<int> own(np + 1, 0);
    int seen = 0;
    for (int f = 0; f < in.F; ++f) {
        if (f % T == 0) own[f / T] = seen;
        for (int m = 0; m < 3; ++m) seen = std::max(seen, in.tedge[3 * f + m] + 1);
    }
    own[np] = seen;
    const int nth = (int)std::max(1u, std::min({16u, std::thread::hardware_concurrency(), (unsigned)((np + 7) / 8)}));
    if (nth == 1) {
        PatchSet S;
        S.soff.assign(1, 0);
        S.T = T;
        build_range(S, in, own, T, 0, np);
        S.ok = np > 0 && S.max_r <= 65535;
        return S;
    }
    // no exception leaves a thread: it is thrown again here.  A thread that cannot be started is done without
    std::vector<PatchSet> part(nth);
    std::vector<std::exception_ptr> failed(nth);
    auto work = [&](int t) noexcept {
        try {
            part[t].soff.assign(1, 0);
            build_range(part[t], in, own, T, (int)((long long)np * t / nth), (int)((long long)np * (t + 1) / nth));
        } catch (...) {
            failed[t] = std::current_exception();
        }
    };
    {
        std::vector<std::thread> th;
        th.reserve(nth);
        try {
            while ((int)th.size() < nth - 1) th.emplace_back(work, (int)th.size());
        } catch (...) {
        }
        for (int t = (int)th.size(); t < nth; ++t) work(t);
        for (auto &t : th) t.join();
    }
    for (const std::exception_ptr &e : failed)
        if (e) std::rethrow_exception(e);
    PatchSet S;
    S.soff.assign(1, 0);
    S.T = T;
    size_t nv = 0, nx = 0, nrow = 0;
    for (const PatchSet &Q : part) { nv += Q.val.size(); nx += Q.xlist.size(); nrow += Q.row_loc.size(); }
    S.val.reserve(nv); S.col.reserve(nv); S.xlist.reserve(nx); S.row_loc.reserve(nrow); S.tloc.reserve(4 * (size_t)in.F);
    for (PatchSet &Q : part) {
        const int x = (int)S.xlist.size(), r = (int)S.row_loc.size(), s = (int)S.soff.size() - 1;
        const long long o = (long long)S.col.size() / 2;
        for (FieldPatch P : Q.patch) {
            P.x0 += x; P.row0 += r; P.slice0 += s;
            S.patch.push_back(P);
        }
        S.xlist.insert(S.xlist.end(), Q.xlist.begin(), Q.xlist.end());
        S.tloc.insert(S.tloc.end(), Q.tloc.begin(), Q.tloc.end());
        S.row_loc.insert(S.row_loc.end(), Q.row_loc.begin(), Q.row_loc.end());
        for (size_t k = 1; k < Q.soff.size(); ++k) S.soff.push_back(o + Q.soff[k]);
        S.col.insert(S.col.end(), Q.col.begin(), Q.col.end());
        S.val.insert(S.val.end(), Q.val.begin(), Q.val.end());
        S.max_r = std::max(S.max_r, Q.max_r);
        S.max_e = std::max(S.max_e, Q.max_e);
        Q = PatchSet();
    }
    S.ok = np > 0 && S.max_r <= 65535;
    return S;
}

}  // namespace fetdpic
