// Patch tables of the field update on the host: against the mesh and the matrix they are made from, and
// with allocations that fail.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <random>

#include "fetdpic_internal.h"

using namespace fetdpic;

static std::atomic<long long> countdown{-1};
void *operator new(std::size_t n)
{
    if (countdown.load() >= 0 && countdown.fetch_sub(1) == 0) throw std::bad_alloc();
    if (void *p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }

struct Input {
    HostMesh M;
    std::vector<int> te, row, mci;
    std::vector<long long> mrp;
    std::vector<double> mv;
    PatchInput in() const { return {M.nf, te.data(), row.data(), mrp.data(), mci.data(), mv.data()}; }
};

// A jittered rectangle; scattered: its triangles in no order, within one cell of the space-filling curve.
static bool make(Input &I, int nx, int ny, int level, bool scattered)
{
    std::mt19937 g(3);
    std::uniform_real_distribution<double> U(-0.2, 0.2);
    const double h = scattered ? 1e-11 : 1.0;
    std::vector<double> xy;
    std::vector<int> t;
    for (int j = 0; j <= ny; ++j)
        for (int i = 0; i <= nx; ++i) {
            xy.push_back((i + (i > 0 && i < nx ? U(g) : 0.0)) * h);
            xy.push_back((j + (j > 0 && j < ny ? U(g) : 0.0)) * h);
        }
    std::vector<int> cells(nx * ny);
    for (int k = 0; k < nx * ny; ++k) cells[k] = k;
    if (scattered) std::shuffle(cells.begin(), cells.end(), g);
    for (int k : cells) {
        const int a = k / nx * (nx + 1) + k % nx, c = a + nx + 1;
        for (int n : {a, a + 1, c + 1, a, c + 1, c}) t.push_back(n);
    }
    if (scattered) {
        const int n = (int)xy.size() / 2;
        for (double v : {1e3, 1e3, 1001.0, 1e3, 1001.0, 1001.0}) xy.push_back(v);
        for (int k = 0; k < 3; ++k) t.push_back(n + k);
    }
    std::string msg;
    HostMesh &M = I.M;
    if (build_mesh(M, (int)xy.size() / 2, xy.data(), (int)t.size() / 3, t.data(), 0, nullptr, nullptr, 0, nullptr, 0, 0, msg) ||
        build_hodge(M, 1.0, msg) || build_spai(M, level, msg))
        return false;
    for (int e : M.tedge) I.te.push_back(M.einv[e]);
    std::vector<int> free_of(M.ne, -1);
    for (size_t a = 0; a < M.free_edges.size(); ++a) free_of[M.free_edges[a]] = (int)a;
    I.row.assign(M.ne, -1);
    I.mrp.assign(1, 0);
    for (int i = 0; i < M.ne; ++i) {
        const int a = free_of[M.eperm[i]];
        if (a < 0) continue;
        I.row[i] = (int)I.mrp.size() - 1;
        for (long long q = M.m_rp[a]; q < M.m_rp[a + 1]; ++q) { I.mci.push_back(M.einv[M.m_ci[q]]); I.mv.push_back(M.m_v[q]); }
        I.mrp.push_back((long long)I.mci.size());
    }
    return true;
}

// Every table entry against the mesh; every index within its range.
static const char *check(const Input &I, const PatchSet &S)
{
    const int F = I.M.nf, E = I.M.ne;
    std::vector<int> tri(F, 0), edge(E, 0), rows(E, 0);
    for (const FieldPatch &P : S.patch) {
        const int nr = P.ne + P.nx;
        if (P.nt < 1 || P.nt > S.T || nr > S.max_r || P.ne + P.nring > S.max_e || P.nring > P.nx) return "patch sizes";
        if (P.x0 + P.nx > (int)S.xlist.size()) return "xlist range";
        auto global = [&](int l) { return l < P.ne ? P.e0 + l : S.xlist[P.x0 + l - P.ne]; };
        for (int k = 0; k < P.ne; ++k) ++edge[P.e0 + k];
        for (int f = P.t0; f < P.t0 + P.nt; ++f) {
            ++tri[f];
            for (int m = 0; m < 3; ++m) {
                const int l = S.tloc[4 * (size_t)f + m];
                if (l >= P.ne + P.nring || global(l) != I.te[3 * f + m]) return "triangle's edge";
            }
        }
        const int no = (P.nown + 31) / 32, ns = no + (P.nringrow + 31) / 32;
        for (int sl = 0; sl < ns; ++sl)
            for (int lane = 0; lane < 32; ++lane) {
                if (P.row0 + sl * 32 + lane >= (int)S.row_loc.size() || P.slice0 + sl + 1 >= (int)S.soff.size()) return "row range";
                const int loc = S.row_loc[P.row0 + sl * 32 + lane];
                if (loc >= P.ne + P.nring) return "row";
                const bool valid = sl < no ? sl * 32 + lane < P.nown : (sl - no) * 32 + lane < P.nringrow;
                const long long o0 = S.soff[P.slice0 + sl], o1 = S.soff[P.slice0 + sl + 1];
                if (2 * o1 > (long long)S.col.size() || (o1 - o0) % 32) return "slice range";
                const int e = global(loc), r = I.row[e];
                if (valid && r < 0) return "row of no free edge";
                if (valid && sl < no) { if (loc >= P.ne) return "owned row"; ++rows[e]; }
                long long q = valid ? I.mrp[r] : 0;
                const long long q1 = valid ? I.mrp[r + 1] : 0;
                for (long long o = o0 + lane; o < o1; o += 32)
                    for (int k = 0; k < 2; ++k) {
                        const int c = S.col[2 * o + k];
                        const double v = S.val[2 * o + k];
                        if (c >= nr) return "column range";
                        if (q < q1) { if (global(c) != I.mci[q] || v != I.mv[q]) return "entry"; ++q; }
                        else if (v != 0.0) return "padding";
                    }
                if (q != q1) return "entries missing";
            }
    }
    for (int f = 0; f < F; ++f) if (tri[f] != 1) return "triangles covered once";
    for (int e = 0; e < E; ++e) if (edge[e] != 1 || rows[e] != (I.row[e] >= 0)) return "edges covered once";
    return nullptr;
}

int main()
{
    struct { int nx, ny, level; bool scattered; } shapes[] = {{1, 1, 1, false}, {7, 5, 2, false}, {60, 3, 3, false}, {90, 80, 2, false}, {50, 50, 3, true}};
    for (auto &s : shapes) {
        Input I;
        if (!make(I, s.nx, s.ny, s.level, s.scattered)) { printf("no mesh\n"); return 1; }
        for (int T : {1, 64, 129, 704, 1900, 40000}) {
            const PatchSet S = build_patches(I.in(), T);
            const char *bad = S.ok ? check(I, S) : "no tables";
            if (bad) { printf("%d x %d, level %d, T %d: %s\n", s.nx, s.ny, s.level, T, bad); return 1; }
        }
    }
    // worth their while on compact meshes of any level, not on large ones in no order
    struct { int nx, ny, level; bool scattered, pay; } uses[] = {{1, 1, 1, false, true}, {60, 3, 3, false, true}, {90, 80, 1, false, true}, {120, 120, 2, false, true},
                                                                 {50, 50, 6, false, true}, {20, 20, 2, true, true}, {160, 160, 2, true, false}, {64, 64, 4, true, false}};
    for (auto &u : uses) {
        Input I;
        if (!make(I, u.nx, u.ny, u.level, u.scattered)) return 1;
        const PatchSet S = build_patches(I.in(), field_patch_size(I.M.nf, 152));
        if (patches_pay(S, I.M.ne, (long long)I.mci.size()) != u.pay) { printf("%d x %d, level %d: pay\n", u.nx, u.ny, u.level); return 1; }
    }
    // an allocation that fails, in a thread or not, arrives as an exception
    Input I;
    if (!make(I, 90, 80, 2, false)) return 1;
    int thrown = 0;
    for (long long n = 0; n < 1200; n += n < 60 ? 1 : 37) {
        countdown = n;
        try {
            build_patches(I.in(), 64);
        } catch (const std::bad_alloc &) {
            ++thrown;
        }
        countdown = -1;
    }
    printf("thrown %d\n", thrown);
    return thrown < 20;
}
