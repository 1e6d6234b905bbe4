// Host-side check of the routes a solve can take (engine.cpp), built with the system C++ compiler: memory
// is the host's and the kernel table records launches.  One launch for a whole solve, passes throughout,
// passes with the last corrections in one launch, and the wide reductions of levels with few chunks.
// Prints "OK" and exits 0, or the first failed check and exits 1.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <string>
#include <vector>

#include "engine.h"

using namespace mhe;

namespace {

std::vector<std::string> g_log;
int g_cluster = 0, g_resume_cluster = 0;           // what the shape's rules answer
int g_asked_mhe = -1, g_asked_batch = 0, g_asked_N = 0;
int g_solve_resume = -1, g_solve_cluster = 0, g_solve_nlev = 0, g_solve_fused = -1;

#define CHECK(cond)                                            \
    do {                                                       \
        if (!(cond)) {                                         \
            printf("FAIL line %d: %s\n", __LINE__, #cond);     \
            exit(1);                                           \
        }                                                      \
    } while (0)

void* f_alloc(size_t b) { return calloc(1, b ? b : 1); }
void f_release(void* p) { free(p); }
int f_memset0(void* p, size_t b, void*) { memset(p, 0, b); return 0; }
int f_copy(void* d, const void* s, size_t b, void*) { memmove(d, s, b); return 0; }
int f_sync(void*) { return 0; }
int f_error() { return 0; }
void f_convert(float* d, const double* s, long long n, void*) { for (long long i = 0; i < n; ++i) d[i] = (float)s[i]; }
void f_widen(double* d, const float* s, long long n, void*) { for (long long i = 0; i < n; ++i) d[i] = (double)s[i]; }
void f_finalize(int batch, const unsigned long long*, const unsigned int*, int* active, int*, const int*, const int*,
                double, int mode, int, mhe_info*, int* any, unsigned int*, void*)
{
    g_log.push_back("finalize");
    if (mode <= 1) {
        for (int b = 0; b < batch; ++b) active[b] = 1;   // nothing converges
        if (any) *any = 1;
    }
}
const Runtime kFake = {f_alloc, f_release, f_memset0, f_copy, f_finalize, f_convert, f_sync, f_error, nullptr, f_widen};

template <typename T>
void red(const LevelArgs<T>&, int, void*) { g_log.push_back("reduce"); }
template <typename T>
void redw(const LevelArgs<T>&, int, void*) { g_log.push_back("reduce_wide"); }
template <typename T>
void rhs(const LevelArgs<T>&, int, void*) { g_log.push_back("rhs"); }
template <typename T>
void down(const LevelArgs<T>&, int, void*) { g_log.push_back("down"); }
template <typename T>
void resid(const ResidArgs<T>&, void*) { g_log.push_back("resid"); }
void knorm(const KnormArgs&, void*) {}
template <typename T>
void solve(const SolveArgs<T>& p, void*)
{
    g_log.push_back("solve");
    g_solve_resume = p.resume; g_solve_cluster = p.cluster; g_solve_nlev = p.nlev; g_solve_fused = p.fused_rhs;
    for (int b = 0; b < p.batch; ++b) p.active[b] = 0;
}
int cluster(int, int mhe, int batch, int N)
{
    g_asked_mhe = mhe; g_asked_batch = batch; g_asked_N = N;
    return g_cluster;
}
int resume(int, int mhe, int batch, int N)
{
    g_asked_mhe = mhe; g_asked_batch = batch; g_asked_N = N;
    return g_resume_cluster;
}

ShapeOps ops()
{
    ShapeOps o;
    memset(&o, 0, sizeof(o));
    o.nx = 4; o.nw = 2; o.ny = 2;
    o.reduce64 = red<double>; o.rhs64 = rhs<double>; o.down64 = down<double>; o.resid64 = resid<double>;
    o.reduce32 = red<float>; o.rhs32 = rhs<float>; o.down32 = down<float>; o.resid32 = resid<float>;
    o.knorm = knorm;
    o.reduce64w = redw<double>; o.reduce32w = redw<float>;
    o.wide64 = 12; o.wide32 = 5;
    o.solve64 = solve<double>; o.solve32 = solve<float>; o.solve_mhe32 = solve<float>;
    o.solve_cluster = cluster; o.resume_cluster = resume;
    return o;
}

int count(const char* op)
{
    int n = 0;
    for (const std::string& s : g_log) n += s == op;
    return n;
}

// factor and solve of two instances with `corrections` allowed; what was launched is in g_log
size_t run(int prec, int corrections, int cl, int resumed)
{
    std::vector<int> N = {41, 9};
    const long long S = 48, X = 52, W = 2 * 4 + 48 * 2;
    std::vector<double> A(S * 16), B(S * 8), Q(S * 36), P0(32), l(S * 6), a(S * 4), x0(8), x(X * 4), w(W), lam(X * 4);
    std::vector<mhe_info> info(2);
    mhe_dims d;
    memset(&d, 0, sizeof(d));
    d.nx = 4; d.nw = 2; d.batch = 2; d.N = N.data();
    d.prec = (mhe_precision)prec;
    d.leaf_len = 4; d.branching = 2; d.top_len = 2;
    d.refine_tol = 1e-12; d.max_refine = corrections;
    const ShapeOps o = ops();
    Engine e;
    CHECK(e.init(d, &o, &kFake, nullptr) == MHE_OK);
    g_log.clear();
    g_cluster = cl; g_resume_cluster = resumed; g_solve_resume = -1;
    mhe_matrices m = {A.data(), B.data(), Q.data(), P0.data()};
    mhe_rhs r = {l.data(), a.data(), x0.data()};
    CHECK(e.factor(m, nullptr, nullptr, nullptr, nullptr) == MHE_OK);
    CHECK(e.solve(&r, x.data(), w.data(), lam.data(), info.data(), false) == MHE_OK);
    const size_t L = e.plan.levels.size();
    e.release();
    return L;
}

}  // namespace

int main()
{
    for (int prec : {(int)MHE_FP64, (int)MHE_FP32_IR}) {
        // the whole solve in one launch
        size_t L = run(prec, 9, 4, 2);
        CHECK(count("solve") == 1 && g_solve_resume == 0 && g_solve_cluster == 4 && g_solve_nlev == (int)L);
        CHECK(count("rhs") == 0 && count("down") == 0 && count("resid") == 0 && count("finalize") == 0);
        CHECK(g_asked_batch == 2 && g_asked_N == 41 && g_asked_mhe == 0);
        // four corrections by passes, the fifth and the rest in one launch of the resumed cluster
        L = run(prec, 9, 0, 2);
        CHECK(count("solve") == 1 && g_solve_resume == 1 && g_solve_cluster == 2 && g_solve_fused == 0);
        CHECK(count("rhs") == 5 * (int)L && count("down") == 5 * (int)L);
        CHECK(count("resid") == 5 && count("finalize") == 6);
        // the shape's rule says no: passes to the end, and a residual of the last iterate
        L = run(prec, 9, 0, 0);
        CHECK(count("solve") == 0 && count("rhs") == 10 * (int)L && count("down") == 10 * (int)L);
        CHECK(count("resid") == 10 && count("finalize") == 10);
        // four corrections allowed: nothing is left to resume
        L = run(prec, 4, 0, 2);
        CHECK(count("solve") == 0 && count("resid") == 5 && count("rhs") == 5 * (int)L);
        // levels of at most `wide` chunks (13 at level 0, then 7, ...) take the wider reduction
        CHECK(count("reduce") == (prec == MHE_FP64 ? 1 : 2) && count("reduce_wide") == (int)L - count("reduce"));
    }
    printf("OK\n");
    return 0;
}
