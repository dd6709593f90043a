// Checks that chain-mode dependencies (derive_fused_deps in fused_deps.h) order every pair of
// products of a launch that touch the same memory.
//
// In chain mode a product's tiles wait for whole earlier products and for nothing else, so any
// product may lag behind all that do not wait for it, however unlikely that is on a given
// machine. The check is therefore exact instead of a simulation: from the derived conditions it
// takes the set of products that are complete when one starts (transitively), and requires
// every earlier product to be in it that writes what this one reads, reads or writes what this
// one writes, or accumulates the norm that this one's scales come from.
//
// The lists are those of a solve (both polar chains, each option that changes the products),
// whole, and cut at every stage into windows as serving cuts them.
//
// Usage: chain_order_check; prints "<n> launches, <n> failures", exit status 0 without failures.
#include <cstdio>
#include <set>
#include <vector>

#include "fused_deps.h"

using svt::DepProduct;
using svt::DepResult;

namespace {

int launches = 0, failures = 0;

// Addresses of the solve's buffers and norms (never read through).
enum Buf { X0, X1, Xt0, Xt1, S0, S1, Yp, Zp, Ys, Zs, ZPp, ZSp, B, Sp, Yp8, S80, S81, Ys8, Zs8, BUFS };
char mem[BUFS];
double norms[4];
enum Norm { NS0, NYP, NYS, NOUT };

struct Options {
    int steps;
    bool skip_p;   // Corollary 1's mode
    bool gram;     // first step scaled by the norm of its Y
    bool quintic;  // five-term steps; else cubic ones (after a first one with `gram`)
    bool polish;
    bool copies;   // e4m3 copies beside the outputs
};

DepProduct product(int l, int r, int c, int o, int t, int sym, int chain, int theta, int norm,
                   int f = -1)
{
    auto at = [](int b) -> const void * { return b < 0 ? nullptr : &mem[b]; };
    auto nrm = [](int n) -> const double * { return n < 0 ? nullptr : &norms[n]; };
    return {at(l), at(r), at(c), at(o), at(t), 0, sym, chain, 2, 2, 3, nrm(theta), nrm(norm), at(f)};
}

// One stage (the products of one launch of the unfused solve) after another.
std::vector<std::vector<DepProduct>> solve(const Options &q)
{
    std::vector<std::vector<DepProduct>> st;
    st.push_back({product(Xt0, Xt0, -1, S0, -1, 1, 1, -1, NS0)});
    const int X[2] = {X0, X1}, Xt[2] = {Xt0, Xt1}, S[2] = {S0, S1}, S8[2] = {S80, S81};
    int cur = 0;
    for (int s = 0; s < q.steps; ++s, cur = 1 - cur) {
        const bool first = s == 0, five = q.quintic || (first && q.gram);
        const int np = first && q.gram ? NYP : -1, ns = first && q.gram ? NYS : -1;
        const int ts = first ? (q.gram ? NYS : NS0) : -1;
        const int c = q.copies ? 1 : 0;
        std::vector<DepProduct> a, b, d;
        if (five) {
            if (!q.skip_p)
                a.push_back(product(Xt[cur], Xt[cur], -1, Yp, -1, 1, 0, -1, np, c ? Yp8 : -1));
            a.push_back(product(S[cur], S[cur], -1, Ys, -1, 1, 1, -1, ns, c ? Ys8 : -1));
            if (!q.skip_p)
                b.push_back(product(c ? Yp8 : Yp, c ? Yp8 : Yp, Yp, Zp, -1, 1, 0, np, -1));
            b.push_back(product(c ? Ys8 : Ys, c ? Ys8 : Ys, Ys, Zs, -1, 1, 1, ts, -1, c ? Zs8 : -1));
        } else {
            if (!q.skip_p)
                a.push_back(product(Xt[cur], Xt[cur], -1, Zp, -1, 1, 0, -1, -1));
            a.push_back(product(S[cur], S[cur], -1, Zs, -1, 1, 1, ts, -1));
        }
        if (!q.skip_p)
            d.push_back(product(X[cur], Zp, -1, X[1 - cur], Xt[1 - cur], 0, 0, -1, -1));
        d.push_back(product(c && s ? S8[cur] : S[cur], c && s ? Zs8 : Zs, -1, S[1 - cur], -1, 1, 1, -1,
                            -1, c ? S8[1 - cur] : -1));
        st.push_back(a);
        if (!b.empty())
            st.push_back(b);
        st.push_back(d);
    }
    if (q.polish) {
        std::vector<DepProduct> a, b;
        if (!q.skip_p) {
            a.push_back(product(Xt[cur], Xt[cur], -1, ZPp, -1, 1, 0, -1, -1));
            b.push_back(product(X[cur], ZPp, -1, B, -1, 0, 0, -1, -1));
        }
        a.push_back(product(S[cur], S[cur], -1, ZSp, -1, 1, 1, -1, -1));
        b.push_back(product(S[cur], ZSp, -1, Sp, -1, 1, 1, -1, -1));
        st.push_back(a);
        st.push_back(b);
        st.push_back({product(B, Sp, B, -1, -1, 0, 2, -1, NOUT)});
    }
    return st;
}

bool touches(const void *p, const DepProduct &q, bool write)
{
    if (!p)
        return false;
    return write ? p == q.o || p == q.t || p == q.f : p == q.l || p == q.r || p == q.c;
}

void check(const std::vector<DepProduct> &ps)
{
    ++launches;
    std::vector<DepResult> d;
    if (!svt::derive_fused_deps(ps, false, 8, 8, 0, d)) {
        std::printf("FAIL: refused\n");
        ++failures;
        return;
    }
    std::vector<std::set<int>> done(ps.size());
    for (int j = 0; j < (int)ps.size(); ++j) {
        for (int k = 0; k < 2; ++k) {
            const int i = d[j].dep[k];
            if (i < 0)
                continue;
            if (i >= j || d[j].dep_target[k] != 8 * ps[i].valid) {
                std::printf("FAIL: product %d waits for %d (of %d)\n", j, i, d[j].dep_target[k]);
                ++failures;
                continue;
            }
            done[j].insert(i);
            done[j].insert(done[i].begin(), done[i].end());
        }
        for (int i = 0; i < j; ++i) {
            bool clash = ps[j].theta_src && ps[j].theta_src == ps[i].norm_acc;
            for (const void *b : {ps[i].o, ps[i].t, ps[i].f})
                clash = clash || touches(b, ps[j], false) || touches(b, ps[j], true);
            for (const void *b : {ps[i].l, ps[i].r, ps[i].c})
                clash = clash || touches(b, ps[j], true);
            if (clash && !done[j].count(i)) {
                if (failures < 10)
                    std::printf("FAIL: of %d products, %d may run beside %d\n", (int)ps.size(), j, i);
                ++failures;
            }
        }
    }
}

} // namespace

int main()
{
    for (int steps : {0, 1, 2, 3, 6})
        for (int bits = 0; bits < 32; ++bits) {
            const Options q{steps, (bits & 1) != 0, (bits & 2) != 0, (bits & 4) != 0,
                            (bits & 8) != 0, (bits & 16) != 0};
            if (q.copies && !q.quintic)
                continue;
            const auto st = solve(q);
            for (size_t a = 0; a < st.size(); ++a)
                for (size_t b = a + 1; b <= st.size(); ++b) {
                    std::vector<DepProduct> ps;
                    for (size_t k = a; k < b; ++k)
                        ps.insert(ps.end(), st[k].begin(), st[k].end());
                    check(ps);
                }
        }
    std::printf("%d launches, %d failures\n", launches, failures);
    return failures ? 1 : 0;
}
