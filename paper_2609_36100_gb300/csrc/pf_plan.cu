// Axis plans (radix schedules and division magic) and the x-pass CTA count.
#include <vector>

#include "pf_xpass.cuh"

namespace pf {
int compiled_plan_len(int pid) { return fixed_plan_len(pid); }
int compiled_plan_count() { return kFixedPlans; }

// Form of the FP32 elastic pass that is run untuned (pf_internal.h lists
// them).  The stages over three fields are the fastest single-CTA form (us a
// launch against the fused one: 14.6 / 18.6 at 96, 23.1 / 24.7 at 128, 51.7 /
// 53.7 at 160, 165 / 229 at 256) except where a radix-16 first stage meets a
// last radix of at most 4, which the fused form holds in few registers (8.7 /
// 9.9 at 64 = 16 4, 82 / 89 at 192 = 16 4 3).  A three-field tile of 8 columns no
// longer fits beside another one above 512 points: the cluster form
// (3.1 / 6.2 ms at 640).
template <int PID = 1>
static int elastic_form(int pid) {
    if constexpr (PID > kFixedPlans) {
        return 0;
    } else {
        if (pid != PID) return elastic_form<PID + 1>(pid);
        using Rad = typename FixedPlan<PID>::Rad;
        if (RadInfo<Rad>::count < 2) return 0;
        if (FixedPlan<PID>::N > 512) return 2;
        return RadInfo<Rad>::first == 16 && RadInfo<Rad>::last <= 4 ? 0 : 1;
    }
}
int default_elastic_form(const AxisPlan& pz) { return elastic_form(fixed_plan_id(pz)); }

// plan of the cluster form: one of those it is compiled for
template <int PID = 1>
static int cluster_plan(int n) {
    if constexpr (PID > kBothWidths)
        return 0;
    else
        return FixedPlan<PID>::N == n ? PID : cluster_plan<PID + 1>(n);
}
int default_elastic_plan(const AxisPlan& pz) { return default_elastic_form(pz) == 2 ? cluster_plan(pz.n) : 0; }

// plan from an explicit radix order (each radix in {2,3,4,5,6,8,9,10,12,15,16}, product n)
bool make_axis_plan_radices(int n, const int* rad, int nr, AxisPlan& p) {
    if (nr < 1 || nr > kMaxRadices) return false;
    long long prod = 1;
    for (int s = 0; s < nr; ++s) {
        if (rad[s] < 2 || rad[s] > 16 || rad[s] == 7 || rad[s] == 11 || rad[s] == 13 || rad[s] == 14) return false;
        prod *= rad[s];
    }
    if (prod != n) return false;
    p.n = n;
    p.nst = nr;
    p.has16 = 0;
    for (int s = 0; s < nr; ++s)
        if (rad[s] > 8) p.has16 = 1;
    unsigned Ns = 1;
    for (int s = 0; s < nr; ++s) {
        p.rad[s] = rad[s];
        p.mulm[s] = magic_u32((unsigned)(n / rad[s]));
        p.mulN[s] = magic_u32(Ns);
        Ns *= (unsigned)rad[s];
    }
    return true;
}

namespace {
// arithmetic instructions per point of a radix-R stage, with twiddles and as
// the first stage (in tenths)
int stage_cost(int r, bool first) {
    switch (r) {
        case 2: return first ? 20 : 31;  // behind 4 4 in the place of 8 2
        case 3: return first ? 40 : 67;
        case 4: return first ? 40 : 60;
        case 5: return first ? 64 : 96;
        case 6: return first ? 60 : 93;
        case 8: return first ? 70 : 90;
        case 9: return first ? 98 : 133;
        case 10: return first ? 84 : 120;
        case 12: return first ? 80 : 117;
        case 15: return first ? 104 : 141;
        default: return first ? 101 : 120;  // behind 8 8 at 64 and 8 4 at 32
    }
}

// descending radix lists of product n: the fewest stages, of those the
// cheapest, of those the largest first radix; or the cheapest, of those the
// fewest stages (by_cost)
void best_order(int n, int limit, bool by_cost, std::vector<int>& cur, int cost, std::vector<int>& best,
                int& best_cost) {
    if (n == 1) {
        const int ns = (int)cur.size(), nb = (int)best.size();
        const bool better = by_cost ? cost < best_cost || (cost == best_cost && ns < nb)
                                    : ns < nb || (ns == nb && cost < best_cost);
        if (best.empty() || better) {
            best = cur;
            best_cost = cost;
        }
        return;
    }
    if (!by_cost && !best.empty() && cur.size() >= best.size()) return;
    for (int r : {16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2}) {
        if (r > limit || n % r) continue;
        cur.push_back(r);
        best_order(n / r, r, by_cost, cur, cost + stage_cost(r, cur.size() == 1), best, best_cost);
        cur.pop_back();
    }
}
}  // namespace

// default schedule.  FP32 (prefer16): the fewest stages, since a stage is a
// trip through shared memory and a barrier, of those the fewest instructions.
// FP64 passes take the time of their FP64 instructions: the fewest of those,
// with radices of at most 12 (wider ones spill).  Lines of up to 48 points in
// both precisions at most radix 8, so that a tile still gives work to a few
// warps (FP32, 30 points: radix 15 left one half-warp of it busy; FP64 step of
// a cube, ms: 30 = 10 3 1.20 and 6 5 0.96, 36 = 12 3 1.61 and 6 6 1.28, 40 = 10 4
// 1.66 and 5 4 2 1.31, 48 = 12 4 1.66 and 6 4 2 1.40).
bool make_axis_plan(int n, AxisPlan& p, bool prefer16) {
    int m = n;
    for (int q : {2, 3, 5})
        while (m % q == 0) m /= q;
    if (n < 2 || m != 1) return false;
    std::vector<int> cur, best;
    int cost = 0;
    best_order(n, n <= 48 ? 8 : (prefer16 ? 16 : 12), !prefer16, cur, 0, best, cost);
    return make_axis_plan_radices(n, best.data(), (int)best.size(), p);
}

int x_pass_blocks(const Geo& g, int f64) {
    const int P = f64 ? x_rows<double>(g) : x_rows<float>(g);
    const int npairs = g.nz * g.ny / 2;
    return (npairs + P - 1) / P;
}

}  // namespace pf
