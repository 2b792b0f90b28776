// plan.cu -- host-side planning: padded geometry, tiling, interpolation tap
// tables grouped per tile, and the binomial checkpoint schedule.
#include <math.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "internal.h"

namespace wave {

Dims make_dims(const wave_grid_t& g)
{
    Dims d;
    d.ndim = g.ndim;
    d.nx = g.nx;
    d.ny = g.ndim == 3 ? g.ny : 1;
    d.nz = g.nz;
    d.nb = g.nb;
    d.nt = g.nt;
    d.Nx = g.nx + 2 * g.nb;
    d.Ny = g.ndim == 3 ? g.ny + 2 * g.nb : 1;
    d.Nz = g.nz + 2 * g.nb;
    d.P = (d.Nx + 31) / 32 * 32;
    d.cell = (long long)d.Nz * d.Ny * d.P;
    d.phys = (long long)d.nx * d.ny * d.nz;
    d.h = g.h;
    d.dt = g.dt;
    d.vref = g.vref;
    return d;
}

// Variants picked by wave_autotune, per (padded grid, shot count).
namespace {
std::mutex g_tuned_mu;
std::map<std::tuple<int, int, int>, std::pair<int, int>> g_tuned;
}  // namespace

void remember_tuning(const Dims& d, int nshot, int vf, int va)
{
    std::lock_guard<std::mutex> lock(g_tuned_mu);
    g_tuned[std::make_tuple(d.Nx, d.Nz, nshot)] = std::make_pair(vf, va);
}

// A CTA sets its tile up once and then takes its group's shots one after the
// other; 3 CTAs fit an SM.  Larger groups spread the set-up over more shots,
// smaller ones fill the GPU and shorten the chain: with groups of 4 throughout, 8
// shots of 592 x 336 (210 CTAs on 456 slots) ran at 10.7 / 14.6 us per step, with
// singly (840 CTAs) at 6.4 / 7.8 us.  Model of a step (us) with N CTAs: the chain
// of one CTA, a little longer with neighbours on the SM, or the GPU's rate over
// all of them, whichever is longer; 36 timings (592 x 336 with 1 to 32 shots, 1280 x
// 580 with 1 and 4, groups of 1, 2 and 4) lie within 10 % but for 24.5 and 32.6 us
// (predicted 21.7 and 27.5) at 32 shots singly.
int shot_group(const Dims& d, int nshot, bool adjoint, float* step_us)
{
    static const float kChain[2][3][2] = {{{4.6f, 0.0f}, {6.2f, 0.0021f}, {9.4f, 0.006f}},
                                          {{5.6f, 0.0019f}, {8.0f, 0.0035f}, {13.3f, 0.005f}}};
    static const float kRate[2][3][2] = {{{0.9f, 0.0062f}, {1.0f, 0.0104f}, {3.5f, 0.0172f}},
                                         {{1.3f, 0.0078f}, {1.5f, 0.0122f}, {5.5f, 0.0172f}}};
    const float tiles = (float)((d.Nx + kTX - 1) / kTX) * ((d.Nz + 15) / 16);
    int best = 4;
    float least = 0.0f;
    for (int k = nshot > 1 ? 2 : 1; k >= 0; --k) {
        const int g = 1 << k;
        const float n = tiles * ((nshot + g - 1) / g), *c = kChain[adjoint][k];
        const auto rate = [&](int j) { return kRate[adjoint][j][0] + kRate[adjoint][j][1] * n; };
        // a group larger than the batch is as long as the batch and does the work of a group of its size
        float chain = c[0], gpu = rate(k);
        if (nshot < g) {
            chain = kChain[adjoint][0][0] + (c[0] - kChain[adjoint][0][0]) * (nshot - 1) / (g - 1);
            gpu = nshot == 3 ? 0.5f * (rate(1) + rate(2)) : rate(nshot - 1);
        }
        const float t = std::max(chain + c[1] * n, gpu);
        if (least == 0.0f || t < least) {
            best = g;
            least = t;
        }
    }
    if (step_us) *step_us = least;
    return best;
}

Tiling choose_tiling(const Dims& d, int nshot)
{
    Tiling t;
    t.TX = kTX;
    t.vf = t.va = t.v3 = -1;
    if (d.ndim == 2) {
        t.TY = 1;
        t.TZc = kTZc2;
        t.vf = current_variant(0);
        t.va = current_variant(1);
        t.set_f = variant_forced(0);
        t.set_a = variant_forced(1);
        // an explicit wave_set_variant wins over a tuned choice
        std::lock_guard<std::mutex> lock(g_tuned_mu);
        auto it = g_tuned.find(std::make_tuple(d.Nx, d.Nz, nshot));
        if (it != g_tuned.end()) {
            if (!variant_forced(0)) t.vf = it->second.first;
            if (!variant_forced(1)) t.va = it->second.second;
            t.set_f = t.set_a = true;
        }
        if (nshot > 0) {
            if (!t.set_f) t.vf = group_variant(false, shot_group(d, nshot, false, nullptr));
            if (!t.set_a) t.va = group_variant(true, shot_group(d, nshot, true, nullptr));
        }
    } else {
        t.TY = 8;
        t.TZc = 4;  // divides every 3D variant's planes per CTA (32, 64, 76, 96)
        t.v3 = current_variant(2);
    }
    t.ncx = (d.Nx + t.TX - 1) / t.TX;
    t.ncy = (d.Ny + t.TY - 1) / t.TY;
    t.ncz = (d.Nz + t.TZc - 1) / t.TZc;
    return t;
}

int gradient_accumulators(const Tiling& t, int ndim, int nshot)
{
    if (ndim != 2) return nshot;
    const Variant2D v = variant_info(1, t.va);
    if (v.kind == 5) {
        const int ntz = (t.ncz * t.TZc + v.TZ - 1) / v.TZ;
        return persistent_slots(t.va, t.ncx, ntz, nshot);
    }
    return v.kind == 2 || v.kind == 4 || v.kind == 7 ? (nshot + v.G - 1) / v.G : nshot;
}

// Interpolation taps of one point: bilinear (2D) / trilinear (3D) weights on
// the padded grid, dropping taps of weight zero; x, y, z: their grid indices.
struct PointTap {
    int x, y, z;
    float w;
};

static bool point_taps(const Dims& d, const float* c, PointTap* tap, int* n)
{
    const int nax = d.ndim;
    const int nphys[3] = {d.nx, nax == 2 ? d.nz : d.ny, d.nz}, npad[3] = {d.Nx, nax == 2 ? d.Nz : d.Ny, d.Nz};
    int i0[3] = {0, 0, 0};
    double fr[3];
    const double h = d.h;
    for (int a = 0; a < nax; ++a) {
        const double x = c[a];
        if (!(x >= 0.0 && x <= (nphys[a] - 1) * h)) return false;  // also rejects NaN
        const double f = x / h + d.nb;
        int i = (int)f;  // f >= 0: the floor
        if (i > npad[a] - 2) i = npad[a] - 2;
        i0[a] = i;
        fr[a] = f - i;
    }
    int k = 0;
    for (int corner = 0; corner < (1 << nax); ++corner) {
        double ww = 1.0;
        int at[3] = {0, 0, 0};
        for (int a = 0; a < nax; ++a) {
            const int up = (corner >> a) & 1;
            at[a] = i0[a] + up;
            ww *= up ? fr[a] : 1.0 - fr[a];
        }
        if (ww == 0.0) continue;
        tap[k].x = at[0];
        tap[k].y = nax == 2 ? 0 : at[1];
        tap[k].z = nax == 2 ? at[1] : at[2];
        tap[k].w = (float)ww;
        ++k;
    }
    *n = k;
    return true;
}

wave_status_t build_taps(const Dims& d, const Tiling& t, int nshot, int npts, const float* xyz, bool count_only,
                         HostTaps& out)
{
    out = HostTaps();
    out.npts = npts;
    const long long cps = t.cells_per_shot();
    const long long npts_all = (long long)nshot * npts;
    out.npt_start = (size_t)npts_all + 1;
    PointTap tap[8];
    int n = 0;
    if (count_only) {
        for (long long pt = 0; pt < npts_all; ++pt) {
            if (!point_taps(d, xyz + pt * d.ndim, tap, &n)) return WAVE_ERR_GEOMETRY;
            out.ntap += n;
        }
        return WAVE_OK;
    }
    // the taps in point order, and how many each cell holds
    struct Item {
        int cell, idx, ab;
        float w;
    };
    std::vector<Item> item;
    item.reserve(npts_all * (d.ndim == 3 ? 2 : 4));
    out.pt_start.resize(npts_all + 1);
    out.cell_start.assign(nshot * cps + 1, 0);
    for (int s = 0; s < nshot; ++s) {
        for (int p = 0; p < npts; ++p) {
            const long long pt = (long long)s * npts + p;
            out.pt_start[pt] = (int)item.size();
            if (!point_taps(d, xyz + pt * d.ndim, tap, &n)) return WAVE_ERR_GEOMETRY;
            for (int k = 0; k < n; ++k) {
                // cells in (shot, cx, cy, cz) order with cz fastest
                const long long cell =
                    (((long long)s * t.ncx + tap[k].x / t.TX) * t.ncy + tap[k].y / t.TY) * t.ncz + tap[k].z / t.TZc;
                item.push_back({(int)cell, (int)(((long long)tap[k].z * d.Ny + tap[k].y) * d.P + tap[k].x),
                                (int)((long long)s * d.nt * npts + p), tap[k].w});
                ++out.cell_start[cell + 1];
            }
        }
    }
    out.pt_start[npts_all] = (int)item.size();
    const size_t ntap = out.ntap = item.size();
    // Stable counting sort of the taps by cell.
    for (long long i = 0; i < nshot * cps; ++i) out.cell_start[i + 1] += out.cell_start[i];
    std::vector<int> fill(out.cell_start.begin(), out.cell_start.end() - 1), order(ntap);
    for (size_t j = 0; j < ntap; ++j) order[fill[item[j].cell]++] = (int)j;
    // Inside a cell, taps of the same grid point become adjacent (stable by
    // point order), so one thread can own each injected point.
    const auto before = [&](int x, int y) { return item[x].idx < item[y].idx; };
    for (size_t b = 0; b < ntap;) {
        const size_t e = out.cell_start[item[order[b]].cell + 1];
        if (!std::is_sorted(order.begin() + b, order.begin() + e, before))
            std::stable_sort(order.begin() + b, order.begin() + e, before);
        b = e;
    }
    out.idx.resize(ntap);
    out.w.resize(ntap);
    out.ab.resize(ntap);
    out.slot.resize(ntap);
    for (size_t pos = 0; pos < ntap; ++pos) {
        const Item& it = item[order[pos]];
        out.idx[pos] = it.idx;
        out.w[pos] = it.w;
        out.ab[pos] = it.ab;
        out.slot[pos] = order[pos];
    }
    return WAVE_OK;
}

// ---------------------------------------------------------------------------
// Binomial checkpointing (after Griewank & Walther's optimal reversal with a
// fixed number of snapshots), written over "macro positions": the state at
// position p, S_j(p) = (u^j, u^{j-1}), serves the adjoint steps j and j - 1.
// Unlike a reversal that needs the state *before* each step, every adjoint
// pair here needs the state *at* its own position, so a snapshot serves its
// position directly.  rev(a, b, s) runs the adjoint pairs of positions
// b, b-1, ..., a (a only if a > 0) with the state at a restorable and s free
// slots.  Cost model (macro advances):
//   T(0, s) = 0,  T(l, 0) = l (l + 1) / 2,
//   T(l, s) = min_{1<=m<=l}  m + T(l - m, s - 1) + T(m - 1, s).
// The split cost is convex in m and its last minimiser grows with l, so each
// row is filled with a pointer that only moves forward.  With s >= l this is a
// single sweep.  Among equally cheap splits the last leaves the longest stretches
// between saves, so forward and adjoint steps alternate less often (nt = 2000, 64
// slots: 36 runs of steps of one kind, 88 with the first minimiser; nt = 4000, 1536
// slots: 4 and 62), and each run of the on-chip loop loads its state once.
namespace {

struct CostTable {
    int L = 0, S = 0;
    std::vector<std::vector<long long>> T;
    std::vector<std::vector<int>> opt;
};

CostTable build_costs(int L, int S)
{
    CostTable c;
    c.L = L;
    c.S = S;
    c.T.assign(S + 1, std::vector<long long>(L + 1, 0));
    c.opt.assign(S + 1, std::vector<int>(L + 1, 0));
    for (int l = 0; l <= L; ++l) c.T[0][l] = (long long)l * (l + 1) / 2;
    for (int s = 1; s <= S; ++s) {
        int m = 1;
        for (int l = 1; l <= L; ++l) {
            if (m > l) m = l;
            auto f = [&](int mm) { return mm + c.T[s - 1][l - mm] + c.T[s][mm - 1]; };
            while (m + 1 <= l && f(m + 1) <= f(m)) ++m;
            c.T[s][l] = f(m);
            c.opt[s][l] = m;
        }
    }
    return c;
}

struct Emitter {
    const CostTable& c;
    Schedule& sch;
    int at = 0;                   // macro position held by the working state
    std::vector<int> slot_of;     // slot holding the state of a macro position (-1: none)
    std::vector<int> free_slots;
    bool finalized = false;

    void ensure_at(int a)
    {
        if (at == a) return;
        const int slot = a == 0 ? -1 : slot_of[a];
        sch.actions.push_back({kRestore, slot, a});
        at = a;
    }
    void advance(int a, int b)
    {
        sch.actions.push_back({kAdvance, a, b});
        sch.advances += b - a;
        sch.fwd_steps += sch.state_of(b) - sch.state_of(a);
        at = b;
    }
    void adjoint_pair(int p)
    {
        if (!finalized) {
            sch.actions.push_back({kFinalize, 0, 0});
            finalized = true;
        }
        sch.actions.push_back({kAdjointPair, p, p});
    }
    void rev(int a, int b, int s)
    {
        const int l = b - a;
        if (l == 0) {
            if (a > 0) {
                ensure_at(a);
                adjoint_pair(a);
            }
            return;
        }
        if (s == 0) {
            for (int p = b; p >= a && p > 0; --p) {
                ensure_at(a);
                if (p > a) advance(a, p);
                adjoint_pair(p);
            }
            return;
        }
        const int m = c.opt[std::min(s, c.S)][l];
        const int cpos = a + m;
        ensure_at(a);
        advance(a, cpos);
        const int slot = free_slots.back();
        free_slots.pop_back();
        sch.actions.push_back({kSave, slot, cpos});
        slot_of[cpos] = slot;
        rev(cpos, b, s - 1);
        slot_of[cpos] = -1;
        free_slots.push_back(slot);
        rev(a, cpos - 1, s);
    }
};

}  // namespace

Schedule make_schedule(int nt, int nsnap)
{
    Schedule sch;
    sch.K = nt - 1;
    if (sch.K < 1) return sch;
    sch.jmin = (sch.K % 2 == 1) ? 1 : 2;
    sch.L = (sch.K - sch.jmin) / 2 + 1;
    const int S = std::max(0, std::min(nsnap, sch.L));
    sch.nsnap = S;
    static std::mutex mu;
    static std::map<std::pair<int, int>, CostTable> cache;
    std::lock_guard<std::mutex> lock(mu);  // held while the cached table is in use
    auto key = std::make_pair(sch.L, S);
    auto it = cache.find(key);
    if (it == cache.end()) {
        if (cache.size() > 16) cache.clear();
        it = cache.emplace(key, build_costs(sch.L, S)).first;
    }
    Emitter e{it->second, sch};
    e.slot_of.assign(sch.L + 1, -1);
    for (int i = S - 1; i >= 0; --i) e.free_slots.push_back(i);
    e.rev(0, sch.L, S);
    return sch;
}

}  // namespace wave

extern "C" int wave_shot_group(const wave_grid_t* g, int nshot, int adjoint, float* step_us)
{
    return wave::shot_group(wave::make_dims(*g), nshot, adjoint != 0, step_us);
}
