// step2d_chip.cu -- many 2D time steps in one launch, the wavefield kept on chip.
//
// A thread-block cluster of C CTAs owns one shot: CTA r holds the rows
// [z0[r], z0[r+1]) of the padded grid, its two time levels in shared memory
// (each with a 4-row halo above and below).  A step reads u^n from one level,
// writes u^{n+1} over u^{n-1} in the other and sends its outermost 4 rows to
// the neighbours' halos through distributed shared memory, counted on their
// mbarriers; global memory sees only what leaves the loop: gather slots, stored
// levels, and in the adjoint the forward level it reads for the imaging
// condition.  A cluster barrier per step would wait for the step's global stores
// to reach L2; the mbarriers wait for the halo rows alone.  A CTA overwrites a
// neighbour's halo of u^{n-1} only after it has received that neighbour's border
// rows of u^n, which were computed from that halo.
//
// A thread marches down (or up) one quad column (4 x points) of its rows with
// the 9-row z window in registers.  The row code has no branches: the loop over
// a thread's rows is unrolled, and with both a sponge and an interior form of
// the update, or two marching directions, its code left the instruction cache
// (warps stalled on instructions for 1.5 of 8 cycles per issue, 0.2 without).
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "chip.h"
#include "stencil.cuh"
#include "step_common.cuh"
#include "tma.cuh"

namespace wave {

namespace {

__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// 16 bytes into another CTA's shared memory, counted on its mbarrier: the data
// is visible to a thread that has seen the barrier's phase complete.  (This and
// the predicated stores read no memory and nothing in the step reads what they
// write, so they need no memory clobber, which would keep the next row's loads
// behind them.)
__device__ __forceinline__ void st_async4_if(uint32_t pred, uint32_t a, float4 v, uint32_t bar)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %6, 0;\n\t"
        "@p st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];\n\t}" ::"r"(a),
        "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar), "r"(pred));
}
// Predicated global accesses: a branch around each would cost more than the access.
__device__ __forceinline__ void st_global4_if(bool pred, float* p, float4 v)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p st.global.v4.f32 [%0], {%1, %2, %3, %4};\n\t}" ::"l"(p),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"((uint32_t)pred));
}
__device__ __forceinline__ void st_global_bf16x4_if(bool pred, __nv_bfloat16* p, const float* o)
{
    __nv_bfloat162 lo = __floats2bfloat162_rn(o[0], o[1]);
    __nv_bfloat162 hi = __floats2bfloat162_rn(o[2], o[3]);
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p st.global.v2.b32 [%0], {%1, %2};\n\t}" ::"l"(p),
                 "r"(*reinterpret_cast<uint32_t*>(&lo)), "r"(*reinterpret_cast<uint32_t*>(&hi)), "r"((uint32_t)pred));
}
__device__ __forceinline__ float4 ldg4_if(bool pred, const float* p)
{
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (pred) v = ld4(p);
    return v;
}
__device__ __forceinline__ uint2 ldg_bf16x4_if(bool pred, const __nv_bfloat16* p)
{
    uint2 v = make_uint2(0u, 0u);
    if (pred) v = __ldg(reinterpret_cast<const uint2*>(p));
    return v;
}
__device__ __forceinline__ void cluster_arrive()
{
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// Bounded wait (as mbar_wait) on a phase that other CTAs' st.async complete.  Their
// complete_tx releases at cluster scope; try_wait without a scope acquires at CTA
// scope only, which does not synchronise with it: neither the halo rows nor the
// order of a neighbour's reads before this CTA's next writes would be guaranteed.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* b, uint32_t parity)
{
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(b)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

constexpr int kAhead = 3;  // rows by which the loads of the forward level run ahead (imaging)
__device__ __forceinline__ void cp_async4(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// This CTA's taps of one list, compacted from the shot's cell-sorted list in
// its order (taps of one grid point stay adjacent).
struct ChipTaps {
    int* off;    // position in a level's shared-memory array
    int* gi;     // flat index in the shot's field
    int* ref;    // injection: amplitude base; gather: slot
    float* fac;  // injection: factor; gather: weight
    int* j;      // position in the whole list
    int* to;     // injection: where the amount of the tap's grid point goes (-1: the point's earlier tap has it)
    int n;
};

__device__ int compact_taps(const ChipArgs& a, const TapList& l, bool inject, int shot, int za, int zb, ChipTaps& t,
                            int* scan, int cap)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    t.n = 0;
    if (!l.cell_start) return 0;
    const int b = l.cell_start[shot * a.cps], e = l.cell_start[(shot + 1) * a.cps];
    const int per = (e - b + nt - 1) / nt;
    const int lo = min(b + tid * per, e), hi = min(lo + per, e);
    int cnt = 0;
    for (int j = lo; j < hi; ++j) {
        const int z = l.idx[j] / a.P;
        cnt += z >= za && z < zb;
    }
    __syncthreads();
    scan[tid] = cnt;
    __syncthreads();
    for (int d = 1; d < nt; d <<= 1) {  // inclusive prefix sum
        const int v = tid >= d ? scan[tid - d] : 0;
        __syncthreads();
        scan[tid] += v;
        __syncthreads();
    }
    int at = scan[tid] - cnt;
    for (int j = lo; j < hi; ++j) {
        const int i = l.idx[j], z = i / a.P;
        if (z < za || z >= zb) continue;
        if (at < cap) {
            const int x = i - z * a.P;
            t.off[at] = (z - za + 4) * (a.Q + 2) * 4 + 4 + x;

            if (t.gi) t.gi[at] = i;
            t.ref[at] = inject ? l.ab[j] : l.slot[j];
            t.fac[at] = inject ? l.fac[j] : l.gw[j];
            if (t.j) t.j[at] = j;
        }
        ++at;
    }
    const int total = min(scan[nt - 1], cap);
    __syncthreads();
    return total;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// One thread's share of a step: nr (RB or RB - 1) rows of a quad column, the
// arithmetic of stencil.cuh (same operations in the same order) on pairs of
// points where the pairs lie in even registers, which is all of it but the odd
// x neighbours.  p: centre of the first row in the level read; st: stride of the
// march (float4s, negative upwards); the level written, the model and, with EPS,
// the sponge factors eps and 1 / (1 + eps) lie at fixed distances from p;
// otherwise the factors are formed from the squared depths fx (x) and fz (z).
// adds: rows with injected points; their amounts lie in row *slot of addb.
template <int RB, int MODE, bool EPS>
__device__ __forceinline__ void chip_rows(const float4* __restrict__ p, int st, int nr, float4* __restrict__ dst, int dk,
                                          float ceps, const float4* kp, float (*gr)[4], const float* fx,
                                          const float* __restrict__ fz, int sz, uint32_t sends, uint32_t to,
                                          uint32_t bar, bool keep, float* g32, __nv_bfloat16* g16, int gs,
                                          const float* u32, const __nv_bfloat16* u16, float4* f32, uint2* f16, uint32_t adds,
                                          const float4* __restrict__ addb, const int* __restrict__ slot, int ss)
{
    constexpr bool IMG = MODE == kChipAdjF32 || MODE == kChipAdjBF16, F16 = MODE == kChipAdjBF16;
    float4 w9[9];
    const float4* pw = p - 4 * st;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        w9[k] = *pw;
        pw += st;
    }
    const Quad c1 = quad(kC1), c2 = quad(kC2), c3 = quad(kC3), c4 = quad(kC4);
#pragma unroll
    for (int j = 0; j < RB; ++j) {
        w9[(j + 8) % 9] = *pw;
        const float4 A = p[-1], B = w9[(j + 4) % 9], C = p[1];
        const Quad cen = quad(B), um = quad(dst[0]);
        const float w[12] = {A.x, A.y, A.z, A.w, B.x, B.y, B.z, B.w, C.x, C.y, C.z, C.w};
        Quad lap = lap_x(w, 2.0f * kC0);
        // z
        lap = fma(c1, quad(w9[(j + 3) % 9]) + quad(w9[(j + 5) % 9]), lap);
        lap = fma(c2, quad(w9[(j + 2) % 9]) + quad(w9[(j + 6) % 9]), lap);
        lap = fma(c3, quad(w9[(j + 1) % 9]) + quad(w9[(j + 7) % 9]), lap);
        lap = fma(c4, quad(w9[j % 9]) + quad(w9[(j + 8) % 9]), lap);
        const Quad kap = quad(IMG ? p[dk] : kp[IMG ? 0 : j]);
        Quad eps, inv;
        if (EPS) {
            eps = quad(p[dk + (IMG ? sz : 0)]);
            inv = quad(p[dk + (IMG ? 2 * sz : sz)]);
        } else {
            const float z = *fz;
            const Quad dd = {make_float2(fmaxf(fx[0], z), fmaxf(fx[1], z)), make_float2(fmaxf(fx[2], z), fmaxf(fx[3], z))};
            eps = kap * quad(ceps) * dd;
            const Quad nx = fma(eps, quad(-1.0f), quad(-1.0f));  // -(1 + eps)
            const Quad r = {make_float2(rcp_approx(-nx.a.x), rcp_approx(-nx.a.y)),
                            make_float2(rcp_approx(-nx.b.x), rcp_approx(-nx.b.y))};
            inv = fma(r, fma(nx, r, quad(1.0f)), r);
            fz += sz;
        }
        Quad t = {make_float2(fmaf(2.0f, cen.a.x, -um.a.x), fmaf(2.0f, cen.a.y, -um.a.y)),
                  make_float2(fmaf(2.0f, cen.b.x, -um.b.x), fmaf(2.0f, cen.b.y, -um.b.y))};
        Quad out = fma(kap, lap, fma(eps, um, t)) * inv;
        if ((adds >> j) & 1u) out = out + quad(addb[*slot]);  // the row's injected points
        slot += ss;
        // (points past Nx stay zero: the model is zero there)
        const float4 o4 = make_float4(out.a.x, out.a.y, out.b.x, out.b.y);
        const bool live = j < RB - 1 || nr == RB;
        if (live) *dst = o4;
        st_async4_if((sends >> j) & 1u, to, o4, bar);
        to += (uint32_t)(st * 16);
        if (MODE == kChipFwdBF16) {
            const float o[4] = {o4.x, o4.y, o4.z, o4.w};
            st_global_bf16x4_if(live, g16 + j * gs, o);
        } else {
            st_global4_if(keep && live, g32 + j * gs, o4);
        }
        if (IMG) {
            Quad uf;
            if (F16) {
                float u[4];
                unpack_bf16x4(f16[F16 ? j % kAhead : 0], u);
                uf = {make_float2(u[0], u[1]), make_float2(u[2], u[3])};
                if (j + kAhead < RB) f16[F16 ? j % kAhead : 0] = ldg_bf16x4_if(j + kAhead < nr, u16 + (j + kAhead) * gs);
            } else {
                uf = quad(f32[IMG && !F16 ? j % kAhead : 0]);
                if (j + kAhead < RB) f32[IMG && !F16 ? j % kAhead : 0] = ldg4_if(j + kAhead < nr, u32 + (j + kAhead) * gs);
            }
            // gr holds minus the gradient
            const Quad d2 = fma(quad(-2.0f), cen, out) + um;
            if (live) {
                Quad g = {make_float2(gr[IMG ? j : 0][0], gr[IMG ? j : 0][1]),
                          make_float2(gr[IMG ? j : 0][2], gr[IMG ? j : 0][3])};
                g = fma(uf, d2, g);
                gr[IMG ? j : 0][0] = g.a.x;
                gr[IMG ? j : 0][1] = g.a.y;
                gr[IMG ? j : 0][2] = g.b.x;
                gr[IMG ? j : 0][3] = g.b.y;
            }
        }
        pw += st;
        p += st;
        dst += st;
    }
}

// MODE: forward steps, adjoint steps without imaging, or with the forward
// level read from FP32 or BF16.
template <int RB, int NT, int MODE, bool EPS>
__global__ void __launch_bounds__(NT, 1) k_chip2d(const __grid_constant__ ChipArgs a)
{
    constexpr bool ADJ = MODE != kChipForward && MODE != kChipFwdBF16, IMG = MODE == kChipAdjF32 || MODE == kChipAdjBF16;
    constexpr bool F16 = MODE == kChipAdjBF16;
    extern __shared__ __align__(16) float4 sm[];
    __shared__ __align__(8) uint64_t halo[2];  // per level: the neighbours' rows have arrived
    __shared__ int side_taps;                  // bit 0 / 1: injected taps in the first / last 4 rows
    const int tid = threadIdx.x, rank = blockIdx.x, shot = blockIdx.y;
    const int za = a.z0[rank], R = a.z0[rank + 1] - za;
    const int Q = a.Q, LD = Q + 2, level = (a.Rmax + 8) * LD, pts = a.Rmax * LD;  // in float4s
    // shared memory: two levels (a zero quad before and after each row), with
    // imaging the model, with EPS the sponge factors, the squared depths along z,
    // then the tap lists
    float4* ksm = sm + 2 * level;
    float4* esm = ksm + (IMG ? pts : 0);
    float4* ism = esm + (EPS ? pts : 0);
    float* zsm = reinterpret_cast<float*>(ism + (EPS ? pts : 0));
    const bool inl = a.add_rows > 0;  // injection in the row loop; otherwise after it, between barriers
    float4* addb = reinterpret_cast<float4*>(zsm + ((a.Rmax + 3) & ~3));  // [2][add_rows][LD]
    int* slot = reinterpret_cast<int*>(addb + 2 * a.add_rows * LD);       // [Rmax] first float4 of a row in addb
    ChipTaps ti, tg;
    float *xa, *xb, *xu, *addp, *acc;  // per injected tap, [2] by step parity: amplitudes; forward level; amount; [1] imaging
    int* scan;
    {
        const int ci = a.cap_inj;
        int* p = slot + a.Rmax;
        auto take = [&](int n) {
            int* r = p;
            p += n;
            return r;
        };
        ti.off = take(ci);
        ti.gi = take(ci);
        ti.ref = take(ci);
        ti.fac = reinterpret_cast<float*>(take(ci));
        ti.to = take(ci);
        xa = reinterpret_cast<float*>(take(2 * ci));
        xb = reinterpret_cast<float*>(take(2 * ci));
        const int cf = inl ? 0 : ci, cg = inl || !IMG ? 0 : ci;
        addp = reinterpret_cast<float*>(take(2 * cf));
        xu = reinterpret_cast<float*>(take(2 * cg));
        acc = reinterpret_cast<float*>(take(cg));
        ti.j = take(cg);
        if (!cg) ti.j = nullptr;
        tg.off = take(a.cap_gat);
        tg.ref = take(a.cap_gat);
        tg.fac = reinterpret_cast<float*>(take(a.cap_gat));
        tg.gi = tg.j = tg.to = nullptr;
        scan = p;
    }
    // thread (chunk c, quad q): nr rows of the strip from r0, points 4q .. 4q+3
    const int c = tid / Q, q = tid - c * Q;
    const bool owner = c < a.NC;
    const int r0 = owner ? c * R / a.NC : 0, nr = owner ? (c + 1) * R / a.NC - r0 : 0;
    // the last chunk marches upwards, so both borders are computed and sent first
    const bool back = c > 0 && c == a.NC - 1;
    const int rb = back ? r0 + nr - 1 : r0, sg = back ? -1 : 1;
    const int gx = 4 * q;
    const long long so = (long long)shot * a.cell;
    const float* gcur = a.cur >= 0 ? a.pool + (long long)a.cur * a.field + so : nullptr;
    const float* gprev = a.prev >= 0 ? a.pool + (long long)a.prev * a.field + so : nullptr;

    if (tid == 0) {
        mbar_init(&halo[0], 1);
        mbar_init(&halo[1], 1);
        fence_mbar_init();
        side_taps = 0;
    }
    // the strip of u^n with its halo rows, the strip of u^{n-1}; zeros elsewhere
    for (int i = tid; i < 2 * level; i += blockDim.x) sm[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    for (int i = tid; i < (R + 8) * Q; i += blockDim.x) {
        const int r = i / Q, qq = i - r * Q, gz = za - 4 + r;
        if (gz < 0 || gz >= a.Nz) continue;
        const int o = gz * a.P + 4 * qq;
        const bool mine = r >= 4 && r < R + 4;
        if (gcur) sm[r * LD + qq + 1] = *reinterpret_cast<const float4*>(gcur + o);
        if (gprev && mine) sm[level + r * LD + qq + 1] = *reinterpret_cast<const float4*>(gprev + o);
        if (mine && (IMG || EPS)) {
            const float4 k = ld4(a.kap + o);
            const int m = (r - 4) * LD + qq, dz = sponge_depth(gz, a.nb, a.nz);
            if (IMG) ksm[m] = k;
            if (EPS) {
                float ev[4], iv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int dd = max(sponge_depth(4 * qq + e, a.nb, a.nx), dz);
                    ev[e] = f4(k, e) * a.ceps * (float)(dd * dd);
                    iv[e] = rcp_sponge(1.0f + ev[e]);
                }
                esm[m] = make_float4(ev[0], ev[1], ev[2], ev[3]);
                ism[m] = make_float4(iv[0], iv[1], iv[2], iv[3]);
            }
        }
    }
    for (int r = tid; r < R; r += blockDim.x) {
        const int dz = sponge_depth(za + r, a.nb, a.nz);
        zsm[r] = (float)(dz * dz);
        slot[r] = -1;
    }
    for (int i = tid; i < 2 * a.add_rows * LD; i += blockDim.x) addb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    ti.n = compact_taps(a, a.inj, true, shot, za, za + R, ti, scan, a.cap_inj);
    tg.n = compact_taps(a, a.gat, false, shot, za, za + R, tg, scan, a.cap_gat);
    if (inl) {
        // rows with injected points, numbered in row order
        for (int t = tid; t < ti.n; t += blockDim.x) slot[ti.gi[t] / a.P - za] = 0;
        __syncthreads();
        if (tid == 0)
            for (int r = 0, k = 0; r < R; ++r)
                if (slot[r] == 0) slot[r] = (k++) * LD;
    } else {
        // a border that holds injected points is sent after the injection, the others as they are computed
        for (int t = tid; t < ti.n; t += blockDim.x) {
            const int lr = ti.gi[t] / a.P - za;
            if (lr < 4) atomicOr(&side_taps, 1);
            if (lr >= R - 4) atomicOr(&side_taps, 2);
            if (IMG) acc[t] = a.tacc[ti.j[t]];
        }
    }
    __syncthreads();
    for (int t = tid; t < ti.n; t += blockDim.x) {
        const int gi = ti.gi[t], z = gi / a.P;
        ti.to[t] = t > 0 && ti.gi[t - 1] == gi ? -1 : (inl ? slot[z - za] * 4 + 4 + gi - z * a.P : t);
    }
    // the threads of an inner chunk take the first taps: those of a border chunk have neighbours waiting
    const int t0 = (tid + (int)blockDim.x - (a.NC > 2 ? Q : 0)) % (int)blockDim.x;
    const int late = side_taps;
    const bool has_up = rank > 0, has_dn = rank + 1 < a.C;
    const bool send_up = has_up && !(late & 1), send_dn = has_dn && !(late & 2);

    const int go = (za + rb) * a.P + gx;
    float4 kp[IMG ? 1 : RB];
    float gr[IMG ? RB : 1][4];
    uint32_t sends = 0, adds = 0;  // bit j: the thread's row j goes to a neighbour, has injected points
    float fx[4];         // squared sponge depth along x
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int d = sponge_depth(gx + e, a.nb, a.nx);
        fx[e] = (float)(d * d);
    }
#pragma unroll
    for (int j = 0; j < RB; ++j) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const int o = go + sg * j * a.P, lr = rb + sg * j;
        if (!IMG) kp[IMG ? 0 : j] = j < nr ? ld4(a.kap + o) : z;
        if (IMG) {
            const float4 v = j < nr ? *reinterpret_cast<const float4*>(a.pool + (long long)a.g_buf * a.field + so + o) : z;
            gr[IMG ? j : 0][0] = -v.x;
            gr[IMG ? j : 0][1] = -v.y;
            gr[IMG ? j : 0][2] = -v.z;
            gr[IMG ? j : 0][3] = -v.w;
        }
        // (the plan sees to it that a thread feeds one neighbour at most)
        if (inl && j < nr && slot[lr] >= 0) adds |= 1u << j;
        if (j < nr && ((send_up && lr < 4) || (send_dn && lr >= R - 4))) sends |= 1u << j;
    }
    const int at = (rb + 4) * LD + q + 1;  // the first row in a level
    const bool down = r0 + nr > R - 4;     // which neighbour
    const uint32_t sbase = smem_u32(sm), hbase = smem_u32(halo);
    const int Rup = has_up ? za - a.z0[rank - 1] : 0;
    // byte addresses that take a row of this strip (float4 index) to the neighbours' halo rows
    const uint32_t up = has_up ? mapa(sbase, rank - 1) + (uint32_t)(Rup * LD) * 16u : 0;
    const uint32_t dn = has_dn ? mapa(sbase, rank + 1) - (uint32_t)(R * LD) * 16u : 0;
    const uint32_t upb = has_up ? mapa(hbase, rank - 1) : 0, dnb = has_dn ? mapa(hbase, rank + 1) : 0;
    const uint32_t halo_bytes = (uint32_t)((has_up ? 1 : 0) + (has_dn ? 1 : 0)) * 64u * Q;
    const bool border = owner && nr > 0 && (r0 < 4 || r0 + nr > R - 4);
    // Injection runs two steps ahead: while step i is computed, the amplitudes of
    // step i + 2 are copied to shared memory and the amounts of step i + 1 are
    // summed (one thread per grid point, its taps in list order).  Fetched and
    // summed within their own step they were the longest chain of it (0.5 us of
    // 2.1 us per step with 201 receivers, 2.3 us in the adjoint).
    auto fetch_taps = [&](int i) {
        if (ti.n == 0 || i >= a.nsteps) return;
        const int n = ADJ ? a.first - i : a.first + i, b = (i & 1) * a.cap_inj;
        for (int t = t0; t < ti.n; t += blockDim.x) {
            const long long r = (long long)ti.ref[t] + (long long)n * a.inj.npts;
            cp_async4(xa + b + t, a.amp_a + r);
            if (a.amp_b) cp_async4(xb + b + t, a.amp_b + r);
        }
    };
    auto fetch_uf = [&](int i) {  // the forward level at the taps (injection between barriers)
        if (!IMG || inl || ti.n == 0 || i >= a.nsteps) return;
        float* x = xu + (i & 1) * a.cap_inj;
        for (int t = tid; t < ti.n; t += blockDim.x) {
            if (F16) cp_async4(x + t, a.uf16 + (long long)(a.first - i) * a.field + so + (ti.gi[t] & ~1));
            else cp_async4(x + t, a.pool + (long long)a.tab[i] * a.field + so + ti.gi[t]);
        }
    };
    auto sum_taps = [&](int i) {
        if (ti.n == 0 || i >= a.nsteps) return;
        const int b = (i & 1) * a.cap_inj;
        float* out = inl ? reinterpret_cast<float*>(addb + (i & 1) * a.add_rows * LD) : addp + b;
        for (int t = t0; t < ti.n; t += blockDim.x) {
            const int o = ti.to[t];
            if (o < 0) continue;
            float add = 0.0f;
            int s = t;
            do {
                add = fmaf(ti.fac[s], a.amp_b ? xa[b + s] - xb[b + s] : xa[b + s], add);
                ++s;
            } while (s < ti.n && ti.to[s] < 0);
            out[o] = add;
        }
    };
    fetch_taps(0);
    fetch_taps(1);
    fetch_uf(0);
    cp_async_done();
    __syncthreads();
    sum_taps(0);
    // every CTA of the cluster has set up its shared memory before the first remote write
    cluster_arrive();
    cluster_wait();
    bool alive = true;
    // the forward level of the next rows, kAhead rows ahead (with imaging)
    float4 f32[IMG && !F16 ? kAhead : 1];
    uint2 f16[F16 ? kAhead : 1];
    const float* u32 = nullptr;
    const __nv_bfloat16* u16 = nullptr;
    auto open_level = [&](int i) {
        if (!IMG || i >= a.nsteps) return;
        const int n = a.first - i;
        if (F16) u16 = a.uf16 + (long long)n * a.field + so + go;
        else u32 = a.pool + (long long)a.tab[i] * a.field + so + go;
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            if (k >= nr) continue;
            if (F16) f16[F16 ? k : 0] = __ldg(reinterpret_cast<const uint2*>(u16 + sg * k * a.P));
            else f32[IMG && !F16 ? k : 0] = ld4(u32 + sg * k * a.P);
        }
        if (i + 1 < a.nsteps && tid < R) {  // the level after it is on its way into L2 meanwhile
            if (F16) {
                prefetch_l2(a.uf16 + (long long)(n - 1) * a.field + so + (za + tid) * a.P, (uint32_t)(Q * 8 + 15) & ~15u);
            } else {
                prefetch_l2(a.pool + (long long)a.tab[i + 1] * a.field + so + (za + tid) * a.P, (uint32_t)Q * 16u);
            }
        }
    };
    open_level(0);

    for (int i = 0; i < a.nsteps; ++i) {
        const float4* src = sm + (i & 1) * level;
        float4* dst = sm + (1 - (i & 1)) * level;
        const uint32_t dsto = (uint32_t)(1 - (i & 1)) * level * 16u, dstb = (uint32_t)(1 - (i & 1)) * 8u;
        const int n = ADJ ? a.first - i : a.first + i;
        // where this level is kept, if it is: a pool buffer, a row of the BF16 store, or nowhere
        int keep = i == a.nsteps - 1 ? a.out_last : (i == a.nsteps - 2 ? a.out_prev : -1);
        if (!ADJ && keep < 0) keep = a.keep_mode == kKeepTable ? a.tab[i] : (a.keep_mode == kKeepRows ? a.row0 + n + 1 : -1);
        float* g32 = a.pool + (long long)max(keep, 0) * a.field + so;
        __nv_bfloat16* g16 = MODE == kChipFwdBF16 ? a.st16 + (long long)(n + 1) * a.field + so : nullptr;
        fetch_taps(i + 2);
        fetch_uf(i + 1);
        sum_taps(i + 1);
        // gathers of the level the last step made
        if (tg.n > 0 && i > 0 && (ADJ || n - 1 >= a.rec_from)) {
            float* row = a.slots + (long long)n * a.gat.ntap;
            const float* lev = reinterpret_cast<const float*>(src);
            for (int t = t0; t < tg.n; t += blockDim.x) row[tg.ref[t]] = tg.fac[t] * lev[tg.off[t]];
        }
        if (a.C > 1) {
            // (after a wait that gave up this barrier's last phase may be open still: no second arrival then)
            if (tid == 0 && alive) mbar_expect_tx(&halo[1 - (i & 1)], halo_bytes);
            // (a thread whose wait gives up records it and goes on: every barrier below stays uniform)
            if (border && i > 0 && alive && !mbar_wait_cluster(&halo[i & 1], (uint32_t)((i - 1) >> 1) & 1u)) {
                alive = false;
                atomicOr(a.err, kErrTimeout);
            }
        }
        if (owner) {
            chip_rows<RB, MODE, EPS>(src + at, sg * LD, nr, dst + at, (int)(ksm + rb * LD + q - (src + at)), a.ceps, kp, gr,
                                     fx, zsm + rb, EPS ? pts : sg, sends,
                                     (down ? dn : up) + dsto + (uint32_t)at * 16u, (down ? dnb : upb) + dstb, keep >= 0,
                                     g32 + go, g16 + go, sg * a.P, u32, u16, f32, f16, adds,
                                     addb + (i & 1) * a.add_rows * LD + q + 1, slot + rb, sg);
            if (keep >= 0 && q == Q - 1)  // the pitch columns of a stored level read as the zero exterior
                for (int j = 0; j < nr; ++j)
                    for (int x = 4 * Q; x < a.P; x += 4)
                        *reinterpret_cast<float4*>(g32 + (za + r0 + j) * a.P + x) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (!inl && ti.n > 0) {
            __syncthreads();
            const int b = (i & 1) * a.cap_inj;
            float* lev = reinterpret_cast<float*>(dst);
            for (int t = tid; t < ti.n; t += blockDim.x) {
                if (ti.to[t] < 0) continue;
                const int gi = ti.gi[t];
                const float add = addp[b + t], v = lev[ti.off[t]] + add;
                lev[ti.off[t]] = v;
                if (keep >= 0) g32[gi] = v;
                if (MODE == kChipFwdBF16) g16[gi] = __float2bfloat16_rn(v);
                if (IMG) {
                    float uf = xu[b + t];
                    if (F16) {
                        const uint32_t w = __float_as_uint(uf);
                        uf = __uint_as_float((gi & 1) ? w & 0xffff0000u : w << 16);
                    }
                    acc[t] -= uf * add;
                }
            }
        }
        open_level(i + 1);
        cp_async_done();
        __syncthreads();
        if (late) {  // borders with injected points (block-uniform)
            for (int t = tid; t < 4 * Q; t += blockDim.x) {
                const int r = t / Q, o = r * LD + t - r * Q + 1, u = o + 4 * LD, d = o + R * LD;
                st_async4_if(has_up && (late & 1), up + dsto + (uint32_t)u * 16u, dst[u], upb + dstb);
                st_async4_if(has_dn && (late & 2), dn + dsto + (uint32_t)d * 16u, dst[d], dnb + dstb);
            }
        }
    }
    if (a.C > 1) {
        // the last rows sent to this CTA have landed, and all of the cluster is here, before any CTA leaves
        if (tid == 0 && alive && a.nsteps > 0 && !mbar_wait_cluster(&halo[a.nsteps & 1], (uint32_t)((a.nsteps - 1) >> 1) & 1u)) {
            alive = false;
            atomicOr(a.err, kErrTimeout);
        }
        cluster_arrive();
        cluster_wait();
        // every CTA has sent its rows by now: one that gave a wait up stays (bounded again) until
        // those on their way to it have landed
        if (tid == 0 && !alive)
            for (int n = a.nsteps; n > 0 && n > a.nsteps - 2; --n)
                mbar_wait_cluster(&halo[n & 1], (uint32_t)((n - 1) >> 1) & 1u);
    }
    const int nl = ADJ ? a.first - a.nsteps : a.first + a.nsteps;  // the index of the next step
    if (tg.n > 0 && a.nsteps > 0 && (ADJ || nl - 1 >= a.rec_from)) {
        const float* lev = reinterpret_cast<const float*>(sm + (a.nsteps & 1) * level);
        float* row = a.slots + (long long)nl * a.gat.ntap;
        for (int t = tid; t < tg.n; t += blockDim.x) row[tg.ref[t]] = tg.fac[t] * lev[tg.off[t]];
    }
    if (IMG) {
        // both sums continue in the next launch, so the order of the additions does
        // not depend on how the steps are split into launches
        float* g = a.pool + (long long)a.g_buf * a.field + so;
        if (owner) {
#pragma unroll
            for (int j = 0; j < RB; ++j) {
                if (j >= nr) break;
                *reinterpret_cast<float4*>(g + go + sg * j * a.P) =
                    make_float4(-gr[IMG ? j : 0][0], -gr[IMG ? j : 0][1], -gr[IMG ? j : 0][2], -gr[IMG ? j : 0][3]);
            }
        }
        if (!inl)
            for (int t = tid; t < ti.n; t += blockDim.x) a.tacc[ti.j[t]] = acc[t];
    }
}

// Adds the taps' imaging terms to the gradient accumulators (injection between
// barriers): the first tap of a grid point holds the point's sum.
__global__ void k_chip_tap_gradient(TapList l, long long per_shot, long long cell, const float* __restrict__ tacc,
                                    float* __restrict__ g)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= l.ntap) return;
    const long long shot = l.ab[j] / per_shot;
    if (j > 0 && l.idx[j - 1] == l.idx[j] && l.ab[j - 1] / per_shot == shot) return;
    g[shot * cell + l.idx[j]] += tacc[j];
}

// ---------------------------------------------------------------------------
// Host side.

typedef void (*ChipKernel)(const ChipArgs);

struct ChipShape {
    int RB;         // rows per thread
    int NT[kChipModes];  // largest block per mode
    bool eps;       // sponge factors in shared memory
    ChipKernel k[kChipModes];
};

// The register file (16384 per scheduler) bounds the block: 4 warps per
// scheduler leave 128 registers a thread, 5 leave 96, 6 leave 80.  A thread
// holds 4 RB model values (with imaging 4 RB gradient values instead, the model
// in shared memory), the 36-value z window and about 35 others.  What exceeds the
// cap spills (bytes of stores / loads per thread): with imaging 8 rows 136 / 156, 7
// rows 72 / 116 (FP32 level; 68 / 88 BF16), 6 rows 60 / 68; without, 10 rows 44 / 44, 4
// rows 44 / 52 and 2 rows 48 / 52 at their 5 and 6 warps, 5 to 8 rows 28 at most.  The cap
// is the shape's, also for a plan of fewer threads (448 of 512 for 592 x 336 on 16 CTAs).
// Of 260 random problems (30 to 700 x 30 to 400 points, sponges of 0 to 40 cells, 1 to 24
// shots) forward steps took 2 rows in 210, 3 in 15, 4 in 13, and 5 to 10 in 2 to 4 each,
// launches kept 5; the shapes of 4, 5 and 6 rows that form the factors were
// not taken forward, the one of 4 rows not at all.
template <int RB, int NF, int NA, bool EPS>
constexpr ChipShape shape()
{
    return {RB,
            {NF, NF, NF, NA, NA},
            EPS,
            {k_chip2d<RB, NF, kChipForward, EPS>, k_chip2d<RB, NF, kChipFwdBF16, EPS>, k_chip2d<RB, NF, kChipAdjoint, EPS>,
             k_chip2d<RB, NA, kChipAdjF32, EPS>, k_chip2d<RB, NA, kChipAdjBF16, EPS>}};
}
const ChipShape kShapes[] = {shape<2, 768, 640, true>(),   shape<3, 640, 640, true>(),  shape<4, 640, 512, true>(),
                             shape<5, 512, 512, true>(),   shape<6, 512, 512, true>(),  shape<4, 640, 512, false>(),
                             shape<5, 512, 512, false>(),  shape<6, 512, 512, false>(), shape<7, 512, 512, false>(),
                             shape<8, 512, 512, false>(),  shape<10, 512, 384, false>()};
constexpr int kShapeCount = sizeof(kShapes) / sizeof(kShapes[0]);

constexpr int kMaxAddRows = 4;
constexpr size_t kMaxSmem = 226 * 1024;  // dynamic; the kernel has a few static bytes beside it

cudaLaunchConfig_t chip_config(const ChipPlan& p, int nshot, cudaStream_t s, cudaLaunchAttribute* at)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.C, nshot);
    cfg.blockDim = dim3(p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = p.C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

// Clusters of this shape that the current device runs at once (0: none).  The
// answer depends on the device, the kernel and the launch shape alone, so it is
// kept per process; shared memory counts in steps of 8 KB.
int resident_clusters(ChipKernel k, int C, int threads, size_t smem)
{
    static std::mutex mu;
    static std::map<std::tuple<int, ChipKernel, int, int, int>, int> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    const int step = (int)((smem + 8191) / 8192);
    std::lock_guard<std::mutex> lock(mu);
    const auto key = std::make_tuple(dev, k, C, threads, step);
    auto it = known.find(key);
    if (it != known.end()) return it->second;
    int n = 0;
    ChipPlan p;
    p.C = C;
    p.threads = threads;
    p.smem = std::min(kMaxSmem, (size_t)step * 8192);
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = chip_config(p, 1, nullptr, at);
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess)
        n = 0;
    (void)cudaGetLastError();
    if (known.size() > 4096) known.clear();
    known[key] = n;
    return n;
}

// Time of one step (us) of a wave of clusters, k of whose CTAs share an SM:
// the exchange and the barriers, the chain of one thread's rows, and the issue
// slots of the SM's warps.  Least squares over 92 splits of eleven problems (91 x
// 69 to 592 x 336 points, 1 to 7 shots, C = 2 ... 16, RB = 2 ... 10); 8 to 10 % rms.
float step_model(int mode, const ChipShape& shape, int warps, float k)
{
    const int RB = shape.RB;
    static const float c[kChipModes][3] = {{1.05f, 0.10f, 0.0555f},   // forward
                                           {0.95f, 0.095f, 0.0615f},  // forward, every level in BF16
                                           {1.05f, 0.10f, 0.0555f},   // adjoint
                                           {0.90f, 0.175f, 0.091f},   // adjoint with imaging, FP32
                                           {1.20f, 0.12f, 0.085f}};   // adjoint with imaging, BF16
    float t = c[mode][0] + c[mode][1] * RB + c[mode][2] * k * warps * RB / 4.0f;
    if (!shape.eps) t *= 1.15f;  // the sponge factors formed at every point (3.6 us where the fit has 3.1)
    return RB >= 10 && mode <= kChipAdjoint ? 1.13f * t : t;  // 10 rows spill at 128 registers
}

// First row of strip r of C.
int strip_start(int Nz, int C, int r) { return (int)((long long)Nz * r / C); }

// Fills h.strip_taps and h.strip_rows, which depend on the problem alone: one pass over
// the taps, and per shot 136 strips (1 + 2 + ... + 16) from running sums over the rows.
// (Counted anew for every split that chip_plan weighed, the taps of 1000 shots of 91 x
// 69 points with 200 receivers took 96 ms of host time, the tap build itself 51.)
void count_strips(HostTaps& h, const Dims& d, int nshot, long long cps)
{
    if (!h.strip_taps.empty()) return;
    h.strip_taps.assign(kMaxCluster + 1, 0);
    h.strip_rows.assign(kMaxCluster + 1, 0);
    if (h.idx.empty()) return;
    int start[kMaxCluster + 1][kMaxCluster + 1];
    for (int C = 1; C <= kMaxCluster; ++C)
        for (int r = 0; r <= C; ++r) start[C][r] = strip_start(d.Nz, C, r);
    std::vector<int> row(d.Nz), taps(d.Nz + 1, 0), rows(d.Nz + 1, 0);
    for (int s = 0; s < nshot; ++s) {
        std::fill(row.begin(), row.end(), 0);
        for (int j = h.cell_start[s * cps]; j < h.cell_start[(s + 1) * cps]; ++j) ++row[h.idx[j] / d.P];
        for (int z = 0; z < d.Nz; ++z) {
            taps[z + 1] = taps[z] + row[z];
            rows[z + 1] = rows[z] + (row[z] > 0);
        }
        for (int C = 1; C <= kMaxCluster; ++C)
            for (int r = 0; r < C; ++r) {
                const int a = start[C][r], b = start[C][r + 1];
                h.strip_taps[C] = std::max(h.strip_taps[C], taps[b] - taps[a]);
                h.strip_rows[C] = std::max(h.strip_rows[C], rows[b] - rows[a]);
            }
    }
}

// Whether no thread holds rows of both borders of its strip.
bool one_sided(int Nz, int C, int NC)
{
    for (int R = Nz / C; R <= (Nz + C - 1) / C; ++R)
        for (int c = 0; c < NC; ++c)
            if (c * R / NC < 4 && (c + 1) * R / NC > R - 4) return false;
    return true;
}

}  // namespace

thread_local ChipForce t_force;  // of calls from this host thread; set by tests only

ChipPlan chip_plan(const Dims& d, const Tiling& t, int nshot, int mode, HostTaps& inj, HostTaps& gat)
{
    ChipPlan best;
    if (d.ndim != 2 || nshot < 1 || nshot > 65535) return best;
    const int Q = (d.Nx + 3) / 4;
    const bool img = mode == kChipAdjF32 || mode == kChipAdjBF16;
    float least = 0.0f;
    for (int C = 1; C <= kMaxCluster; ++C) {
        const int R = (d.Nz + C - 1) / C;
        if (C > 1 && d.Nz / C < 4) break;  // a strip feeds its neighbours' 4-row halos
        if (t_force.C && C != t_force.C) continue;
        for (int k = 0; k < kShapeCount; ++k) {
            if (t_force.shape >= 0 && k != t_force.shape) continue;
            const int NT = kShapes[k].NT[mode];
            const int NC = (R + kShapes[k].RB - 1) / kShapes[k].RB;
            const int threads = (NC * Q + 31) / 32 * 32;
            // (a thread's rows are the kernel's RB, or one fewer)
            if (C > 1 && !one_sided(d.Nz, C, NC)) continue;
            if (threads > NT || (R + NC - 1) / NC != kShapes[k].RB || d.Nz / C / NC < kShapes[k].RB - 1) continue;
            const size_t pts = (size_t)((img ? 1 : 0) + (kShapes[k].eps ? 2 : 0)) * R * (Q + 2);
            const size_t levels = 16 * (2 * (size_t)(R + 8) * (Q + 2) + pts) + 8 * (size_t)(R + 4);
            if (levels > kMaxSmem) continue;
            ChipPlan p;
            p.C = C;
            p.shape = k;
            p.mode = mode;
            p.NC = NC;
            p.threads = threads;
            p.Rmax = R;
            for (int r = 0; r <= C; ++r) p.z0[r] = strip_start(d.Nz, C, r);
            const float one = step_model(mode, kShapes[k], threads / 32, 1.0f);
            if (best.C && one >= least) continue;
            count_strips(inj, d, nshot, t.cells_per_shot());
            count_strips(gat, d, nshot, t.cells_per_shot());
            const int inj_rows = inj.strip_rows[C];
            p.cap_inj = inj.strip_taps[C];
            p.cap_gat = gat.strip_taps[C];
            // injection in the row loop where the points lie in few rows (surface lines):
            // 2 rows of amounts each; many rows (a borehole) take the barriers
            p.add_rows = inj_rows <= kMaxAddRows ? inj_rows : 0;
            p.smem = levels + 16 * (size_t)2 * p.add_rows * (Q + 2) +
                     4 * ((size_t)(p.add_rows ? 9 : img ? 15 : 11) * p.cap_inj + 3 * p.cap_gat + threads);
            if (p.smem > kMaxSmem) continue;
            const int res = resident_clusters(kShapes[k].k[mode], C, threads, p.smem);
            const int alone = resident_clusters(kShapes[k].k[mode], C, threads, kMaxSmem);  // one CTA per SM
            if (res < 1 || alone < 1) continue;
            const int waves = (nshot + res - 1) / res, wide = std::min(nshot, res);
            const float time = waves * step_model(mode, kShapes[k], threads / 32, std::max(1.0f, (float)wide / alone));
            if (best.C && time >= least) continue;
            p.step_us = least = time;
            best = p;
        }
    }
    return best;
}

cudaError_t launch_chip(const ChipPlan& p, ChipArgs& a, int nshot, cudaStream_t s)
{
    a.C = p.C;
    a.NC = p.NC;
    a.Rmax = p.Rmax;
    a.Q = (a.Nx + 3) / 4;
    a.cap_inj = p.cap_inj;
    a.cap_gat = p.cap_gat;
    a.add_rows = p.add_rows;
    std::copy(p.z0, p.z0 + p.C + 1, a.z0);
    const ChipKernel k = kShapes[p.shape].k[p.mode];
    if (resident_clusters(k, p.C, p.threads, p.smem) < 1) return cudaErrorInvalidConfiguration;  // sets the attributes too
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = chip_config(p, nshot, s, at);
    count_step_launch();
    if (t_force.refuse) cfg.dynamicSmemBytes = (size_t)1 << 30;
    cudaEvent_t stop;
    const bool timed = profile_sample(p.mode >= kChipAdjoint, s, &stop, a.nsteps);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, a);
    if (timed) profile_close(stop, s);
    return e;
}

void launch_chip_tap_gradient(const TapList& l, int nt, long long cell, const float* tacc, float* g, cudaStream_t s)
{
    if (l.ntap == 0) return;
    count_launch();
    k_chip_tap_gradient<<<(l.ntap + 255) / 256, 256, 0, s>>>(l, (long long)nt * l.npts, cell, tacc, g);
}

}  // namespace wave

extern "C" int wave_chip_force(int shape, int clusters, int refuse)
{
    wave::t_force.shape = shape;
    wave::t_force.C = clusters;
    wave::t_force.refuse = refuse != 0;
    return wave::kShapeCount;
}
