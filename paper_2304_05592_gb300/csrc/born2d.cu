// born2d.cu -- one linearised (Born) 2D time step of every shot in one kernel:
// the background level u^{n+1} and the scattered level p^{n+1}, whose secondary
// source -dm v^2 (u^{n+1} - 2 u^n + u^{n-1}) is formed from the background
// values while they are in registers.
//
// Memory bound: u^n, u^{n-1}, p^n, p^{n-1} are read and u^{n+1}, p^{n+1} written
// once, 24 bytes per point and step, where two launches of the direct kernel
// moved 36 (the scattered step read three background levels again) and kept a
// third background level, 130 MB in all for 32 shots of 592 x 336 against 104 MB
// here and 129 MB of L2.
//
// As in the shot-group step (k_step2d_sgt) a CTA works through up to 4 shots of one 128
// x 16 tile: the model, dm v^2 and the sponge factors are set up once, each
// shot's two halo tiles and two previous levels arrive by TMA into a two-stage
// ring, and consecutive steps are chained by programmatic dependent launch.
#include <atomic>

#include "internal.h"
#include "stencil.cuh"
#include "step_common.cuh"
#include "tma.cuh"

namespace wave {

namespace {

constexpr int kBTZ = 16, kBBZ = 8, kBG = 4, kBRows = kBTZ / kBBZ;
constexpr int kBSW = kTX + 8, kBHalo = (kBTZ + 8) * kBSW, kBTile = kBTZ * kTX;
constexpr int kBStage = 2 * kBHalo + 2 * kBTile;  // floats
static_assert(kBHalo % 32 == 0 && kBTile % 32 == 0, "sub-buffers must stay 128-byte aligned");

__global__ void __launch_bounds__(32 * kBBZ, 2) k_born2d(const __grid_constant__ StepMaps mp, const StepArgs a,
                                                          const int p_buf, const int pprev_buf, float* pnew_all)
{
    extern __shared__ unsigned char dyn[];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ int taprng[kBG][4];  // per shot: source and receiver tap ranges
    float* st = reinterpret_cast<float*>(dyn + ((128u - (smem_u32(dyn) & 127u)) & 127u));
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * 32 + tx;
    // (x tiles, shot groups, z tiles): the top tile rows, which hold the taps, run first
    const int tzi = blockIdx.z, x0 = blockIdx.x * kTX, z0 = tzi * kBTZ;
    const int s0 = blockIdx.y * a.group, ns = min(a.group, a.nshot - s0);  // a.group <= kBG
    const int lx = 4 * tx, gx = x0 + lx, nvalid = min(4, a.Nx - gx);
    auto issue = [&](int i) {
        float* sb = st + (i & 1) * kBStage;
        uint64_t* b = &bar[i & 1];
        mbar_expect_tx(b, kBStage * 4u);
        tma_load_4d(sb, &mp.halo_f, b, x0 - 4, z0 - 4, s0 + i, a.u_buf);
        tma_load_4d(sb + kBHalo, &mp.halo_f, b, x0 - 4, z0 - 4, s0 + i, p_buf);
        tma_load_4d(sb + 2 * kBHalo, &mp.tile_f, b, x0, z0, s0 + i, a.prev_buf);
        tma_load_4d(sb + 2 * kBHalo + kBTile, &mp.tile_f, b, x0, z0, s0 + i, pprev_buf);
    };
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    if (tid < ns) {
        const int kcell = kBTZ / a.TZc;
        const int cbase = ((s0 + tid) * a.ncx + (int)blockIdx.x) * a.ncz;
        const int c0 = tzi * kcell, c1 = min(c0 + kcell, a.ncz);
        taprng[tid][0] = a.inj.cell_start ? a.inj.cell_start[cbase + c0] : 0;
        taprng[tid][1] = a.inj.cell_start ? a.inj.cell_start[cbase + c1] : 0;
        taprng[tid][2] = a.gat.cell_start ? a.gat.cell_start[cbase + c0] : 0;
        taprng[tid][3] = a.gat.cell_start ? a.gat.cell_start[cbase + c1] : 0;
    }
    __syncthreads();
    // up to griddepcontrol.wait only arrays that no step writes are read
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int off[kBRows];
    bool live[kBRows], pad[kBRows];
    float kv[kBRows][4], dv[kBRows][4], eps[kBRows][4], inv[kBRows][4];
#pragma unroll
    for (int rr = 0; rr < kBRows; ++rr) {
        const int gz = z0 + ty + rr * kBBZ;
        off[rr] = gz * a.P + gx;
        live[rr] = gz < a.Nz && nvalid > 0;
        pad[rr] = gz < a.Nz && nvalid <= 0 && gx < a.P;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 k4 = live[rr] ? ld4(a.kap + off[rr]) : zero, d4 = live[rr] ? ld4(a.dmv + off[rr]) : zero;
        const int dz = sponge_depth(gz, a.nb, a.nz);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int dd = max(sponge_depth(gx + e, a.nb, a.nx), dz);
            kv[rr][e] = f4(k4, e);
            dv[rr][e] = f4(d4, e);
            eps[rr][e] = kv[rr][e] * a.ceps * (float)(dd * dd);
            inv[rr][e] = rcp_sponge(1.0f + eps[rr][e]);
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid == 0 && ns > 0) issue(0);

    // (a thread whose wait gives up records it and does no further work, but
    // passes every block barrier below, which are uniform)
    bool alive = true;
    for (int i = 0; i < ns; ++i) {
        if (tid == 0 && alive && i + 1 < ns) {
            fence_proxy_async();
            issue(i + 1);  // into the stage shot i - 1 used (released by the barrier after it)
        }
        if (alive && !mbar_wait(&bar[i & 1], (uint32_t)(i >> 1) & 1u)) {
            alive = false;
            atomicOr(a.err, kErrTimeout);
            if (tid == 0)  // copies issued by this CTA may still land in its shared memory
                for (int j = i; j < i + 2 && j < ns; ++j) mbar_wait(&bar[j & 1], (uint32_t)(j >> 1) & 1u);
        }
        const size_t so = (size_t)(s0 + i) * a.cell;
        float* un = a.unew + so;
        float* pn = pnew_all + so;
        const float* sb = st + (i & 1) * kBStage;
        auto step = [&](const float* halo, const float* tile, int rr, const float* src, float* cen, float* um, float* out) {
            const int r = ty + rr * kBBZ;
            const float* row = halo + (r + 4) * kBSW + lx;
            const float4 A = lds4(row), B = lds4(row + 4), C = lds4(row + 8), o = lds4(tile + r * kTX + lx);
            const float w[12] = {A.x, A.y, A.z, A.w, B.x, B.y, B.z, B.w, C.x, C.y, C.z, C.w};
            float lap[4];
            lap4(w, [&](int k, float4& Up, float4& Dn) {
                Up = lds4(row + 4 - k * kBSW);
                Dn = lds4(row + 4 + k * kBSW);
            }, lap);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                cen[e] = w[e + 4];
                um[e] = f4(o, e);
            }
            update4(cen, um, lap, kv[rr], eps[rr], inv[rr], src, out);
        };
        auto put = [&](float* p, int rr, const float* v) {  // points past Nx stay the zero exterior
            *reinterpret_cast<float4*>(p + off[rr]) = make_float4(v[0], nvalid > 1 ? v[1] : 0.0f, nvalid > 2 ? v[2] : 0.0f,
                                                                   nvalid > 3 ? v[3] : 0.0f);
        };
        float up[kBRows][4], d2[kBRows][4];  // u^{n+1}; u^{n-1} - 2 u^n
        const float zero4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int rr = 0; rr < kBRows; ++rr) {
            if (!alive) break;
            if (!live[rr]) {
                if (pad[rr]) {
                    *reinterpret_cast<float4*>(un + off[rr]) = make_float4(0.f, 0.f, 0.f, 0.f);
                    *reinterpret_cast<float4*>(pn + off[rr]) = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                continue;
            }
            float cen[4], um[4];
            step(sb, sb + 2 * kBHalo, rr, zero4, cen, um, up[rr]);
#pragma unroll
            for (int e = 0; e < 4; ++e) d2[rr][e] = fmaf(-2.0f, cen[e], um[e]);
            put(un, rr, up[rr]);
        }
        const int ib = taprng[i][0], ie = taprng[i][1], gb = taprng[i][2], ge = taprng[i][3];
        if (ie > ib) {
            // the sources: one thread per grid point adds its taps in list order; the secondary
            // source of the points' owners must include them
            __syncthreads();
            for (int j = ib + tid; j < ie; j += 32 * kBBZ) {
                const int k = a.inj.idx[j];
                if (j > ib && a.inj.idx[j - 1] == k) continue;
                float add = 0.0f;
                for (int jj = j; jj < ie && a.inj.idx[jj] == k; ++jj)
                    add = fmaf(a.inj.fac[jj], a.amp_a[(long long)a.inj.ab[jj] + (long long)a.amp_row * a.inj.npts], add);
                un[k] += add;
            }
            __syncthreads();
#pragma unroll
            for (int rr = 0; rr < kBRows; ++rr) {
                if (!live[rr]) continue;
                const float4 v = *reinterpret_cast<const float4*>(un + off[rr]);
#pragma unroll
                for (int e = 0; e < 4; ++e) up[rr][e] = f4(v, e);
            }
        }
#pragma unroll
        for (int rr = 0; rr < kBRows; ++rr) {
            if (!alive || !live[rr]) continue;
            float src[4], cen[4], um[4], out[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) src[e] = dv[rr][e] * (up[rr][e] + d2[rr][e]);
            step(sb + kBHalo, sb + 2 * kBHalo + kBTile, rr, src, cen, um, out);
            put(pn, rr, out);
        }
        // the stage is refilled by shot i + 2's copies, and the gathers read other threads' points
        if (ge > gb || i + 2 < ns) __syncthreads();
        if (ge > gb) {
            float* row = a.slots + (long long)a.slot_row * a.gat.ntap;
            for (int j = gb + tid; j < ge; j += 32 * kBBZ) row[a.gat.slot[j]] = a.gat.gw[j] * pn[a.gat.idx[j]];
        }
    }
}

}  // namespace

void launch_born2d(const StepArgs& a, int p_buf, int pprev_buf, float* pnew, const StepMaps* maps, cudaStream_t s)
{
    constexpr size_t smem = (size_t)2 * kBStage * 4 + 128;
    count_step_launch();
    cudaEvent_t stop;
    const bool timed = profile_sample(false, s, &stop);
    static std::atomic<bool> configured[64];  // kernel attributes are per device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || !configured[dev].load()) {
        cudaFuncSetAttribute(k_born2d, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (dev >= 0 && dev < 64) configured[dev].store(true);
    }
    cudaLaunchConfig_t cfg = {};
    const int group = a.group < 1 ? kBG : (a.group > kBG ? kBG : a.group);
    StepArgs args = a;
    args.group = group;
    cfg.gridDim = dim3(a.ncx, (a.nshot + group - 1) / group, (a.Nz + kBTZ - 1) / kBTZ);
    cfg.blockDim = dim3(32, kBBZ);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_born2d, *maps, args, p_buf, pprev_buf, pnew);
    if (e != cudaSuccess) note_cuda_error(e);  // the caller's cudaGetLastError check reports it
    if (timed) profile_close(stop, s);
}

}  // namespace wave
