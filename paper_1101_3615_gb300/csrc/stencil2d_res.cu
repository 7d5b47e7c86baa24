// Cluster-resident 2D time stepping (sm_103a): many time levels per launch.
//
// A field whose grid fits the shared memory of one thread-block cluster stays there for a whole
// segment of time levels.  The cluster's CTAs own contiguous strips of grid rows (full width); a launch
// loads the two levels of the state, the medium and the pointwise operands once, advances a segment (the
// checkpoint stride; up to twice that in calls without checkpoints), and writes the two last levels back.  Per level a CTA computes its rows
// from the level in shared memory, writes the new level over the older one, and stores its first and
// last four rows into the neighbouring CTAs' halo rows as well (asynchronous distributed-shared-memory
// stores that complete on the neighbour's mbarrier, so data and signal travel together and no store
// is waited for).  One field per cluster: the incident field (writing Dtt u^n of every level to
// device memory), a Born field (reading it), or an adjoint field (reading it, with the image and its
// Kahan compensation resident too).
//
// What bounds it: per level the shared-memory loads of the taps and the instruction issue of one CTA
// per SM, plus the halo exchange (about half a microsecond) -- not memory.  The one-level kernels
// are bound by launch and first-load latency on such grids.  Measured, whole calls, one-level kernels ->
// here: F on 77 x 103, 1 shot, 3 trials, nt = 200 1.79 -> 0.366 ms; H on 141 x 141, 4 shots, nt = 800 12.8 ->
// 2.77 ms; four H in a chain on 241 x 281, 6 shots, nt = 400 38.2 -> 11.0 ms; F* on 277 x 423, 12 shots,
// 2 data sets, nt = 700 29.1 -> 15.6 ms.
//
// The two halves of the halo exchange need no second barrier: the rows whose update reads a
// neighbour's halo rows are exactly the rows sent to that neighbour, so the arrival of all their
// bytes also says that the halo rows of the level they were computed from have been read.
//
// Every cell update is the arithmetic of stencil2d.cu, operation for operation (x taps, then z taps,
// in first-difference form; explicit roundings), so the fields are the same bits.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace probe {

namespace {

constexpr int kResThreads = 512;
constexpr int kResPadMax = 64;  // sponge table of at most 17 KB

// 16 bytes from global to shared memory without passing through registers
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// The two halves of a cluster barrier that orders no memory
__device__ __forceinline__ void cluster_arrive_relaxed() {
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait;" ::: "memory"); }

struct Strip {  // rows of one CTA
    int z0, rows;
};
__host__ __device__ __forceinline__ Strip strip_of(int Nz, int C, int rank) {
    const int base = Nz / C, rem = Nz % C;
    return {rank * base + (rank < rem ? rank : rem), base + (rank < rem ? 1 : 0)};
}

__host__ __device__ __forceinline__ int res_groups(int Nx) { return (Nx + 3) / 4; }
__host__ __device__ __forceinline__ int res_pitch(int Nx) { return 4 * (res_groups(Nx) + 2); }
// Rows of the largest strip, rounded up to whole blocks of RB
__host__ __device__ __forceinline__ int res_rows(int Nz, int C, int RB) {
    return ((Nz + C - 1) / C + RB - 1) / RB * RB;
}
// Sponge factors G = 1 / (1 + e) by (rho_z, rho_x): one per distinct pair, and a last column of
// zeros for the pitch columns
__host__ __device__ __forceinline__ int res_gtab(int pad) { return ((pad + 1) * (pad + 2) + 3) / 4 * 4; }
// Resident planes besides the two levels: s; dm (Born); image and compensation (adjoint)
__host__ __device__ __forceinline__ int res_planes(int mode, bool kahan) {
    return mode == RES_INC ? 1 : (mode == RES_BORN ? 2 : (kahan ? 3 : 2));
}

size_t res_smem(int mode, bool kahan, int Nz, int Nx, int pad, int C, int RB, int nsteps) {
    const size_t rp = res_rows(Nz, C, RB), gx4 = 4 * res_groups(Nx);
    return 4 * (2 * (rp + 8) * res_pitch(Nx) + res_planes(mode, kahan) * rp * gx4 + 2 * gx4 + rp + res_gtab(pad) +
                nsteps);
}

template <int MODE, bool KAHAN, int RB>
__global__ void __launch_bounds__(kResThreads, 1) k_res2d(const __grid_constant__ ResParams2D p) {
    extern __shared__ __align__(128) float smem[];
    __shared__ __align__(8) uint64_t bars[2];
    const int C = p.C, tid = threadIdx.x, nthr = blockDim.x;
    const int rank = (C > 1) ? (int)cluster_ctarank() : 0;
    const int unit = blockIdx.x / C;
    const int shot = unit / p.nfield, b = unit - shot * p.nfield;
    const Strip me = strip_of(p.Nz, C, rank);
    const int R = me.rows, z0 = me.z0;
    const int gx = res_groups(p.Nx), PW = res_pitch(p.Nx), PX = 4 * gx;
    const int RP = res_rows(p.Nz, C, RB), BR = RP + 8;
    float* S = smem + 2 * BR * PW;
    float* A1 = S + RP * PX;    // Born: dm; adjoint: image
    float* A2 = A1 + RP * PX;   // adjoint with Kahan: compensation
    float* xt = S + res_planes(MODE, KAHAN) * RP * PX;  // cx rho_x^2 of every column
    int* xr = reinterpret_cast<int*>(xt + PX);          // rho_x of every column, pad + 1 past the grid
    float* gt = xt + 2 * PX;                            // G by (rho_z, rho_x)
    int* band = reinterpret_cast<int*>(gt + res_gtab(p.pad));  // adjoint: injection band of every row
    float* wl = gt + res_gtab(p.pad) + RP;              // incident: w[n] / (h_z h_x) of every level
    const bool up = rank > 0, dn = rank < C - 1;
    const long long F = p.F;
    // two levels in shared memory, level k of the launch in the (k & 1)-th: the first to be differentiated at smem
    const float* in0 = p.in + ((long long)unit * 2 + p.pin) * F;
    const float* in1 = p.in + ((long long)unit * 2 + (p.pin ^ 1)) * F;
    float* gimg = (MODE == RES_ADJ) ? p.img + (long long)unit * F : nullptr;
    float* gcmp = (MODE == RES_ADJ && KAHAN) ? p.comp + (long long)unit * F : nullptr;

    // Everything the segment reads from memory but Dtt, as asynchronous copies, a warp per row: no
    // thread waits for a load before it issues its next, and the tables below are made meanwhile.
    // Cells off the grid are zero in both levels (a neighbour's rows arrive after the cluster barrier).
    const int warp = tid >> 5, lane = tid & 31, nwarp = nthr >> 5;
    for (int r = warp; r < BR; r += nwarp) {
        const int z = z0 - 4 + r;
        const bool row0 = z >= 0 && z < p.Nz && r < R + 8, row1 = r >= 4 && r < R + 4;
        for (int g = lane; g < gx + 2; g += 32) {
            const bool col = g >= 1 && g <= gx;
            float* lv = smem + r * PW + 4 * g;
            const long long off = (long long)z * p.P + 4 * (g - 1);
            if (row0 && col)
                cp_async16(lv, in0 + off);
            else
                st4(lv, make_float4(0.f, 0.f, 0.f, 0.f));
            if (row1 && col) {
                const int q = (r - 4) * PX + 4 * (g - 1);
                cp_async16(lv + BR * PW, in1 + off);
                cp_async16(S + q, p.s + off);
                if (MODE == RES_BORN) cp_async16(A1 + q, p.dm + (long long)b * F + off);
                if (MODE == RES_ADJ) cp_async16(A1 + q, gimg + off);
                if (MODE == RES_ADJ && KAHAN) cp_async16(A2 + q, gcmp + off);
            } else {
                st4(lv + BR * PW, make_float4(0.f, 0.f, 0.f, 0.f));
            }
        }
    }
    for (int i = tid; i < PX; i += nthr) {
        const int rx = max(max(p.pad - i, i - (p.pad + p.nx - 1)), 0);
        xt[i] = __fmul_rn(p.cx, (float)(rx * rx));
        xr[i] = i < p.Nx ? rx : p.pad + 1;
    }
    for (int i = tid; i < (p.pad + 1) * (p.pad + 2); i += nthr) {
        const int rz = i / (p.pad + 2), rx = i - rz * (p.pad + 2);
        float G = 1.f, am = 1.f;
        sponge_pair(__fmaf_rn(p.cz, (float)(rz * rz), __fmul_rn(p.cx, (float)(rx * rx))), G, am);
        gt[i] = rx <= p.pad ? G : 0.f;
    }
    if (MODE == RES_INC)
        for (int i = tid; i < p.nsteps; i += nthr) wl[i] = p.wavelet[p.n0 + i] * p.vol_inv;
    if (MODE == RES_ADJ)
        for (int i = tid; i < R; i += nthr) band[i] = p.rrow ? p.rrow[z0 + i] : -1;
    const unsigned rx_bytes = (unsigned)((up ? 4 : 0) + (dn ? 4 : 0)) * gx * 16u;
    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        fence_mbar_init();
        // level k + 1 arrives while this CTA works on level k
        if (C > 1 && p.nsteps >= 2) mbar_arm_tx(&bars[1], rx_bytes);
        if (C > 1 && p.nsteps >= 3) mbar_arm_tx(&bars[0], rx_bytes);
    }
    uint32_t halo_up = 0, halo_dn = 0, bar_up = 0, bar_dn = 0;  // neighbours' halo rows (of the first level) and bars[0]
    if (up) {
        const int rows_up = strip_of(p.Nz, C, rank - 1).rows;
        halo_up = mapa_rank(smem_u32(smem + (rows_up + 4) * PW + 4), (uint32_t)(rank - 1));
        bar_up = mapa_rank(smem_u32(&bars[0]), (uint32_t)(rank - 1));
    }
    if (dn) {
        halo_dn = mapa_rank(smem_u32(smem + 4), (uint32_t)(rank + 1));
        bar_dn = mapa_rank(smem_u32(&bars[0]), (uint32_t)(rank + 1));
    }
    const int nrb = (R + RB - 1) / RB, ntask = nrb * gx;
    const int dq = nthr / gx, dr = nthr - dq * gx;
    const int t0q = tid / gx, t0r = tid - t0q * gx;
    // row block of task order q: the strip's first and last blocks come first (their rows travel)
    auto block_of = [&](int q) { return q == 0 ? 0 : (q == 1 ? nrb - 1 : q - 1); };
    // receivers sampled by this CTA (rows z0 .. z0 + R - 1); each thread keeps its first one
    const bool sample = MODE != RES_ADJ && p.data != nullptr;
    const int rbeg = sample ? p.rec_ptr[z0] : 0, rend = sample ? p.rec_ptr[z0 + R] : 0;
    auto rec_off = [&](int r) { return (p.rec_zx[2 * r] - z0 + 4) * PW + 4 + p.rec_zx[2 * r + 1]; };
    int my_rec = -1, my_off = 0;
    if (rbeg + tid < rend) {
        my_rec = p.rec_idx[rbeg + tid];
        my_off = rec_off(my_rec);
    }
    float* dout = sample ? p.data + (long long)shot * p.dss + (long long)b * p.dts : nullptr;
    float* dtt = p.dtt ? p.dtt + (long long)shot * p.dtt_shot_stride : nullptr;
    const int sz = (MODE == RES_INC) ? p.src_zx[2 * shot] : -1, sx = (MODE == RES_INC) ? p.src_zx[2 * shot + 1] : -1;

    // Dtt of a thread's first task of a level, fetched one level ahead
    float4 dpre[RB];
    auto fetch_dtt = [&](int k, int q, int g, float4 d[RB]) {
        const int r0 = block_of(q) * RB;
        const float* src = dtt + (long long)(MODE == RES_ADJ ? p.slot0 - k : p.slot0 + k) * F + 4 * g;
#pragma unroll
        for (int r = 0; r < RB; ++r)
            d[r] = (r0 + r < R) ? __ldg(reinterpret_cast<const float4*>(src + (long long)(z0 + r0 + r) * p.P))
                                : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    if (MODE != RES_INC && tid < ntask) fetch_dtt(0, t0q, t0r, dpre);

    cp_async_wait_all();
    if (C > 1)
        cluster_sync_all();
    else
        __syncthreads();

    for (int k = 0; k < p.nsteps; ++k) {
        const float* cur = smem + (k & 1) * BR * PW;
        float* oth = smem + ((k + 1) & 1) * BR * PW;
        const uint32_t oth_off = (uint32_t)((k + 1) & 1) * BR * PW * 4u, oth_bar = (uint32_t)((k + 1) & 1) * 8u;
        const bool last = k + 1 == p.nsteps;
        const int n = (MODE == RES_ADJ) ? p.n0 - k : p.n0 + k;
        int q = t0q, g = t0r;
        for (int t = tid; t < ntask; t += nthr) {
            const int r0 = block_of(q) * RB, x = 4 * g;
            float4 D[RB];
            if (MODE != RES_INC) {
                if (t == tid) {
#pragma unroll
                    for (int r = 0; r < RB; ++r) D[r] = dpre[r];
                } else {
                    fetch_dtt(k, q, g, D);
                }
            }
            const float* c0 = cur + (r0 + 4) * PW + 4 + x;
            P4 L[RB], cc[RB];
#pragma unroll
            for (int r = 0; r < RB; ++r) {  // x taps: 11 shared differences for 4 cells
                const float4 a = ld4(c0 + r * PW - 4), m = ld4(c0 + r * PW), e = ld4(c0 + r * PW + 4);
                const float v[12] = {a.x, a.y, a.z, a.w, m.x, m.y, m.z, m.w, e.x, e.y, e.z, e.w};
                float d[11], o[4];
#pragma unroll
                for (int i = 0; i < 11; ++i) d[i] = v[i + 1] - v[i];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float acc = p.cxm[0] * (d[4 + j] - d[3 + j]);
#pragma unroll
                    for (int mm = 1; mm < 4; ++mm) acc = fmaf(p.cxm[mm], d[4 + j + mm] - d[3 + j - mm], acc);
                    o[j] = acc;
                }
                L[r] = p4(o[0], o[1], o[2], o[3]);
                cc[r] = p4(m);
            }
            {  // z taps: differences of neighbouring rows, shared by the RB rows
                P4 d[RB + 7];
                P4 prev = p4(ld4(c0 - 4 * PW));
#pragma unroll
                for (int i = 0; i < RB + 7; ++i) {
                    const P4 nx = (i >= 3 && i < 3 + RB) ? cc[(i >= 3 && i < 3 + RB) ? i - 3 : 0] : p4(ld4(c0 + (i - 3) * PW));
                    d[i] = p4sub(nx, prev);
                    prev = nx;
                }
#pragma unroll
                for (int r = 0; r < RB; ++r)
#pragma unroll
                    for (int mm = 0; mm < 4; ++mm) {
                        const float w = p.czm[mm];
                        L[r] = p4fma(p4(w, w, w, w), p4sub(d[r + 4 + mm], d[r + 3 - mm]), L[r]);
                    }
            }
            const int zb = z0 + r0;
            const P4 ex = p4(ld4(xt + x));
            const int4 ix = *reinterpret_cast<const int4*>(xr + x);
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                if (r0 + r >= R) break;
                const int z = zb + r;
                const int qo = (r0 + r) * PX + x;
                float* op = oth + (r0 + r + 4) * PW + 4 + x;
                if (MODE == RES_INC && z == sz) {
                    const float4 l = f4(L[r]);
                    float a[4] = {l.x, l.y, l.z, l.w};
                    add_lane(a, sx - x, wl[k]);
                    L[r] = p4(a[0], a[1], a[2], a[3]);
                }
                if (MODE == RES_ADJ && band[r0 + r] >= 0) {  // receiver injection R^T r^n of the segment
                    const float4 in = __ldg(reinterpret_cast<const float4*>(
                        p.inj + (((long long)k * p.nshots + shot) * p.nfield + b) * p.inj_block +
                        (long long)band[r0 + r] * p.P + x));
                    L[r] = p4add(L[r], p4(in));
                }
                if (MODE == RES_BORN) L[r] = p4fma(p4neg(p4(ld4(A1 + qo))), p4(D[r]), L[r]);
                // u = G (2c - a- u_old + s L), a- = 1 - e; G = a- = 1 off the sponge, G = 0 off the grid
                const P4 Fo = p4mul(p4(ld4(S + qo)), L[r]);
                const int rz = max(max(p.pad - z, z - (p.pad + p.nz - 1)), 0);
                const float ez = (float)(rz * rz);
                const P4 am = p4sub(p4(1.f, 1.f, 1.f, 1.f), p4fma(p4(p.cz, p.cz, p.cz, p.cz), p4(ez, ez, ez, ez), ex));
                const float* gz = gt + rz * (p.pad + 2);
                const P4 G = p4(gz[ix.x], gz[ix.y], gz[ix.z], gz[ix.w]);
                const float4 o = f4(p4mul(
                    G, p4add_one(Fo, p4fma(p4neg(am), p4(ld4(op)), p4add(cc[r], cc[r])), p.one)));
                st4(op, o);
                if (!last) {
                    if (up && r0 + r < 4)
                        st_async4(halo_up + oth_off + (uint32_t)((r0 + r) * PW + x) * 4u, o, bar_up + oth_bar);
                    if (dn && r0 + r >= R - 4)
                        st_async4(halo_dn + oth_off + (uint32_t)((r0 + r - (R - 4)) * PW + x) * 4u, o, bar_dn + oth_bar);
                }
                if (MODE == RES_INC && dtt) {
                    const float i2 = p.inv_dt2;
                    st4(dtt + (long long)(p.slot0 + k) * F + (long long)z * p.P + x, f4(p4mul(Fo, p4(i2, i2, i2, i2))));
                }
                if (MODE == RES_ADJ) {  // img -= Dtt u^{n-1} mu^n
                    float4 iv = ld4(A1 + qo);
                    const float4 t = make_float4(__fmul_rn(-D[r].x, o.x), __fmul_rn(-D[r].y, o.y),
                                                 __fmul_rn(-D[r].z, o.z), __fmul_rn(-D[r].w, o.w));
                    if (KAHAN) {
                        float4 cv = ld4(A2 + qo);
                        kahan4(iv, cv, t.x, t.y, t.z, t.w);
                        st4(A2 + qo, cv);
                    } else {  // scalar: a packed product and sum may be contracted into one rounding
                        iv = make_float4(__fadd_rn(iv.x, t.x), __fadd_rn(iv.y, t.y), __fadd_rn(iv.z, t.z),
                                         __fadd_rn(iv.w, t.w));
                    }
                    st4(A1 + qo, iv);
                }
            }
            q += dq;
            g += dr;
            if (g >= gx) {
                g -= gx;
                ++q;
            }
        }
        if (sample) {  // level n at the receivers
            if (my_rec >= 0) dout[(long long)n * p.nr + my_rec] = cur[my_off];
            for (int i = rbeg + tid + nthr; i < rend; i += nthr) {
                const int r = p.rec_idx[i];
                dout[(long long)n * p.nr + r] = cur[rec_off(r)];
            }
        }
        if (MODE != RES_INC && !last && tid < ntask) fetch_dtt(k + 1, t0q, t0r, dpre);
        bool ok = true;
        if (C > 1 && !last) {  // the neighbours' rows of the new level
            ok = mbar_wait_bounded(&bars[(k + 1) & 1], (uint32_t)((k >> 1) & 1));
            if (tid == 0 && k + 3 < p.nsteps) mbar_arm_tx(&bars[(k + 1) & 1], rx_bytes);
        }
        if (__syncthreads_or(!ok)) {
            if (tid == 0) set_dev_error(p.err, DEVERR_TIMEOUT);
            break;
        }
    }
    // No CTA leaves while a neighbour's stores may still be on their way to it.
    if (C > 1) cluster_arrive_relaxed();
    // both levels back, the image with them
    const float *c0 = smem + (p.nsteps & 1) * BR * PW, *c1 = smem + ((p.nsteps & 1) ^ 1) * BR * PW;
    for (int r = warp; r < R; r += nwarp)
        for (int g = lane; g < gx; g += 32) {
            const long long off = (long long)(z0 + r) * p.P + 4 * g;
            if (p.out) {
                st4(p.out + ((long long)unit * 2 + p.pout) * F + off, ld4(c0 + (r + 4) * PW + 4 + 4 * g));
                st4(p.out + ((long long)unit * 2 + (p.pout ^ 1)) * F + off, ld4(c1 + (r + 4) * PW + 4 + 4 * g));
            }
            if (MODE == RES_ADJ) st4(gimg + off, ld4(A1 + r * PX + 4 * g));
            if (MODE == RES_ADJ && KAHAN) st4(gcmp + off, ld4(A2 + r * PX + 4 * g));
        }
    if (C > 1) cluster_wait();
}

void res_config(int C, int threads, size_t smem, int units, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr) {
    cfg = {};
    cfg.gridDim = dim3((unsigned)(C * units));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

// A plan is made before its first launch, so the kernel's limits (raised to the most that any plan
// uses) are set here and not with each launch.
template <int MODE, bool KAHAN, int RB>
int res_clusters(int C, int threads, size_t smem) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    res_config(C, threads, smem, 1, cfg, attr);
    int n = 0;
    auto kernel = k_res2d<MODE, KAHAN, RB>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmemMax) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <int MODE, bool KAHAN, int RB>
cudaError_t res_launch(const ResPlan& pl, const ResParams2D& p, int units, cudaStream_t st) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    res_config(pl.C, pl.threads, res_smem(MODE, KAHAN, p.Nz, p.Nx, p.pad, pl.C, RB, p.nsteps), units, cfg, attr);
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, k_res2d<MODE, KAHAN, RB>, p);
}

template <int MODE, bool KAHAN>
int res_clusters_rb(int RB, int C, int threads, size_t smem) {
    if (RB == 1) return res_clusters<MODE, KAHAN, 1>(C, threads, smem);
    return RB == 4 ? res_clusters<MODE, KAHAN, 4>(C, threads, smem) : res_clusters<MODE, KAHAN, 2>(C, threads, smem);
}

template <int MODE, bool KAHAN>
cudaError_t res_launch_rb(const ResPlan& pl, const ResParams2D& p, int units, cudaStream_t st) {
    if (pl.RB == 1) return res_launch<MODE, KAHAN, 1>(pl, p, units, st);
    return pl.RB == 4 ? res_launch<MODE, KAHAN, 4>(pl, p, units, st) : res_launch<MODE, KAHAN, 2>(pl, p, units, st);
}

}  // namespace

bool res2d_fits(int mode, bool kahan, int Nz, int Nx, int pad, int nsteps) {
    int C = 16;
    while (C > 1 && Nz / C < 4) C /= 2;  // the most CTAs share the planes
    return pad <= kResPadMax && res_smem(mode, kahan, Nz, Nx, pad, C, 2, nsteps) <= kResSmemMax;
}

// Candidate cluster sizes (not only powers of two: with 9 CTAs the chip holds 15 clusters, as with 8,
// and a strip is an eighth lower; 241 x 281, 6 shots, Krylov trials 13.4 -> 11.1 ms; 11, 13 and 15 have
// not been timed) and rows per
// thread for fields of an Nz x Nx grid, each with the number of
// clusters that the chip holds at once and the estimated time of one level of one wave of clusters.
// The model (microseconds), fitted on 77 x 103 to 277 x 423 grids, C = 1 to 16, within about 15 %:
// exchange and barriers 0.55 (0.3 in a single CTA); then per round of tasks, with w warps,
// max(0.73, 0.45 + 0.078 w) with four rows per thread, max(0.32, 0.2 + 0.045 w) with two,
// max(0.22, 0.1 + 0.034 w) with one; Born 1.17, adjoint 1.4 times that.  More rows per thread share more
// differences, fewer make a shorter chain: 77 x 103, clusters of 16, a level of the incident field
// 1.24, 0.93 and 0.79 us with four, two and one; 241 x 281 1.65, 1.89 and 1.85.
std::vector<ResPlan> plan_res2d(int mode, bool kahan, int Nz, int Nx, int pad, int nsteps) {
    std::vector<ResPlan> out;
    const int gx = res_groups(Nx);
    for (int C : {1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 16}) {
        if (C > 1 && Nz / C < 4) break;  // a halo row must belong to the adjacent strip
        for (int RB : {4, 2, 1}) {
            const size_t sm = res_smem(mode, kahan, Nz, Nx, pad, C, RB, nsteps);
            if (sm > kResSmemMax) continue;
            const int rows = (Nz + C - 1) / C, ntask = (rows + RB - 1) / RB * gx;
            const int rounds = (ntask + kResThreads - 1) / kResThreads;
            ResPlan pl;
            pl.C = C;
            pl.RB = RB;
            pl.threads = std::min(kResThreads, ((ntask + rounds - 1) / rounds + 31) / 32 * 32);
            switch (mode) {
                case RES_INC: pl.clusters = res_clusters_rb<RES_INC, false>(RB, C, pl.threads, sm); break;
                case RES_BORN: pl.clusters = res_clusters_rb<RES_BORN, false>(RB, C, pl.threads, sm); break;
                default:
                    pl.clusters = kahan ? res_clusters_rb<RES_ADJ, true>(RB, C, pl.threads, sm)
                                        : res_clusters_rb<RES_ADJ, false>(RB, C, pl.threads, sm);
            }
            if (pl.clusters < 1) continue;
            const double f = mode == RES_INC ? 1.0 : (mode == RES_BORN ? 1.17 : 1.4), w = pl.threads / 32;
            const double task = RB == 4   ? std::max(0.73, 0.45 + 0.078 * w)
                                : RB == 2 ? std::max(0.32, 0.2 + 0.045 * w)
                                          : std::max(0.22, 0.1 + 0.034 * w);
            pl.us = (C > 1 ? 0.55 : 0.3) + f * rounds * task;
            out.push_back(pl);
        }
    }
    return out;
}

cudaError_t launch_res2d(int mode, bool kahan, const ResPlan& pl, const ResParams2D& p0, cudaStream_t st) {
    ResParams2D p = p0;
    p.C = pl.C;
    p.one = 1.f;
    const int units = p.nshots * p.nfield;
    if (units <= 0 || p.nsteps <= 0) return cudaSuccess;
    switch (mode) {
        case RES_INC: return res_launch_rb<RES_INC, false>(pl, p, units, st);
        case RES_BORN: return res_launch_rb<RES_BORN, false>(pl, p, units, st);
        case RES_ADJ:
            return kahan ? res_launch_rb<RES_ADJ, true>(pl, p, units, st) : res_launch_rb<RES_ADJ, false>(pl, p, units, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace probe
