// 3D time-stepping kernels with the z taps in registers (sm_103a).
//
// As in stencil3d.cu a CTA marches 64 (x) x 16 (y) columns through a chunk of z planes and one thread
// updates 4 consecutive x cells per plane.  Here
//   * a thread keeps the nine values of its column that the z taps need in a register queue (the plane
//     loop is unrolled by nine, so the queue never moves): the z taps cost no shared-memory loads and no
//     ring-slot arithmetic;
//   * everything a plane needs comes by TMA: the halo'd plane tile (72 x 24) through a ring of nine
//     slots, the pointwise operands (64 x 16 each) through a ring of three or two stages, issued by a
//     producer warp against per-slot full / empty mbarriers; halo slots and barrier phases are constants
//     inside the unrolled loop;
//   * the adjoint touches the image (and Dtt u) every third step only: the step that computes mu^n also
//     holds mu^{n+1} (the differentiated level) and mu^{n+2} (the level it overwrites), so it adds the
//     imaging terms of all three, in the order in which the single steps would.
//
// What bounds it: issue and operand latency at two CTAs (18 warps) per SM below DRAM -- 300 instructions
// per warp and plane, issue active half of the cycles, DRAM 5.1 to 5.8 TB/s in the adjoint and 4.2 in
// the incident step (168 x 256 x 296, 4 shots, 4 trials).  Measured against the kernels of
// stencil3d.cu as they were tuned, whole calls: H on 296^3 (padded), 8 shots, 4 trials, 60 levels 528 ->
// 465 ms; H on 116 x 101 x 141, 3 shots 45.2 -> 34.7 ms; F on 168^3, 4 shots, 2 trials 42.9 -> 38.8 ms.
// Slower variants: two trials per CTA, two rows per thread, a refill by the last compute warp.  At the 96
// registers that two CTAs per SM leave, every instantiation spills (16 to 84 bytes stored per thread).
//
// The per-cell arithmetic is that of cells3 in stencil3d.cu, operation for operation: same bits.
#include "common.cuh"
#include "internal.h"

namespace probe {

namespace {

constexpr int kQH = 9;                   // halo ring slots = planes of the z queue
constexpr int kQHX = kTX + 8;            // 72
constexpr int kQHalo = kQHX * (kTY3D + 8);  // floats of a halo'd plane tile
constexpr int kQTile = kTX * kTY3D;      // floats of a plain plane tile
constexpr unsigned kQHaloB = kQHalo * 4u, kQTileB = kQTile * 4u;

// Operand tiles per stage: the older level, s, then (Born) Dtt u and dm or (adjoint with NI imaging
// terms) NI planes of Dtt u and the image; stages so that two CTAs share an SM.
template <int MODE, int NI>
struct QOps {
    static constexpr int N = MODE == STEP3_BORN ? 4 : (MODE == STEP3_ADJ && NI ? 3 + NI : 2);
    static constexpr int STAGES = N <= 4 ? 3 : 2;
    static constexpr int FLOATS = N * kQTile;
    static constexpr size_t SMEM = ((size_t)kQH * kQHalo + (size_t)STAGES * FLOATS) * 4;
};

__device__ __forceinline__ float q_sponge_e(const ModelStep3D& M, int z, int y, int x) {
    const int rz = max(max(M.pad - z, z - (M.pad + M.nz - 1)), 0);
    const int ry = max(max(M.pad - y, y - (M.pad + M.ny - 1)), 0);
    const int rx = max(max(M.pad - x, x - (M.pad + M.nx - 1)), 0);
    return __fmaf_rn(M.cz, (float)(rz * rz), __fmaf_rn(M.cy, (float)(ry * ry), __fmul_rn(M.cx, (float)(rx * rx))));
}

template <int MODE, int NI>
__global__ void __launch_bounds__(kThreads + 32, 2) k_step3d_q(const __grid_constant__ StepParams3D p) {
    using O = QOps<MODE, NI>;
    constexpr bool INC = MODE == STEP3_INC || MODE == STEP3_INC_SAMPLE;
    constexpr bool SAMPLE = MODE == STEP3_BORN || MODE == STEP3_INC_SAMPLE;
    constexpr bool ADJ = MODE == STEP3_ADJ;
    constexpr int NO = O::STAGES;
    extern __shared__ __align__(128) float smem[];
    __shared__ __align__(8) uint64_t hfull[kQH], hempty[kQH], ofull[NO], oempty[NO];
    __shared__ int srec[kZCMax3D + 1];  // sampling: receiver CSR bounds of the planes; adjoint: injection bands
    const ModelStep3D& M = p.m;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // grid.x: field fastest, then (shots_inner) the shots, then the column tile and the chunk, then
    // (otherwise) the shots
    int t = blockIdx.x;
    const int b = t % M.nfield;
    t /= M.nfield;
    int shot = 0;
    if (M.shots_inner) {
        shot = t % M.nshots;
        t /= M.nshots;
    }
    const int txi = t % M.tiles_x;
    t /= M.tiles_x;
    const int tyi = t % M.tiles_y;
    t /= M.tiles_y;
    const int zc = t % M.zchunks;
    if (!M.shots_inner) shot = t / M.zchunks;
    const int x0 = txi * kTX, y0 = tyi * kTY3D, z0 = zc * M.ZC;
    const int nloc = min(z0 + M.ZC, M.Nz) - z0;
    const int n = p.n;
    const int pc = ADJ ? ((n + 1) & 1) : (n & 1), po = pc ^ 1;
    float* hring = smem;                  // [kQH][kQHalo]
    float* oring = smem + kQH * kQHalo;   // [NO][O::FLOATS]

    if (tid == 0) {
        for (int i = 0; i < kQH; ++i) {
            mbar_init(&hfull[i], 1);
            mbar_init(&hempty[i], kThreads / 32);
        }
        for (int i = 0; i < NO; ++i) {
            mbar_init(&ofull[i], 1);
            mbar_init(&oempty[i], kThreads / 32);
        }
        fence_mbar_init();
    }
    if (SAMPLE && tid <= nloc) srec[tid] = M.rec_ptr[(tyi * M.tiles_x + txi) * M.Nz + z0 + tid];
    if (ADJ && tid < nloc) srec[tid] = (M.rrow && M.inj) ? M.rrow[z0 + tid] : -1;
    __syncthreads();

    if (warp == kThreads / 32) {  // ---------------- producer warp
        if (lane != 0) return;
        const int vol = shot * M.nvol_shot + 2 * b;
        auto halo = [&](int k, int slot) {
            mbar_expect_tx(&hfull[slot], kQHaloB);
            tma_load_4d(hring + slot * kQHalo, &M.tm, x0 - 4, y0 - 4, z0 - 4 + k, vol + pc, &hfull[slot]);
        };
        const bool own = MODE == STEP3_BORN || (ADJ && NI && !M.seg_first);  // dm, or the image to add to
        const unsigned obytes = kQTileB * (unsigned)(O::N - ((ADJ && NI && !own) ? 1 : 0));
        int hs = 0, os = 0;
        uint32_t hph = 1, oph = 1;  // a fresh barrier passes a wait for the phase before its first
        for (int k = 0; k < 8; ++k, ++hs) halo(k, hs);
        for (int i = 0; i < nloc; ++i) {
            const int z = z0 + i;
            if (!mbar_wait_bounded(&oempty[os], oph)) {
                set_dev_error(p.err, DEVERR_TIMEOUT);
                return;
            }
            float* st = oring + os * O::FLOATS;
            mbar_expect_tx(&ofull[os], obytes);
            tma_load_4d(st, &M.tm_prev, x0, y0, z, vol + po, &ofull[os]);
            tma_load_4d(st + kQTile, &M.tm_s, x0, y0, z, 0, &ofull[os]);
            if (MODE == STEP3_BORN)
                tma_load_4d(st + 2 * kQTile, &M.tm_d, x0, y0, z, shot * M.d_slots + M.d_slot, &ofull[os]);
            if (ADJ)
                for (int c = 0; c < NI; ++c)  // Dtt u^{m-1} of m = n + NI - 1 - c
                    tma_load_4d(st + (2 + c) * kQTile, &M.tm_d, x0, y0, z, shot * M.d_slots + M.d_slot + NI - 1 - c,
                                &ofull[os]);
            if (own)
                tma_load_4d(st + (O::N - 1) * kQTile, &M.tm_own, x0, y0, z, ADJ ? shot * M.nfield + b : b, &ofull[os]);
            if (++os == NO) {
                os = 0;
                oph ^= 1u;
            }
            if (!mbar_wait_bounded(&hempty[hs], hph)) {
                set_dev_error(p.err, DEVERR_TIMEOUT);
                return;
            }
            halo(i + 8, hs);
            if (++hs == kQH) {
                hs = 0;
                hph ^= 1u;
            }
        }
        return;
    }

    // ---------------- consumer warps
    const int lx = (tid & 15) << 2, ly = tid >> 4;
    const int x = x0 + lx, y = y0 + ly;
    const bool col_ok = (x < M.Nx) && (y < M.Ny);
    const bool tile_in = x0 >= M.pad && x0 + kTX <= M.pad + M.nx && y0 >= M.pad && y0 + kTY3D <= M.pad + M.ny;
    // sponge factors of the column on the planes where z is not in the sponge (G = 0 past the grid)
    float4 Gc, Ac;
    {
        float g[4], a[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            g[j] = 1.f;
            a[j] = 1.f;
            sponge_pair(q_sponge_e(M, M.pad, y, x + j), g[j], a[j]);
            if (x + j >= M.Nx) g[j] = 0.f;
        }
        Gc = make_float4(g[0], g[1], g[2], g[3]);
        Ac = make_float4(a[0], a[1], a[2], a[3]);
    }
    const int sz = INC ? M.src[3 * shot] : -1;
    const bool src_row = INC && M.src[3 * shot + 1] == y;
    const int src_j = INC ? M.src[3 * shot + 2] - x : 0;
    const float fsrc = INC ? __fmul_rn(M.wavelet[n], M.vol_inv) : 0.f;  // added below: not to be fused into the sum
    const long long plane = (long long)M.Ny * M.P;
    const long long off0 = ((long long)z0 * M.Ny + y) * M.P + x;
    float* outp = M.state + (long long)(shot * M.nvol_shot + 2 * b + po) * M.F + off0;
    float* auxp = nullptr;  // incident: where Dtt u^n goes; adjoint: the image
    if (INC && M.Dout) auxp = M.Dout + (long long)shot * M.Dout_shot_stride + off0;
    if (ADJ && NI) auxp = M.img + (long long)(shot * M.nfield + b) * M.F + off0;
    float* dout = SAMPLE ? M.data + (long long)shot * M.dss + (long long)b * M.dts + (long long)n * M.nr : nullptr;
    const float* hbase = hring + (ly + 4) * kQHX + lx + 4;
    const float* obase = oring + ly * kTX + lx;
    const float one = p.one;

    P4 q[kQH];  // the column's values, ring plane k in q[k % 9]
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        ok = ok && mbar_wait_bounded(&hfull[k], 0u);
        q[k] = p4(ld4(hbase + k * kQHalo));
    }
    __syncwarp();
    if (lane == 0)
        for (int k = 0; k < 4; ++k) mbar_arrive(&hempty[k]);  // planes below the chunk: only the columns were needed
    uint32_t par = 0;  // parity of iz / 9
    for (int base = 0; base < nloc && ok; base += kQH, par ^= 1u) {
#pragma unroll
        for (int u = 0; u < kQH; ++u) {
            const int iz = base + u;
            if (iz >= nloc) break;
            const int z = z0 + iz;
            const int sn = (u + 8) % kQH, sc = (u + 4) % kQH;  // newest and current plane
            const int so = NO == 3 ? u % 3 : iz & 1;            // operand stage, its iz / NO-th use
            const uint32_t opar = NO == 3 ? (((u / 3) & 1) ? (par ^ 1u) : par) : (uint32_t)((iz >> 1) & 1);
            // plane k = iz + 8 is the (iz + 8) / 9-th use of its slot
            ok = mbar_wait_bounded(&hfull[sn], u == 0 ? par : (par ^ 1u)) && mbar_wait_bounded(&ofull[so], opar);
            if (!ok) {
                set_dev_error(p.err, DEVERR_TIMEOUT);
                break;
            }
            const float* cur = hbase + sc * kQHalo;
            q[sn] = p4(ld4(hbase + sn * kQHalo));
            if (SAMPLE) {  // receivers of this plane, from its staged tile
                const int rend = srec[iz + 1];
                for (int i = srec[iz] + tid; i < rend; i += kThreads) {
                    const int r = M.rec_idx[i];
                    dout[r] = (hring + sc * kQHalo)[(M.rec_zyx[3 * r + 1] - y0 + 4) * kQHX + (M.rec_zyx[3 * r + 2] - x0 + 4)];
                }
            }
            if (col_ok) {
                const P4 cc = q[sc];
                P4 acc;
                {  // x taps in first-difference form (11 shared differences for the 4 cells)
                    const float4 a = ld4(cur - 4), c = f4(cc), d = ld4(cur + 4);
                    const float v[12] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w, d.x, d.y, d.z, d.w};
                    float dx[11], L[4];
#pragma unroll
                    for (int i = 0; i < 11; ++i) dx[i] = v[i + 1] - v[i];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float s = M.cxm[0] * (dx[4 + j] - dx[3 + j]);
#pragma unroll
                        for (int m = 1; m < 4; ++m) s = fmaf(M.cxm[m], dx[4 + j + m] - dx[3 + j - m], s);
                        L[j] = s;
                    }
                    acc = p4(L[0], L[1], L[2], L[3]);
                }
#pragma unroll
                for (int k = 1; k <= 4; ++k) {
                    const P4 up = p4(ld4(cur - k * kQHX)), dn = p4(ld4(cur + k * kQHX));
                    const float w = M.ly[k - 1];
                    acc = p4fma(p4(w, w, w, w), p4add(p4sub(up, cc), p4sub(dn, cc)), acc);
                }
#pragma unroll
                for (int k = 1; k <= 4; ++k) {
                    const P4 up = q[(u + 4 - k + kQH) % kQH], dn = q[(u + 4 + k) % kQH];
                    const float w = M.lz[k - 1];
                    acc = p4fma(p4(w, w, w, w), p4add(p4sub(up, cc), p4sub(dn, cc)), acc);
                }
                const float* st = obase + so * O::FLOATS;
                if (INC && z == sz && src_row) {
                    const float4 l = f4(acc);
                    float a[4] = {l.x, l.y, l.z, l.w};
                    add_lane(a, src_j, fsrc);
                    acc = p4(a[0], a[1], a[2], a[3]);
                }
                if (MODE == STEP3_BORN) acc = p4fma(p4neg(p4(ld4(st + 3 * kQTile))), p4(ld4(st + 2 * kQTile)), acc);
                if (ADJ && srec[iz] >= 0)  // receiver injection of the segment's band buffer
                    acc = p4add(acc, p4(ld4(M.inj + ((long long)(M.inj_slot * M.nshots + shot) * M.nfield + b) * M.inj_block +
                                            (long long)srec[iz] * plane + (long long)y * M.P + x)));
                const P4 Fo = p4mul(p4(ld4(st + kQTile)), acc);
                const P4 prev = p4(ld4(st));
                const P4 c2 = p4add(cc, cc);
                float4 o;
                if (z < M.pad || z >= M.pad + M.nz) {  // z sponge: factors of the cell
                    float g[4], a[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        g[j] = 1.f;
                        a[j] = 1.f;
                        sponge_pair(q_sponge_e(M, z, y, x + j), g[j], a[j]);
                        if (x + j >= M.Nx) g[j] = 0.f;
                    }
                    o = f4(p4mul(p4(g[0], g[1], g[2], g[3]),
                                 p4add_one(Fo, p4fma(p4neg(p4(a[0], a[1], a[2], a[3])), prev, c2), one)));
                } else if (tile_in) {
                    o = f4(p4add_one(Fo, p4sub(c2, prev), one));
                } else {
                    o = f4(p4mul(p4(Gc), p4add_one(Fo, p4fma(p4neg(p4(Ac)), prev, c2), one)));
                }
                st4(outp, o);
                if (INC && auxp) {
                    const float i2 = M.inv_dt2;
                    st4(auxp, f4(p4mul(Fo, p4(i2, i2, i2, i2))));
                }
                if (ADJ && NI) {  // img -= Dtt u^{m-1} mu^m, m = n + NI - 1 .. n; scalar: two roundings each
                    float4 iv = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (!M.seg_first) iv = ld4(st + (O::N - 1) * kQTile);
#pragma unroll
                    for (int c = 0; c < NI; ++c) {
                        const int age = NI - 1 - c;  // mu^{n + age}
                        const float4 mu = age == 0 ? o : (age == 1 ? f4(cc) : f4(prev)), d = ld4(st + (2 + c) * kQTile);
                        const float4 tm = make_float4(__fmul_rn(-d.x, mu.x), __fmul_rn(-d.y, mu.y),
                                                      __fmul_rn(-d.z, mu.z), __fmul_rn(-d.w, mu.w));
                        if (c == 0 && M.seg_first)
                            iv = tm;
                        else
                            iv = make_float4(__fadd_rn(iv.x, tm.x), __fadd_rn(iv.y, tm.y), __fadd_rn(iv.z, tm.z),
                                             __fadd_rn(iv.w, tm.w));
                    }
                    st4(auxp, iv);
                }
            }
            outp += plane;
            if (auxp) auxp += plane;
            __syncwarp();
            if (lane == 0) {  // this warp is done with the current plane and its operands
                mbar_arrive(&hempty[sc]);
                mbar_arrive(&oempty[so]);
            }
        }
    }
}

template <int MODE, int NI>
cudaError_t launch_q(const StepParams3D& p, cudaStream_t st) {
    const ModelStep3D& M = p.m;
    const size_t sm = QOps<MODE, NI>::SMEM;
    // set on every launch (a host-side attribute, no stream work): no shared state between threads
    cudaError_t e = cudaFuncSetAttribute(k_step3d_q<MODE, NI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)(M.tiles_x * M.tiles_y * M.zchunks * M.nshots * M.nfield);
    if (grid == 0) return cudaSuccess;
    k_step3d_q<MODE, NI><<<grid, kThreads + 32, sm, st>>>(p);
    return cudaGetLastError();
}

}  // namespace

// terms: imaging terms added by an adjoint step (0 to 3); p.m.d_slot is the Dtt slot of this step's own.
cudaError_t launch_step3d_q(int mode, int terms, const StepParams3D& p0, cudaStream_t st) {
    StepParams3D p = p0;
    p.one = 1.f;
    switch (mode) {
        case STEP3_INC: return launch_q<STEP3_INC, 0>(p, st);
        case STEP3_INC_SAMPLE: return launch_q<STEP3_INC_SAMPLE, 0>(p, st);
        case STEP3_BORN: return launch_q<STEP3_BORN, 0>(p, st);
        case STEP3_ADJ:
            switch (terms) {
                case 0: return launch_q<STEP3_ADJ, 0>(p, st);
                case 1: return launch_q<STEP3_ADJ, 1>(p, st);
                case 2: return launch_q<STEP3_ADJ, 2>(p, st);
                case 3: return launch_q<STEP3_ADJ, 3>(p, st);
            }
    }
    return cudaErrorInvalidValue;
}

}  // namespace probe
