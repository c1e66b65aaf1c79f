// sweep_pair_k: two explicit steps per pass with per-cell conductivity (the
// counterpart of sweep_pair), for grids whose ghost layers hold every face.
//
// The face coefficients of a plane serve both steps, so no warp should form
// them twice: a block of 6 warps steps R W = 12 neighbouring rows of 128 cells
// (or 24 of 64, 48 of 32: a row takes 32, 16 or 8 lanes, so narrow grids fill
// their warps), each thread 4 cells of 2 rows, and every row is stepped twice
// by the same thread. Only the outer rows and lanes are redundant (12 of 10
// rows, 128 of 120 cells; nothing at a non-periodic face). The first step's
// field goes to the neighbouring rows' threads through shared memory, two
// planes, one barrier a plane; x neighbours come by shuffle.
// Order of an iteration (plane q): the second step's first five terms at plane
// q - 1, whose coefficients are then dead; the first step at q, which forms the
// coefficients of q; the loads of q + 2; the second step's last term (the
// +z face), its store, and the first step's rows into shared memory.
// Without the sharing (a warp alone with its ring rows recomputed, as
// sweep_pair) it was no faster than the one-step pass: 507 against 503 GLUPS
// at 512^3. Bound by latency at 12 warps an SM (168 registers; issue 51%, FMA
// pipe 25% with packed halves, MUFU for the 3.75 reciprocals a cell, DRAM 48%);
// one row a thread with 16 or 20 warps was 20% slower, blocks of 4 or 12 warps
// 4%, the plain and the edge body in one loop 6% (every live register has to
// agree where they meet).
// Measured on one GB300, us a step against the one-step column march: 512^3
// fp32 267 -> 213, bf16 246 -> 220; 333x250x187 fp32 42.2 -> 32.9, bf16 42.2
// -> 31.5; 40x300x500 28.7 -> 15.7; 128^3 6.2 -> 4.9.
#pragma once

#include "wfa_sweep_pair.cuh"

namespace wfa {

// Weights of the 4 cells of a row: x faces as left / right pairs.
struct RowW {
    f2 xm0, xm1, xp0, xp1;
};

// The 4 cells of one row: flux_sum's first five terms in its order, from the
// x neighbours and the differences to the y neighbours and the lower plane.
__device__ __forceinline__ void pair_acc5(const RowW& w, const f2 (&ym)[2], const f2 (&yp)[2], const f2 (&gm)[2],
                                          const f2 (&t)[2], const f2 (&tym)[2], const f2 (&typ)[2], const f2 (&zm)[2],
                                          float xl, float xr, f2 (&acc)[2]) {
    float t0, t1, t2, t3;
    f2_get(t[0], t0, t1);
    f2_get(t[1], t2, t3);
    acc[0] = f2_mul(w.xm0, f2_make(__fsub_rn(xl, t0), __fsub_rn(t0, t1)));
    acc[1] = f2_mul(w.xm1, f2_make(__fsub_rn(t1, t2), __fsub_rn(t2, t3)));
    acc[0] = f2_fma(w.xp0, f2_make(__fsub_rn(t1, t0), __fsub_rn(t2, t1)), acc[0]);
    acc[1] = f2_fma(w.xp1, f2_make(__fsub_rn(t3, t2), __fsub_rn(xr, t3)), acc[1]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        acc[i] = f2_fma(ym[i], f2_sub(tym[i], t[i]), acc[i]);
        acc[i] = f2_fma(yp[i], f2_sub(typ[i], t[i]), acc[i]);
        acc[i] = f2_fma(gm[i], zm[i], acc[i]);
    }
}
// A face weight with its upwind part, half by half: a packed add of a packed
// product is contracted into one fma (measured: last-bit differences).
__device__ __forceinline__ f2 adv1(f2 g, float adv) {
    float a, b;
    f2_get(g, a, b);
    return f2_make(__fadd_rn(a, adv), __fadd_rn(b, adv));
}
template <bool ADV> __device__ __forceinline__ void add_adv(f2 (&o)[2], const f2 (&g)[2], float adv) {
#pragma unroll
    for (int i = 0; i < 2; ++i) o[i] = ADV ? adv1(g[i], adv) : g[i];
}

struct PairKCfg {
    static constexpr int R = 2;        // rows a thread steps
    static constexpr int W = 6;        // warps a block
    static constexpr int BLOCKS = 2;   // blocks per SM the register budget targets
};

// How a grid is cut: lx lanes (32, 16 or 8) take a row's tile of 4 lx cells,
// so a warp takes 32 / lx rows at a time. A tile's outer lanes (and a block's
// outer rows) hold the ring that the second step needs, except at a
// non-periodic face, where nothing lies beyond.
struct PairTiles {
    int lx;           // lanes a row
    int gx, gy;       // tiles along x and y
    int sx, sy;       // cells and rows from one tile to the next
};
__host__ __device__ inline PairTiles pair_k_tiles(const SweepCoef& c) {
    PairTiles t;
    const int per = c.periodic[0] ? 8 : 0;   // ring cells beyond the row's ends
    t.lx = c.n[0] + per <= 32 ? 8 : c.n[0] + per <= 64 ? 16 : 32;
    t.sx = 4 * t.lx - 8;
    t.sy = PairKCfg::R * PairKCfg::W * (32 / t.lx) - 2;
    const int ex = c.n[0] + per - 8, ey = c.n[1] + (c.periodic[1] ? 0 : -2);
    t.gx = ex <= t.sx ? 1 : (ex + t.sx - 1) / t.sx;
    t.gy = ey <= t.sy ? 1 : (ey + t.sy - 1) / t.sy;
    return t;
}

// Planes [z0, z1) of tile (bx, by): called by a whole block of W warps.
// sm: 2 planes of (R W 32 / lx + 2) rows of 4 lx floats.
template <typename S, bool PER, bool RAG, bool ADV, int R, int W>
__device__ __forceinline__ void pair_k_run(const SweepCoef& c, const void* tin, void* tout, const float* __restrict__ rk,
                                           const PairTiles& tl, int bx, int by, int z0, int z1, float* sm) {
    constexpr int E = sizeof(S);
    const int nx = c.n[0], ny = c.n[1], nz = c.n[2];
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int LX = tl.lx, xi = lane & (LX - 1);
    const int rows = R * W * (32 / LX);                       // the block's rows
    const int r0 = R * (wy * (32 / LX) + lane / LX);          // this thread's first of them
    const bool perx = PER && c.periodic[0], pery = PER && c.periodic[1], perz = PER && c.periodic[2];
    const int gx = bx * tl.sx + (perx ? -4 : 0) + 4 * xi;
    const int y0 = by * tl.sy + (pery ? -1 : 0) + r0;
    const long long sy = c.sy, sz = c.sz;   // elements
    const int lx = !RAG && perx ? (gx < 0 ? gx + nx : gx < nx ? gx : min(gx - nx, nx)) : min(gx, (nx + 3) & ~3);
    const S* const tX = (const S*)tin;
    // rows past n_y + 1 (the last block's) are read as that row: never stored
    const int yl = min(y0, ny + 1);
    const S* tP = tX + lx + yl * sy + (z0 - 1) * sz;          // this lane's group, row y0, plane q
    const float* rP = rk + lx + yl * sy + (z0 - 1) * sz;
    S* oP = (S*)tout + gx + y0 * sy + (z0 - 2) * sz;
    // x faces: what lies beyond the row's ends (the value and 1/k of the ghost cell)
    const int el = perx ? -8 : nx - 1 - gx;
    const bool x_first = !perx && gx == 0, x_last = el == 3;
    const float tb0 = c.tb[0], tb1 = c.tb[1];
    const float kg0 = c.bkind[0] == WFA_BC_DIRICHLET ? 0.0f : INFINITY, kg1 = c.bkind[1] == WFA_BC_DIRICHLET ? 0.0f : INFINITY;
    // rows this thread stores: inside its tile's ring, or at a face the tile ends at
    const bool mine_x = gx < nx && (xi >= 1 || x_first) && (xi <= LX - 2 || (!perx && gx + 4 >= nx));
    unsigned mine = 0;
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const int r = r0 + j, y = y0 + j;
        if (mine_x && y < ny && (r >= 1 || (!pery && y == 0)) && (r <= rows - 2 || (!pery && y == ny - 1))) mine |= 1u << j;
    }
    const bool edge_xy = __any_sync(0xffffffffu, y0 < 1 || y0 + R >= ny);
    const bool copies = RAG && perx && (gx < 4 || gx + 3 >= nx - 4);   // its cells have x copies (see sweep_pair)
    float* const own = sm + (1 + r0) * 4 * LX + 4 * xi;       // row r0 of slot 0
    const int slot_f = (rows + 2) * 4 * LX;
    const f2 tcx = f2_make(c.tcd[0], c.tcd[0]), tcy = f2_make(c.tcd[1], c.tcd[1]), tcz = f2_make(c.tcd[2], c.tcd[2]);

    RowBuf<S> T0[R], T1[R], H[2];            // T at planes q and q + 1, the rows beyond at q
    RowBuf<float> K0[R], K1[R], KH[2];       // 1/k likewise
    f2 D[R][2], G0[R][2], G1[R][2];          // T(q - 1) - T(q); z faces between planes q - 2, q - 1 and q - 1, q
    f2 S0[R][2], S1[R][2], DS[R][2];         // first step's field at q - 1 and q; S(q - 2) - S(q - 1)
    f2 WY[R + 1][2];                         // plane q - 1: y faces,
    RowW WX[R];                              // x faces
    int q = z0 - 1;
    auto load_wrapped = [&](RowBuf<S>& t, RowBuf<float>& k, int j, int z) {
        if (!PER) {
            t.load(reinterpret_cast<const char*>(tP + j * sy + (z - q) * sz));
            k.load_rk(reinterpret_cast<const char*>(rP + j * sy + (z - q) * sz));
            return;
        }
        int y = yl + j;
        if (pery) y = y < 0 ? y + ny : y >= ny ? y - ny : y;
        if (perz) z = z < 0 ? z + nz : z >= nz ? z - nz : z;
        const long long row = y * sy + z * sz;
        t.load(reinterpret_cast<const char*>(tX + row + lx));
        k.load_rk(reinterpret_cast<const char*>(rk + row + lx));
    };
#pragma unroll
    for (int j = 0; j < R; ++j) {
        f2 u[2], v[2], ku[2], kv[2];
        load_wrapped(T1[j], K1[j], j, q - 1);
        load_wrapped(T0[j], K0[j], j, q);
        T1[j].get(u);
        T0[j].get(v);
        K1[j].get(ku);
        K0[j].get(kv);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            D[j][i] = f2_sub(u[i], v[i]);
            G1[j][i] = pair_face(ku[i], kv[i], tcz);
            S0[j][i] = S1[j][i] = DS[j][i] = G0[j][i] = 0;
        }
        WX[j].xm0 = WX[j].xm1 = WX[j].xp0 = WX[j].xp1 = 0;
        load_wrapped(T1[j], K1[j], j, q + 1);
    }
#pragma unroll
    for (int j = 0; j <= R; ++j) WY[j][0] = WY[j][1] = 0;
    load_wrapped(H[0], KH[0], -1, q);
    load_wrapped(H[1], KH[1], R, q);
    // the rows beyond the block's: a y face's value where the block ends at one
    // (elsewhere they feed no stored row); the first slot read: finite
    for (int i = threadIdx.x; i < slot_f; i += 32 * W) {
        const int row = i / (4 * LX);
        const float v = row == 0 ? c.tb[2] : row == rows + 1 ? c.tb[3] : 0.0f;
        sm[i] = v;
        sm[slot_f + i] = v;
    }
    __syncthreads();

    auto plane = [&](auto edge_tag, RowBuf<S>(&Tc)[R], RowBuf<S>(&Tn)[R], RowBuf<float>(&Kc)[R], RowBuf<float>(&Kn)[R],
                     f2(&Sc)[R][2], f2(&Sn)[R][2], f2(&Ga)[R][2], f2(&Gb)[R][2], int slot) {
        constexpr bool EDGE = decltype(edge_tag)::value;
        const int p = q - 1;
        // ---- second step at plane p = q - 1, all but the term of plane q: Sc
        // (and its neighbour rows from the other warps), DS, the faces of plane p
        f2 acc2[R][2];
        {
            f2 nb[2][2];
            const float4 lo = *reinterpret_cast<const float4*>(own + (slot ^ 1) * slot_f - 4 * LX);
            const float4 hi = *reinterpret_cast<const float4*>(own + (slot ^ 1) * slot_f + R * 4 * LX);
            nb[0][0] = f2_make(lo.x, lo.y);
            nb[0][1] = f2_make(lo.z, lo.w);
            nb[1][0] = f2_make(hi.x, hi.y);
            nb[1][1] = f2_make(hi.z, hi.w);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                float xl = __shfl_up_sync(0xffffffffu, f2_hi(Sc[j][1]), 1, LX),
                      xr = __shfl_down_sync(0xffffffffu, f2_lo(Sc[j][0]), 1, LX);
                xl = x_first ? tb0 : xl;
                xr = x_last ? tb1 : xr;
                f2 ym[2], yp[2], gm[2];
                add_adv<ADV>(ym, WY[j], c.adv[2]);
                add_adv<ADV>(yp, WY[j + 1], c.adv[3]);
                add_adv<ADV>(gm, Ga[j], c.adv[4]);
                pair_acc5(WX[j], ym, yp, gm, Sc[j], j == 0 ? nb[0] : Sc[j > 0 ? j - 1 : 0],
                          j == R - 1 ? nb[1] : Sc[j < R - 1 ? j + 1 : 0], DS[j], xl, xr, acc2[j]);
            }
        }
        // ---- first step at plane q -> Sn, with the faces of plane q
        {
            f2 t[2], lo[2], k[2], h[2];
            H[0].get(lo);
            Tc[0].get(t);
            KH[0].get(h);
            Kc[0].get(k);
            WY[0][0] = pair_face(h[0], k[0], tcy);
            WY[0][1] = pair_face(h[1], k[1], tcy);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                f2 up[2], tn[2], ku[2], kn[2], acc[2], v[2], ym[2], yp[2], gm[2], gp[2];
                if (j == R - 1) {
                    H[1].get(up);
                    KH[1].get(ku);
                } else {
                    Tc[j + 1 < R ? j + 1 : 0].get(up);
                    Kc[j + 1 < R ? j + 1 : 0].get(ku);
                }
                Tn[j].get(tn);
                Kn[j].get(kn);
                float xl = __shfl_up_sync(0xffffffffu, f2_hi(t[1]), 1, LX),
                      xr = __shfl_down_sync(0xffffffffu, f2_lo(t[0]), 1, LX);
                float kl = __shfl_up_sync(0xffffffffu, f2_hi(k[1]), 1, LX),
                      kr = __shfl_down_sync(0xffffffffu, f2_lo(k[0]), 1, LX);
                xl = x_first ? tb0 : xl;
                xr = x_last ? tb1 : xr;
                kl = x_first ? kg0 : kl;
                kr = x_last ? kg1 : kr;
                float k0, k1, k2, k3;
                f2_get(k[0], k0, k1);
                f2_get(k[1], k2, k3);
                const float x0 = rcp_approx(__fadd_rn(kl, k0)), x1 = rcp_approx(__fadd_rn(k0, k1)),
                            x2 = rcp_approx(__fadd_rn(k1, k2)), x3 = rcp_approx(__fadd_rn(k2, k3)),
                            x4 = rcp_approx(__fadd_rn(k3, kr));
                WX[j].xm0 = f2_mul(tcx, f2_make(x0, x1));
                WX[j].xm1 = f2_mul(tcx, f2_make(x2, x3));
                WX[j].xp0 = f2_mul(tcx, f2_make(x1, x2));
                WX[j].xp1 = f2_mul(tcx, f2_make(x3, x4));
                if (ADV) {
                    WX[j].xm0 = adv1(WX[j].xm0, c.adv[0]);
                    WX[j].xm1 = adv1(WX[j].xm1, c.adv[0]);
                    WX[j].xp0 = adv1(WX[j].xp0, c.adv[1]);
                    WX[j].xp1 = adv1(WX[j].xp1, c.adv[1]);
                }
                f2 gz[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    WY[j + 1][i] = pair_face(k[i], ku[i], tcy);
                    gz[i] = pair_face(k[i], kn[i], tcz);
                }
                add_adv<ADV>(ym, WY[j], c.adv[2]);
                add_adv<ADV>(yp, WY[j + 1], c.adv[3]);
                add_adv<ADV>(gm, Gb[j], c.adv[4]);
                add_adv<ADV>(gp, gz, c.adv[5]);
                pair_acc5(WX[j], ym, yp, gm, t, lo, up, D[j], xl, xr, acc);
#pragma unroll
                for (int i = 0; i < 2; ++i) v[i] = round2<S>(f2_add(t[i], f2_fma(gp[i], f2_sub(tn[i], t[i]), acc[i])));
                const int y = y0 + j;
                const bool ghost = EDGE && ((!pery && (y < 0 || y >= ny)) || (!perz && (q < 0 || q >= nz)));
                if (RAG) {
                    v[0] = f2_make(f2_lo(v[0]), el == 0 ? f2_hi(t[0]) : f2_hi(v[0]));
                    v[1] = f2_make(el == 1 ? f2_lo(t[1]) : f2_lo(v[1]), el == 2 ? f2_hi(t[1]) : f2_hi(v[1]));
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    Sn[j][i] = ghost ? t[i] : v[i];
                    D[j][i] = f2_sub(t[i], tn[i]);
                    Ga[j][i] = gz[i];
                    lo[i] = t[i];
                    t[i] = up[i];
                    k[i] = ku[i];
                }
            }
        }
        if (q < z1) {   // plane q + 2 and the outer rows of plane q + 1
            if (EDGE && PER) {
#pragma unroll
                for (int j = 0; j < R; ++j) load_wrapped(Tc[j], Kc[j], j, q + 2);
                load_wrapped(H[0], KH[0], -1, q + 1);
                load_wrapped(H[1], KH[1], R, q + 1);
            } else {
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    Tc[j].load(reinterpret_cast<const char*>(tP + 2 * sz + j * sy));
                    Kc[j].load_rk(reinterpret_cast<const char*>(rP + 2 * sz + j * sy));
                }
                H[0].load(reinterpret_cast<const char*>(tP + sz - sy));
                H[1].load(reinterpret_cast<const char*>(tP + sz + R * sy));
                KH[0].load_rk(reinterpret_cast<const char*>(rP + sz - sy));
                KH[1].load_rk(reinterpret_cast<const char*>(rP + sz + R * sy));
            }
            if ((lane & 7) == 0 && q + 4 <= z1 + 1) {
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    if (E == 4 || (lane & 15) == 0) prefetch_l2(tP + 4 * sz + j * sy);
                    prefetch_l2(rP + 4 * sz + j * sy);
                }
            }
        }
        // ---- second step's last term, its store; this plane's rows for the other warps
#pragma unroll
        for (int j = 0; j < R; ++j) {
            f2 gp[2];
            add_adv<ADV>(gp, Gb[j], c.adv[5]);
            float o[4];
            f2_get(f2_add(Sc[j][0], f2_fma(gp[0], f2_sub(Sn[j][0], Sc[j][0]), acc2[j][0])), o[0], o[1]);
            f2_get(f2_add(Sc[j][1], f2_fma(gp[1], f2_sub(Sn[j][1], Sc[j][1]), acc2[j][1])), o[2], o[3]);
            if ((mine >> j & 1u) && p >= z0) {
                pair_put<S, RAG>(o, nx - gx, reinterpret_cast<char*>(oP + j * sy));
                if (RAG && PER && copies) pair_put_copies<S>(o, gx, nx, reinterpret_cast<char*>(oP + j * sy));
            }
            float v[4];
            f2_get(Sn[j][0], v[0], v[1]);
            f2_get(Sn[j][1], v[2], v[3]);
            *reinterpret_cast<float4*>(own + slot * slot_f + j * 4 * LX) = make_float4(v[0], v[1], v[2], v[3]);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                DS[j][i] = f2_sub(Sc[j][i], Sn[j][i]);
            }
        }
        __syncthreads();
        ++q;
        tP += sz;
        rP += sz;
        oP += sz;
    };
    // first and last plane of the plain body (no ghost row or plane, nothing wraps)
    const int qa = edge_xy ? z1 + 1 : 0, qb = min(z1, nz - (PER ? 3 : 1));
    for (;;) {
        for (; q >= qa && q < qb;) {
            plane(std::false_type{}, T0, T1, K0, K1, S0, S1, G0, G1, 0);
            plane(std::false_type{}, T1, T0, K1, K0, S1, S0, G1, G0, 1);
        }
        if (q > z1) break;
        plane(std::true_type{}, T0, T1, K0, K1, S0, S1, G0, G1, 0);
        if (q > z1) break;
        plane(std::true_type{}, T1, T0, K1, K0, S1, S0, G1, G0, 1);
        if (q > z1) break;
    }
}

template <typename S, bool PER, bool RAG, bool ADV>
__global__ void __launch_bounds__(32 * PairKCfg::W, PairKCfg::BLOCKS)
    sweep_pair_k(const __grid_constant__ SweepArgs a, const __grid_constant__ PairTiles tl) {
    __shared__ __align__(16) float sm[2 * (PairKCfg::R * PairKCfg::W + 2) * 128];
    const void* tin = a.tin;
    const float* rk = a.rk;
    grid_wait(tin, rk);
    const int z0 = blockIdx.z * a.zchunk;
    pair_k_run<S, PER, RAG, ADV, PairKCfg::R, PairKCfg::W>(a.c, tin, a.tout, rk, tl, blockIdx.x, blockIdx.y, z0,
                                                           min(z0 + a.zchunk, a.c.n[2]), sm);
}

template <typename S, bool ADV>
cudaError_t pair_k_dispatch(const SweepArgs& a, const PairTiles& tl, dim3 grid, cudaStream_t st) {
    const dim3 block(32 * PairKCfg::W);
    const bool per = a.c.periodic[0] || a.c.periodic[1] || a.c.periodic[2], rag = a.c.n[0] % 4 != 0;
    if (per && rag) return launch_overlapped(sweep_pair_k<S, true, true, ADV>, grid, block, st, !a.fresh_k, a, tl);
    if (per) return launch_overlapped(sweep_pair_k<S, true, false, ADV>, grid, block, st, !a.fresh_k, a, tl);
    if (rag) return launch_overlapped(sweep_pair_k<S, false, true, ADV>, grid, block, st, !a.fresh_k, a, tl);
    return launch_overlapped(sweep_pair_k<S, false, false, ADV>, grid, block, st, !a.fresh_k, a, tl);
}

// z chunks of a launch of `tiles` blocks a chunk: whole waves of resident
// blocks against the planes a chunk steps but does not store. At most 1024
// chunks (three waves of the smallest tile count; the loop runs at every launch).
// cost_out: the planes a resident block steps, about a microsecond each on one
// GB300 (see default_choice).
inline int pair_k_chunk(int nz, long long tiles, long long resident, double* cost_out = nullptr) {
    int best = nz;
    double cost = 1e300;
    for (int n = 1; n <= std::min((nz + 3) / 4, 1024); ++n) {
        const int zc = (nz + n - 1) / n;
        const double waves = (double)((tiles * ((nz + zc - 1) / zc) + resident - 1) / resident);
        if (waves * (zc + 4) < cost * 0.995) {
            cost = waves * (zc + 4);
            best = zc;
        }
    }
    if (cost_out) *cost_out = cost;
    return best;
}

// One pass of two steps with per-cell k (a.c.halo_bc: the ghost layers hold every face).
template <typename S>
cudaError_t pair_k_launch(const SweepArgs& a_in, cudaStream_t st, int nsm, const cudaEvent_t* ev) {
    SweepArgs a = a_in;
    const PairTiles tl = pair_k_tiles(a.c);
    a.zchunk = a_in.zchunk > 0 ? std::min(a_in.zchunk, a.c.n[2])
                               : pair_k_chunk(a.c.n[2], (long long)tl.gx * tl.gy, (long long)nsm * PairKCfg::BLOCKS);
    const dim3 grid(tl.gx, tl.gy, (a.c.n[2] + a.zchunk - 1) / a.zchunk);
    const bool adv = a.c.adv[0] != 0.0f || a.c.adv[1] != 0.0f || a.c.adv[2] != 0.0f || a.c.adv[3] != 0.0f ||
                     a.c.adv[4] != 0.0f || a.c.adv[5] != 0.0f;
    if (ev) cudaEventRecord(ev[0], st);
    const cudaError_t e = adv ? pair_k_dispatch<S, true>(a, tl, grid, st) : pair_k_dispatch<S, false>(a, tl, grid, st);
    if (ev) cudaEventRecord(ev[1], st);
    return e;
}

}  // namespace wfa
