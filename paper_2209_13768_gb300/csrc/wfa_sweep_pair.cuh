// sweep_pair: two explicit steps per pass over the grid (Sec. 1.1.1,
// Eq. expl_form applied twice) with uniform conductivity, so a pass reads and
// writes the field once for two steps (4 B a cell update in fp32 instead of 8;
// Eqs. A_eff and t_it_min).
//
// A warp owns 120 x cells (30 lanes of 4; the lanes at both ends hold the ring
// that the second step needs) of 4 rows and marches z. Per plane it takes the
// first step of 6 rows (its 4 and one either side) and the second of its 4
// rows, one plane behind. Everything between the two steps stays in
// registers: x neighbours come from the next lanes by shuffle, y neighbours
// are the thread's own rows, z neighbours the thread's previous planes. No
// shared memory and no barrier; the planes are loaded half an iteration
// before they are used and prefetched into L2 two planes before that.
// What it costs is redundant work: (6 + 4) / 8 rows x 128 / 120 cells = 1.33
// cell updates for each kept one, plus two planes a z chunk.
//
// Why this split. The single pass runs at 0.92 of the copy bandwidth, so only
// fewer bytes a step help; staged two-step passes (shared-memory or TMA
// planes) lost because they spent 80 instructions an update. Here an update
// takes 17 warp instructions a lane (ncu), because
//  * each difference across a face is formed once and used by both its cells
//    (the sign goes into the weight: the same bits), 10 instead of 13 fp32
//    operations a cell;
//  * add, multiply and fma work on pairs of cells (f32x2), which halves their
//    issue slots (not their pipe time).
// 4 rows: 3 or 2 rows (fewer registers, more warps) were 6% and 10% slower,
// 6 rows with 8 warps an SM 1% slower; sharing the x differences pays 1%
// (fp32) and 3% (bf16) against recomputing them. Bound by instruction latency
// at 12 warps an SM (issue 57%, fp32 DRAM 63%; bf16 issue 69%, half of it
// converting), not by memory any more.
// Measured on one GB300, us a step, against the one-step column march with
// its boundary launch: 1024x1024x512 advection-diffusion fp32 728 -> 401,
// bf16 657 -> 387 (16 cells a thread: 467); 512^3 fp32 212 -> 118; 256^3
// 46.6 -> 25.0; 128^3 8.1 -> 6.4.
//
// Boundaries. Warps and planes away from the faces run the plain body; the
// others the same body with weights, self terms and ghost rows chosen by
// select (no branch inside a row: branches there cost 40%). A Dirichlet value
// comes from the halo's ghost layer, a zero-flux face has weight 0. Periodic
// axes wrap the rows, planes and groups that are read, so no copies are
// stored (ragged rows: the 4 columns beyond a row's ends only) and a buffer's
// other periodic copies are stale after this pass (TWINS_NONE, TWINS_X). The fixed
// per-cell expression is that of every other kernel, rounded to the storage
// type after each step, so a pass gives bitwise the field of two single
// steps.
#pragma once

#include <type_traits>

#include "wfa_sweep_col.cuh"

namespace wfa {

// Two fp32 values in one 64-bit register pair: add / mul / fma.rn.f32x2 round
// each half exactly as the scalar instruction does and take one issue slot.
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_make(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_get(f2 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ float f2_lo(f2 v) {
    float a, b;
    f2_get(v, a, b);
    return a;
}
__device__ __forceinline__ float f2_hi(f2 v) {
    float a, b;
    f2_get(v, a, b);
    return b;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ f2 unpack2(unsigned u) {
    return f2_make(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}
// Coefficients of two faces from the sums of their cells' 1/k.
__device__ __forceinline__ f2 pair_face(f2 ra, f2 rb, f2 tcd) {
    float a, b;
    f2_get(f2_add(ra, rb), a, b);
    return f2_mul(tcd, f2_make(rcp_approx(a), rcp_approx(b)));
}

// A row as loaded: fp32 pairs, or bf16 words converted where they are first used.
template <typename S> struct RowBuf;
template <> struct RowBuf<float> {
    float4 q;
    __device__ __forceinline__ void load(const char* p) { q = ld_f4(p); }
    __device__ __forceinline__ void load_rk(const char* p) { q = __ldg(reinterpret_cast<const float4*>(p)); }   // see ldrk
    __device__ __forceinline__ void get(f2 (&o)[2]) const { o[0] = f2_make(q.x, q.y); o[1] = f2_make(q.z, q.w); }
};
template <> struct RowBuf<__nv_bfloat16> {
    uint2 q;
    __device__ __forceinline__ void load(const char* p) { q = ld_u2(p); }
    __device__ __forceinline__ void get(f2 (&o)[2]) const { o[0] = unpack2(q.x); o[1] = unpack2(q.y); }
};
template <typename S> __device__ __forceinline__ f2 round2(f2 v) {
    if constexpr (sizeof(S) == 4) return v;
    return unpack2(pack_bf16x2(f2_lo(v), f2_hi(v)));
}

// Face weights of a thread's 4 cells, the upper faces' negated.
struct PairW {
    f2 xm0, xm1, nxp0, nxp1, ym, nyp, zm, nzp;
};

// The 4 cells of one row: dm = T_y- - T_C, dp = T_C - T_y+, ez = T_z- - T_C,
// fz = T_C - T_z+, xl / xr the x neighbours of the row's ends. A difference
// is shared by the two cells of a face: its negative is exact and goes into
// the weight, so flux_sum's terms keep their bits and order.
__device__ __forceinline__ void pair_acc(const PairW& w, const f2 (&t)[2], const f2 (&dm)[2], const f2 (&dp)[2],
                                         const f2 (&ez)[2], const f2 (&fz)[2], float xl, float xr, f2 (&acc)[2]) {
    float t0, t1, t2, t3;
    f2_get(t[0], t0, t1);
    f2_get(t[1], t2, t3);
    const float l0 = __fsub_rn(xl, t0), l1 = __fsub_rn(t0, t1), l2 = __fsub_rn(t1, t2), l3 = __fsub_rn(t2, t3),
                l4 = __fsub_rn(t3, xr);
    acc[0] = f2_mul(w.xm0, f2_make(l0, l1));
    acc[1] = f2_mul(w.xm1, f2_make(l2, l3));
    acc[0] = f2_fma(w.nxp0, f2_make(l1, l2), acc[0]);
    acc[1] = f2_fma(w.nxp1, f2_make(l3, l4), acc[1]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        acc[i] = f2_fma(w.ym, dm[i], acc[i]);
        acc[i] = f2_fma(w.nyp, dp[i], acc[i]);
        acc[i] = f2_fma(w.zm, ez[i], acc[i]);
        acc[i] = f2_fma(w.nzp, fz[i], acc[i]);
    }
}

// Where a non-periodic face may be near: the y / z weights of row y at plane
// z and the self terms (zero-flux faces that meet advection) of its cells, by
// select, so the edge body stays free of branches like the plain one.
__device__ __forceinline__ PairW edge_weights(const SweepCoef& c, PairW w, int y, int z) {
    const float ym = !c.periodic[1] && y == 0 ? c.w_bd[2] : c.w_in[2];
    const float yp = !c.periodic[1] && y == c.n[1] - 1 ? c.w_bd[3] : c.w_in[3];
    const float zm = !c.periodic[2] && z == 0 ? c.w_bd[4] : c.w_in[4];
    const float zp = !c.periodic[2] && z == c.n[2] - 1 ? c.w_bd[5] : c.w_in[5];
    w.ym = f2_make(ym, ym);
    w.nyp = f2_make(-yp, -yp);
    w.zm = f2_make(zm, zm);
    w.nzp = f2_make(-zp, -zp);
    return w;
}
__device__ __forceinline__ void edge_self(const SweepCoef& c, const f2 (&t)[2], f2 (&acc)[2], int gx, int y, int z) {
    float tv[4], av[4];
    f2_get(t[0], tv[0], tv[1]);
    f2_get(t[1], tv[2], tv[3]);
    f2_get(acc[0], av[0], av[1]);
    f2_get(acc[1], av[2], av[3]);
    // self_term's sum: x, then y, then z (s_lo / s_hi are 0 where no term applies)
    const float sy = y == 0 ? c.s_lo[1] : y == c.n[1] - 1 ? c.s_hi[1] : 0.0f;
    const float sz = z == 0 ? c.s_lo[2] : z == c.n[2] - 1 ? c.s_hi[2] : 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float sx = gx + i == 0 ? c.s_lo[0] : gx + i == c.n[0] - 1 ? c.s_hi[0] : 0.0f;
        const float s = __fadd_rn(__fadd_rn(sx, sy), sz);
        const float v = __fmaf_rn(s, tv[i], av[i]);
        av[i] = s != 0.0f ? v : av[i];
    }
    acc[0] = f2_make(av[0], av[1]);
    acc[1] = f2_make(av[2], av[3]);
}

constexpr int PAIR_TX = 120;   // cells a warp updates along x

// Registers decide: 168 a thread for 12 warps an SM (65 to 80 words spilled in
// fp32, 21 to 28 in bf16), as blocks of 1 or 2 warps so that no tail of a
// larger block holds them (fp32 2 warps 1366 GLUPS, 4 warps 1355; bf16 1 warp
// 1382, 4 warps 1355).
template <typename S> struct PairCfg {
    static constexpr int R = 4;                              // rows a warp updates
    static constexpr int WPB = sizeof(S) == 4 ? 2 : 1;       // warps a block
    static constexpr int BLOCKS = sizeof(S) == 4 ? 5 : 11;   // blocks per SM the register budget targets
};

// Stores the 4 new cells of a group whose first is x (`left` = n_x - x) at p.
template <typename S, bool RAG>
__device__ __forceinline__ void pair_put(const float (&o)[4], int left, char* p) {
    if (!RAG || left >= 4) {
        StoreVec<S, 4>(o).store(reinterpret_cast<S*>(p));
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < left) reinterpret_cast<S*>(p)[i] = from_f32<S>(o[i]);
    }
}
// The copies of the first and last 4 cells of a row one period (n_x cells) away.
template <typename S>
__device__ __forceinline__ void pair_put_copies(const float (&o)[4], int gx, int nx, char* p) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int x = gx + i;
        if (x < 4 && x < nx) reinterpret_cast<S*>(p)[i + nx] = from_f32<S>(o[i]);
        if (x < nx && x >= nx - 4) reinterpret_cast<S*>(p)[i - nx] = from_f32<S>(o[i]);
    }
}

// PER: some axis is periodic. RAG: n_x is not a multiple of 4 (a row's last
// group holds cells beyond the face).
template <typename S, bool PER, bool RAG, int R, int WPB, int BLOCKS>
__global__ void __launch_bounds__(32 * WPB, BLOCKS) sweep_pair(const __grid_constant__ SweepArgs a) {
    constexpr int E = sizeof(S);
    const SweepCoef& c = a.c;
    const void* tin = a.tin;
    const float* rk = a.rk;
    grid_wait(tin, rk);
    const int nx = c.n[0], ny = c.n[1], nz = c.n[2];
    const int lane = threadIdx.x;
    const int gx = blockIdx.x * PAIR_TX - 4 + 4 * lane;
    const int y0 = WPB == 1 ? (int)blockIdx.y * R : __shfl_sync(0xffffffffu, (int)(blockIdx.y * WPB + threadIdx.y) * R, 0);
    if (y0 >= ny) return;
    const int z0 = blockIdx.z * a.zchunk, z1 = min(z0 + a.zchunk, nz);
    const bool perx = PER && c.periodic[0], pery = PER && c.periodic[1], perz = PER && c.periodic[2];
    const long long sy = c.sy * E, sz = c.sz * E;
    // Where this lane's group is read: beyond a row's end from its halo; across
    // a periodic x face one period away, or (where a period is no whole number
    // of groups) from the halo's copies, which the RAG passes store
    const int lx = !RAG && perx ? (gx < 0 ? gx + nx : gx < nx ? gx : min(gx - nx, nx)) : min(gx, (nx + 3) & ~3);
    const char* const tX = reinterpret_cast<const char*>((const S*)tin);   // cell (0, 0, 0)
    const char* tP = tX + (long long)lx * E + y0 * sy + (z0 - 1) * sz;       // this lane's group, row y0, plane q
    char* oP = reinterpret_cast<char*>((S*)a.tout) + (long long)gx * E + y0 * sy + (z0 - 2) * sz;
    // x faces: the weights of cells 0 and n_x - 1, and the face values that
    // stand for the neighbour beyond them in the second step
    const int el = perx ? -8 : nx - 1 - gx;   // cell n_x - 1 in this lane's group (if 0 <= el < 4)
    const bool x_first = !perx && gx == 0, x_last = el == 3;
    const float wp_in = -c.w_in[1], wp_bd = -c.w_bd[1];
    PairW w;
    w.xm0 = f2_make(x_first ? c.w_bd[0] : c.w_in[0], c.w_in[0]);
    w.xm1 = f2_make(c.w_in[0], c.w_in[0]);
    w.nxp0 = f2_make(RAG && el == 0 ? wp_bd : wp_in, RAG && el == 1 ? wp_bd : wp_in);
    w.nxp1 = f2_make(RAG && el == 2 ? wp_bd : wp_in, el == 3 ? wp_bd : wp_in);
    w.ym = f2_make(c.w_in[2], c.w_in[2]);
    w.nyp = f2_make(-c.w_in[3], -c.w_in[3]);
    w.zm = f2_make(c.w_in[4], c.w_in[4]);
    w.nzp = f2_make(-c.w_in[5], -c.w_in[5]);
    const bool mine = lane >= 1 && lane <= 30 && gx < nx;   // this lane's cells are stored
    // edge body: a row of the tile or its ring on or beyond a y face, or
    // (zero-flux faces with advection) a cell of the tile or its ring on an x face
    const bool x_tile = blockIdx.x == 0 || (int)(blockIdx.x + 1) * PAIR_TX + 4 >= nx - 1;
    const bool edge_xy = y0 <= 1 || y0 + R >= ny - 1 || (c.any_self && !perx && x_tile);
    const bool copies = RAG && perx && mine && (gx < 4 || gx + 3 >= nx - 4);   // its cells have x copies

    // rows y0-1 .. y0+R: T at plane q and the rows beyond (H), at q + 1,
    // T(q - 1) - T(q) (D); the same for the first step's field S (planes q - 1, q)
    RowBuf<S> T0[R + 2], T1[R + 2], H[2];
    f2 D[R + 2][2], S0[R + 2][2], S1[R + 2][2], DS[R][2];
    int q = z0 - 1;   // plane of the first step
    // row y0 + j of plane z, both wrapped across periodic faces
    auto load_wrapped = [&](RowBuf<S>& t, int j, int z) {
        if (!PER) {
            t.load(tP + j * sy + (z - q) * sz);
            return;
        }
        int y = y0 + j;
        if (pery) y = y < 0 ? y + ny : y >= ny ? y - ny : y;
        if (perz) z = z < 0 ? z + nz : z >= nz ? z - nz : z;
        t.load(tX + (long long)lx * E + y * sy + z * sz);
    };
#pragma unroll
    for (int j = 0; j < R + 2; ++j) {
        f2 u[2], v[2];
        load_wrapped(T1[j], j - 1, q - 1);
        load_wrapped(T0[j], j - 1, q);
        T1[j].get(u);
        T0[j].get(v);
        D[j][0] = f2_sub(u[0], v[0]);
        D[j][1] = f2_sub(u[1], v[1]);
        S0[j][0] = S0[j][1] = S1[j][0] = S1[j][1] = 0;
        load_wrapped(T1[j], j - 1, q + 1);
    }
    load_wrapped(H[0], -2, q);
    load_wrapped(H[1], R + 1, q);

    auto plane = [&](auto edge_tag, RowBuf<S>(&Tc)[R + 2], RowBuf<S>(&Tn)[R + 2], f2(&Sc)[R + 2][2], f2(&Sn)[R + 2][2]) {
        constexpr bool EDGE = decltype(edge_tag)::value;
        // ---- first step at plane q -> Sn
        {
            f2 t[2], dm[2], h[2];
            H[0].get(h);
            Tc[0].get(t);
            dm[0] = f2_sub(h[0], t[0]);
            dm[1] = f2_sub(h[1], t[1]);
#pragma unroll
            for (int j = 0; j < R + 2; ++j) {
                f2 up[2], tn[2], dp[2], fz[2], acc[2], v[2];
                if (j == R + 1) H[1].get(up);
                else Tc[j + 1 < R + 2 ? j + 1 : 0].get(up);
                Tn[j].get(tn);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    dp[i] = f2_sub(t[i], up[i]);
                    fz[i] = f2_sub(t[i], tn[i]);
                }
                const float xl = __shfl_up_sync(0xffffffffu, f2_hi(t[1]), 1),
                            xr = __shfl_down_sync(0xffffffffu, f2_lo(t[0]), 1);
                const int y = y0 - 1 + j;
                pair_acc(EDGE ? edge_weights(c, w, y, q) : w, t, dm, dp, D[j], fz, xl, xr, acc);
                if (EDGE) edge_self(c, t, acc, gx, y, q);
#pragma unroll
                for (int i = 0; i < 2; ++i) v[i] = round2<S>(f2_add(t[i], acc[i]));
                // ghost rows, planes and (in a row's last group) cells keep their value
                const bool ghost = EDGE && ((!pery && (y < 0 || y >= ny)) || (!perz && (q < 0 || q >= nz)));
                if (RAG) {
                    v[0] = f2_make(f2_lo(v[0]), el == 0 ? f2_hi(t[0]) : f2_hi(v[0]));
                    v[1] = f2_make(el == 1 ? f2_lo(t[1]) : f2_lo(v[1]), el == 2 ? f2_hi(t[1]) : f2_hi(v[1]));
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    Sn[j][i] = ghost ? t[i] : v[i];
                    D[j][i] = fz[i];
                    t[i] = up[i];
                    dm[i] = dp[i];
                }
            }
        }
        if (q < z1) {   // plane q + 2 and the outer rows of plane q + 1
            if (EDGE && PER) {
#pragma unroll
                for (int j = 0; j < R + 2; ++j) load_wrapped(Tc[j], j - 1, q + 2);
                load_wrapped(H[0], -2, q + 1);
                load_wrapped(H[1], R + 1, q + 1);
            } else {
#pragma unroll
                for (int j = 0; j < R + 2; ++j) Tc[j].load(tP + 2 * sz + (j - 1) * sy);
                H[0].load(tP + sz - 2 * sy);
                H[1].load(tP + sz + (R + 1) * sy);
            }
            if ((lane & (E == 4 ? 7 : 15)) == 0 && q + 4 <= z1 + 1) {
#pragma unroll
                for (int j = 0; j < R; ++j) prefetch_l2(tP + 4 * sz + j * sy);
            }
        }
        // ---- second step at plane p = q - 1 from Sc (p), Sn (q), DS = S(p-1) - S(p)
        const int p = q - 1;
        if (p >= z0) {
            f2 dm[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) dm[i] = f2_sub(Sc[0][i], Sc[1][i]);
#pragma unroll
            for (int j = 1; j <= R; ++j) {
                f2 dp[2], fz[2], acc[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    dp[i] = f2_sub(Sc[j][i], Sc[j + 1][i]);
                    fz[i] = f2_sub(Sc[j][i], Sn[j][i]);
                }
                float xl = __shfl_up_sync(0xffffffffu, f2_hi(Sc[j][1]), 1),
                      xr = __shfl_down_sync(0xffffffffu, f2_lo(Sc[j][0]), 1);
                xl = x_first ? c.tb[0] : xl;
                xr = x_last ? c.tb[1] : xr;
                const int y = y0 - 1 + j;
                pair_acc(EDGE ? edge_weights(c, w, y, p) : w, Sc[j], dm, dp, DS[j - 1], fz, xl, xr, acc);
                if (EDGE) edge_self(c, Sc[j], acc, gx, y, p);
                float o[4];
                f2_get(f2_add(Sc[j][0], acc[0]), o[0], o[1]);
                f2_get(f2_add(Sc[j][1], acc[1]), o[2], o[3]);
                if (mine && y < ny) pair_put<S, RAG>(o, nx - gx, oP + (j - 1) * sy);
                if (RAG && PER && copies && y < ny) pair_put_copies<S>(o, gx, nx, oP + (j - 1) * sy);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    DS[j - 1][i] = fz[i];
                    dm[i] = dp[i];
                }
            }
        } else {
#pragma unroll
            for (int j = 1; j <= R; ++j)
#pragma unroll
                for (int i = 0; i < 2; ++i) DS[j - 1][i] = f2_sub(Sc[j][i], Sn[j][i]);
        }
        ++q;
        tP += sz;
        oP += sz;
    };
    // planes q - 1 .. q + 2 inside the domain (nothing wraps), q and q - 1 away from its z faces
    auto plain = [&]() { return !edge_xy && q >= 2 && q < nz - (PER ? 2 : 1); };
    for (;;) {
        if (plain()) plane(std::false_type{}, T0, T1, S0, S1);
        else plane(std::true_type{}, T0, T1, S0, S1);
        if (q > z1) break;
        if (plain()) plane(std::false_type{}, T1, T0, S1, S0);
        else plane(std::true_type{}, T1, T0, S1, S0);
        if (q > z1) break;
    }
}

// One pass of two steps.
template <typename S>
cudaError_t pair_launch(const SweepArgs& a_in, cudaStream_t st, int nsm, const cudaEvent_t* ev) {
    using Cfg = PairCfg<S>;
    SweepArgs a = a_in;
    const int gxb = (a.c.n[0] + PAIR_TX - 1) / PAIR_TX, gyb = (a.c.n[1] + Cfg::R * Cfg::WPB - 1) / (Cfg::R * Cfg::WPB);
    const long long tiles = (long long)gxb * gyb, resident = (long long)nsm * Cfg::BLOCKS;
    // z chunks: about four waves of blocks, between 4 planes (a chunk steps two
    // planes more than it stores) and 16 (fp32) or 24 (bf16). Measured us a
    // step: 256^3 fp32 24.9 at 8, 26.4 at 16; 512^3 fp32 118 at 12 to 24, 128 at
    // 8; 1024x1024x512 bf16 387 at 24, 399 at 16; 128^3 6.4 at 4, 9.8 at 16
    constexpr int ZMAX = sizeof(S) == 4 ? 16 : 24;
    const long long want = std::max<long long>(1, (4 * resident + tiles - 1) / tiles);
    int nch = (int)std::min<long long>(std::max<long long>(want, (a.c.n[2] + ZMAX - 1) / ZMAX), (a.c.n[2] + 3) / 4);
    nch = std::min(nch, 65535);
    if (a_in.zchunk > 0) nch = (a.c.n[2] + a_in.zchunk - 1) / a_in.zchunk;
    a.zchunk = (a.c.n[2] + nch - 1) / nch;
    nch = (a.c.n[2] + a.zchunk - 1) / a.zchunk;
    const dim3 grid(gxb, gyb, nch), block(32, Cfg::WPB);   // gyb: see pair_applies
    if (ev) cudaEventRecord(ev[0], st);
    cudaError_t e;
    const bool per = a.c.periodic[0] || a.c.periodic[1] || a.c.periodic[2], rag = a.c.n[0] % 4 != 0;
    if (per && rag) e = launch_overlapped(sweep_pair<S, true, true, Cfg::R, Cfg::WPB, Cfg::BLOCKS>, grid, block, st, !a.fresh_k, a);
    else if (per) e = launch_overlapped(sweep_pair<S, true, false, Cfg::R, Cfg::WPB, Cfg::BLOCKS>, grid, block, st, !a.fresh_k, a);
    else if (rag) e = launch_overlapped(sweep_pair<S, false, true, Cfg::R, Cfg::WPB, Cfg::BLOCKS>, grid, block, st, !a.fresh_k, a);
    else e = launch_overlapped(sweep_pair<S, false, false, Cfg::R, Cfg::WPB, Cfg::BLOCKS>, grid, block, st, !a.fresh_k, a);
    if (ev) cudaEventRecord(ev[1], st);
    return e;
}

}  // namespace wfa
