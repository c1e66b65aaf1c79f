// Implicit (backward-Euler) time steps solved by classic conjugate gradients
// (Sec. 1.1.2, Eq. impl_form), in the same face-flux form as the explicit
// sweep, diffusion only (with advection the system is not symmetric and CG
// does not apply).
//
// One step solves, for every cell that is not held,
//   T'_C + sum_f c_f (T'_C - T'_D) + sum_{Dirichlet faces} d_f (T'_C - Tb_f) = T_C
// with c_f = dt K_f / h_a^2 (K_f the harmonic-mean face conductivity) and
// d_f = 2 dt k_C / h_a^2; held cells keep their value. Moving the known
// values (Dirichlet faces, held neighbours) to the right-hand side leaves a
// symmetric positive definite system A y = b on the free cells, solved from
// y = T by classic CG with its two inner products per iteration:
//
//   q = A p,  alpha = r.r / p.q,  x += alpha p,  r -= alpha q,
//   beta = r.r' / r.r,  p = r + beta p
//
// GB300 mapping. The field x is the grid's fp32 buffer, updated in place;
// r, p (two buffers) and q are fp32 work vectors in the same padded layout.
// Each iteration is two HBM-bound kernels and a one-block control kernel:
//   cg_dir    p = r + beta p_old on the fly (for the cell and its six
//             neighbours), the block partials of p.(A p), and the x += alpha p
//             of the iteration before (its p is read here anyway); reads r,
//             p_old and x, writes p and x (20 B a cell); per-cell k: reads 1/k
//             and writes q = A p too (28 B);
//   cg_res    r -= alpha q and the block partials of r.r: uniform k forms
//             q = A p again (cg_res_u: reads p and r, writes r, 12 B), per-cell
//             k reads it (cg_res_k: q and r, writes r, 12 B);
//   cg_ctl_iter  r.r, beta and the convergence test from the partials.
// 32 B a cell and iteration (40 with per-cell k); storing q and updating x in
// cg_res takes 40 (44). cg_xfin adds the last iteration's alpha p.
// Every scalar is computed on the device, so no host round trip sits between
// iterations: a whole call is one graph launch whose conditional WHILE nodes
// loop over the time steps and the iterations (device loops, below); where
// those cannot be built, captured runs of iterations are replayed with the
// host reading the convergence flag between runs, one run ahead.
// Periodic axes read the neighbour across the boundary from a twin copy
// that every writer of a boundary cell also stores one cell beyond the
// opposite face; non-periodic boundary faces take a ghost value that makes
// the interior expression exact, only in warps that hold a boundary cell.
// cg_pipe is the pipelined alternative (Chronopoulos and Gear): one kernel
// and one reduction an iteration.
// Inner products: fp32 products summed per plane, a compensated fp32 sum over
// a thread's planes, fp64 above that (the block, the fixed-order sum over
// blocks); the GPU's fp64 rate is low, so no fp64 arithmetic sits in the
// hot loops.
#include <type_traits>
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <new>

#include "wfa_internal.cuh"
#include "wfa_sweep_pair.cuh"

namespace wfa {

constexpr int CG_TX = 16, CG_TY = 16;   // cg_init / cg_pipe block: 64 x 16 cells, 4 x cells a thread
constexpr int CG_THREADS = 256;
constexpr int CG_CTL = 512;             // threads of the one-block control kernels (16 warps: see block_sum)
constexpr int CG_MAX_PART = 16384;      // per-block partials of one launch
constexpr int CG_FOLD = 512;            // most blocks of cg_dir whose partials every block of cg_res sums
constexpr int CG_R = 2, CG_W = 4;       // cg_dir / cg_res_u: rows a thread, most warps of a block
constexpr int CG_NRUN = 4;              // captured runs of 1, 2, 4 and 8 iterations
constexpr int CG_RUN_LEN[CG_NRUN] = {1, 2, 4, 8};

// Solver scalars on the device (56 bytes; read back as one block).
struct CgState {   // fits one 64-byte pinned word
    double rr;        // r.r of the current residual
    double bb;        // b.b of the step's right-hand side
    double alpha, beta;
    double tol2;      // rtol^2
    int done;         // converged, iteration limit reached, or breakdown
    int iter;         // iterations of the current step
    int max_iter;
    unsigned ticket;  // blocks of the current launch that have finished
    int pending;      // classic CG: x lacks the last iteration's alpha p (1), or only its periodic twins (2)
};

static_assert(sizeof(CgState) <= 64, "CgState is read back into a 64-byte pinned word");

struct CgCoef {
    int n[3];
    int periodic[3];
    int dface[6];     // face carries a Dirichlet value (on the face)
    int held[6];      // face holds its outer cell layer
    long long sy, sz; // element strides of the padded layout
    float tb[6];      // Dirichlet face values
    float cu[3];      // uniform k: dt k / h_a^2
    float du;         // uniform k: 1 + 2 (cu[0] + cu[1] + cu[2]), an interior row's diagonal
    float tcd[3];     // per-cell k: 2 dt / h_a^2 (c_f = tcd / (1/k_C + 1/k_D))
};

struct CgArgs {
    CgCoef c;
    float* x;          // domain origins (cell (0,0,0)) of the padded arrays
    const float* rk;   // 1/k, or nullptr for uniform k
    float* r;
    float* p0;
    float* p1;
    float* q;
    double* part;      // per-block partials, two arrays of CG_MAX_PART: p.q and r.r (cg_init: r.r and b.b)
    CgState* s;
    float* r2;         // pipelined CG: second r, w and s buffers (r, w and s ping-pong, read at
    float* w2;         // neighbours: r in r / r2, w in q / w2, s in p1 / s2; p in p0)
    float* s2;
    int zchunk;        // planes per block
    int nblk;          // blocks of this launch
    int lanes;         // cg_dir / cg_res_u: threads side by side along x (32, 16 or 8)
    int dblk;          // partials of p.q that cg_res sums itself (0: the last block of cg_dir has)
    int q_twins;       // cg_dir also writes q's periodic twins (q is the pipelined solver's first w)
};

__device__ __forceinline__ long long cg_at(const CgCoef& c, int x, int y, int z) {
    return x + (long long)y * c.sy + (long long)z * c.sz;
}

__device__ __forceinline__ bool cg_held(const CgCoef& c, int x, int y, int z) {
    return (c.held[0] && x == 0) || (c.held[1] && x == c.n[0] - 1) || (c.held[2] && y == 0) ||
           (c.held[3] && y == c.n[1] - 1) || (c.held[4] && z == 0) || (c.held[5] && z == c.n[2] - 1);
}
// The same over the faces of mask FM (bit f: face f); the caller knows that
// the cell is on no face outside FM.
template <int FM>
__device__ __forceinline__ bool cg_held_m(const CgCoef& c, int x, int y, int z) {
    return ((FM & 1) && c.held[0] && x == 0) || ((FM & 2) && c.held[1] && x == c.n[0] - 1) ||
           ((FM & 4) && c.held[2] && y == 0) || ((FM & 8) && c.held[3] && y == c.n[1] - 1) ||
           ((FM & 16) && c.held[4] && z == 0) || ((FM & 32) && c.held[5] && z == c.n[2] - 1);
}

__device__ __forceinline__ void ld4(const float* p, float v[4]) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}

// Store 4 cells of row (gx.., y, z), the ones inside the domain, plus the
// periodic twins of those on a periodic face.
__device__ __forceinline__ void st4_row(float* o, int gx, int nx, const float v[4]) {
    if (gx + 3 < nx) {
        *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (gx + i < nx) o[i] = v[i];
    }
}

__device__ __forceinline__ void st4_twins(float* base, const CgCoef& c, int gx, int y, int z, const float v[4]) {
    const int nx = c.n[0];
    st4_row(base + cg_at(c, gx, y, z), gx, nx, v);
    if (c.periodic[1] && (y == 0 || y == c.n[1] - 1)) st4_row(base + cg_at(c, gx, y == 0 ? c.n[1] : -1, z), gx, nx, v);
    if (c.periodic[2] && (z == 0 || z == c.n[2] - 1)) st4_row(base + cg_at(c, gx, y, z == 0 ? c.n[2] : -1), gx, nx, v);
    if (c.periodic[0]) {
        if (gx == 0) base[cg_at(c, nx, y, z)] = v[0];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (gx + i == nx - 1) base[cg_at(c, -1, y, z)] = v[i];
    }
}

// Compensated (Kahan) fp32 running sum: a thread's share of an inner product
// without per-plane fp64 arithmetic (the GPU's fp64 rate is a small fraction
// of its fp32 rate); the block and the blocks are then summed in fp64.
struct KahanF {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float v) {
        const float y = __fsub_rn(v, c);
        const float t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// Block sum of one double per thread (fixed shuffle trees: the warps, then the
// first warp over their sums); the result is valid in thread 0. A dependent
// fp64 add takes some 60 cycles here, so the chain is kept short.
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nw = (blockDim.x * blockDim.y + 31) / 32;
    if ((tid & 31) == 0) red[tid >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (tid < 32) {
        t = tid < nw ? red[tid] : 0.0;
        for (int o = nw > 8 ? 8 : 4; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    }
    __syncthreads();
    return t;
}

// Publish this block's partial; true in every thread of the last block of
// the launch to do so (which then owns the finish and resets the ticket).
__device__ __forceinline__ bool publish(const CgArgs& a, double* slot, double v, bool* last) {
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    if (tid == 0) {
        *slot = v;
        __threadfence();
        const unsigned t = atomicAdd(&a.s->ticket, 1u);
        *last = t == (unsigned)a.nblk - 1;
        if (t == (unsigned)a.nblk - 1) __threadfence();
    }
    __syncthreads();
    return *last;
}

// Fixed-order sum of n partials by the whole block; valid in thread 0.
__device__ __forceinline__ double sum_partials(const double* part, int n, double* red) {
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int nt = blockDim.x * blockDim.y;
    double t = 0.0;
#pragma unroll 8
    for (int i = tid; i < n; i += nt) t += __ldcg(part + i);
    return block_sum(t, red);
}

template <bool KVAR>
struct CgOcc {
    static constexpr int blocks = KVAR ? 3 : 4;
};

// Boundary faces a thread's cells touch (non-periodic axes only). A face is
// taken as a ghost neighbour that makes the interior formula exact: across a
// Dirichlet face (value 0 in A) p_ghost = -p_C, across a zero-flux face
// p_ghost = p_C, with the ghost's conductivity that of the cell (so the face
// coefficient is tcd / (2 r_C): twice it is the Dirichlet coefficient
// 2 k_C dt / h^2). Held cells are masked (q = 0).
struct CgEdge {
    int ih;            // index 0..3 of the thread's cell on the +x face (4: none)
    unsigned bits;     // 1: cell 0 on the -x face, 2: the row on the -y face, 4: on the +y face
};

__device__ __forceinline__ CgEdge cg_edge(const CgCoef& c, int gx, int gy) {
    CgEdge e;
    const int nx = c.n[0], ny = c.n[1];
    e.ih = (!c.periodic[0] && gx <= nx - 1 && nx - 1 - gx < 4) ? nx - 1 - gx : 4;
    e.bits = ((!c.periodic[0] && gx == 0) ? 1u : 0u) | ((!c.periodic[1] && gy == 0) ? 2u : 0u) |
             ((!c.periodic[1] && gy == ny - 1) ? 4u : 0u);
    return e;
}

// ghost value across face f of a cell holding v: -v (Dirichlet face) or v
__device__ __forceinline__ float ghost(const CgCoef& c, int f, float v) { return c.dface[f] ? -v : v; }

// r = dt acc(T) and the b terms of the 4 cells of a thread at plane z. EDGE
// (warp-uniform) puts ghost values across boundary faces (2 Tb - T_C across a
// Dirichlet face, T_C across a zero-flux face, the cell's own 1/k), adds the
// known values to b (Dirichlet faces: d_f Tb; held neighbours: c_f T_D) and
// masks held cells and cells beyond the x end; without it every neighbour
// is a free cell inside the domain or across a periodic face. FM: the faces
// (bit f: face f) whose boundary or held layer may be near the warp's cells
// (x faces only for warps away from the y and z faces); the others are not
// looked at.
template <bool KVAR, bool EDGE, int FM = 63>
__device__ __forceinline__ void cg_r4(const CgCoef& c, const CgEdge& e, int gx, int gy, int z, const float tc[4],
                                      const float tm[4], const float tp[4], const float ym[4], const float yp[4],
                                      float xm, float xp, const float kc[4], const float km[4], const float kp[4],
                                      const float kym[4], const float kyp[4], float kxm, float kxp, float rv[4],
                                      float& sr, float& sb) {
    const int nx = c.n[0], ny = c.n[1], nz = c.n[2];
    const bool zlo = EDGE && (FM & 16) && !c.periodic[2] && z == 0,
               zhi = EDGE && (FM & 32) && !c.periodic[2] && z == nz - 1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float t[6] = {i == 0 ? xm : tc[i - 1], i == 3 ? xp : tc[i + 1], ym[i], yp[i], tm[i], tp[i]};
        float k[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (KVAR) {
            k[0] = i == 0 ? kxm : kc[i - 1];
            k[1] = i == 3 ? kxp : kc[i + 1];
            k[2] = kym[i];
            k[3] = kyp[i];
            k[4] = km[i];
            k[5] = kp[i];
        }
        float bs = tc[i];
        if (EDGE) {
            const int xi = gx + i;
            const bool bd[6] = {(FM & 1) && i == 0 && (e.bits & 1u) != 0, (FM & 2) && i == e.ih,
                                (FM & 4) && (e.bits & 2u) != 0, (FM & 8) && (e.bits & 4u) != 0, zlo, zhi};
            // a neighbour inside the domain is held only through its own axis's face
            const bool hn[6] = {(FM & 1) && c.held[0] && xi == 1, (FM & 2) && c.held[1] && xi == nx - 2,
                                (FM & 4) && c.held[2] && gy == 1, (FM & 8) && c.held[3] && gy == ny - 2,
                                (FM & 16) && c.held[4] && z == 1, (FM & 32) && c.held[5] && z == nz - 2};
#pragma unroll
            for (int f = 0; f < 6; ++f) {
                if (!((FM >> f) & 1)) continue;
                const float cf = KVAR ? face_r(kc[i], bd[f] ? kc[i] : k[f], c.tcd[f >> 1]) : c.cu[f >> 1];
                if (hn[f]) bs = __fmaf_rn(cf, t[f], bs);
                if (bd[f]) {
                    if (c.dface[f]) bs = __fmaf_rn(__fmul_rn(2.0f, cf), c.tb[f], bs);
                    t[f] = c.dface[f] ? __fsub_rn(__fmul_rn(2.0f, c.tb[f]), tc[i]) : tc[i];
                    k[f] = kc[i];
                }
            }
        }
        float acc;
        if (KVAR) {
            acc = __fmul_rn(face_r(kc[i], k[0], c.tcd[0]), __fsub_rn(t[0], tc[i]));
            acc = __fmaf_rn(face_r(kc[i], k[1], c.tcd[0]), __fsub_rn(t[1], tc[i]), acc);
            acc = __fmaf_rn(face_r(kc[i], k[2], c.tcd[1]), __fsub_rn(t[2], tc[i]), acc);
            acc = __fmaf_rn(face_r(kc[i], k[3], c.tcd[1]), __fsub_rn(t[3], tc[i]), acc);
            acc = __fmaf_rn(face_r(kc[i], k[4], c.tcd[2]), __fsub_rn(t[4], tc[i]), acc);
            acc = __fmaf_rn(face_r(kc[i], k[5], c.tcd[2]), __fsub_rn(t[5], tc[i]), acc);
        } else {
            acc = __fmul_rn(c.cu[0], __fadd_rn(__fsub_rn(t[0], tc[i]), __fsub_rn(t[1], tc[i])));
            acc = __fmaf_rn(c.cu[1], __fadd_rn(__fsub_rn(t[2], tc[i]), __fsub_rn(t[3], tc[i])), acc);
            acc = __fmaf_rn(c.cu[2], __fadd_rn(__fsub_rn(t[4], tc[i]), __fsub_rn(t[5], tc[i])), acc);
        }
        if (EDGE) {
            const bool isfree = gx + i < nx && gy < ny && !cg_held_m<FM>(c, gx + i, gy, z);
            rv[i] = isfree ? acc : 0.0f;
            sr = __fmaf_rn(rv[i], rv[i], sr);
            if (isfree) sb = __fmaf_rn(bs, bs, sb);
        } else {
            rv[i] = acc;
            sr = __fmaf_rn(acc, acc, sr);
            sb = __fmaf_rn(bs, bs, sb);
        }
    }
}

// ---------------------------------------------------------------- cg_init --
// r = b - A T (dt times the explicit step's accumulation), b.b and r.r, on
// a column-march layout (4 x cells a thread, z queue). The
// field's periodic twins are current (refresh_halo before the first step,
// cg_xfin after every step). b adds to T the known values: Dirichlet
// faces and held neighbours. O32: every array is under 4 GiB, so the loop
// addresses its planes by a 32-bit byte offset from the array's start (one
// integer add an address); otherwise by a 64-bit one.
template <bool KVAR, bool O32>
__global__ void __launch_bounds__(CG_TX * CG_TY, CgOcc<KVAR>::blocks) cg_init(const __grid_constant__ CgArgs a) {
    __shared__ double red[CG_TX * CG_TY / 32];
    const CgCoef& c = a.c;
    const float* __restrict__ xv = a.x;
    const float* __restrict__ rk = a.rk;
    const int nx = c.n[0], ny = c.n[1], nz = c.n[2];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int gx = blockIdx.x * 64 + 4 * tx, gy = blockIdx.y * CG_TY + ty;
    const int z0 = blockIdx.z * a.zchunk, z1 = min(z0 + a.zchunk, nz);
    const bool perx = c.periodic[0], pery = c.periodic[1], perz = c.periodic[2];
    KahanF rr, bb;
    if (gx < nx && gy < ny) {
        const long long sy = c.sy, sz = c.sz;
        const long long row = cg_at(c, gx, gy, 0);
        // fast cells: no boundary face and no held neighbour (two cells from
        // every non-periodic face); inner_y: the same along y only
        const bool inner_y = pery || (gy > 1 && gy < ny - 2);
        const bool inner_xy = gx + 3 < nx && (perx || (gx > 1 && gx + 5 < nx)) && inner_y;
        const CgEdge edge = cg_edge(c, gx, gy);
        float tm[4], tc[4], km[4], kc[4];
        ld4(xv + row + (long long)(z0 - 1) * sz, tm);
        ld4(xv + row + (long long)z0 * sz, tc);
        if (KVAR) {
            ld4(rk + row + (long long)(z0 - 1) * sz, km);
            ld4(rk + row + (long long)z0 * sz, kc);
        }
        using OT = typename std::conditional<O32, unsigned, unsigned long long>::type;
        const long long org = HALO * sz + HALO * sy + HALO;   // elements before the domain origin
        const char* const xB = reinterpret_cast<const char*>(xv - org);
        const char* const kB = KVAR ? reinterpret_cast<const char*>(rk - org) : nullptr;
        char* const rB = reinterpret_cast<char*>(a.r - org);
        auto F = [](const char* b, OT o) { return reinterpret_cast<const float*>(b + o); };
        OT o = (OT)((org + row + (long long)z0 * sz) * 4);   // plane z, this thread's first cell
        const OT dz = (OT)(sz * 4), dy = (OT)(sy * 4);
        const bool twins = perx || pery || perz;
        for (int z = z0; z < z1; ++z) {
            if ((tx & 7) == 0) prefetch_l2(F(xB, o + 3 * dz));
            float tp[4], ym[4], yp[4];
            ld4(F(xB, o + dz), tp);
            ld4(F(xB, o - dy), ym);
            ld4(F(xB, o + dy), yp);
            const float xm = __ldg(F(xB, o - 4u)), xp = __ldg(F(xB, o + 16u));
            float kp[4], kym[4], kyp[4], kxm = 0.0f, kxp = 0.0f;
            if (KVAR) {
                ld4(F(kB, o + dz), kp);
                ld4(F(kB, o - dy), kym);
                ld4(F(kB, o + dy), kyp);
                kxm = __ldg(F(kB, o - 4u));
                kxp = __ldg(F(kB, o + 16u));
            }
            float rv[4];
            float sr = 0.0f, sb = 0.0f;
            const bool inner_z = perz || (z > 1 && z < nz - 2);
            const bool fast = inner_xy && inner_z;
            const unsigned am = __activemask();
            if (__all_sync(am, fast))   // warp-uniform choice
                cg_r4<KVAR, false>(c, edge, gx, gy, z, tc, tm, tp, ym, yp, xm, xp, kc, km, kp, kym, kyp, kxm, kxp, rv,
                                   sr, sb);
            else if (__all_sync(am, inner_y && inner_z))   // near an x face only
                cg_r4<KVAR, true, 3>(c, edge, gx, gy, z, tc, tm, tp, ym, yp, xm, xp, kc, km, kp, kym, kyp, kxm, kxp,
                                     rv, sr, sb);
            else
                cg_r4<KVAR, true>(c, edge, gx, gy, z, tc, tm, tp, ym, yp, xm, xp, kc, km, kp, kym, kyp, kxm, kxp, rv,
                                  sr, sb);
            if (twins)   // the same for every thread
                st4_twins(a.r, c, gx, gy, z, rv);
            else
                st4_row(reinterpret_cast<float*>(rB + o), gx, nx, rv);
            rr.add(sr);
            bb.add(sb);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                tm[i] = tc[i];
                tc[i] = tp[i];
                if (KVAR) {
                    km[i] = kc[i];
                    kc[i] = kp[i];
                }
            }
            o += dz;
        }
    }
    const int blk = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    const double rs = block_sum(rr.value(), red);
    const double bsum = block_sum(bb.value(), red);
    if (threadIdx.x == 0 && threadIdx.y == 0) {   // summed by cg_ctl_start
        a.part[blk] = rs;
        a.part[CG_MAX_PART + blk] = bsum;
    }
}

// ---------------------------------------------------------------- q = A p --
// q = A p for the 4 cells of a thread at plane z, and their p.q (cells inside
// the domain). EDGE (chosen warp-uniformly) puts ghost values across
// boundary faces and masks held cells and cells beyond the x end; without
// it every neighbour is inside the domain or across a periodic face. Both
// evaluate the same expression, so an interior cell gets the same bits
// either way.
template <bool KVAR, bool EDGE>
__device__ __forceinline__ float cg_q4(const CgCoef& c, const CgEdge& e, int gx, int gy, int z, const float pc[4],
                                       const float pm[4], const float pp[4], const float ym[4], const float yp[4],
                                       float xm, float xp, const float kc[4], const float km[4], const float kp[4],
                                       const float kym[4], const float kyp[4], float kxm, float kxp, float q[4]) {
    float psum = 0.0f;
    const bool zlo = EDGE && !c.periodic[2] && z == 0,
               zhi = EDGE && !c.periodic[2] && z == c.n[2] - 1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float pw = i == 0 ? xm : pc[i - 1], pe = i == 3 ? xp : pc[i + 1];
        float y0 = ym[i], y1 = yp[i], z0 = pm[i], z1 = pp[i];
        float kw = 0.0f, ke = 0.0f, ky0 = 0.0f, ky1 = 0.0f, kz0 = 0.0f, kz1 = 0.0f;
        if (KVAR) {
            kw = i == 0 ? kxm : kc[i - 1];
            ke = i == 3 ? kxp : kc[i + 1];
            ky0 = kym[i];
            ky1 = kyp[i];
            kz0 = km[i];
            kz1 = kp[i];
        }
        if (EDGE) {
            if (i == 0 && (e.bits & 1u)) { pw = ghost(c, 0, pc[i]); kw = kc[i]; }
            if (i == e.ih) { pe = ghost(c, 1, pc[i]); ke = kc[i]; }
            if ((e.bits & 2u)) { y0 = ghost(c, 2, pc[i]); ky0 = kc[i]; }
            if ((e.bits & 4u)) { y1 = ghost(c, 3, pc[i]); ky1 = kc[i]; }
            if (zlo) { z0 = ghost(c, 4, pc[i]); kz0 = kc[i]; }
            if (zhi) { z1 = ghost(c, 5, pc[i]); kz1 = kc[i]; }
        }
        float qi;
        if (KVAR) {
            const float r0 = kc[i];
            float acc = __fmul_rn(face_r(r0, kw, c.tcd[0]), __fsub_rn(pc[i], pw));
            acc = __fmaf_rn(face_r(r0, ke, c.tcd[0]), __fsub_rn(pc[i], pe), acc);
            acc = __fmaf_rn(face_r(r0, ky0, c.tcd[1]), __fsub_rn(pc[i], y0), acc);
            acc = __fmaf_rn(face_r(r0, ky1, c.tcd[1]), __fsub_rn(pc[i], y1), acc);
            acc = __fmaf_rn(face_r(r0, kz0, c.tcd[2]), __fsub_rn(pc[i], z0), acc);
            acc = __fmaf_rn(face_r(r0, kz1, c.tcd[2]), __fsub_rn(pc[i], z1), acc);
            qi = __fadd_rn(pc[i], acc);
        } else {
            float acc = __fmul_rn(c.du, pc[i]);
            acc = __fmaf_rn(-c.cu[0], __fadd_rn(pw, pe), acc);
            acc = __fmaf_rn(-c.cu[1], __fadd_rn(y0, y1), acc);
            qi = __fmaf_rn(-c.cu[2], __fadd_rn(z0, z1), acc);
        }
        if (EDGE) {
            const bool isfree = gx + i < c.n[0] && gy < c.n[1] && !cg_held(c, gx + i, gy, z);
            qi = isfree ? qi : 0.0f;
            psum = isfree ? __fmaf_rn(pc[i], qi, psum) : psum;
        } else {
            psum = __fmaf_rn(pc[i], qi, psum);
        }
        q[i] = qi;
    }
    return psum;
}

// Row operands of a thread: 4 cells of two rows as pairs.
__device__ __forceinline__ void ldp(const float* p, f2 (&v)[2]) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = f2_make(t.x, t.y);
    v[1] = f2_make(t.z, t.w);
}
__device__ __forceinline__ void unp(const f2 (&v)[2], float o[4]) {
    f2_get(v[0], o[0], o[1]);
    f2_get(v[1], o[2], o[3]);
}
// v = r + beta p_old, both as loaded. On the first iteration p_old is r itself
// and beta 0, so that no load waits behind a branch.
__device__ __forceinline__ void pnew_pairs(const float4& r, const float4& o, f2 beta, f2 (&v)[2]) {
    v[0] = f2_fma(beta, f2_make(o.x, o.y), f2_make(r.x, r.y));
    v[1] = f2_fma(beta, f2_make(o.z, o.w), f2_make(r.z, r.w));
}
__device__ __forceinline__ float4 ldv(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ f2 lo2(const float4& v) { return f2_make(v.x, v.y); }
__device__ __forceinline__ f2 hi2(const float4& v) { return f2_make(v.z, v.w); }

// q = A p of one interior row (every neighbour a free cell), cg_q4's
// expression on pairs; uniform k.
__device__ __forceinline__ void cg_row_u(const CgCoef& c, const f2 (&pc)[2], const f2 (&pm)[2], const f2 (&pp)[2],
                                         const f2 (&ym)[2], const f2 (&yp)[2], float xm, float xp, f2 (&q)[2]) {
    float v[4];
    unp(pc, v);
    const f2 n0 = f2_make(-c.cu[0], -c.cu[0]), n1 = f2_make(-c.cu[1], -c.cu[1]), n2 = f2_make(-c.cu[2], -c.cu[2]);
    const f2 x[2] = {f2_make(__fadd_rn(xm, v[1]), __fadd_rn(v[0], v[2])), f2_make(__fadd_rn(v[1], v[3]), __fadd_rn(v[2], xp))};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        f2 acc = f2_mul(f2_make(c.du, c.du), pc[i]);
        acc = f2_fma(n0, x[i], acc);
        acc = f2_fma(n1, f2_add(ym[i], yp[i]), acc);
        q[i] = f2_fma(n2, f2_add(pm[i], pp[i]), acc);
    }
}
// Per-cell k: gm / gp the faces below and above the row, zm / zp along z.
__device__ __forceinline__ void cg_row_k(const CgCoef& c, const f2 (&pc)[2], const f2 (&pm)[2], const f2 (&pp)[2],
                                         const f2 (&ym)[2], const f2 (&yp)[2], float xm, float xp, const f2 (&kc)[2],
                                         float kxm, float kxp, const f2 (&gm)[2], const f2 (&gp)[2], const f2 (&zm)[2],
                                         const f2 (&zp)[2], f2 (&q)[2]) {
    float v[4], k[4];
    unp(pc, v);
    unp(kc, k);
    const float x0 = face_r(kxm, k[0], c.tcd[0]), x1 = face_r(k[0], k[1], c.tcd[0]), x2 = face_r(k[1], k[2], c.tcd[0]),
                x3 = face_r(k[2], k[3], c.tcd[0]), x4 = face_r(k[3], kxp, c.tcd[0]);
    f2 acc[2];
    acc[0] = f2_mul(f2_make(x0, x1), f2_make(__fsub_rn(v[0], xm), __fsub_rn(v[1], v[0])));
    acc[1] = f2_mul(f2_make(x2, x3), f2_make(__fsub_rn(v[2], v[1]), __fsub_rn(v[3], v[2])));
    acc[0] = f2_fma(f2_make(x1, x2), f2_make(__fsub_rn(v[0], v[1]), __fsub_rn(v[1], v[2])), acc[0]);
    acc[1] = f2_fma(f2_make(x3, x4), f2_make(__fsub_rn(v[2], v[3]), __fsub_rn(v[3], xp)), acc[1]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        acc[i] = f2_fma(gm[i], f2_sub(pc[i], ym[i]), acc[i]);
        acc[i] = f2_fma(gp[i], f2_sub(pc[i], yp[i]), acc[i]);
        acc[i] = f2_fma(zm[i], f2_sub(pc[i], pm[i]), acc[i]);
        acc[i] = f2_fma(zp[i], f2_sub(pc[i], pp[i]), acc[i]);
        q[i] = f2_add(pc[i], acc[i]);
    }
}

// What a thread of cg_dir / cg_res_u covers: 4 x cells of CG_R rows; a.lanes
// (32, 16 or 8) threads lie side by side along x, so narrow grids fill their warps.
struct CgPlace {
    int gx, gy;            // first cell and row
    long long row;         // its place in memory at plane 0 (threads beyond a row or the rows read its halo)
    int lane, lanes;       // position along x, shuffle width
    bool rows, in;         // some row of the warp, some cell of the thread inside the domain
    bool ends;             // first or last lane: its outer x neighbour is another thread group's
    int eo;                // that neighbour's offset from the first cell
    bool inner_y;          // warp: every row away from the y faces
    bool xlo, xhi;         // the thread's first / last cell lies on a (non-periodic) x face
    bool ragged;           // warp: some thread's cells reach beyond the x end or into a held x layer
    int ih;                // index of its cell on the +x face, 4 when none
    unsigned dead;         // bit i: cell i is beyond the x end or in a held x layer
    __device__ __forceinline__ CgPlace(const CgArgs& a) {
        const CgCoef& c = a.c;
        const int nx = c.n[0], ny = c.n[1];
        lanes = a.lanes;
        lane = threadIdx.x & (lanes - 1);
        const int tile = blockDim.x / lanes;   // row groups of a block
        gx = (blockIdx.x * lanes + lane) * 4;
        gy = (blockIdx.y * tile + threadIdx.x / lanes) * CG_R;
        row = min(gx, (nx + 3) & ~3) + (long long)min(gy, ny) * c.sy;
        in = gx < nx && gy < ny;
        rows = __any_sync(0xffffffffu, in);
        ends = lane == 0 || lane == lanes - 1;
        eo = lane == 0 ? -1 : 4;
        const bool iy = gy + CG_R <= ny && (c.periodic[1] || (gy > 0 && gy + CG_R < ny));
        inner_y = __all_sync(0xffffffffu, !in || iy);
        ih = !c.periodic[0] && gx < nx && nx - 1 - gx < 4 ? nx - 1 - gx : 4;
        xlo = !c.periodic[0] && gx == 0;
        xhi = ih == 3;
        dead = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (gx + i >= nx || (c.held[0] && gx + i == 0) || (c.held[1] && gx + i == nx - 1)) dead |= 1u << i;
        ragged = __any_sync(0xffffffffu, dead != 0);
    }
};

// q = A p of a thread's rows at plane z and their p.q. Away from the y and z
// faces the pair form serves every warp: across an x face the neighbour is the
// ghost value (cg_q4's) put in its place, and cells that are not free get
// q = 0; next to a y or z face cg_q4 goes row by row. zf: the faces towards
// z - 1 on entry, towards z + 1 on return; kz: 1/k of the first row at z - 1.
// dot takes the 4 products of each row at a time: what a plain fp32 sum of them
// rounds off is all that the compensated sum does not see.
template <bool KVAR>
__device__ __forceinline__ void cg_rows(const CgCoef& c, const CgPlace& t, int z, f2 (&pc)[CG_R][2],
                                         const f2 (&pm)[CG_R][2], const f2 (&pp)[CG_R][2], const f2 (&h)[2][2],
                                         const float (&e)[CG_R], f2 (&kc)[KVAR ? CG_R : 1][2],
                                         f2 (&zf)[KVAR ? CG_R : 1][2], const f2 (&kp)[KVAR ? CG_R : 1][2],
                                         const f2 (&kh)[2][2], const float (&ke)[CG_R], const float* kz, f2 (&q)[CG_R][2],
                                        KahanF& dot) {
    constexpr unsigned FULL = 0xffffffffu;
    const int ny = c.n[1], nz = c.n[2];
    float xm[CG_R], xp[CG_R], kxm[CG_R], kxp[CG_R];
    const float g0 = c.dface[0] ? -1.0f : 1.0f, g1 = c.dface[1] ? -1.0f : 1.0f;
#pragma unroll
    for (int j = 0; j < CG_R; ++j) {
        const float u = __shfl_up_sync(FULL, f2_hi(pc[j][1]), 1, t.lanes);
        const float d = __shfl_down_sync(FULL, f2_lo(pc[j][0]), 1, t.lanes);
        xm[j] = t.lane == 0 ? e[j] : u;
        xp[j] = t.lane == t.lanes - 1 ? e[j] : d;
        xm[j] = t.xlo ? __fmul_rn(g0, f2_lo(pc[j][0])) : xm[j];
        xp[j] = t.xhi ? __fmul_rn(g1, f2_hi(pc[j][1])) : xp[j];
        kxm[j] = kxp[j] = 0.0f;
        if (KVAR) {
            const int jk = KVAR ? j : 0;
            const float ku = __shfl_up_sync(FULL, f2_hi(kc[jk][1]), 1, t.lanes);
            const float kd = __shfl_down_sync(FULL, f2_lo(kc[jk][0]), 1, t.lanes);
            kxm[j] = t.lane == 0 ? ke[j] : ku;
            kxp[j] = t.lane == t.lanes - 1 ? ke[j] : kd;
            kxm[j] = t.xlo ? f2_lo(kc[jk][0]) : kxm[j];
            kxp[j] = t.xhi ? f2_hi(kc[jk][1]) : kxp[j];
        }
    }
    if (t.ragged) {   // the +x face inside the thread's cells: the ghost goes into the cell beyond it
#pragma unroll
        for (int j = 0; j < CG_R; ++j) {
            float v[4], k[4];
            unp(pc[j], v);
            if (KVAR) unp(kc[KVAR ? j : 0], k);
#pragma unroll
            for (int i = 2; i >= 0; --i)
                if (t.ih == i) {
                    v[i + 1] = __fmul_rn(g1, v[i]);
                    if (KVAR) k[i + 1] = k[i];
                }
            pc[j][0] = f2_make(v[0], v[1]);
            pc[j][1] = f2_make(v[2], v[3]);
            if (KVAR) {
                kc[KVAR ? j : 0][0] = f2_make(k[0], k[1]);
                kc[KVAR ? j : 0][1] = f2_make(k[2], k[3]);
            }
        }
    }
    const f2(&pr)[CG_R][2] = pc;
    const f2(&kr)[KVAR ? CG_R : 1][2] = kc;
    f2 gp[KVAR ? CG_R : 1][2];
    if (KVAR) {
        const f2 tz = f2_make(c.tcd[2], c.tcd[2]);
#pragma unroll
        for (int j = 0; j < (KVAR ? CG_R : 1); ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) gp[j][i] = pair_face(kc[j][i], kp[j][i], tz);
    }
    if (t.inner_y && (c.periodic[2] || (z > 0 && z < nz - 1))) {
        f2 gy[2][2];
        const f2 ty = f2_make(c.tcd[1], c.tcd[1]);
        if (KVAR) {
#pragma unroll
            for (int i = 0; i < 2; ++i) gy[0][i] = pair_face(kh[0][i], kc[0][i], ty);
        }
#pragma unroll
        for (int j = 0; j < CG_R; ++j) {
            const int jk = KVAR ? j : 0;
            const f2(&ym)[2] = j == 0 ? h[0] : pr[j > 0 ? j - 1 : 0];
            const f2(&yp)[2] = j == CG_R - 1 ? h[1] : pr[j < CG_R - 1 ? j + 1 : 0];
            if (KVAR) {
                const f2(&kn)[2] = j == CG_R - 1 ? kh[1] : kr[KVAR && j < CG_R - 1 ? j + 1 : 0];
#pragma unroll
                for (int i = 0; i < 2; ++i) gy[1][i] = pair_face(kc[jk][i], kn[i], ty);
                cg_row_k(c, pc[j], pm[j], pp[j], ym, yp, xm[j], xp[j], kc[jk], kxm[j], kxp[j], gy[0], gy[1], zf[jk], gp[jk],
                         q[j]);
#pragma unroll
                for (int i = 0; i < 2; ++i) gy[0][i] = gy[1][i];
            } else {
                cg_row_u(c, pc[j], pm[j], pp[j], ym, yp, xm[j], xp[j], q[j]);
            }
            if (t.ragged) {
                float v[4];
                unp(q[j], v);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (t.dead >> i & 1u) v[i] = 0.0f;
                q[j][0] = f2_make(v[0], v[1]);
                q[j][1] = f2_make(v[2], v[3]);
            }
            const f2 d = f2_fma(pc[j][1], q[j][1], f2_mul(pc[j][0], q[j][0]));
            dot.add(t.in ? __fadd_rn(f2_lo(d), f2_hi(d)) : 0.0f);
        }
    } else {
#pragma unroll
        for (int j = 0; j < CG_R; ++j) {
            const int y = t.gy + j, jk = KVAR ? j : 0;
            const CgEdge edge = cg_edge(c, t.gx, y);
            float pcv[4], pmv[4], ppv[4], ymv[4], ypv[4], kcv[4], kmv[4], kpv[4], kymv[4], kypv[4], qv[4];
            unp(pc[j], pcv);
            unp(pm[j], pmv);
            unp(pp[j], ppv);
            unp(j == 0 ? h[0] : pr[j > 0 ? j - 1 : 0], ymv);
            unp(j == CG_R - 1 ? h[1] : pr[j < CG_R - 1 ? j + 1 : 0], ypv);
            if (KVAR) {
                ld4(kz + (long long)j * c.sy, kmv);   // the plane below is not kept
                unp(kc[jk], kcv);
                unp(kp[jk], kpv);
                unp(j == 0 ? kh[0] : kr[KVAR && j > 0 ? j - 1 : 0], kymv);
                unp(j == CG_R - 1 ? kh[1] : kr[KVAR && j < CG_R - 1 ? j + 1 : 0], kypv);
            }
            const float sj = cg_q4<KVAR, true>(c, edge, t.gx, y, z, pcv, pmv, ppv, ymv, ypv, xm[j], xp[j], kcv, kmv, kpv, kymv,
                                               kypv, kxm[j], kxp[j], qv);
            dot.add(t.in && y < ny ? sj : 0.0f);
            q[j][0] = f2_make(qv[0], qv[1]);
            q[j][1] = f2_make(qv[2], qv[3]);
        }
    }
#pragma unroll
    for (int j = 0; j < (KVAR ? CG_R : 1); ++j)
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (KVAR) zf[j][i] = gp[j][i];
}

// Where a thread's cells lie: byte offset from the start of the padded arrays
// (the same in all of them; O32: every array is under 4 GiB, so an address is
// one 32-bit add from the array's base).
template <bool O32>
struct CgAddr {
    using OT = typename std::conditional<O32, unsigned, unsigned long long>::type;
    long long org;         // elements before the domain origin
    OT o, dy, dz;          // first cell at the current plane, row and plane strides
    __device__ __forceinline__ CgAddr(const CgCoef& c, const CgPlace& t, int z)
        : org(HALO * c.sz + HALO * c.sy + HALO), o((OT)((org + t.row + (long long)z * c.sz) * 4)), dy((OT)(c.sy * 4)),
          dz((OT)(c.sz * 4)) {}
    template <typename T>
    __device__ __forceinline__ char* base(T* p) const { return reinterpret_cast<char*>(const_cast<float*>(p) - org); }
};
template <typename OT>
__device__ __forceinline__ const float* cg_f(const char* b, OT o) { return reinterpret_cast<const float*>(b + o); }

// Store a row's cells at byte offset o; twins: the array keeps its periodic twins.
template <typename OT>
__device__ __forceinline__ void cg_put(char* b, OT o, const CgCoef& c, const CgPlace& t, int j, const f2 (&v)[2]) {
    if (!t.in || (j > 0 && t.gy + j >= c.n[1])) return;
    float w[4];
    unp(v, w);
    st4_row(reinterpret_cast<float*>(b + o), t.gx, c.n[0], w);
}
__device__ __forceinline__ void cg_put_twins(float* dom, int z, const CgCoef& c, const CgPlace& t, int j, const f2 (&v)[2]) {
    if (!t.in || t.gy + j >= c.n[1]) return;
    float w[4];
    unp(v, w);
    st4_twins(dom, c, t.gx, t.gy + j, z, w);
}

// ----------------------------------------------------------------- cg_dir --
// One iteration's direction: p = r + beta p_old, p.(A p), and the update of x
// that the previous iteration left pending, x += alpha_old p_old (p_old is
// read here anyway). STOREQ: q = A p is stored for cg_res_k (per-cell k); with
// uniform k cg_res_u forms it again from p, which costs less than its 8 bytes.
// Bound by HBM with uniform k and close to it with per-cell k: what decides is
// loads in flight, so every load of a plane is issued before its first use (a
// branch around p_old's loads alone: 618 us instead of 471 on 512^3), a thread
// has CG_R rows whose y neighbours and faces are its own registers, x
// neighbours come by shuffle, and an address is one add (O32; 64-bit address
// arithmetic: +30 us with per-cell k). Warps on an x face run the same body
// with ghost values (cg_rows). Lanes along x: as many of 16 or 8 as fill their
// tiles best (wfa_implicit_step); chunks of 32 planes 2%, of 64 planes 10% slower.
// 512^3, uniform k: 444 us (2.8 GB, 6.3 TB/s) + cg_res_u 254 us (1.68 GB, 6.6
// TB/s), where q stored and x updated with r took 371 + 481 us; 390 x 322 x
// 257, per-cell k: 197 us (1.03 GB, 5.2 TB/s) + cg_res_k 66 us for 183 + 123.
template <bool KVAR, bool STOREQ, bool O32>
__global__ void __launch_bounds__(32 * CG_W, 16 / CG_W) cg_dir(const __grid_constant__ CgArgs a) {
    __shared__ double red[CG_W];
    __shared__ bool last;
    const CgCoef& c = a.c;
    if (a.s->done) return;
    const int iter = a.s->iter;
    const double rr = a.s->rr;
    const bool first = iter == 0;
    const int par = iter & 1;   // iteration i reads p[i mod 2], writes p[(i + 1) mod 2]
    const float* __restrict__ rv = a.r;
    const float* __restrict__ po = first ? a.r : par ? a.p1 : a.p0;
    const float bs = first ? 0.0f : (float)a.s->beta;
    const f2 beta = f2_make(bs, bs);
    const float alpha = (float)a.s->alpha;
    const f2 al = f2_make(alpha, alpha);
    float* __restrict__ pn = par ? a.p0 : a.p1;
    const float* __restrict__ rk = a.rk;
    const int z0 = blockIdx.z * a.zchunk, z1 = min(z0 + a.zchunk, c.n[2]);
    const CgPlace t(a);
    const bool twins = c.periodic[0] || c.periodic[1] || c.periodic[2];
    KahanF dot;
    if (t.rows) {
        using OT = typename CgAddr<O32>::OT;
        const CgAddr<O32> A(c, t, z0);
        const OT dy = A.dy, dz = A.dz;
        OT o = A.o;
        const char *const rB = A.base(rv), *const oB = A.base(po), *const kB = KVAR ? A.base(rk) : nullptr;
        char *const xB = A.base(a.x), *const pB = A.base(pn), *const qB = STOREQ ? A.base(a.q) : nullptr;
        f2 pm[CG_R][2], pc[CG_R][2], pp[CG_R][2], zf[KVAR ? CG_R : 1][2], kc[KVAR ? CG_R : 1][2], kp[KVAR ? CG_R : 1][2];
        // x += alpha_old p_old of a thread's row
        auto xadd = [&](int j, OT oj, const float4& x, const float4& old) {
            const f2 v[2] = {f2_fma(al, lo2(old), lo2(x)), f2_fma(al, hi2(old), hi2(x))};
            cg_put(xB, oj, c, t, j, v);
        };
#pragma unroll
        for (int j = 0; j < CG_R; ++j) {
            const OT oj = o + j * dy;
            const float4 r0 = ldv(cg_f(rB, oj - dz)), o0 = ldv(cg_f(oB, oj - dz)), r1 = ldv(cg_f(rB, oj)), o1 = ldv(cg_f(oB, oj));
            pnew_pairs(r0, o0, beta, pm[j]);
            pnew_pairs(r1, o1, beta, pc[j]);
            if (!first) xadd(j, oj, *reinterpret_cast<const float4*>(xB + oj), o1);
            if constexpr (KVAR) {
                f2 km[2];
                ldp(cg_f(kB, oj - dz), km);
                ldp(cg_f(kB, oj), kc[j]);
#pragma unroll
                for (int i = 0; i < 2; ++i) zf[j][i] = pair_face(km[i], kc[j][i], f2_make(c.tcd[2], c.tcd[2]));
            }
        }
        for (int z = z0; z < z1; ++z, o += dz) {
            float4 rn[CG_R], on[CG_R], xn[CG_R], rh[2], oh[2];
            float e[CG_R], eo[CG_R], ke[CG_R];
            f2 h[2][2], kh[2][2];
            const bool xup = !first && z + 1 < z1;
#pragma unroll
            for (int j = 0; j < CG_R; ++j) {
                const OT oj = o + dz + j * dy;
                rn[j] = ldv(cg_f(rB, oj));
                on[j] = ldv(cg_f(oB, oj));
                xn[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (xup) xn[j] = *reinterpret_cast<const float4*>(xB + oj);
                if constexpr (KVAR) ldp(cg_f(kB, oj), kp[j]);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const OT oj = j == 0 ? o - dy : o + CG_R * dy;
                rh[j] = ldv(cg_f(rB, oj));
                oh[j] = ldv(cg_f(oB, oj));
                if constexpr (KVAR) ldp(cg_f(kB, oj), kh[j]);
            }
#pragma unroll
            for (int j = 0; j < CG_R; ++j) {
                e[j] = eo[j] = ke[j] = 0.0f;
                if (t.ends) {
                    const OT oj = o + j * dy + (OT)(t.eo * 4);
                    e[j] = __ldg(cg_f(rB, oj));
                    eo[j] = __ldg(cg_f(oB, oj));
                    if constexpr (KVAR) ke[j] = __ldg(cg_f(kB, oj));
                }
            }
            if ((threadIdx.x & 7) == 0) {   // one thread per 128-byte line asks L2 for plane z + 3
#pragma unroll
                for (int j = 0; j < CG_R; ++j) {
                    const OT oj = o + 3 * dz + j * dy;
                    prefetch_l2(cg_f(rB, oj));
                    if (!first) {
                        prefetch_l2(cg_f(oB, oj));
                        prefetch_l2(xB + oj);
                    }
                    if constexpr (KVAR) prefetch_l2(cg_f(kB, oj));
                }
            }
#pragma unroll
            for (int j = 0; j < CG_R; ++j) {
                pnew_pairs(rn[j], on[j], beta, pp[j]);
                e[j] = __fmaf_rn(bs, eo[j], e[j]);
                if (xup) xadd(j, o + dz + j * dy, xn[j], on[j]);
            }
            pnew_pairs(rh[0], oh[0], beta, h[0]);
            pnew_pairs(rh[1], oh[1], beta, h[1]);
            f2 q[CG_R][2];
            cg_rows<KVAR>(c, t, z, pc, pm, pp, h, e, kc, zf, kp, kh, ke, KVAR ? cg_f(kB, o - dz) : nullptr, q, dot);
#pragma unroll
            for (int j = 0; j < CG_R; ++j) {
                if (twins) {
                    cg_put_twins(pn, z, c, t, j, pc[j]);
                    if (STOREQ && a.q_twins) cg_put_twins(a.q, z, c, t, j, q[j]);
                } else {
                    cg_put(pB, o + j * dy, c, t, j, pc[j]);
                }
                if (STOREQ && !(twins && a.q_twins)) cg_put(qB, o + j * dy, c, t, j, q[j]);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    pm[j][i] = pc[j][i];
                    pc[j][i] = pp[j][i];
                    if constexpr (KVAR) kc[j][i] = kp[j][i];
                }
            }
        }
    }
    const double bsum = block_sum(dot.value(), red);
    const int blk = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    if (a.dblk) {
        if (threadIdx.x == 0) a.part[blk] = bsum;
        return;
    }
    if (!publish(a, a.part + blk, bsum, &last)) return;
    const double pq = sum_partials(a.part, a.nblk, red);
    if (threadIdx.x == 0) {
        CgState* s = a.s;
        const bool ok = pq > 0.0 && pq < INFINITY;   // else p = 0 (exact solution) or a breakdown
        s->alpha = ok ? rr / pq : 0.0;
        if (!ok) s->done = 1;
        s->pending = !ok && !first ? 2 : 0;
        s->ticket = 0;
    }
}

// ---------------------------------------------------------------- cg_pipe --
// One iteration of Chronopoulos and Gear's CG in one kernel and one
// reduction (the reduction-limited variant Sec. 3.2 points to): with alpha,
// beta of this iteration,
//   s = w + beta s,  p = r + beta p,  x += alpha p,  r' = r - alpha s,
//   w' = A r',  gamma' = r'.r',  delta' = w'.r'
// and the last block forms beta' = gamma' / gamma and
// alpha' = gamma' / (delta' - beta' gamma' / alpha). r' is needed at the
// neighbours of each cell, so it is formed there from r, w and s (three
// arrays with their x / y halo); r, w and s ping-pong between two buffers, p
// is read and written only at its own cell.
template <bool KVAR>
struct PipeOcc {
    static constexpr int blocks = KVAR ? 2 : 3;
};

struct RNew {
    const float* r;
    const float* w;
    const float* s;
    float alpha, beta;
    bool first;   // beta = 0: s = w (s is not read)
};

// r' and s at 4 cells of one row
__device__ __forceinline__ void rnew4(const RNew& R, long long o, float rn[4], float sn[4], float rv[4]) {
    ld4(R.r + o, rv);
    ld4(R.w + o, sn);
    if (!R.first) {
        float so[4];
        ld4(R.s + o, so);
#pragma unroll
        for (int i = 0; i < 4; ++i) sn[i] = __fmaf_rn(R.beta, so[i], sn[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) rn[i] = __fmaf_rn(-R.alpha, sn[i], rv[i]);
}
__device__ __forceinline__ float rnew1(const RNew& R, long long o) {
    float sv = __ldg(R.w + o);
    if (!R.first) sv = __fmaf_rn(R.beta, __ldg(R.s + o), sv);
    return __fmaf_rn(-R.alpha, sv, __ldg(R.r + o));
}

template <bool KVAR>
__global__ void __launch_bounds__(CG_TX * CG_TY, PipeOcc<KVAR>::blocks) cg_pipe(const __grid_constant__ CgArgs a) {
    __shared__ double red[CG_TX * CG_TY / 32];
    __shared__ bool last;
    const CgCoef& c = a.c;
    if (a.s->done) return;
    const int par = a.s->iter & 1;   // iteration i reads r, w [i mod 2], writes [(i + 1) mod 2]
    RNew R;
    R.r = par ? a.r2 : a.r;
    R.w = par ? a.w2 : a.q;
    R.s = par ? a.s2 : a.p1;
    R.alpha = (float)a.s->alpha;
    R.beta = (float)a.s->beta;
    R.first = a.s->iter == 0;
    float* __restrict__ r_out = par ? a.r : a.r2;
    float* __restrict__ w_out = par ? a.q : a.w2;
    float* __restrict__ pv = a.p0;
    float* __restrict__ sv = par ? a.p1 : a.s2;
    float* __restrict__ xv = a.x;
    const float* __restrict__ rk = a.rk;
    const int nx = c.n[0], ny = c.n[1], nz = c.n[2];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int gx = blockIdx.x * 64 + 4 * tx, gy = blockIdx.y * CG_TY + ty;
    const int z0 = blockIdx.z * a.zchunk, z1 = min(z0 + a.zchunk, nz);
    const bool perx = c.periodic[0], pery = c.periodic[1], perz = c.periodic[2];
    KahanF gam, del;
    if (gx < nx && gy < ny) {
        const long long sy = c.sy, sz = c.sz;
        const long long row = cg_at(c, gx, gy, 0);
        const bool inner_xy = gx + 3 < nx && (perx || (gx > 0 && gx + 4 < nx)) && (pery || (gy > 0 && gy < ny - 1));
        const CgEdge edge = cg_edge(c, gx, gy);
        float rm[4], rc[4], sc[4], rvc[4], km[4], kc[4], tmp[4];
        rnew4(R, row + (long long)(z0 - 1) * sz, rm, tmp, rvc);
        rnew4(R, row + (long long)z0 * sz, rc, sc, rvc);
        if (KVAR) {
            ld4(rk + row + (long long)(z0 - 1) * sz, km);
            ld4(rk + row + (long long)z0 * sz, kc);
        }
        for (int z = z0; z < z1; ++z) {
            const long long o = row + (long long)z * sz;
            if ((tx & 7) == 0) {   // one thread per 128-byte line asks L2 for plane z + 3
                prefetch_l2(R.r + o + 3 * sz);
                prefetch_l2(R.w + o + 3 * sz);
                if (!R.first) prefetch_l2(R.s + o + 3 * sz);
            }
            float rp[4], sp_[4], rvp[4], ym[4], yp[4], t4[4], t5[4];
            rnew4(R, o + sz, rp, sp_, rvp);
            rnew4(R, o - sy, ym, t4, t5);
            rnew4(R, o + sy, yp, t4, t5);
            const float xm = rnew1(R, o - 1), xp = rnew1(R, o + 4);
            float kp[4], kym[4], kyp[4], kxm = 0.0f, kxp = 0.0f;
            if (KVAR) {
                ld4(rk + o + sz, kp);
                ld4(rk + o - sy, kym);
                ld4(rk + o + sy, kyp);
                kxm = __ldg(rk + o - 1);
                kxp = __ldg(rk + o + 4);
            }
            float wn[4];
            const bool fast = inner_xy && (perz || (z > 0 && z < nz - 1));
            const bool interior = __all_sync(__activemask(), fast);
            const float dsum = interior
                                   ? cg_q4<KVAR, false>(c, edge, gx, gy, z, rc, rm, rp, ym, yp, xm, xp, kc, km, kp, kym,
                                                        kyp, kxm, kxp, wn)
                                   : cg_q4<KVAR, true>(c, edge, gx, gy, z, rc, rm, rp, ym, yp, xm, xp, kc, km, kp, kym,
                                                       kyp, kxm, kxp, wn);
            float gsum = 0.0f;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                gsum = (interior || gx + i < nx) ? __fmaf_rn(rc[i], rc[i], gsum) : gsum;   // held cells: r' = 0
            gam.add(gsum);
            del.add(dsum);
            // own cells at plane z: p, x, and the new s, r, w
            float pn[4], xn[4];
            ld4(xv + o, xn);
            if (R.first) {
#pragma unroll
                for (int i = 0; i < 4; ++i) pn[i] = rvc[i];
            } else {
                ld4(pv + o, pn);
#pragma unroll
                for (int i = 0; i < 4; ++i) pn[i] = __fmaf_rn(R.beta, pn[i], rvc[i]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) xn[i] = __fmaf_rn(R.alpha, pn[i], xn[i]);
            st4_row(pv + o, gx, nx, pn);
            st4_twins(sv, c, gx, gy, z, sc);
            st4_twins(xv, c, gx, gy, z, xn);
            st4_twins(r_out, c, gx, gy, z, rc);
            st4_twins(w_out, c, gx, gy, z, wn);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                rm[i] = rc[i];
                rc[i] = rp[i];
                sc[i] = sp_[i];
                rvc[i] = rvp[i];
                if (KVAR) {
                    km[i] = kc[i];
                    kc[i] = kp[i];
                }
            }
        }
    }
    const double gs = block_sum(gam.value(), red);
    const double ds = block_sum(del.value(), red);
    const int blk = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    if (threadIdx.x == 0 && threadIdx.y == 0) a.part[CG_MAX_PART + blk] = ds;
    if (!publish(a, a.part + blk, gs, &last)) return;
    const double G = sum_partials(a.part, a.nblk, red);
    const double Dl = sum_partials(a.part + CG_MAX_PART, a.nblk, red);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        CgState* st = a.s;
        const double beta = st->rr > 0.0 ? G / st->rr : 0.0;
        const double den = st->alpha > 0.0 ? Dl - beta * G / st->alpha : 0.0;
        st->iter += 1;
        st->beta = beta;
        st->rr = G;
        if (den > 0.0 && den < INFINITY) {
            st->alpha = G / den;
        } else {
            st->alpha = 0.0;
            st->done = 1;   // r' = 0 (exact solution) or a breakdown
        }
        if (G <= st->tol2 * st->bb || st->iter >= st->max_iter || !(G == G)) st->done = 1;
        st->ticket = 0;
    }
}

// ----------------------------------------------------------------- cg_res --
// The new residual and its r.r (cg_ctl_iter sums the partials); x takes its
// alpha p later (the next cg_dir, or cg_xfin after the last iteration).

// alpha = r.r / p.q as cg_dir's last block left it, or, on a small grid, from
// the blocks' partials in every block of cg_res: a load and a short sum at its
// start for the ticket and the tail at cg_dir's end (3 us of an iteration's 19
// on 64^3). False: p = 0 or a breakdown, which ends the solve.
__device__ __forceinline__ bool cg_alpha(const CgArgs& a, double* red, float (&sh)[2], float* alpha) {
    if (!a.dblk) {
        *alpha = (float)a.s->alpha;
        return true;
    }
    const double rr = a.s->rr;
    const int iter = a.s->iter;
    const double pq = sum_partials(a.part, a.dblk, red);
    if (threadIdx.x == 0) {
        const bool ok = pq > 0.0 && pq < INFINITY;
        const double al = ok ? rr / pq : 0.0;
        sh[0] = (float)al;
        sh[1] = ok ? 1.0f : 0.0f;
        if (blockIdx.x + blockIdx.y + blockIdx.z == 0) {   // the others neither read these nor, without ok, go on
            a.s->alpha = al;
            if (!ok) {
                a.s->pending = iter > 0 ? 2 : 0;
                a.s->done = 1;
            }
        }
    }
    __syncthreads();
    *alpha = sh[0];
    return sh[1] != 0.0f;
}

// r -= alpha q over the domain cells (4 along x per item), q stored by cg_dir.
__global__ void __launch_bounds__(CG_THREADS) cg_res_k(const __grid_constant__ CgArgs a) {
    __shared__ double red[CG_THREADS / 32];
    __shared__ float sh[2];
    const CgCoef& c = a.c;
    if (a.s->done) return;
    float alpha;
    if (!cg_alpha(a, red, sh, &alpha)) return;
    const int nx = c.n[0], ny = c.n[1], nz = c.n[2];
    const int xg = (nx + 3) / 4;
    const long long items = (long long)xg * ny * nz;
    KahanF rr;
    // item it = (x group, y, z); one division at the start, then the stride
    // is added digit by digit (no 64-bit division in the loop)
    const long long it0 = blockIdx.x * (long long)CG_THREADS + threadIdx.x;
    const long long stride = (long long)gridDim.x * CG_THREADS;
    const int dxg = (int)(stride % xg);
    const long long drow = stride / xg;
    const int dy = (int)(drow % ny), dz = (int)(drow / ny);
    int ixg = (int)(it0 % xg), y = (int)((it0 / xg) % ny), z = (int)(it0 / xg / ny);
    for (long long it = it0; it < items; it += stride) {
        const int gx = 4 * ixg;
        const long long o = cg_at(c, gx, y, z);
        float qv[4], rv[4];
        ld4(a.q + o, qv);
        ld4(a.r + o, rv);
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            rv[i] = __fmaf_rn(-alpha, qv[i], rv[i]);
            if (gx + i < nx) s = __fmaf_rn(rv[i], rv[i], s);
        }
        rr.add(s);
        st4_twins(a.r, c, gx, y, z, rv);
        ixg += dxg;
        y += dy;
        z += dz;
        if (ixg >= xg) {
            ixg -= xg;
            ++y;
        }
        if (y >= ny) {
            y -= ny;
            ++z;
        }
    }
    const double bsum = block_sum(rr.value(), red);
    if (threadIdx.x == 0) a.part[CG_MAX_PART + blockIdx.x] = bsum;
}

// r -= alpha A p with A p formed from p again (uniform k), on cg_dir's layout.
template <bool O32>
__global__ void __launch_bounds__(32 * CG_W, 24 / CG_W) cg_res_u(const __grid_constant__ CgArgs a) {
    __shared__ double red[CG_W];
    __shared__ float sh[2];
    const CgCoef& c = a.c;
    if (a.s->done) return;
    float alpha;
    if (!cg_alpha(a, red, sh, &alpha)) return;
    const f2 nal = f2_make(-alpha, -alpha);
    const float* __restrict__ p = (a.s->iter & 1) ? a.p0 : a.p1;
    const int z0 = blockIdx.z * a.zchunk, z1 = min(z0 + a.zchunk, c.n[2]);
    const CgPlace t(a);
    const bool twins = c.periodic[0] || c.periodic[1] || c.periodic[2];
    KahanF rr;
    if (t.rows) {
        using OT = typename CgAddr<O32>::OT;
        const CgAddr<O32> A(c, t, z0);
        const OT dy = A.dy, dz = A.dz;
        OT o = A.o;
        const char* const pB = A.base(p);
        char* const rB = A.base(a.r);
        f2 pm[CG_R][2], pc[CG_R][2], pp[CG_R][2];
        f2 kd[1][2] = {{0, 0}}, zf[1][2] = {{0, 0}};
        const f2 kh[2][2] = {{0, 0}, {0, 0}};
        const float ke[CG_R] = {};
        const bool row1 = t.in && t.gy + 1 < c.n[1];
#pragma unroll
        for (int j = 0; j < CG_R; ++j) {
            ldp(cg_f(pB, o + j * dy - dz), pm[j]);
            ldp(cg_f(pB, o + j * dy), pc[j]);
        }
        for (int z = z0; z < z1; ++z, o += dz) {
            f2 h[2][2], r[CG_R][2], q[CG_R][2];
            float e[CG_R];
#pragma unroll
            for (int j = 0; j < CG_R; ++j) {
                ldp(cg_f(pB, o + dz + j * dy), pp[j]);
                const float4 v = *reinterpret_cast<const float4*>(rB + (o + j * dy));
                r[j][0] = lo2(v);
                r[j][1] = hi2(v);
            }
            ldp(cg_f(pB, o - dy), h[0]);
            ldp(cg_f(pB, o + CG_R * dy), h[1]);
#pragma unroll
            for (int j = 0; j < CG_R; ++j) {
                e[j] = 0.0f;
                if (t.ends) e[j] = __ldg(cg_f(pB, o + j * dy + (OT)(t.eo * 4)));
            }
            if ((threadIdx.x & 7) == 0) {
#pragma unroll
                for (int j = 0; j < CG_R; ++j) {
                    prefetch_l2(cg_f(pB, o + 3 * dz + j * dy));
                    prefetch_l2(rB + (o + 2 * dz + j * dy));
                }
            }
            KahanF pq;   // not used here
            cg_rows<false>(c, t, z, pc, pm, pp, h, e, kd, zf, kd, kh, ke, nullptr, q, pq);
#pragma unroll
            for (int j = 0; j < CG_R; ++j) {
                r[j][0] = f2_fma(nal, q[j][0], r[j][0]);
                r[j][1] = f2_fma(nal, q[j][1], r[j][1]);
                float s = 0.0f;   // 4 products a compensated addition, as in cg_rows
                if (j == 0 ? t.in : row1) {
                    float v[4];
                    unp(r[j], v);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float u = i == 0 || t.gx + i < c.n[0] ? v[i] : 0.0f;
                        s = __fmaf_rn(u, u, s);
                    }
                }
                rr.add(s);
                if (twins) cg_put_twins(a.r, z, c, t, j, r[j]);
                else cg_put(rB, o + j * dy, c, t, j, r[j]);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    pm[j][i] = pc[j][i];
                    pc[j][i] = pp[j][i];
                }
            }
        }
    }
    const double bsum = block_sum(rr.value(), red);
    if (threadIdx.x == 0) a.part[CG_MAX_PART + blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)] = bsum;
}

// ---------------------------------------------------------- device loops --
// The whole call as one graph launch: an outer conditional WHILE node over the
// time steps, an inner one over the CG iterations of a step. One thread of a
// control kernel sets each loop's condition; both loops also stop on their
// own counters (max_iter + 2 iterations, n steps), whatever the solver
// scalars say, so neither can run on without bound.
struct CgLoop {
    long long steps_left;    // time steps still to take
    long long steps_limit;   // n: the outer loop's own bound
    long long steps_done;
    long long total_iters;   // CG iterations of all steps
    double last_rr, last_bb; // the last step's r.r and b.b
    unsigned inner_count;    // iterations run in the current step (the inner loop's own bound)
    unsigned pad;
};
static_assert(sizeof(CgLoop) <= 64, "CgLoop is read back into a 64-byte pinned word");

// The scalar work after cg_init: r.r and b.b from the blocks' partials, the
// solver's state for a new step. L is null in the host-checked runs.
__global__ void __launch_bounds__(CG_CTL) cg_ctl_start(const __grid_constant__ CgArgs a, CgLoop* L,
                                                       cudaGraphConditionalHandle inner, double tol2, int max_iter) {
    __shared__ double red[CG_CTL / 32];
    const double R = sum_partials(a.part, a.nblk, red);
    const double B = sum_partials(a.part + CG_MAX_PART, a.nblk, red);
    if (threadIdx.x == 0) {
        CgState* s = a.s;
        s->rr = R;
        s->bb = B;
        s->alpha = 0.0;
        s->beta = 0.0;
        s->tol2 = tol2;
        s->iter = 0;
        s->max_iter = max_iter;
        s->pending = 0;
        const int done = (R <= tol2 * B || max_iter <= 0 || !(R == R)) ? 1 : 0;
        s->done = done;
        s->ticket = 0;
        if (L) {
            L->inner_count = 0;
            cudaGraphSetConditional(inner, done ? 0u : 1u);
        }
    }
}

// The scalar work after cg_res: r.r from the blocks' partials, beta and the
// convergence test. It is a kernel of its own in the device loop anyway (the
// loop's condition), so cg_res ends without a ticket and a last block's tail.
__global__ void __launch_bounds__(CG_CTL) cg_ctl_iter(const __grid_constant__ CgArgs a, CgLoop* L,
                                                      cudaGraphConditionalHandle inner, int max_iter) {
    __shared__ double red[CG_CTL / 32];
    CgState* s = a.s;
    int done = s->done, iter = s->iter;
    const double rr = s->rr, lim = s->tol2 * s->bb;
    const int mi = s->max_iter;
    const unsigned k = L ? L->inner_count + 1 : 0;
    const double R = sum_partials(a.part + CG_MAX_PART, a.nblk, red);
    if (threadIdx.x != 0) return;
    if (!done) {
        iter += 1;
        done = (R <= lim || iter >= mi || !(R == R)) ? 1 : 0;
        s->iter = iter;
        s->rr = R;
        s->beta = rr > 0.0 ? R / rr : 0.0;
        s->pending = 1;
        s->done = done;
    }
    if (L) {
        L->inner_count = k;
        cudaGraphSetConditional(inner, (!done && k < (unsigned)max_iter + 2u) ? 1u : 0u);
    }
}

// The pipelined method's (cg_pipe has done the scalar work).
__global__ void cg_ctl_pipe(CgState* s, CgLoop* L, cudaGraphConditionalHandle inner, int max_iter) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        const unsigned k = ++L->inner_count;
        cudaGraphSetConditional(inner, (!s->done && k < (unsigned)max_iter + 2u) ? 1u : 0u);
    }
}

__global__ void cg_ctl_step(CgState* s, CgLoop* L, cudaGraphConditionalHandle outer) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        L->total_iters += s->iter;
        L->last_rr = s->rr;
        L->last_bb = s->bb;
        L->steps_left -= 1;
        L->steps_done += 1;
        cudaGraphSetConditional(outer, (L->steps_left > 0 && L->steps_done < L->steps_limit) ? 1u : 0u);
    }
}

// ---------------------------------------------------------------- cg_xfin --
// The end of a classic step: the pending x += alpha p, with x's periodic twins
// (they feed the next step's cg_init; cg_dir's updates leave them stale), and
// the step's bookkeeping (L: device loops).
__global__ void __launch_bounds__(CG_THREADS) cg_xfin(const __grid_constant__ CgArgs a, CgLoop* L, cudaGraphConditionalHandle outer) {
    const CgCoef& c = a.c;
    const int pending = a.s->pending;
    if (pending) {
        const float alpha = (float)a.s->alpha;
        const float* __restrict__ p = (a.s->iter & 1) ? a.p1 : a.p0;   // written by iteration iter - 1
        const int nx = c.n[0], ny = c.n[1], nz = c.n[2];
        const int xg = (nx + 3) / 4;
        const long long items = (long long)xg * ny * nz;
        const long long it0 = blockIdx.x * (long long)CG_THREADS + threadIdx.x;
        const long long stride = (long long)gridDim.x * CG_THREADS;
        const int dxg = (int)(stride % xg);
        const long long drow = stride / xg;
        const int dy = (int)(drow % ny), dz = (int)(drow / ny);
        int ixg = (int)(it0 % xg), y = (int)((it0 / xg) % ny), z = (int)(it0 / xg / ny);
        for (long long it = it0; it < items; it += stride) {
            const int gx = 4 * ixg;
            const long long o = cg_at(c, gx, y, z);
            const float4 x = *reinterpret_cast<const float4*>(a.x + o);
            float xv[4] = {x.x, x.y, x.z, x.w}, pv[4];
            if (pending == 1) {
                ld4(p + o, pv);
#pragma unroll
                for (int i = 0; i < 4; ++i) xv[i] = __fmaf_rn(alpha, pv[i], xv[i]);
            }
            st4_twins(a.x, c, gx, y, z, xv);
            ixg += dxg;
            y += dy;
            z += dz;
            if (ixg >= xg) {
                ixg -= xg;
                ++y;
            }
            if (y >= ny) {
                y -= ny;
                ++z;
            }
        }
    }
    if (L && blockIdx.x == 0 && threadIdx.x == 0) {
        const CgState* s = a.s;
        L->total_iters += s->iter;
        L->last_rr = s->rr;
        L->last_bb = s->bb;
        L->steps_left -= 1;
        L->steps_done += 1;
        cudaGraphSetConditional(outer, (L->steps_left > 0 && L->steps_done < L->steps_limit) ? 1u : 0u);
    }
}

// ------------------------------------------------------------------ host --
struct CgWork {
    float* r = nullptr;
    float* p[2] = {nullptr, nullptr};
    float* q = nullptr;
    double* part = nullptr;
    CgState* s = nullptr;
    CgState* h[2] = {nullptr, nullptr};   // pinned read-back slots
    cudaEvent_t ev[2] = {nullptr, nullptr};
    float* extra[3] = {nullptr, nullptr, nullptr};   // pipelined CG: r2, w2, s2 (allocated on first use)
    CgLoop* loop = nullptr;            // device loop counters
    cudaGraphExec_t loop_exec = nullptr;   // the whole call as one graph (device loops)
    CgArgs loop_key;
    int loop_kvar = -1, loop_method = -1, loop_max_iter = -1;
    double loop_tol2 = -1.0;
    bool loop_broken = false;          // building it failed once: host loop from then on
    cudaGraphExec_t exec[CG_NRUN] = {nullptr, nullptr, nullptr, nullptr};
    cudaStream_t cap = nullptr;   // capture stream (the grid's own may be the legacy default stream)
    CgArgs key;        // arguments the graph was captured with
    int kvar = -1;
    int method = -1;   // WFA_CG_CLASSIC / WFA_CG_PIPELINED of the captured graphs
    int init_grid[3] = {0, 0, 0};   // cg_init, cg_pipe
    int dir_grid[3] = {0, 0, 0};    // cg_dir, cg_res_u
    int dir_threads = 0, dir_chunk = 0, dir_lanes = 0;
    int upd_blocks = 0;
    long long prev_iters = 0;   // iterations the last step needed (sizes the first run of the next)
    bool o32 = false;           // every array under 4 GiB: cg_init takes 32-bit byte offsets
};

void free_cg(wfa_grid_s* g) {
    CgWork* w = static_cast<CgWork*>(g->cg);
    if (!w) return;
    cudaStreamSynchronize(g->stream);
    for (cudaGraphExec_t e : w->exec)
        if (e) cudaGraphExecDestroy(e);
    if (w->cap) cudaStreamDestroy(w->cap);
    for (int b = 0; b < 2; ++b) {
        if (w->ev[b]) cudaEventDestroy(w->ev[b]);
        pinned_release(w->h[b]);
        padded_free(w->p[b], 4, g->stream);
    }
    if (w->loop_exec) cudaGraphExecDestroy(w->loop_exec);
    dev_free(w->loop, g->stream);
    for (float* e : w->extra) padded_free(e, 4, g->stream);
    padded_free(w->r, 4, g->stream);
    padded_free(w->q, 4, g->stream);
    dev_free(w->part, g->stream);
    dev_free(w->s, g->stream);
    delete w;
    g->cg = nullptr;
}

static int cg_workspace(wfa_grid_s* g, CgWork** out) {
    if (g->cg) {
        *out = static_cast<CgWork*>(g->cg);
        return WFA_OK;
    }
    CgWork* w = new (std::nothrow) CgWork();
    if (!w) {
        set_error("host allocation failed");
        return WFA_ERR_OOM;
    }
    g->cg = w;
    const size_t fb = field_elems(g) * sizeof(float);
    // WFA_CG_ADDR=64 takes the kernels of larger arrays here too (a second
    // compilation of the same arithmetic, for comparison)
    const char* addr = getenv("WFA_CG_ADDR");
    w->o32 = fb < ((size_t)1 << 32) && !(addr && strcmp(addr, "64") == 0);
    // padded arrays in the field's layout (see lead_bytes)
    cudaError_t e = padded_alloc((void**)&w->r, fb, 4, g->stream);
    for (int b = 0; b < 2 && e == cudaSuccess; ++b) e = padded_alloc((void**)&w->p[b], fb, 4, g->stream);
    if (e == cudaSuccess) e = padded_alloc((void**)&w->q, fb, 4, g->stream);
    if (e == cudaSuccess) e = dev_alloc((void**)&w->part, 2 * CG_MAX_PART * sizeof(double), g->stream);
    if (e == cudaSuccess) e = dev_alloc((void**)&w->s, sizeof(CgState), g->stream);
    // the halos and held cells of the work vectors stay 0 (finite) for good
    for (float* v : {w->r, w->p[0], w->p[1], w->q})
        if (e == cudaSuccess) e = cudaMemsetAsync(v, 0, fb, g->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(w->s, 0, sizeof(CgState), g->stream);
    for (int b = 0; b < 2 && e == cudaSuccess; ++b) {
        w->h[b] = static_cast<CgState*>(pinned_word());
        if (!w->h[b]) e = cudaErrorMemoryAllocation;
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&w->ev[b], cudaEventDisableTiming);
    }
    if (e != cudaSuccess) {
        const int rc = cuda_fail(e, "implicit solver workspace");
        free_cg(g);
        return rc;
    }
    *out = w;
    return WFA_OK;
}

static void cg_coef(const wfa_grid_s* g, double dt, CgCoef* c) {
    memset(c, 0, sizeof *c);
    for (int a = 0; a < 3; ++a) {
        c->n[a] = g->n[a];
        c->periodic[a] = g->bc_kind[2 * a] == WFA_BC_PERIODIC;
        const double ih2 = 1.0 / (g->h[a] * g->h[a]);
        c->cu[a] = (float)(dt * g->k_uniform * ih2);
        c->tcd[a] = (float)(2.0 * dt * ih2);
    }
    c->du = 1.0f + 2.0f * (c->cu[0] + c->cu[1] + c->cu[2]);
    for (int f = 0; f < 6; ++f) {
        c->dface[f] = g->bc_kind[f] == WFA_BC_DIRICHLET;
        c->held[f] = g->bc_kind[f] == WFA_BC_DIRICHLET_CELL;
        c->tb[f] = (float)g->bc_value[f];
    }
    c->sy = g->px;
    c->sz = g->px * g->py;
}

// A kernel of the solver with its grid and arguments, launched on a stream or
// added to a graph.
struct CgKernel {
    const void* fn;
    dim3 grid, block;
    CgArgs a;
    cudaError_t run(cudaStream_t st, void** args = nullptr) const {
        void* own[] = {const_cast<CgArgs*>(&a)};
        return cudaLaunchKernel(fn, grid, block, args ? args : own, 0, st);
    }
};
struct CgLaunch {
    CgKernel init, start, dir, res, iter, pipe;
    CgLaunch(const CgWork* w, const CgArgs& base, bool kvar, int method) {
        const bool storeq = kvar || method == WFA_CG_PIPELINED;
        if (w->o32)
            dir.fn = kvar ? (const void*)cg_dir<true, true, true>
                          : storeq ? (const void*)cg_dir<false, true, true> : (const void*)cg_dir<false, false, true>;
        else
            dir.fn = kvar ? (const void*)cg_dir<true, true, false>
                          : storeq ? (const void*)cg_dir<false, true, false> : (const void*)cg_dir<false, false, false>;
        dir.grid = dim3(w->dir_grid[0], w->dir_grid[1], w->dir_grid[2]);
        dir.block = dim3(w->dir_threads);
        dir.a = base;
        dir.a.lanes = w->dir_lanes;
        dir.a.zchunk = w->dir_chunk;
        dir.a.nblk = w->dir_grid[0] * w->dir_grid[1] * w->dir_grid[2];
        if (method != WFA_CG_PIPELINED && dir.a.nblk <= CG_FOLD) dir.a.dblk = dir.a.nblk;
        res = dir;
        res.fn = w->o32 ? (const void*)cg_res_u<true> : (const void*)cg_res_u<false>;
        if (kvar) {
            res.fn = (const void*)cg_res_k;
            res.grid = dim3(w->upd_blocks);
            res.block = dim3(CG_THREADS);
            res.a.nblk = w->upd_blocks;
        }
        iter.fn = (const void*)cg_ctl_iter;
        iter.grid = dim3(1);
        iter.block = dim3(CG_CTL);
        iter.a = res.a;
        pipe.fn = kvar ? (const void*)cg_pipe<true> : (const void*)cg_pipe<false>;
        pipe.grid = dim3(w->init_grid[0], w->init_grid[1], w->init_grid[2]);
        pipe.block = dim3(CG_TX, CG_TY);
        pipe.a = base;
        pipe.a.nblk = w->init_grid[0] * w->init_grid[1] * w->init_grid[2];
        init = pipe;
        init.fn = kvar ? (w->o32 ? (const void*)cg_init<true, true> : (const void*)cg_init<true, false>)
                       : (w->o32 ? (const void*)cg_init<false, true> : (const void*)cg_init<false, false>);
        start = iter;
        start.fn = (const void*)cg_ctl_start;
        start.a = init.a;
    }
};

static int cg_capture(wfa_grid_s* g, CgWork* w, const CgArgs& base, bool kvar, int method) {
    if (w->exec[0] && w->kvar == (int)kvar && w->method == method && memcmp(&w->key, &base, sizeof base) == 0)
        return WFA_OK;
    for (cudaGraphExec_t& e : w->exec)
        if (e) {
            cudaGraphExecDestroy(e);
            e = nullptr;
        }
    const CgLaunch kl(w, base, kvar, method);
    if (!w->cap) WFA_CUDA(cudaStreamCreateWithFlags(&w->cap, cudaStreamNonBlocking));
    const cudaStream_t st = w->cap;
    for (int k = 0; k < CG_NRUN; ++k) {
        WFA_CUDA(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
        cudaError_t e = cudaSuccess;
        for (int it = 0; it < CG_RUN_LEN[k] && e == cudaSuccess; ++it) {
            if (method == WFA_CG_PIPELINED) {   // one kernel, one reduction an iteration
                e = kl.pipe.run(st);
                continue;
            }
            e = kl.dir.run(st);
            if (e == cudaSuccess) e = kl.res.run(st);
            if (e == cudaSuccess) {
                CgLoop* none = nullptr;
                cudaGraphConditionalHandle h0 = 0;
                int mi = 0;
                void* args[] = {const_cast<CgArgs*>(&kl.iter.a), &none, &h0, &mi};
                e = kl.iter.run(st, args);
            }
        }
        cudaGraph_t gr = nullptr;
        const cudaError_t e2 = cudaStreamEndCapture(st, &gr);
        if (e == cudaSuccess) e = e2;
        if (e == cudaSuccess) e = cudaGraphInstantiate(&w->exec[k], gr, 0);
        if (gr) cudaGraphDestroy(gr);
        if (e != cudaSuccess) {
            w->exec[k] = nullptr;
            return cuda_fail(e, "implicit solver graph");
        }
    }
    w->key = base;
    w->kvar = kvar;
    w->method = method;
    return WFA_OK;
}

// Kernel node of `fn` with the given arguments, depending on `dep` (if any).
static cudaError_t add_kernel(cudaGraph_t gr, cudaGraphNode_t* node, cudaGraphNode_t dep, const void* fn, dim3 grid,
                              dim3 block, void** args) {
    cudaKernelNodeParams kp = {};
    kp.func = const_cast<void*>(fn);
    kp.gridDim = grid;
    kp.blockDim = block;
    kp.sharedMemBytes = 0;
    kp.kernelParams = args;
    return cudaGraphAddKernelNode(node, gr, dep ? &dep : nullptr, dep ? 1 : 0, &kp);
}

// Conditional WHILE node depending on `dep`; its body graph is returned.
static cudaError_t add_while(cudaGraph_t gr, cudaGraphNode_t* node, cudaGraphNode_t dep, cudaGraphConditionalHandle h,
                             cudaGraph_t* body) {
    cudaGraphNodeParams np = {};
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = h;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    cudaError_t e = cudaGraphAddNode(node, gr, dep ? &dep : nullptr, nullptr, dep ? 1 : 0, &np);
    if (e == cudaSuccess) *body = np.conditional.phGraph_out[0];
    return e;
}

// outer WHILE (steps) { cg_init; cg_ctl_start; [pipelined: cg_dir];
//   inner WHILE (iterations) { classic: cg_dir, cg_res, cg_ctl_iter | pipelined: cg_pipe, cg_ctl_pipe };
//   classic: cg_xfin | pipelined: cg_ctl_step }
static cudaError_t build_loop_graph(CgWork* w, const CgArgs& base, bool kvar, int method, double tol2,
                                    int max_iter, cudaGraphExec_t* out) {
    cudaGraph_t top = nullptr;
    cudaError_t e = cudaGraphCreate(&top, 0);
    if (e != cudaSuccess) return e;
    cudaGraphConditionalHandle ho = 0, hi = 0;
    cudaGraph_t outer = nullptr, inner = nullptr;
    cudaGraphNode_t n_outer = nullptr, n = nullptr, prev = nullptr;
    const CgLaunch kl(w, base, kvar, method);
    CgArgs up = base;
    up.nblk = w->upd_blocks;
    CgState* st = w->s;
    CgLoop* L = w->loop;
    auto arg = [](const CgKernel& k) { return const_cast<CgArgs*>(&k.a); };
    void* a_init[] = {arg(kl.init)};
    void* a_dir[] = {arg(kl.dir)};
    void* a_res[] = {arg(kl.res)};
    void* a_pipe[] = {arg(kl.pipe)};
    void* a_start[] = {arg(kl.start), &L, &hi, &tol2, &max_iter};
    void* a_iter[] = {arg(kl.iter), &L, &hi, &max_iter};
    void* a_pctl[] = {&st, &L, &hi, &max_iter};
    void* a_step[] = {&st, &L, &ho};
    void* a_fin[] = {&up, &L, &ho};
    e = cudaGraphConditionalHandleCreate(&ho, top, 1, cudaGraphCondAssignDefault);
    if (e == cudaSuccess) e = add_while(top, &n_outer, nullptr, ho, &outer);
    if (e == cudaSuccess) e = add_kernel(outer, &n, nullptr, kl.init.fn, kl.init.grid, kl.init.block, a_init);
    prev = n;
    if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&hi, outer, 0, 0);
    if (e == cudaSuccess) e = add_kernel(outer, &n, prev, kl.start.fn, kl.start.grid, kl.start.block, a_start);
    prev = n;
    if (e == cudaSuccess && method == WFA_CG_PIPELINED) {
        e = add_kernel(outer, &n, prev, kl.dir.fn, kl.dir.grid, kl.dir.block, a_dir);
        prev = n;
    }
    cudaGraphNode_t n_inner = nullptr;
    if (e == cudaSuccess) e = add_while(outer, &n_inner, prev, hi, &inner);
    if (e == cudaSuccess) {
        cudaGraphNode_t ip = nullptr;
        if (method == WFA_CG_PIPELINED) {
            e = add_kernel(inner, &ip, nullptr, kl.pipe.fn, kl.pipe.grid, kl.pipe.block, a_pipe);
        } else {
            e = add_kernel(inner, &ip, nullptr, kl.dir.fn, kl.dir.grid, kl.dir.block, a_dir);
            if (e == cudaSuccess) e = add_kernel(inner, &ip, ip, kl.res.fn, kl.res.grid, kl.res.block, a_res);
        }
        if (e == cudaSuccess)
            e = method == WFA_CG_PIPELINED
                    ? add_kernel(inner, &ip, ip, (const void*)cg_ctl_pipe, dim3(1), dim3(32), a_pctl)
                    : add_kernel(inner, &ip, ip, kl.iter.fn, kl.iter.grid, kl.iter.block, a_iter);
    }
    if (e == cudaSuccess)
        e = method == WFA_CG_PIPELINED
                ? add_kernel(outer, &n, n_inner, (const void*)cg_ctl_step, dim3(1), dim3(32), a_step)
                : add_kernel(outer, &n, n_inner, (const void*)cg_xfin, dim3(w->upd_blocks), dim3(CG_THREADS), a_fin);
    if (e == cudaSuccess) e = cudaGraphInstantiate(out, top, 0);
    cudaGraphDestroy(top);
    return e;
}

}  // namespace wfa

using namespace wfa;

int wfa_implicit_step(wfa_grid g, double dt, long long n, double rtol, int max_iter, long long* iters,
                      double* rel_res) {
    NvtxRange nvtx_("wfa_implicit_step");
    if (!g) {
        set_error("NULL grid");
        return WFA_ERR_ARG;
    }
    if (!(dt >= 0.0) || !std::isfinite(dt) || n < 0 || !(rtol >= 0.0) || !std::isfinite(rtol) || max_iter < 0) {
        set_error("wfa_implicit_step: need dt >= 0 (finite), n >= 0, rtol >= 0 (finite), max_iter >= 0");
        return WFA_ERR_ARG;
    }
    if (g->storage != WFA_F32) {
        set_error("wfa_implicit_step: the implicit solver needs fp32 storage");
        return WFA_ERR_ARG;
    }
    if (!g->field_set || !g->coeffs_set) {
        set_error("set the field and the coefficients before an implicit step");
        return WFA_ERR_STATE;
    }
    if (g->u[0] != 0.0 || g->u[1] != 0.0 || g->u[2] != 0.0) {
        set_error("wfa_implicit_step: advection makes the system non-symmetric; CG needs u = 0");
        return WFA_ERR_ARG;
    }
    for (int a = 0; a < 3; ++a)
        if ((g->bc_kind[2 * a] == WFA_BC_PERIODIC) != (g->bc_kind[2 * a + 1] == WFA_BC_PERIODIC)) {
            set_error("axis %d: a periodic face needs a periodic opposite face", a);
            return WFA_ERR_BC;
        }
    if (has_exchange_face(g)) {   // a slab's CG would need the other slabs' inner products
        set_error("wfa_implicit_step: exchange faces are for the explicit step only");
        return WFA_ERR_BC;
    }
    if (iters) *iters = 0;
    if (rel_res) *rel_res = 0.0;
    if (n == 0) return WFA_OK;
    if (g->halo_dirty || !(g->thin[g->cur] & HAS_LAYER)) {   // held layers carry their value before the first solve
        int rc = refresh_halo(g, g->cur);
        if (rc) return rc;
        g->halo_dirty = false;
    }
    int rc = prepare_coeff_halo(g);
    if (rc) return rc;
    CgWork* w = nullptr;
    rc = cg_workspace(g, &w);
    if (rc) return rc;

    const bool kvar = g->k != nullptr;
    const long long off = domain_offset(g);
    CgArgs base;
    memset(&base, 0, sizeof base);
    cg_coef(g, dt, &base.c);
    base.x = static_cast<float*>(g->T[g->cur]) + off;
    base.rk = kvar ? g->r + off : nullptr;
    base.r = w->r + off;
    base.p0 = w->p[0] + off;
    base.p1 = w->p[1] + off;
    base.q = w->q + off;
    base.part = w->part;
    base.s = w->s;
    int nsm = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (nsm <= 0) nsm = 1;
    {   // cg_init / cg_pipe grid: 64 x 16 columns, z chunks of about 16 planes,
        // many waves of blocks so the last wave's tail is short; chunks down to
        // 2 planes only where 16 would leave SMs idle (small grids)
        const int gxb = (g->n[0] + 63) / 64, gyb = (g->n[1] + CG_TY - 1) / CG_TY;
        const long long cols = (long long)gxb * gyb;
        const long long resident = (long long)nsm * (kvar ? CgOcc<true>::blocks : CgOcc<false>::blocks);
        long long nch = std::max<long long>(1, resident * 16 / cols);
        long long cap = std::max(1, g->n[2] / 16);
        if (cols * cap < resident) cap = std::max(1, g->n[2] / 2);
        nch = std::min(nch, cap);
        nch = std::min<long long>(nch, std::max<long long>(1, CG_MAX_PART / cols));
        base.zchunk = (int)((g->n[2] + nch - 1) / nch);
        nch = (g->n[2] + base.zchunk - 1) / base.zchunk;
        if (cols * nch > CG_MAX_PART) {
            set_error("wfa_implicit_step: grid too large for the partial-sum buffer");
            return WFA_ERR_ARG;
        }
        w->init_grid[0] = gxb;
        w->init_grid[1] = gyb;
        w->init_grid[2] = (int)nch;
        // cg_dir / cg_res_u: CG_R rows a thread; chunks of about 16 planes, shorter
        // where that leaves SMs idle. Tiles of 64 x 16 cells (16 lanes along x, CG_W
        // warps); 32 x 32 (8 lanes) or 64 x 8 (2 warps) where those hold enough
        // more cells of the grid; 32 lanes and no more warps than rows ask for where
        // the rows are few. us an iteration, 64 x 16 / as chosen, uniform k:
        // 130x258x200 92 / 80, 200x200x200 96 / 86, 70x260x300 91 / 78, 321x200x100
        // 73.6 / 69.2, 1000x2x1000 124 / 43, 500x8x700 50 / 37; nothing between
        // them where all are full: 512x512x128 227.5, 228.1, 231.3
        auto fill = [&](int l, int w) {
            const int tx = 4 * l, ty = CG_R * w * 32 / l;
            return (double)g->n[0] * g->n[1] /
                   ((double)((g->n[0] + tx - 1) / tx * tx) * ((g->n[1] + ty - 1) / ty * ty));
        };
        int lanes = g->n[0] > 32 ? 16 : 8, warps = CG_W;
        if (g->n[1] <= CG_R * CG_W && g->n[0] > 64) {
            lanes = 32;
        } else if (lanes == 16) {
            if (fill(8, CG_W) > 1.05 * fill(16, CG_W)) lanes = 8;
            else if (fill(16, 2) > 1.035 * fill(16, CG_W) &&   // twice the tiles: only where their partials have room
                     (long long)((g->n[0] + 63) / 64) * ((g->n[1] + 7) / 8) <= CG_MAX_PART)
                warps = 2;
        }
        if (lanes == 32) warps = std::min(warps, (g->n[1] + CG_R - 1) / CG_R);
        const long long bx = (g->n[0] + 4 * lanes - 1) / (4 * lanes);
        const int rows = CG_R * warps * 32 / lanes, by = (g->n[1] + rows - 1) / rows;
        const long long dcols = bx * by;
        const long long dres = (long long)nsm * 16 / warps;   // resident blocks
        long long dch = std::max(1, g->n[2] / 16);
        if (dcols * dch < dres) dch = std::min<long long>(g->n[2], std::max<long long>(dch, dres / dcols));
        dch = std::min<long long>(dch, std::max<long long>(1, CG_MAX_PART / dcols));
        w->dir_chunk = (int)((g->n[2] + dch - 1) / dch);
        dch = (g->n[2] + w->dir_chunk - 1) / w->dir_chunk;
        w->dir_grid[0] = (int)bx;
        w->dir_grid[1] = by;
        w->dir_grid[2] = (int)dch;
        w->dir_lanes = lanes;
        w->dir_threads = 32 * warps;
        if (dcols * dch > CG_MAX_PART) {
            set_error("wfa_implicit_step: grid too large for the partial-sum buffer");
            return WFA_ERR_ARG;
        }
        const long long items = (long long)((g->n[0] + 3) / 4) * g->n[1] * g->n[2];
        w->upd_blocks = (int)std::max<long long>(1, std::min<long long>((items + CG_THREADS - 1) / CG_THREADS, nsm * 4LL));
    }
    const int method = g->cg_method;
    if (method == WFA_CG_PIPELINED) {   // three more work vectors: r, w and s ping-pong
        const size_t fb = field_elems(g) * sizeof(float);
        for (float*& e : w->extra)
            if (!e) {
                WFA_CUDA(padded_alloc((void**)&e, fb, 4, g->stream));
                WFA_CUDA(cudaMemsetAsync(e, 0, fb, g->stream));
            }
        base.r2 = w->extra[0] + off;
        base.w2 = w->extra[1] + off;
        base.s2 = w->extra[2] + off;
        base.q_twins = 1;
    }
    rc = cg_capture(g, w, base, kvar, method);
    if (rc) return rc;

    const int per_iter = method == WFA_CG_PIPELINED ? 1 : 3;   // kernels an iteration (host-checked runs)

    // The device-loop graph: every step and iteration without a host round
    // trip (WFA_CG_LOOP=host keeps the host-checked runs below).
    const char* loop_pick = getenv("WFA_CG_LOOP");
    if (!(loop_pick && strcmp(loop_pick, "host") == 0) && !w->loop_broken) {
        const double tol2 = rtol * rtol;
        if (!w->loop) {
            WFA_CUDA(dev_alloc((void**)&w->loop, sizeof(CgLoop), g->stream));
        }
        if (!w->loop_exec || w->loop_kvar != (int)kvar || w->loop_method != method || w->loop_max_iter != max_iter ||
            w->loop_tol2 != tol2 || memcmp(&w->loop_key, &base, sizeof base) != 0) {
            if (w->loop_exec) cudaGraphExecDestroy(w->loop_exec);
            w->loop_exec = nullptr;
            const cudaError_t e = build_loop_graph(w, base, kvar, method, tol2, max_iter, &w->loop_exec);
            if (e != cudaSuccess) {   // no conditional nodes here: host-checked runs from now on
                cudaGetLastError();
                w->loop_exec = nullptr;
                w->loop_broken = true;
            } else {
                w->loop_key = base;
                w->loop_kvar = kvar;
                w->loop_method = method;
                w->loop_max_iter = max_iter;
                w->loop_tol2 = tol2;
            }
        }
        if (w->loop_exec) {
            CgLoop L0;
            memset(&L0, 0, sizeof L0);
            L0.steps_left = n;
            L0.steps_limit = n;
            CgLoop* h = reinterpret_cast<CgLoop*>(w->h[0]);
            memcpy(h, &L0, sizeof L0);
            WFA_CUDA(cudaMemcpyAsync(w->loop, h, sizeof(CgLoop), cudaMemcpyHostToDevice, g->stream));
            WFA_CUDA(cudaGraphLaunch(w->loop_exec, g->stream));
            WFA_CUDA(cudaMemcpyAsync(h, w->loop, sizeof(CgLoop), cudaMemcpyDeviceToHost, g->stream));
            WFA_CUDA(cudaStreamSynchronize(g->stream));
            CgLoop Lr;
            memcpy(&Lr, h, sizeof Lr);
            if (Lr.steps_done != n) {
                set_error("wfa_implicit_step: the device loop ran %lld of %lld steps", Lr.steps_done, n);
                return WFA_ERR_STATE;
            }
            const int extra_per_step = method == WFA_CG_PIPELINED ? 4 : 3;   // init, start, [the first cg_dir], end of the step
            g->launches += extra_per_step * n + (method == WFA_CG_PIPELINED ? 2LL : 3LL) * Lr.total_iters;
            w->prev_iters = n > 0 ? Lr.total_iters / n : 0;
            g->halo_dirty = true;
            g->steps_done += n;
            if (iters) *iters = Lr.total_iters;
            if (rel_res) *rel_res = Lr.last_bb > 0.0 ? sqrt(Lr.last_rr / Lr.last_bb) : sqrt(Lr.last_rr);
            return WFA_OK;
        }
    }

    const CgLaunch kl(w, base, kvar, method);
    long long total = 0;
    double last_rel = 0.0;
    for (long long step = 0; step < n; ++step) {
        {
            CgLoop* none = nullptr;
            cudaGraphConditionalHandle h0 = 0;
            double tol2 = rtol * rtol;
            void* args[] = {const_cast<CgArgs*>(&kl.start.a), &none, &h0, &tol2, &max_iter};
            WFA_CUDA(kl.init.run(g->stream));
            WFA_CUDA(kl.start.run(g->stream, args));
            g->launches += 2;
        }
        if (method == WFA_CG_PIPELINED) {
            // w = A r, delta = w.r and alpha = r.r / delta: the first half of a
            // classic iteration (q = A p with p = r), q keeping its twins
            WFA_CUDA(kl.dir.run(g->stream));
            g->launches += 1;
        }
        // Runs of captured iterations with one run queued ahead of the flag
        // check, so the GPU does not wait for the host: the first run as long
        // as the last step needed (rounded up to 1, 2, 4 or 8), then 2, then 8s.
        // Iterations after convergence are kernels that return at once.
        long long queued = 0, launched = 0;
        auto enqueue = [&]() -> int {
            int k = CG_NRUN - 1;
            if (launched == 0) {
                const long long want = w->prev_iters > 0 ? w->prev_iters : CG_RUN_LEN[CG_NRUN - 1];
                k = 0;
                while (k < CG_NRUN - 1 && CG_RUN_LEN[k] < want) ++k;
            } else if (launched == 1) {
                k = 1;
            }
            WFA_CUDA(cudaGraphLaunch(w->exec[k], g->stream));
            WFA_CUDA(cudaMemcpyAsync(w->h[launched & 1], w->s, sizeof(CgState), cudaMemcpyDeviceToHost, g->stream));
            WFA_CUDA(cudaEventRecord(w->ev[launched & 1], g->stream));
            g->launches += per_iter * CG_RUN_LEN[k];
            queued += CG_RUN_LEN[k];
            ++launched;
            return WFA_OK;
        };
        rc = enqueue();
        if (rc) return rc;
        CgState st;
        memset(&st, 0, sizeof st);
        for (long long k = 0;; ++k) {
            if (launched == k + 1 && queued < max_iter) {
                rc = enqueue();
                if (rc) return rc;
            }
            WFA_CUDA(cudaEventSynchronize(w->ev[k & 1]));
            memcpy(&st, w->h[k & 1], sizeof st);
            if (st.done) break;
            if (launched == k + 1) {   // nothing left in flight, yet not done
                set_error("wfa_implicit_step: the solver did not report completion");
                return WFA_ERR_STATE;
            }
        }
        WFA_CUDA(cudaStreamSynchronize(g->stream));   // the run queued ahead has ended (no-op kernels)
        if (method != WFA_CG_PIPELINED) {
            CgArgs fa = base;
            fa.nblk = w->upd_blocks;
            cg_xfin<<<w->upd_blocks, CG_THREADS, 0, g->stream>>>(fa, nullptr, cudaGraphConditionalHandle());
            WFA_CUDA(cudaGetLastError());
            g->launches += 1;
        }
        total += st.iter;
        w->prev_iters = st.iter;
        last_rel = st.bb > 0.0 ? sqrt(st.rr / st.bb) : sqrt(st.rr);
    }
    g->halo_dirty = true;   // periodic copies and ghost layers of the field are stale
    g->steps_done += n;
    if (iters) *iters = total;
    if (rel_res) *rel_res = last_rel;
    return WFA_OK;
}

int wfa_set_cg_method(wfa_grid g, int method) {
    if (!g || (method != WFA_CG_CLASSIC && method != WFA_CG_PIPELINED)) {
        set_error("wfa_set_cg_method: NULL grid or unknown method %d", method);
        return WFA_ERR_ARG;
    }
    g->cg_method = method;
    return WFA_OK;
}
