// lbm_kernels.cuh -- CUDA kernels of the GB300 colour-gradient LBM library.
//
//   k_step_fused   one full time step (pull-stream + boundaries, moments, S2I4
//                  colour gradient, omega_eff, collision, perturbation,
//                  recolouring, store) in a single pass.  Each thread block owns
//                  a strip of W columns and marches up a range of rows; source
//                  rows (all planes, with a margin in x) arrive in shared-memory
//                  slots by TMA loads, so every stored population is read from
//                  HBM once per step.
//   k_step_tile    the same step, bit-identical, of a small lattice: a block owns a
//                  tile and pulls it and the nodes around it from global memory.
//   k_tp_moments / k_tp_collide
//                  the same step as two plain node-parallel kernels with a
//                  global scratch field (psi, q u) in between: the reference
//                  GPU path (equal to the fused one but for rounding).
//   k_init, k_fields, k_diag, k_slug_profile, k_advance, k_set_times   support kernels.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

constexpr long long WAIT_LIMIT_CYCLES = 4000000000LL;   // ~2 s at 2 GHz

// Resident fused-kernel blocks per SM the register allocation is sized for
// (0: the per-variant choice of FusedCfg::MINB).
#ifndef LBM_FUSED_MIN_BLOCKS
#define LBM_FUSED_MIN_BLOCKS 0
#endif
// 1: each fused step is launched as a programmatic dependent of the previous one.
#ifndef LBM_FUSED_PDL
#define LBM_FUSED_PDL 1
#endif
// ------------------------------------------------------------------ loaders

// Stored values from global memory around one row: pulls of nodes of row y read rows y - 1,
// y and y + 1 (wrapped periodically when the loader is made).  Three row pointers and 32-bit
// plane offsets: one address instruction per load.
template <typename T>
struct RowLoader {
    const float *rho_m, *rho_c, *rho_p;   // plane 0, interior column 0, of rows y - 1, y, y + 1
    const T *dev_m, *dev_c, *dev_p;
    int rho_plane, dev_plane, y;
    int slip;   // free-slip walls
    SplitC q;
    __device__ __forceinline__ RowLoader(const SimDesc &d, int b, int row) {
        const int ny = d.ph.ny;
        auto wrap = [&](int ys) { return ys < 0 ? ys + ny : (ys >= ny ? ys - ny : ys); };
        const float *r = d.rho + b * d.rho_buf + d.ghost;
        const T *v = reinterpret_cast<const T *>(d.dev) + b * d.dev_buf + d.ghost;
        rho_m = r + wrap(row - 1) * d.rho_row, rho_c = r + wrap(row) * d.rho_row, rho_p = r + wrap(row + 1) * d.rho_row;
        dev_m = v + wrap(row - 1) * d.dev_row, dev_c = v + wrap(row) * d.dev_row, dev_p = v + wrap(row + 1) * d.dev_row;
        rho_plane = (int)d.rho_plane;
        dev_plane = (int)d.dev_plane;
        y = row;
        slip = d.wet.slip;
        q = split_consts(d.ph);
    }
    __device__ __forceinline__ float rho(int k, int xs, int ys) const {
        const int dy = ys - y;
        return (dy < 0 ? rho_m : (dy == 0 ? rho_c : rho_p))[k * rho_plane + xs];
    }
    static constexpr bool SPLIT = SplitStore<T>::value;
    // stored value r^k_i of node (xs, ys): the deviation itself, or the split-form residual
    __device__ __forceinline__ float res(int k, int i, int xs, int ys) const {
        const int dy = ys - y;
        return Codec<T>::dec((dy < 0 ? dev_m : (dy == 0 ? dev_c : dev_p))[(k * 8 + i - 1) * dev_plane + xs]);
    }
    // split-form shift h_i of node (xs, ys) (0 without the split form)
    __device__ __forceinline__ float shift(int i, int xs, int ys) const {
        if (!SPLIT) return 0.0f;
        return split_shift(q, i, rho(0, xs, ys), rho(1, xs, ys), rho(2, xs, ys), rho(3, xs, ys), rho(4, xs, ys));
    }
    __device__ __forceinline__ float own_shift_sum(int xs, int ys) const {
        return SPLIT ? 4.0f * rho(2, xs, ys) * (q.dph1 + q.dph2) : 0.0f;
    }
    // stored deviation d^k_i of node (xs, ys), decoded from the split form for 16-bit storage
    __device__ __forceinline__ float dev(int k, int i, int xs, int ys) const {
        const float r = res(k, i, xs, ys);
        if (!SPLIT) return r;
        const float sh = shift(i, xs, ys);
        return k == 0 ? __fadd_rn(r, sh) : __fsub_rn(r, sh);
    }
};

// psi on a solid wall row: W-weighted mean of the in-domain fluid nodes next
// to it on the adjacent fluid row (Sec. 2.4 extrapolation).  `psi_of(X)`
// returns psi of the fluid node in column X of that row.
template <class PsiOf>
__device__ __forceinline__ float wall_psi(const Phys &p, int X, const PsiOf &psi_of) {
    float num = 0.0f, den = 0.0f;
#pragma unroll
    for (int dx = -1; dx <= 1; dx++) {
        const int Xp = X + dx;
        if (p.bc_x == BC_PERIODIC || (Xp >= 0 && Xp < p.nx)) {
            const float wgt = dx == 0 ? (1.0f / 9.0f) : (1.0f / 36.0f);
            num += wgt * psi_of(Xp);
            den += wgt;
        }
    }
    return den > 0.0f ? num / den : 0.0f;
}

// S2I4 gradient (Eq. (eq:colorGradient)) summed in opposite pairs so that a
// uniform field gives exactly zero.  v(dx, dy) returns the field at x + (dx, dy).
template <class V>
__device__ __forceinline__ void s2i4(const V &v, float &gx, float &gy) {
    const float e = v(1, 0), wv = v(-1, 0), n = v(0, 1), s = v(0, -1);
    const float ne = v(1, 1), nw = v(-1, 1), sw = v(-1, -1), se = v(1, -1);
    const float a = ne - sw, b = se - nw;
    gx = (1.0f / 3.0f) * (e - wv) + (1.0f / 12.0f) * (a + b);
    gy = (1.0f / 3.0f) * (n - s) + (1.0f / 12.0f) * (a - b);
}

// ------------------------------------------------------------ fused kernel

// Rows of open-column values computed at a time, and the values kept of such a node (two
// densities, eight non-rest parts).
constexpr int OPEN_ROWS = 32;
constexpr int OPEN_VALUES = 10;

// Side columns of a row of an odd lattice, in shared memory between the pass that collides it
// and the next one, which stores them: columns 0 .. 7 and, from the second place on,
// nx - 8 .. nx - 1 (nx - 9 is even: pairs of columns start at even places), per plane.
template <typename T>
struct SideCols {
    static constexpr int NS = ScalarPlanes<T>::value, PITCH = 10;
    static constexpr int DEV_AT = NS * PITCH * 4;                             // bytes, of a side
    static constexpr int BYTES = (DEV_AT + 16 * PITCH * (int)sizeof(T) + 15) / 16 * 16;
    static constexpr int FLOATS = 2 * BYTES / 4;                              // of a row
};

template <typename T, int CV, int W, int NSLOT, bool ODD>
struct FusedCfg {
    static constexpr int GMEM = 8;                           // ghost columns kept in memory
    static constexpr int G = 16 / (int)sizeof(T);            // halo columns loaded each side
    static constexpr int BOXW = W + 2 * G;                   // TMA box width (elements)
    static constexpr int NS = ScalarPlanes<T>::value;          // FP32 node planes per row
    static constexpr int RHO_BYTES = ((NS * BOXW * 4 + 127) / 128) * 128;
    static constexpr int DEV_BYTES = 16 * BOXW * (int)sizeof(T);
    static constexpr int SLOT_BYTES = ((RHO_BYTES + DEV_BYTES + 127) / 128) * 128;
    static constexpr int RING = W + 4;                       // columns x0-2 .. x0+W+1
    static constexpr bool QRING = (CV & CV_MRT) && (CV & CV_HERMITE);
    static constexpr bool WET = (CV & CV_WET) != 0;
    // shared floats: rings of what neighbouring threads read, psi and q u of the newest
    // row and the one before (a slower thread may still read that one); psi of the lower
    // wall; the edge lanes' values of the last four rows (two columns a side next to
    // walls); the paired constants; open columns of two chunks of rows
    static constexpr int QX_OFF = 3 * RING;
    static constexpr int QY_OFF = QX_OFF + (QRING ? 2 * RING : 0);
    static constexpr int HIST_OFF = ((QY_OFF + (QRING ? 2 * RING : 0)) + 3) / 4 * 4;
    static constexpr int CONST_OFF = HIST_OFF + 2 * 4 * 32 * 4;
    static constexpr int OPEN_OFF = CONST_OFF + (int)sizeof(Consts<f2>) / 4;
    static constexpr int SIDE_OFF = ((CV & CV_OPEN) ? OPEN_OFF + 4 * OPEN_ROWS * OPEN_VALUES + 3 : OPEN_OFF + 3) / 4 * 4;
    static constexpr int RING_FLOATS = SIDE_OFF + (ODD ? 2 * SideCols<T>::FLOATS : 0);
    static constexpr int DESC_BYTES = ((int)sizeof(SimDesc) + 127) / 128 * 128;
    static constexpr int RING_BYTES = ((RING_FLOATS * 4 + 15) / 16) * 16;
    static constexpr int SMEM = DESC_BYTES + NSLOT * SLOT_BYTES + RING_BYTES + NSLOT * 8 + 16;
    static constexpr uint32_t TX_BYTES = (uint32_t)(NS * BOXW * 4 + DEV_BYTES);
    // Blocks per SM the registers are sized for: 6 blocks of 2 warps are 3 warps on each
    // scheduler, 168 registers a thread (so are 5 blocks).  That holds both columns' state of
    // periodic BGK and MRT lattices; other variants spill some (FP16 open BGK 84 bytes stored and
    // 48 loaded, MRT with the Hermite source 28 to 220 stored) and are still faster than
    // without spills at 4 blocks and up to 255 registers.  us a step of 2048 x 512 with 6 and with
    // 4: FP32 BGK 27.6 and 30.7, FP16 27.9 and 31.6, open 39.8 and 41.7, MRT + Hermite 45.2 and 47.8,
    // wet 47.1 and 50.9; only 16-bit open MRT + Hermite is a little slower (59.8 and 59.5).  How
    // many of them a plan uses: plan_blocks, plan_for.
    static constexpr int MINB = LBM_FUSED_MIN_BLOCKS > 0 ? LBM_FUSED_MIN_BLOCKS : 6;
    static_assert(BOXW <= 256, "TMA box dimension limit");
    static_assert((BOXW * sizeof(T)) % 16 == 0 && (BOXW * 4) % 16 == 0, "TMA inner box bytes");
    static_assert(G <= GMEM && G >= 3, "halo must cover the stencil and fit the memory ghost");
    static_assert(NSLOT >= 2, "one row is read while the next ones arrive");
    static_assert(W / 2 >= 2 * OPEN_ROWS, "one thread per side and row of a chunk");
};

// Two neighbouring columns' values of one shared-memory row: `at` points at the first.
template <typename T>
__device__ __forceinline__ f2 pair_at(const T *at);
template <>
__device__ __forceinline__ f2 pair_at<float>(const float *at) {
    const float2 v = *reinterpret_cast<const float2 *>(at);
    return f2{v.x, v.y};
}
template <>
__device__ __forceinline__ f2 pair_at<__half>(const __half *at) {
    const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(at));
    return f2{v.x, v.y};
}
template <>
__device__ __forceinline__ f2 pair_at<__nv_bfloat16>(const __nv_bfloat16 *at) {
    const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(at));
    return f2{v.x, v.y};
}
__device__ __forceinline__ void pair_to(float *at, f2 v) { *reinterpret_cast<float2 *>(at) = make_float2(v.x, v.y); }
__device__ __forceinline__ void pair_to(__half *at, f2 v) {
    *reinterpret_cast<__half2 *>(at) = __floats2half2_rn(v.x, v.y);
}
__device__ __forceinline__ void pair_to(__nv_bfloat16 *at, f2 v) {
    *reinterpret_cast<__nv_bfloat162 *>(at) = __floats2bfloat162_rn(v.x, v.y);
}

// What one stored row r adds, in the two columns of one thread, to the nodes of rows
// r + 1 (links 2, 5, 6), r (links 1, 3, less the node's own deviations) and r - 1
// (links 4, 7, 8).  u^k_i = phi^k_i (rho_k(source) - rho_k(x, r)) + d^k_i(source) is
// taken relative to the column's own density in row r, so that every term is a
// small difference; moving the reference to the node's own row later costs one
// density difference per row.  T_i = u^r_i + u^b_i.  h_*: sums of the split-form shifts
// of the same links (16-bit storage).
struct RowTerms {
    f2 own[2];                    // densities of (x, r)
    f2 up[2], mid[2], dn[2];      // per colour: sums of u over the links into rows r + 1, r, r - 1
    f2 T1, T2, T3, T4, T5, T6, T7, T8;
    f2 h_up, h_mid, h_dn;
};

// `rp`, `dp`: the thread's first column in planes 0 of the row's densities and deviations,
// `rs`, `ds`: the distances of their planes.  In shared memory each stored value of a row is
// read in this one pass only.
template <typename T>
__device__ __forceinline__ RowTerms row_terms(const float *rp, int rs, const T *dp, int ds, const Consts<f2> &K) {
    RowTerms R;
    f2 west[2], east[2];
    auto half = [&](int k, f2 &T1, f2 &T2, f2 &T3, f2 &T4, f2 &T5, f2 &T6, f2 &T7, f2 &T8) {
        const f2 own = pair_at(rp + k * rs);
        west[k] = f2{rp[k * rs - 1], own.x};
        east[k] = f2{own.y, rp[k * rs + 2]};
        R.own[k] = own;
        const f2 phi1 = k == 0 ? K.phr : K.phb;
        const f2 dW = west[k] - own, dE = east[k] - own;
        // phi_2 times a density step, added to a deviation.  16-bit storage holds phi_2 as a
        // constant (2048 x 128 FP16 14.3 us a step, 14.9 with the quarter of phi_1's product
        // that FP32 storage takes, where the constant costs 12.78 against 12.67).
        f2 pW, pE;
        if (!SplitStore<T>::value) pW = phi1 * dW, pE = phi1 * dE;
        auto diag = [&](f2 step, f2 product, f2 dev) {
            if (SplitStore<T>::value) return fmav(k == 0 ? K.phr2 : K.phb2, step, dev);
            return fmav(lit<f2, LIT_QUARTER>(), product, dev);
        };
        const T *d = dp + (8 * k - 1) * ds;   // direction i at d + i * ds
        auto at = [&](int i, int dx) { return Codec<T>::dec(d[i * ds + dx]); };
        const f2 o1 = pair_at(d + 1 * ds), o3 = pair_at(d + 3 * ds);
        T1 = fmav(phi1, dW, f2{at(1, -1), o1.x});
        T3 = fmav(phi1, dE, f2{o3.y, at(3, 2)});
        f2 out = o1 + o3;
        R.mid[k] = T1 + T3;
        const f2 o5 = pair_at(d + 5 * ds), o6 = pair_at(d + 6 * ds);
        T5 = diag(dW, pW, f2{at(5, -1), o5.x});
        T6 = diag(dE, pE, f2{o6.y, at(6, 2)});
        out = out + (o5 + o6);
        T2 = pair_at(d + 2 * ds);
        T4 = pair_at(d + 4 * ds);
        out = out + (T2 + T4);
        R.up[k] = T2 + (T5 + T6);
        const f2 o7 = pair_at(d + 7 * ds), o8 = pair_at(d + 8 * ds);
        T8 = diag(dW, pW, f2{at(8, -1), o8.x});
        T7 = diag(dE, pE, f2{o7.y, at(7, 2)});
        out = out + (o7 + o8);
        R.dn[k] = T4 + (T7 + T8);
        R.mid[k] = R.mid[k] - out;
    };
    f2 b1, b2, b3, b4, b5, b6, b7, b8;
    half(0, R.T1, R.T2, R.T3, R.T4, R.T5, R.T6, R.T7, R.T8);
    half(1, b1, b2, b3, b4, b5, b6, b7, b8);
    R.T1 = R.T1 + b1, R.T2 = R.T2 + b2, R.T3 = R.T3 + b3, R.T4 = R.T4 + b4;
    R.T5 = R.T5 + b5, R.T6 = R.T6 + b6, R.T7 = R.T7 + b7, R.T8 = R.T8 + b8;
    R.h_up = R.h_mid = R.h_dn = lit<f2, LIT_ZERO>();
    if (SplitStore<T>::value) {
        // the shift of direction i is m dphi_c + (c_i . G) / |c_i| rest_c, rest_c = rho_r phi^r_c
        // + rho_b phi^b_c; phi_2 = phi_1 / 4 for both colours.  The node's own eight shifts sum
        // to 4 m (dphi_1 + dphi_2) = 5 m dphi_1.
        const f2 pr = K.phr, pb = K.phb, dph = K.dphi, quarter = lit<f2, LIT_QUARTER>();
        const f2 rW = fmav(pr, west[0], pb * west[1]), rE = fmav(pr, east[0], pb * east[1]);
        const f2 rC = fmav(pr, R.own[0], pb * R.own[1]);
        const float *mp = rp + 2 * rs, *xp = rp + 3 * rs, *yp = rp + 4 * rs;
        const f2 mC = pair_at(mp), xC = pair_at(xp), yC = pair_at(yp);
        const f2 b = yC * rC, mWE = f2{mp[-1], mC.x} + f2{mC.y, mp[2]};
        const f2 xWE = fmav(f2{xp[-1], xC.x}, rW, f2{-xC.y, -xp[2]} * rE);
        const f2 yWE = fmav(f2{yp[-1], yC.x}, rW, f2{yC.y, yp[2]} * rE);
        const f2 D = lit<f2, LIT_DIAG>();
        const f2 even = fmav(D, xWE, dph * fmav(quarter, mWE, mC)), odd = fmav(D, yWE, b);
        R.h_up = even + odd;
        R.h_dn = even - odd;
        R.h_mid = fmav(dph, fmav(lit<f2, LIT_M5>(), mC, mWE), xWE);
    }
    return R;
}

// Terms of a no-slip wall for the row next to it, from that row's own deviations: the
// opposite directions i, j, k of the links out of the wall (an axis, two diagonals); sgn: the
// wall's side in y.
struct WallTerms {
    f2 sum[2], Ti, Tj, Tk, h;
};
template <typename T>
__device__ __forceinline__ WallTerms wall_row_terms(const float *rp, int rs, const T *dp, int ds, const Consts<f2> &K, float dphi,
                                                    int i, int j, int k, float sgn) {
    auto at = [&](int plane) { return pair_at(dp + plane * ds); };
    const f2 ri = at(i - 1), rj = at(j - 1), rk = at(k - 1), bi = at(i + 7), bj = at(j + 7), bk = at(k + 7);
    WallTerms L;
    L.sum[0] = ri + (rj + rk);
    L.sum[1] = bi + (bj + bk);
    L.Ti = ri + bi;
    L.Tj = rj + bj;
    L.Tk = rk + bk;
    L.h = lit<f2, LIT_ZERO>();
    if (SplitStore<T>::value) {
        const f2 rest = fmav(K.phr, pair_at(rp), K.phb * pair_at(rp + rs));
        L.h = fmav(bc<f2>(1.5f * dphi), pair_at(rp + 2 * rs),
                   bc<f2>(sgn * (1.0f + 0.5f * 0.70710678118654752f)) * (pair_at(rp + 4 * rs) * rest));
    }
    return L;
}

// The nodes (x, r) of a thread between the passes over their own row and over row r + 1:
// sums over the links from rows r - 1 and r, and the T_i of those links (relative to the
// nodes' own densities).
struct HalfPulled {
    f2 own[2], acc[2];
    f2 T1, T2, T3, T5, T6, h;
};

// Close the nodes (x, r): add the links from row r + 1 (dn, T4, T7, T8, h_dn) and form the
// new densities and the colour-blind non-rest parts.  S: phi_1 times the density step from
// (x, r) to (x, r + 1) (zero at a wall): it moves the reference of the links from row r + 1,
// once on the axis and a quarter on each diagonal, 1.5 in the sum.
//
// Every product that is added to something is an explicit fused operation, here and in
// row_terms: the compiler fuses a packed product into an addition where it has no other use,
// which made the same sums round differently in different kernels.
struct Step {
    f2 r, b, sum;   // per colour, and of both
};
__device__ __forceinline__ Step step_of(const Consts<f2> &K, const f2 (&from)[2], const f2 (&to)[2]) {
    Step S;
    const f2 dr = to[0] - from[0];
    S.r = K.phr * dr;
    S.b = K.phb * (to[1] - from[1]);
    S.sum = fmav(K.phr, dr, S.b);
    return S;
}
__device__ __forceinline__ Step no_step() {
    const f2 zero = lit<f2, LIT_ZERO>();
    return Step{zero, zero, zero};
}
template <bool SPLIT>
__device__ __forceinline__ void close_node(const Consts<f2> &K, const HalfPulled &H, f2 dn0, f2 dn1, f2 T4, f2 T7, f2 T8,
                                           f2 h_dn, const Step &S, PulledOf<f2> &P) {
    const f2 c15 = lit<f2, LIT_3HALVES>(), quarter = lit<f2, LIT_QUARTER>(), mquarter = lit<f2, LIT_MQUARTER>();
    f2 ar = fmav(c15, S.r, H.acc[0] + dn0);
    f2 ab = fmav(c15, S.b, H.acc[1] + dn1);
    if (SPLIT) {
        const f2 h = H.h + h_dn;
        ar = ar + h;
        ab = ab - h;
    }
    P.rr = H.own[0] + ar;
    P.rb = H.own[1] + ab;
    // rest part of the density change on the axis links
    const f2 R1 = fmav(K.phr, P.rr - H.own[0], K.phb * (P.rb - H.own[1]));
    const f2 up = S.sum - R1;
    P.e1 = H.T1 - R1;
    P.e2 = H.T2 - R1;
    P.e3 = H.T3 - R1;
    P.e4 = T4 + up;
    P.e5 = fmav(mquarter, R1, H.T5);
    P.e6 = fmav(mquarter, R1, H.T6);
    P.e7 = fmav(quarter, up, T7);
    P.e8 = fmav(quarter, up, T8);
}

// Post-collision state of the nodes (x, y) and, with `both`, (x + 1, y) of a lattice of
// descriptor d, and its copies in the ghost columns of a periodic lattice.  out_rho,
// out_dev: where planes 0 of node (x, y) are.  STAGED: of an odd lattice the copies and a lone
// last column go to `side` instead (SideCols).
template <typename T, bool SPLIT, bool STAGED = false>
__device__ __forceinline__ void store_pair(const SimDesc &d, bool per_x, int x, bool both, char *out_rho, char *out_dev, f2 rr, f2 rb,
                                           const Collided<f2> &o, unsigned char *side = nullptr) {
    constexpr int GMEM = 8;   // ghost columns (checked against the descriptor by the kernels)
    const uint32_t ps_rho = (uint32_t)d.rho_plane * 4u, ps_dev = (uint32_t)d.dev_plane * (uint32_t)sizeof(T);
    const long long nx = d.ph.nx;
    auto store = [&](char *qr, char *qd) {
        auto put = [&](char *q, f2 v) { pair_to(reinterpret_cast<float *>(q), v); };
        put(qr, rr);
        put(qr + ps_rho, rb);
        if (SPLIT) {
            put(qr + 2ull * ps_rho, o.m);
            put(qr + 3ull * ps_rho, o.gx);
            put(qr + 4ull * ps_rho, o.gy);
        }
#pragma unroll
        for (int i = 0; i < 8; i++) {
            pair_to(reinterpret_cast<T *>(qd + (unsigned long long)ps_dev * i), o.r[i]);
            pair_to(reinterpret_cast<T *>(qd + (unsigned long long)ps_dev * (i + 8)), o.b[i]);
        }
    };
    if (both) store(out_rho, out_dev);
    if (per_x && (nx & 1) == 0) {
        // the pair's copies in the ghost columns of the other side (both on lattices
        // narrower than two ghosts)
        if (x < GMEM) store(out_rho + nx * 4, out_dev + nx * (long long)sizeof(T));
        if (x >= nx - GMEM) store(out_rho - nx * 4, out_dev - nx * (long long)sizeof(T));
    } else if constexpr (STAGED) {
        using Side = SideCols<T>;
        if (x >= GMEM && x + 1 < nx - GMEM) return;
#pragma unroll 1
        for (int right = x < GMEM ? 0 : 1; right < 2; right++) {
            if (right && x + 1 < nx - GMEM) break;
            const int at = right ? x - ((int)nx - GMEM - 1) : x;
            float *q = reinterpret_cast<float *>(side + right * Side::BYTES) + at;
            T *v = reinterpret_cast<T *>(side + right * Side::BYTES + Side::DEV_AT) + at;
            pair_to(q, rr);
            pair_to(q + Side::PITCH, rb);
            if (SPLIT) {
                pair_to(q + 2 * Side::PITCH, o.m);
                pair_to(q + 3 * Side::PITCH, o.gx);
                pair_to(q + 4 * Side::PITCH, o.gy);
            }
#pragma unroll
            for (int i = 0; i < 8; i++) {
                pair_to(v + i * Side::PITCH, o.r[i]);
                pair_to(v + (i + 8) * Side::PITCH, o.b[i]);
            }
        }
    } else if (!both || (per_x && (x < GMEM || x + 1 >= nx - GMEM))) {
        // odd widths: single columns, in place (g = 0) or as ghost copies
        auto single = [&](int h, auto pick) {
            for (int g = both ? 1 : 0; g < 3; g++) {
                if (g == 1 && !(per_x && x + h < GMEM)) continue;
                if (g == 2 && !(per_x && x + h >= nx - GMEM)) continue;
                const long long to = h + (g == 0 ? 0 : (g == 1 ? nx : -nx));
                char *qr = out_rho + to * 4, *qd = out_dev + to * (long long)sizeof(T);
                *reinterpret_cast<float *>(qr) = pick(rr);
                *reinterpret_cast<float *>(qr + ps_rho) = pick(rb);
                if (SPLIT) {
                    *reinterpret_cast<float *>(qr + 2ull * ps_rho) = pick(o.m);
                    *reinterpret_cast<float *>(qr + 3ull * ps_rho) = pick(o.gx);
                    *reinterpret_cast<float *>(qr + 4ull * ps_rho) = pick(o.gy);
                }
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    *reinterpret_cast<T *>(qd + (unsigned long long)ps_dev * i) = Codec<T>::enc(pick(o.r[i]));
                    *reinterpret_cast<T *>(qd + (unsigned long long)ps_dev * (i + 8)) = Codec<T>::enc(pick(o.b[i]));
                }
            }
        };
        single(0, [](f2 v) { return v.x; });
        if (both) single(1, [](f2 v) { return v.y; });
    }
}

// Nodes beside a strip, link by link: the split form's shift of one link (gc: c_i . G) and the
// colour field.  Every product that is added to something is an explicit fused operation, so
// that such a node has the same bits wherever it is formed.
__device__ __forceinline__ float edge_shift(const Phys &p, bool axis, float rr, float rb, float m, float gc) {
    const float rest = __fmaf_rn(p.phi_r[1], rr, __fmul_rn(p.phi_b[1], rb)) * (axis ? 1.0f : 0.25f);
    return __fmaf_rn(axis ? p.dphi[1] : p.dphi[2], m, __fmul_rn(__fmul_rn(axis ? 1.0f : 0.70710678118654752f, gc), rest));
}
__device__ __forceinline__ float edge_colour(const Phys &p, float rr, float rb) {
    return __fmaf_rn(rr, p.inv_gamma, -rb) / __fmaf_rn(rr, p.inv_gamma, rb);
}

// One link of a node beside a strip, direction i of colour k, on one lane, from global memory:
// lanes 8 k + (i - 1) of a half warp form the node's psi (and q u) by shuffles, with the
// operations of the strip kernel's edge lanes.  `rp`, `dp`: the node's column in planes 0 of a
// row, `rs`, `ds`: the distances of the planes.
struct EdgeLink {
    const Phys &p;
    int i, k, cx, cy;
    bool axis;
    float phi;
    __device__ __forceinline__ EdgeLink(const Phys &p_, int i_, int k_) : p(p_), i(i_), k(k_) {
        cx = (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
        cy = (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
        axis = i <= 4;
        phi = (k == 0 ? p.phi_r[1] : p.phi_b[1]) * (axis ? 1.0f : 0.25f);
    }
    // density and decoded deviation of direction (dx, dy), plane j, at the given column
    template <typename T>
    __device__ __forceinline__ void value(const float *rp, int rs, const T *dp, int ds, int j, int dx, int dy, float &s,
                                          float &dv) const {
        s = rp[k * rs];
        dv = Codec<T>::dec(dp[(k * 8 + j - 1) * ds]);
        if (SplitStore<T>::value) {
            const float gc = (float)dx * rp[3 * rs] + (float)dy * rp[4 * rs];
            const float h = edge_shift(p, axis, rp[0], rp[rs], rp[2 * rs], gc);
            dv = __fadd_rn(dv, k == 0 ? h : -h);
        }
    }
    // the link's source: in the row of y - cy (rp, dp at the node's column there) or, `wall`, in
    // the node's own row: the node itself in the opposite direction, or (free slip) the row's
    // neighbour in the mirrored one
    template <typename T>
    __device__ __forceinline__ void source(const float *rp, int rs, const T *dp, int ds, bool wall, bool slip, float &s,
                                           float &dv) const {
        const int opp = i <= 4 ? ((i + 1) & 3) + 1 : ((i - 3) & 3) + 5;
        const int mir = i == 2 ? 4 : i == 4 ? 2 : i == 5 ? 8 : i == 8 ? 5 : i == 6 ? 7 : i == 7 ? 6 : i;
        const bool back = wall && !slip;
        const int at = back ? 0 : -cx;
        value<T>(rp + at, rs, dp + at, ds, !wall ? i : (slip ? mir : opp), back ? -cx : cx, wall ? -cy : cy, s, dv);
    }
    // the node's own density and deviation (its own shifts sum to 5 m dphi_1: an eighth per lane)
    template <typename T>
    __device__ __forceinline__ void own(const float *rp, int rs, const T *dp, int ds, float &s, float &dv) const {
        s = rp[k * rs];
        dv = Codec<T>::dec(dp[(k * 8 + i - 1) * ds]);
        if (SplitStore<T>::value) dv = __fmaf_rn((k == 0 ? 0.625f : -0.625f) * p.dphi[1], rp[2 * rs], dv);
    }
    // psi and q u from the lanes' links (source density and deviation, own ones)
    template <bool NEED_J>
    __device__ __forceinline__ void node(unsigned lanes, float s, float dv, float own_s, float own_dv, float &psi, float &qx,
                                         float &qy) const {
        const float u = __fmaf_rn(phi, __fsub_rn(s, own_s), dv);
        float v = __fsub_rn(u, own_dv);
        v = __fadd_rn(v, __shfl_xor_sync(lanes, v, 1));
        v = __fadd_rn(v, __shfl_xor_sync(lanes, v, 2));
        v = __fadd_rn(v, __shfl_xor_sync(lanes, v, 4));
        const float mine = __fadd_rn(own_s, v);                       // colour k's new density
        const float other = __shfl_xor_sync(lanes, mine, 8);
        const float rr = k == 0 ? mine : other, rb = k == 0 ? other : mine;
        psi = edge_colour(p, rr, rb);
        qx = qy = 0.0f;
        if (NEED_J) {   // momentum: the shifts and rest parts cancel
            float jx = (float)cx * u, jy = (float)cy * u;
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) {
                jx = __fadd_rn(jx, __shfl_xor_sync(lanes, jx, o));
                jy = __fadd_rn(jy, __shfl_xor_sync(lanes, jy, o));
            }
            const float q = __fmaf_rn(p.q_r, rr, __fmul_rn(p.q_b, rb)), rho = __fadd_rn(rr, rb);
            qx = __fmul_rn(q, __fadd_rn(jx / rho, 0.5f * p.gx));
            qy = __fmul_rn(q, __fadd_rn(jy / rho, 0.5f * p.gy));
        }
    }
};

// Persistent fused step.  Block b processes the work items
// items[item_off[b] .. item_off[b+1]) in order (strip segments, possibly of
// different simulations), so that every block gets an equal share of rows.
//
// Per segment the block marches up a strip of w <= W columns, one thread per two
// neighbouring columns: the arithmetic of both is issued as f32x2 instructions, stored
// values move as pairs, and loop, address and barrier work is shared.
// Source rows arrive by TMA into a ring of NSLOT shared slots.  The pass over row r
//   - reads row r once (the node's own densities and deviations and those entering from
//     the two sides) and splits it into what it adds to the nodes of rows r + 1, r and
//     r - 1 (RowTerms), kept in registers;
//   - closes the nodes of row r - 1 and shares their colour field through a ring;
//   - collides the nodes of row r - 2, whose gradient now has its three rows, and
//     stores them.
// A row's slot is free after its one pass, so NSLOT - 1 rows are in flight.
//
// Bound by the latency of its own instructions: a warp issues once in about six cycles
// (fixed-latency and shared-memory dependencies), so the time goes with instructions per
// node and with warps in flight, and FP32 also with DRAM (5.5 TB/s of halo, state and ghost
// traffic).  Instructions issued per node of the 40-lattice sweep, one column a thread with
// scalar arithmetic and separate pulls of three rows (before): FP32 681, BF16 973; now FP32
// 389, BF16 476.  Microseconds a step before and now: sweep BF16 107.6 and 63.1, FP32 78.9
// and 76.5; eight open channels of mixed storage 293 and 173.
//
// ODD: stages the side columns of odd widths.  The ghost copies of an odd lattice start at odd
// columns, so that no pair is aligned; stored by the thread that has the values, 36 single ones
// more a row, they make the blocks at the sides the last ones.  Here they go through shared
// memory, and in the next pass all threads store a few values each, eight columns of a plane by
// eight threads.  us a step without and with it: FP32 2001 x 2001 130 and 119, 40 of 255 x 256 92
// and 80, FP16 2271 x 911 67.9 and 61.1.  A variant of its own (stage_sides says where), because
// the test in every lattice's kernel cost even widths 1 to 2 % (1280 x 640 23.0 and 23.3).
template <typename T, int CV, int W, int NSLOT, bool ODD>
__global__ void __launch_bounds__(W / 2, (FusedCfg<T, CV, W, NSLOT, ODD>::MINB)) k_step_fused(
    const SimDesc *__restrict__ descs, const WorkItem *__restrict__ items, const int *__restrict__ item_off,
    int n_blocks, int step_offset, int flags, int *__restrict__ err) {
    using Cfg = FusedCfg<T, CV, W, NSLOT, ODD>;
    constexpr int G = Cfg::G, BOXW = Cfg::BOXW, RING = Cfg::RING, NT = W / 2;
    constexpr bool HERMITE = (CV & CV_HERMITE) != 0;
    constexpr bool HERMITE_SRC = Cfg::QRING;
    constexpr bool WET = Cfg::WET;
    constexpr bool OPEN = (CV & CV_OPEN) != 0;
    constexpr bool SPLIT = SplitStore<T>::value;
    static_assert(!(ODD && OPEN), "open lattices have no ghost copies");
    extern __shared__ __align__(128) unsigned char smem[];

    const int tid = threadIdx.x;

    SimDesc &d = *reinterpret_cast<SimDesc *>(smem);
    unsigned char *slots = smem + Cfg::DESC_BYTES;
    float *rings = reinterpret_cast<float *>(slots + NSLOT * Cfg::SLOT_BYTES);
    Consts<f2> &K = *reinterpret_cast<Consts<f2> *>(rings + Cfg::CONST_OFF);
    float *opens = rings + Cfg::OPEN_OFF;
    unsigned char *sides = reinterpret_cast<unsigned char *>(rings + Cfg::SIDE_OFF);
    uint64_t *bars = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(rings) + Cfg::RING_BYTES);

    if (smem_u32(slots) & 127) {   // TMA destinations must be 128-byte aligned
        if (tid == 0) atomicOr(err, ERR_ALIGN);
        return;
    }

    // descriptor of an item into shared memory, its row barriers and constants
    auto prepare = [&](const SimDesc *gd, bool again) {
        const int4 *src = reinterpret_cast<const int4 *>(gd);
        int4 *dst = reinterpret_cast<int4 *>(smem);
        for (int j = tid; j < (int)(sizeof(SimDesc) / 16); j += NT) dst[j] = __ldcv(src + j);
        if (tid == 0) {
            for (int s = 0; s < NSLOT; s++) {
                if (again) mbar_inval(&bars[s]);
                mbar_init(&bars[s], 1);
            }
            fence_mbar_init();
            fence_proxy_async_smem();
            tensormap_acquire(&gd->tmap_rho);
            tensormap_acquire(&gd->tmap_dev);
        }
        __syncthreads();
        if (tid == NT - 1) fill_consts(K, d.ph);
    };
    // Launched as a programmatic dependent of the previous step: the work table and the
    // first item's descriptor are read while that step still runs.  Nothing it writes is
    // touched (state, error word) before every prerequisite grid has completed and its
    // writes are visible.  The descriptors' times are written between chunks of steps: the
    // first step of a chunk reads them again after the wait; a later one is launched by
    // blocks that have all waited for that write themselves.
    // With FUSED_EARLY_NEXT (plan_flags: plans of even pieces or with half the chip idle, one
    // launch per step) the next step may launch at once, its blocks waiting in free slots;
    // otherwise only once this block's work is done (below): on uneven batches
    // and concurrent launch groups the early trigger placed waiting blocks on SMs
    // in the order slots freed and cost 5-16 %.
    const bool any = (int)blockIdx.x < n_blocks;
    const int it_first = any ? item_off[blockIdx.x] : 0, it_end = any ? item_off[blockIdx.x + 1] : 0;
    if (it_first < it_end) prepare(descs + items[it_first].sim, false);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (flags & FUSED_EARLY_NEXT) asm volatile("griddepcontrol.launch_dependents;");

    for (int itx = it_first; itx < it_end; ++itx) {
        const WorkItem it = items[itx];
        const SimDesc *gd = descs + it.sim;
        if (itx > it_first) {
            __syncthreads();   // previous segment fully consumed (all its rows were waited for)
            prepare(gd, true);
        }
        long long t0 = d.t0, t_end = d.t_end;
        if (step_offset == 0 && itx == it_first) {
            t0 = __ldcv(&gd->t0);
            t_end = __ldcv(&gd->t_end);
        }

        const Phys &p = d.ph;   // per-simulation constants, in shared memory
        const long long t = t0 + step_offset;
        if (t >= t_end) continue;   // this simulation has stopped
        const int bsrc = (int)(t & 1), bdst = bsrc ^ 1;
        const int x0 = it.x0, w = it.w, ya = it.ya, yb = it.yb;
        if (d.variant != CV || d.ghost != Cfg::GMEM || w <= 0 || w > W || x0 < 0 || x0 + w > p.nx || (x0 % 8) != 0 ||
            ya < 0 || yb > p.ny || ya >= yb) {
            if (tid == 0) atomicOr(err, ERR_BADITEM);
            continue;
        }
        const bool wall_y = p.bc_y == BC_WALL;
        // source rows r0 .. r_load - 1 are loaded (none lies behind a wall)
        const int r0 = wall_y ? max(ya - 2, 0) : ya - 2;
        const int r_load = wall_y ? min(yb + 2, p.ny) : yb + 2;

        // Load source row r (densities and all 16 deviation planes, columns
        // x0-G .. x0+W+G-1) into slot s.
        auto issue = [&](int r, int s) {
            const int yr = r < 0 ? r + p.ny : (r >= p.ny ? r - p.ny : r);
            unsigned char *dst = slots + s * Cfg::SLOT_BYTES;
            const int xb = x0 + (Cfg::GMEM - G);   // element index of column x0 - G in the padded row
            mbar_arrive_expect_tx(&bars[s], Cfg::TX_BYTES);
            const int brow = bsrc * p.ny + yr;   // row index over both buffers
            tma_load_2d(dst, &gd->tmap_rho, &bars[s], xb, brow * Cfg::NS);
            tma_load_2d(dst + Cfg::RHO_BYTES, &gd->tmap_dev, &bars[s], xb, brow * 16);
        };
        if (tid == 0) {
            for (int m = 0; m < NSLOT && r0 + m < r_load; ++m) issue(r0 + m, m);
        }

        bool ok = true;   // a thread that gave up waiting does not wait again
        const int tc = 2 * tid, x = x0 + tc;            // the thread's first column
        const bool active = tc < w, both = tc + 1 < w;
        const bool last = tid == (w - 1) / 2;            // has the strip's last column
        const bool open_l = OPEN && x0 == 0, open_r = OPEN && x0 + w == p.nx;
        // the outlet column is the first or second one beyond the strip
        const bool open_next = OPEN && x0 + w == p.nx - 1, open_next2 = OPEN && x0 + w == p.nx - 2;
        __syncthreads();   // the constants are in place

        // store pointers of the row collided next
        char *out_rho = reinterpret_cast<char *>(d.rho + bdst * d.rho_buf + (long long)ya * d.rho_row + d.ghost + x);
        char *out_dev = reinterpret_cast<char *>(reinterpret_cast<T *>(d.dev) + bdst * d.dev_buf +
                                                 (long long)ya * d.dev_row + d.ghost + x);

        const f2 zero{0.0f, 0.0f};
        HalfPulled H;        // nodes (x, r - 1) at the start of pass r
        f2 lo0 = zero, lo1 = zero, lo2 = zero, lo5 = zero, lo6 = zero, lo_h = zero;   // row r - 1's terms for row r
        PulledOf<f2> Pc, Pn; // pulled state of rows r - 2 and r - 1
        H.own[0] = H.own[1] = H.acc[0] = H.acc[1] = zero;
        H.T1 = H.T2 = H.T3 = H.T5 = H.T6 = H.h = zero;
        Pn.rr = Pn.rb = Pn.e1 = Pn.e2 = Pn.e3 = Pn.e4 = Pn.e5 = Pn.e6 = Pn.e7 = Pn.e8 = zero;
        // colour field of rows r - 3 (s) and r - 2 (c): the thread's columns, the column west
        // of them and the one east; q u: the x difference of q u_x, and q u_y
        f2 sC = zero, cC = zero, sX = zero, cX = zero, qsC = zero, qcC = zero;
        float sW = 0.0f, sE = 0.0f, cW = 0.0f, cE = 0.0f, qsW = 0.0f, qsE = 0.0f, qcW = 0.0f, qcE = 0.0f;

        auto wall_terms = [&](const unsigned char *sp, int i, int j, int k, float sgn) {
            return wall_row_terms<T>(reinterpret_cast<const float *>(sp) + tc + G, BOXW,
                                     reinterpret_cast<const T *>(sp + Cfg::RHO_BYTES) + tc + G, BOXW, K, p.dphi[1], i, j, k, sgn);
        };
        // side columns of an odd lattice, collided in the pass before
        const bool odd_sides = ODD && (p.nx & 1) && (x0 == 0 || x0 + w > p.nx - 8);
        auto store_sides = [&](int y) {
            using Side = SideCols<T>;
            constexpr int PLANES = Side::NS + 16;
            float *orho = d.rho + bdst * d.rho_buf + (long long)y * d.rho_row + d.ghost;
            T *odev = reinterpret_cast<T *>(d.dev) + bdst * d.dev_buf + (long long)y * d.dev_row + d.ghost;
            const unsigned char *row = sides + (y & 1) * Side::FLOATS * 4;
            auto put = [&](int plane, int right, int from, int col) {
                const unsigned char *s = row + right * Side::BYTES;
                if (plane < Side::NS)
                    orho[plane * d.rho_plane + col] = reinterpret_cast<const float *>(s)[plane * Side::PITCH + from];
                else
                    odev[(plane - Side::NS) * d.dev_plane + col] =
                        reinterpret_cast<const T *>(s + Side::DEV_AT)[(plane - Side::NS) * Side::PITCH + from];
            };
            const int c = tid & 7;
            if (x0 == 0)
                for (int k = tid >> 3; k < PLANES; k += NT / 8) put(k, 0, c, p.nx + c);
            const int col = p.nx - 8 + c;   // (a narrow last strip leaves some to the one before it)
            if (col >= x0 && col < x0 + w)
                for (int k = tid >> 3; k < PLANES; k += NT / 8) put(k, 1, c + 1, c - 8);
            if (x0 + w == p.nx && tid < PLANES) put(tid, 1, 8, p.nx - 1);   // the lone last column itself
        };
        int slot = 0;
        uint32_t phase = 0;
#pragma unroll 1
        for (int r = r0; r < yb + 2; ++r) {
            const int Y = r - 1;                          // row whose nodes this pass closes
            const bool closes = r >= ya && (Y >= 0 || !wall_y);
            const bool wall_row = wall_y && Y >= p.ny;    // Y is the wall above
            const bool by_wall = wall_y && (Y == 0 || Y >= p.ny - 1);
            if (OPEN && (open_l || open_r || open_next || open_next2) && r >= ya && ((r - ya) & (OPEN_ROWS - 1)) == 0) {
                // open columns of rows Y .. Y + OPEN_ROWS - 1 by the general pull with the Zou-He
                // values, one node per thread; row Y's are at slot (Y - ya + 1) mod 2 OPEN_ROWS
                const int side = tid / OPEN_ROWS, Yo = Y + tid % OPEN_ROWS;
                if (side < 2 && (side == 0 ? open_l : open_r || open_next || open_next2) && Yo <= yb && !(wall_y && (Yo < 0 || Yo >= p.ny))) {
                    const RowLoader<T> L(d, bsrc, Yo);
                    Pulled P;
                    pull_node<HERMITE>(p, L, side == 0 ? 0 : p.nx - 1, Yo, t, false, 0.0f, 0.0f, P);
                    float *o = opens + (side * 2 * OPEN_ROWS + ((Yo - ya + 1) & (2 * OPEN_ROWS - 1))) * OPEN_VALUES;
                    o[0] = P.rr;
                    o[1] = P.rb;
#pragma unroll
                    for (int i = 1; i < 9; i++) o[i + 1] = P.e[i];
                }
                __syncthreads();
            }
            Pc = Pn;
            float *ring_psi = rings + (Y & 1) * RING + 2, *ring_qx = ring_psi + Cfg::QX_OFF, *ring_qy = ring_psi + Cfg::QY_OFF;
            if (r < r_load && ok && !mbar_wait_bounded(&bars[slot], phase, WAIT_LIMIT_CYCLES)) ok = false;
            if (r < r_load) {
                const unsigned char *sp = slots + slot * Cfg::SLOT_BYTES;
                if (active) {
                    const RowTerms R = row_terms<T>(reinterpret_cast<const float *>(sp) + tc + G, BOXW,
                                                    reinterpret_cast<const T *>(sp + Cfg::RHO_BYTES) + tc + G, BOXW, K);
                    Step S = step_of(K, H.own, R.own);
                    if (closes) close_node<SPLIT>(K, H, R.dn[0], R.dn[1], R.T4, R.T7, R.T8, R.h_dn, S, Pn);
                    if (wall_y && r == 0) {
                        // links from behind the lower wall: the node's own opposite
                        // populations (no slip), or those of its row travelling on
                        // mirrored (free slip)
                        S = no_step();
                        if (WET && d.wet.slip) {
                            lo0 = R.dn[0], lo1 = R.dn[1];
                            lo2 = R.T4, lo5 = R.T8, lo6 = R.T7, lo_h = R.h_dn;
                        } else {
                            const WallTerms L = wall_terms(sp, 4, 7, 8, -1.0f);
                            lo0 = L.sum[0], lo1 = L.sum[1], lo2 = L.Ti, lo5 = L.Tj, lo6 = L.Tk, lo_h = L.h;
                        }
                    }
                    const f2 mquarter = lit<f2, LIT_MQUARTER>(), m15 = lit<f2, LIT_M3HALVES>();
                    H.own[0] = R.own[0], H.own[1] = R.own[1];
                    H.acc[0] = fmav(m15, S.r, R.mid[0] + lo0);
                    H.acc[1] = fmav(m15, S.b, R.mid[1] + lo1);
                    H.T1 = R.T1;
                    H.T3 = R.T3;
                    H.T2 = lo2 - S.sum;
                    H.T5 = fmav(mquarter, S.sum, lo5);
                    H.T6 = fmav(mquarter, S.sum, lo6);
                    if (SPLIT) H.h = lo_h + R.h_mid;
                    lo0 = R.up[0], lo1 = R.up[1];
                    lo2 = R.T2, lo5 = R.T5, lo6 = R.T6;
                    if (SPLIT) lo_h = R.h_up;
                }
            } else if (active && !wall_row) {
                // the row above is the upper wall (r == ny, row ny - 1 still in its slot)
                f2 dn0 = lo0, dn1 = lo1, T4 = lo2, T7 = lo6, T8 = lo5, h_dn = lo_h;
                if (!(WET && d.wet.slip)) {
                    const WallTerms L = wall_terms(slots + ((p.ny - 1 - r0) % NSLOT) * Cfg::SLOT_BYTES, 2, 5, 6, 1.0f);
                    dn0 = L.sum[0], dn1 = L.sum[1], T4 = L.Ti, T7 = L.Tj, T8 = L.Tk, h_dn = L.h;
                }
                close_node<SPLIT>(K, H, dn0, dn1, T4, T7, T8, h_dn, no_step(), Pn);
            }
            // The columns beside the strip, x0 - 1 and x0 + w, need psi (and q u) only.  The last
            // warp computes them, 16 lanes per side, lane j = 8 k + (i - 1) for colour k's
            // direction i: each adds its link's u of the edge node of row Y from the row that the
            // link's source is in (the values of the rows before are kept in shared memory; a
            // link from behind a wall stands for the missing row), and the sums are reduced with
            // shuffles.  Next to a wall the columns one further out are computed as well (outer):
            // psi of the wall row needs them.
            if (tid >= NT - 32 && !wall_row) {
                const int lane = tid & 31, side = lane >> 4, k = (lane >> 3) & 1, i = (lane & 7) + 1;
                const int cx = (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
                const int cy = (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
                const bool axis = i <= 4;
                const float phi = (k == 0 ? p.phi_r[1] : p.phi_b[1]) * (axis ? 1.0f : 0.25f);
                const bool near = wall_y && (r <= 1 || r >= p.ny - 2);
                for (int outer = 0; outer <= (near ? 1 : 0); outer++) {
                    const int at = side == 0 ? -1 - outer : w + outer, col = G + at;
                    // density and decoded deviation of direction (dx, dy), plane j, at slot column q
                    auto value = [&](const unsigned char *row, int q, int j, int dx, int dy, float &s, float &dv) {
                        const float *rp = reinterpret_cast<const float *>(row) + q;
                        s = rp[k * BOXW];
                        dv = Codec<T>::dec(reinterpret_cast<const T *>(row + Cfg::RHO_BYTES)[(k * 8 + j - 1) * BOXW + q]);
                        if (SPLIT) {
                            const float gc = (float)dx * rp[3 * BOXW] + (float)dy * rp[4 * BOXW];
                            const float h = edge_shift(p, axis, rp[0], rp[BOXW], rp[2 * BOXW], gc);
                            dv += k == 0 ? h : -h;
                        }
                    };
                    // source across a wall next to `row`: the node itself in the opposite direction, or
                    // (free slip) the row's neighbour in the mirrored one
                    auto across = [&](const unsigned char *row, float4 &v) {
                        const bool slip = WET && d.wet.slip;
                        const int opp = i <= 4 ? ((i + 1) & 3) + 1 : ((i - 3) & 3) + 5;
                        const int mir = i == 2 ? 4 : i == 4 ? 2 : i == 5 ? 8 : i == 8 ? 5 : i == 6 ? 7 : i == 7 ? 6 : i;
                        value(row, slip ? col - cx : col, slip ? mir : opp, slip ? cx : -cx, -cy, v.x, v.y);
                    };
                    float4 *hist = reinterpret_cast<float4 *>(rings + Cfg::HIST_OFF) + outer * 128 + lane;
                    float4 now;   // source density, its deviation, own density, own deviation
                    if (r < r_load) {
                        const unsigned char *row = slots + slot * Cfg::SLOT_BYTES;
                        value(row, col - cx, i, cx, cy, now.x, now.y);
                        now.z = reinterpret_cast<const float *>(row)[k * BOXW + col];
                        now.w = Codec<T>::dec(reinterpret_cast<const T *>(row + Cfg::RHO_BYTES)[(k * 8 + i - 1) * BOXW + col]);
                        // (the node's own shifts sum to 5 m dphi_1: an eighth per lane)
                        if (SPLIT)
                            now.w = __fmaf_rn((k == 0 ? 0.625f : -0.625f) * p.dphi[1],
                                              reinterpret_cast<const float *>(row)[2 * BOXW + col], now.w);
                        if (wall_y && r == 0) across(row, hist[3 * 32]);   // stands for row -1
                    } else {
                        across(slots + ((p.ny - 1 - r0) % NSLOT) * Cfg::SLOT_BYTES, now);   // stands for row ny
                    }
                    if (closes && (outer == 0 || by_wall)) {
                        const float4 one = hist[((r - 1) & 3) * 32];
                        const float4 src = cy < 0 ? now : (cy == 0 ? one : hist[((r - 2) & 3) * 32]);
                        const float u = fmav(phi, src.x - one.z, src.y);
                        float v = u - one.w;
                        v += __shfl_xor_sync(0xffffffffu, v, 1);
                        v += __shfl_xor_sync(0xffffffffu, v, 2);
                        v += __shfl_xor_sync(0xffffffffu, v, 4);
                        const float mine = one.z + v;                        // colour k's new density
                        const float other = __shfl_xor_sync(0xffffffffu, mine, 8);
                        const float rr = k == 0 ? mine : other, rb = k == 0 ? other : mine;
                        float jx = 0.0f, jy = 0.0f;
                        if (HERMITE_SRC) {   // momentum: the shifts and rest parts cancel
                            jx = (float)cx * u;
                            jy = (float)cy * u;
#pragma unroll
                            for (int o = 1; o < 16; o <<= 1) {
                                jx += __shfl_xor_sync(0xffffffffu, jx, o);
                                jy += __shfl_xor_sync(0xffffffffu, jy, o);
                            }
                        }
                        if ((lane & 15) == 0 &&
                            !(OPEN && (side == 0 ? open_l : open_r || open_next || (open_next2 && outer)))) {
                            ring_psi[at] = edge_colour(p, rr, rb);
                            if (HERMITE_SRC && outer == 0) {
                                const float q = __fmaf_rn(p.q_r, rr, __fmul_rn(p.q_b, rb)), rho = rr + rb;
                                ring_qx[at] = q * (jx / rho + 0.5f * p.gx);
                                ring_qy[at] = q * (jy / rho + 0.5f * p.gy);
                            }
                        }
                    }
                    hist[(r & 3) * 32] = now;
                }
            }

            f2 nC = zero, qx = zero, qy = zero;
            if (closes && !wall_row && active) {
                if (OPEN && ((open_l && tid == 0) || ((open_r || open_next || open_next2) && last))) {
                    const float *q = opens + ((Y - ya + 1) & (2 * OPEN_ROWS - 1)) * OPEN_VALUES;
                    auto put = [&](f2 &v, float s, bool second) { (second ? v.y : v.x) = s; };
                    auto take = [&](const float *o, bool second) {
                        put(Pn.rr, o[0], second), put(Pn.rb, o[1], second);
                        put(Pn.e1, o[2], second), put(Pn.e2, o[3], second), put(Pn.e3, o[4], second);
                        put(Pn.e4, o[5], second), put(Pn.e5, o[6], second), put(Pn.e6, o[7], second);
                        put(Pn.e7, o[8], second), put(Pn.e8, o[9], second);
                    };
                    // values beyond an open end (x = -1, x = nx) are those of the open column itself
                    // (zero gradient); a neighbouring outlet column's are its own
                    auto beside = [&](const float *o, int at) {
                        ring_psi[at] = colour_field(p, o[0], o[1]);
                        if (HERMITE_SRC && !open_next2) {
                            PulledOf<float> P{o[0], o[1], o[2], o[3], o[4], o[5], o[6], o[7], o[8], o[9]};
                            float jx, jy;
                            momentum_of(P, jx, jy);
                            const float rho = o[0] + o[1], u = p.q_r * o[0] + p.q_b * o[1];
                            ring_qx[at] = u * (jx / rho + 0.5f * p.gx);
                            ring_qy[at] = u * (jy / rho + 0.5f * p.gy);
                        }
                    };
                    if (open_l && tid == 0) {
                        take(q, false);
                        beside(q, -1);
                    }
                    if ((open_r || open_next || open_next2) && last) {
                        if (open_r) take(q + 2 * OPEN_ROWS * OPEN_VALUES, both);
                        beside(q + 2 * OPEN_ROWS * OPEN_VALUES, open_next2 ? w + 1 : w);
                    }
                }
                nC = colour_field_of(K, Pn.rr, Pn.rb);
                if (HERMITE_SRC) {
                    f2 jx, jy;
                    momentum_of(Pn, jx, jy);
                    const f2 rho = Pn.rr + Pn.rb;
                    const f2 q = fmav(K.q_r, Pn.rr, K.q_b * Pn.rb);
                    qx = q * (f2{jx.x / rho.x, jx.y / rho.y} + K.hgx);
                    qy = q * (f2{jy.x / rho.x, jy.y / rho.y} + K.hgy);
                    ring_qx[tc] = qx.x, ring_qy[tc] = qy.x;
                    if (both) ring_qx[tc + 1] = qx.y, ring_qy[tc + 1] = qy.y;
                }
                ring_psi[tc] = nC.x;
                if (both) ring_psi[tc + 1] = nC.y;
            }
            // colour field of the wall row beyond Yn, from that row's own values; q u is zero
            auto wall_fill = [&](int Yn, float *to) {
                const float *f = rings + (Yn & 1) * RING + 2;
                for (int cc = tid - 1; cc <= w; cc += NT)
                    to[cc] = wall_psi(p, x0 + cc, [&](int Xp) { return f[Xp - x0]; });
            };
            if (wall_row) {
                wall_fill(p.ny - 1, ring_psi);
                if (HERMITE_SRC)
                    for (int cc = tid; cc < w + 2; cc += NT) ring_qx[cc - 1] = ring_qy[cc - 1] = 0.0f;
            }
            __syncthreads();   // row Y's colour field is in the ring; row r was read
            if (r < r_load) {
                if (tid == 0 && r + NSLOT < r_load) issue(r + NSLOT, slot);
                if (++slot == NSLOT) {
                    slot = 0;
                    phase ^= 1u;
                }
            }
            if (ODD && odd_sides && r - 3 >= ya) store_sides(r - 3);
            if (!closes) continue;
            if (wall_y && Y == 0 && ya == 0) {   // the wall below row 0
                float *wall = rings + 2 * RING + 2;
                wall_fill(0, wall);
                __syncthreads();
                if (active) {
                    cC = f2{wall[tc], wall[tc + 1]}, cW = wall[tc - 1], cE = wall[tc + 2];
                    cX = qcC = zero;
                    qcW = qcE = 0.0f;
                }
            }
            if (!active) continue;

            // (an odd strip's last pair has its second column beyond the strip: that half holds
            // the edge column, and its results are not stored)
            const float nW = ring_psi[tc - 1], nE = ring_psi[tc + 2];
            if (wall_row) nC = f2{ring_psi[tc], ring_psi[tc + 1]};
            else if (!both) nC.y = ring_psi[tc + 1];
            f2 nX = zero;
            float qnE = 0.0f, qnW = 0.0f;
            if (HERMITE_SRC) {
                if (!both && !wall_row) qx.y = ring_qx[tc + 1], qy.y = ring_qy[tc + 1];
                nX = f2{qx.y - ring_qx[tc - 1], ring_qx[tc + 2] - qx.x};
                qnE = ring_qy[tc + 2];
                qnW = ring_qy[tc - 1];
            }
            if (r - 2 >= ya) {
                // 12 times the S2I4 gradient (Eq. (eq:colorGradient)), from differences only,
                // so that a uniform field gives exactly zero
                const f2 four = lit<f2, LIT_FOUR>();
                auto row_diff = [](f2 m, float west, float east) { return f2{m.y - west, east - m.x}; };
                f2 Fx = fmav(four, row_diff(cC, cW, cE), row_diff(nC, nW, nE) + row_diff(sC, sW, sE));
                const f2 dC = nC - sC;
                f2 Fy = fmav(four, dC, f2{dC.y + (nW - sW), (nE - sE) + dC.x});
                f2 dQx = zero, dQy = zero;
                if (WET) {
                    contact_angle_adjust(d.wet, p, r - 2, Fx.x, Fy.x);
                    contact_angle_adjust(d.wet, p, r - 2, Fx.y, Fy.y);
                }
                if (HERMITE_SRC) {
                    dQx = fmav(four, cX, nX + sX);
                    const f2 dq = qy - qsC;
                    dQy = fmav(four, dq, f2{dq.y + (qnW - qsW), (qnE - qsE) + dq.x});
                }
                Collided<f2> o;
                collide_of<CV, SPLIT, f2>(p, K, Pc, cC, Fx, Fy, dQx, dQy, o);
                store_pair<T, SPLIT, ODD>(d, !OPEN && p.bc_x == BC_PERIODIC, x, both, out_rho, out_dev, Pc.rr, Pc.rb, o,
                                          sides + (r & 1) * SideCols<T>::FLOATS * 4);
                out_rho += d.rho_row * 4;
                out_dev += d.dev_row * (long long)sizeof(T);
            }
            sC = cC, sW = cW, sE = cE;
            cC = nC, cW = nW, cE = nE;
            if (HERMITE_SRC) {
                sX = cX, cX = nX;
                qsC = qcC, qsW = qcW, qsE = qcE;
                qcC = qy, qcW = qnW, qcE = qnE;
            }
        }

        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                atomicOr(err, ERR_TIMEOUT);
                // wait (bounded) for the copies this block still has in flight, so
                // that none lands after the block's shared memory is released: the
                // latest phase issued into each slot (every row was issued by now)
                // covers the earlier ones
                for (int s = 0; s < NSLOT; s++) {
                    const int uses = (r_load - r0 - s + NSLOT - 1) / NSLOT;
                    if (uses > 0) mbar_wait_bounded(&bars[s], (uint32_t)((uses - 1) & 1), WAIT_LIMIT_CYCLES / 4);
                }
            }
            __syncthreads();
            return;
        }
        if (ODD && odd_sides) store_sides(yb - 1);
    }
    // this block's stores are issued: the next step may launch (it still waits
    // for this grid's completion before it reads anything); a block that
    // triggered at its start does not trigger again
    if (!(flags & FUSED_EARLY_NEXT)) asm volatile("griddepcontrol.launch_dependents;");
}

// ------------------------------------------------------------- tile kernel

// Launch shape: columns per tile (two per thread), at most so many rows (one warp each),
// blocks per SM the registers are sized for.
constexpr int TILE_W = 64;
constexpr int TILE_MAX_ROWS = 8;
constexpr int TILE_THREADS = 32 * TILE_MAX_ROWS;
constexpr int TILE_MINB = 2;

// Pulled state of the nodes (x, Y), (x + 1, Y) from global memory by the strip kernel's
// sequence of operations (bit-identical to it).  Y lies in the lattice.
template <typename T, int CV>
__device__ __forceinline__ void pull_pair(const SimDesc &d, const Consts<f2> &K, int b, int x, int Y, PulledOf<f2> &P) {
    constexpr bool SPLIT = SplitStore<T>::value;
    const Phys &p = d.ph;
    const int ny = p.ny, rs = (int)d.rho_plane, ds = (int)d.dev_plane;
    const bool wall_y = p.bc_y == BC_WALL, bottom = wall_y && Y == 0, top = wall_y && Y == ny - 1;
    const bool slip = (CV & CV_WET) && d.wet.slip;
    const float *r = d.rho + b * d.rho_buf + d.ghost + x;
    const T *v = reinterpret_cast<const T *>(d.dev) + b * d.dev_buf + d.ghost + x;
    const float *rp = r + Y * d.rho_row;
    const T *dp = v + Y * d.dev_row;
    const f2 zero{0.0f, 0.0f};
    const RowTerms R = row_terms<T>(rp, rs, dp, ds, K);
    HalfPulled H;
    f2 lo0, lo1, lo2, lo5, lo6, lo_h;
    Step S = no_step();
    if (!bottom) {
        const int Ym = Y > 0 ? Y - 1 : ny - 1;
        const RowTerms A = row_terms<T>(r + Ym * d.rho_row, rs, v + Ym * d.dev_row, ds, K);
        lo0 = A.up[0], lo1 = A.up[1], lo2 = A.T2, lo5 = A.T5, lo6 = A.T6, lo_h = A.h_up;
        S = step_of(K, A.own, R.own);
    } else if (slip) {
        lo0 = R.dn[0], lo1 = R.dn[1], lo2 = R.T4, lo5 = R.T8, lo6 = R.T7, lo_h = R.h_dn;
    } else {
        const WallTerms L = wall_row_terms<T>(rp, rs, dp, ds, K, p.dphi[1], 4, 7, 8, -1.0f);
        lo0 = L.sum[0], lo1 = L.sum[1], lo2 = L.Ti, lo5 = L.Tj, lo6 = L.Tk, lo_h = L.h;
    }
    const f2 mquarter = lit<f2, LIT_MQUARTER>(), m15 = lit<f2, LIT_M3HALVES>();
    H.own[0] = R.own[0], H.own[1] = R.own[1];
    H.acc[0] = fmav(m15, S.r, R.mid[0] + lo0);
    H.acc[1] = fmav(m15, S.b, R.mid[1] + lo1);
    H.T1 = R.T1;
    H.T3 = R.T3;
    H.T2 = lo2 - S.sum;
    H.T5 = fmav(mquarter, S.sum, lo5);
    H.T6 = fmav(mquarter, S.sum, lo6);
    H.h = SPLIT ? lo_h + R.h_mid : zero;
    f2 dn0, dn1, T4, T7, T8, h_dn;
    S = no_step();
    if (!top) {
        const int Yp = Y + 1 < ny ? Y + 1 : 0;
        const RowTerms B = row_terms<T>(r + Yp * d.rho_row, rs, v + Yp * d.dev_row, ds, K);
        dn0 = B.dn[0], dn1 = B.dn[1], T4 = B.T4, T7 = B.T7, T8 = B.T8, h_dn = B.h_dn;
        S = step_of(K, H.own, B.own);
    } else if (slip) {
        dn0 = R.up[0], dn1 = R.up[1], T4 = R.T2, T7 = R.T6, T8 = R.T5, h_dn = R.h_up;
    } else {
        const WallTerms L = wall_row_terms<T>(rp, rs, dp, ds, K, p.dphi[1], 2, 5, 6, 1.0f);
        dn0 = L.sum[0], dn1 = L.sum[1], T4 = L.Ti, T7 = L.Tj, T8 = L.Tk, h_dn = L.h;
    }
    close_node<SPLIT>(K, H, dn0, dn1, T4, T7, T8, h_dn, S, P);
}

// One step of a lattice whose tiles all fit on the chip at once: block (bx, by) owns 64 columns
// by `ty` rows, one thread per two neighbouring columns.  Every thread pulls its nodes straight
// from global memory; the nodes around the tile (colour field and q u only) are pulled by
// blockDim.x / 32 - ty more warps at the same time (by the tile's own warps if there are none);
// after one barrier the tile is collided and stored.  Periodic in x; any walls.
//
// Such a lattice is in L2 and a step is bound by its chain of dependent latencies: a strip's
// block waits for a row load, makes at least five row passes with a barrier each, and stores;
// a tile's block makes one pull, one barrier and one collision.  It loads and pulls the nodes
// around its tile again (1.6 times the nodes with 4 rows), so where the strips' blocks are
// all busy they win.  Microseconds a step, strips and tiles (FP32): 64 x 64 5.8 / 4.3, 200 x
// 200 8.8 / 5.3, 140 x 280 9.9 / 5.3, 256 x 256 9.5 / 6.3, 512 x 256 11.1 / 8.7, 512 x 512
// 12.7 / 16.1.
//
// LONE: between walls, with one column right of the last full tile (nx = 65 mod 128).  The strip
// kernel forms the column beyond that one link by link, and a wall's psi at the last column, a
// corner of the full tile's gradients, is made from both: so does the full tile.  A variant of
// its own, because the test in every lattice's kernel cost 64 x 64 and 140 x 280 1.6 %.
template <typename T, int CV, bool LONE>
__global__ void __launch_bounds__(TILE_THREADS, TILE_MINB) k_step_tile(const SimDesc *__restrict__ gd, int step_offset, int ty,
                                                                        int *__restrict__ err) {
    constexpr bool SPLIT = SplitStore<T>::value, WET = (CV & CV_WET) != 0;
    constexpr bool HERMITE_SRC = (CV & CV_MRT) && (CV & CV_HERMITE);
    constexpr int PITCH = TILE_W + 4;   // columns x0 - 2 .. x0 + TILE_W + 1
    __shared__ SimDesc d;
    __shared__ Consts<f2> K;
    __shared__ __align__(16) float s_psi[(TILE_MAX_ROWS + 2) * PITCH];
    __shared__ __align__(16) float s_qx[HERMITE_SRC ? (TILE_MAX_ROWS + 2) * PITCH : 4], s_qy[HERMITE_SRC ? (TILE_MAX_ROWS + 2) * PITCH : 4];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x >> 5;
    {   // read while the previous step still runs
        const int4 *src = reinterpret_cast<const int4 *>(gd);
        int4 *dst = reinterpret_cast<int4 *>(&d);
        for (int j = tid; j < (int)(sizeof(SimDesc) / 16); j += blockDim.x) dst[j] = __ldcv(src + j);
    }
    __syncthreads();
    if (tid == 0) fill_consts(K, d.ph);
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    long long t0 = d.t0, t_end = d.t_end;
    if (step_offset == 0) {   // written between chunks of steps
        t0 = __ldcv(&gd->t0);
        t_end = __ldcv(&gd->t_end);
    }
    const Phys &p = d.ph;
    const long long t = t0 + step_offset;
    if (t >= t_end) return;   // this simulation has stopped
    if (d.variant != CV || d.ghost != 8 || p.bc_x != BC_PERIODIC || ty < 1 || ty > TILE_MAX_ROWS || ty > warps) {
        if (tid == 0) atomicOr(err, ERR_BADITEM);
        return;
    }
    const int bsrc = (int)(t & 1), bdst = bsrc ^ 1;
    const int x0 = blockIdx.x * TILE_W, y0 = blockIdx.y * ty, nx = p.nx, ny = p.ny;
    const int rows = min(ty, ny - y0);
    if (x0 >= nx || rows <= 0) return;
    const bool wall_y = p.bc_y == BC_WALL;

    PulledOf<f2> P;
    // Where the tile borders on another 128-column strip (or the lattice's end) the strip
    // kernel forms the columns beyond link by link: so does this one, so that a lattice has the
    // same states in tiles, in strips and in a batch.
    const bool edge_l = x0 % FUSED_W == 0, edge_r = (x0 + TILE_W) % FUSED_W == 0 || x0 + TILE_W >= nx;
    const int w = min(TILE_W, nx - x0);
    const bool link_r = edge_r || (LONE && x0 + TILE_W + 1 == nx);
    // pull the nodes of pair `q` (columns x0 + 2 q, + 1), row `row` of the tile, and share
    // their colour field
    auto node = [&](int q, int row, PulledOf<f2> &N) {
        int Y = y0 + row;
        const int x = x0 + 2 * q;
        if ((q < 0 && edge_l) || (edge_r && 2 * q >= w)) return;
        if (Y < 0 || Y >= ny) {
            if (wall_y) return;
            Y = Y < 0 ? Y + ny : Y - ny;
        }
        pull_pair<T, CV>(d, K, bsrc, x, Y, N);
        const int at = (row + 1) * PITCH + 2 * q + 2;
        auto share = [&](float *to, f2 v) {   // (an odd lattice's last pair: the second column is beyond)
            if (link_r && 2 * q + 1 >= w) to[at] = v.x;
            else pair_to(to + at, v);
        };
        share(s_psi, colour_field_of(K, N.rr, N.rb));
        if (HERMITE_SRC) {
            f2 jx, jy;
            momentum_of(N, jx, jy);
            const f2 rho = N.rr + N.rb;
            const f2 u = fmav(K.q_r, N.rr, K.q_b * N.rb);
            share(s_qx, u * (f2{jx.x / rho.x, jx.y / rho.y} + K.hgx));
            share(s_qy, u * (f2{jy.x / rho.x, jy.y / rho.y} + K.hgy));
        }
    };
    const int halo = 2 * (TILE_W / 2 + 2) + 2 * rows;
    const int own_warps = warps > ty ? ty : 0;   // with extra warps, those pull the halo
    if (warp >= own_warps) {
        PulledOf<f2> N;
        for (int h = tid - own_warps * 32; h < halo; h += blockDim.x - own_warps * 32) {
            const int side = TILE_W / 2 + 2;
            if (h < 2 * side) node(h < side ? h - 1 : h - side - 1, h < side ? -1 : rows, N);
            else node((h & 1) ? TILE_W / 2 : -1, (h - 2 * side) >> 1, N);
        }
        // nodes beside strip borders, one per half warp: rows, next column out (the wall rows'
        // psi needs those), of the one or two sides that are borders.  All fit in one round of
        // the extra warps away from walls (with every second half warp left to the side that
        // mostly is none, two rounds: 200 x 200 6.0 us a step, now 5.3).
        const int rs = (int)d.rho_plane, ds = (int)d.dev_plane;
        const unsigned lanes = 0xffffu << (tid & 16);
        const EdgeLink E(p, (tid & 7) + 1, (tid >> 3) & 1);
        // (beside a lone column, two more: the column beyond it in the rows next to the walls)
        const bool lone = LONE && link_r && !edge_r;
        const int sides = (edge_l ? 1 : 0) + (edge_r ? 1 : 0), edges = sides * (rows + 2) * (wall_y ? 2 : 1);
        for (int e = (tid - own_warps * 32) >> 4; e < edges + (lone ? 2 : 0); e += (blockDim.x - own_warps * 32) >> 4) {
            const int j = sides == 2 ? e >> 1 : e;
            int side = sides == 2 ? e & 1 : (edge_l ? 0 : 1), outer = j >= rows + 2, row = j - (outer ? rows + 2 : 0) - 1;
            if (lone && e >= edges) {
                side = 1, outer = 1, row = e == edges ? -y0 : ny - 1 - y0;
                if (row < 0 || row >= rows) continue;
            }
            int Y = y0 + row;
            if (wall_y && (Y < 0 || Y >= ny)) continue;
            if (outer && !(wall_y && (Y == 0 || Y == ny - 1))) continue;
            Y = Y < 0 ? Y + ny : (Y >= ny ? Y - ny : Y);
            const int col = side == 0 ? -1 - outer : w + outer;
            const float *rp = d.rho + bsrc * d.rho_buf + d.ghost + x0 + col;
            const T *dp = reinterpret_cast<const T *>(d.dev) + bsrc * d.dev_buf + d.ghost + x0 + col;
            float s, dv, own_s, own_dv, psi, qx, qy;
            E.own<T>(rp + Y * d.rho_row, rs, dp + Y * d.dev_row, ds, own_s, own_dv);
            int from = Y - E.cy;
            const bool wall = wall_y && (from < 0 || from >= ny);
            from = wall ? Y : (from < 0 ? from + ny : (from >= ny ? from - ny : from));
            E.source<T>(rp + from * d.rho_row, rs, dp + from * d.dev_row, ds, wall, WET && d.wet.slip, s, dv);
            __syncwarp(lanes);
            E.node<HERMITE_SRC>(lanes, s, dv, own_s, own_dv, psi, qx, qy);
            if ((tid & 15) == 0) {
                const int at = (row + 1) * PITCH + col + 2;
                s_psi[at] = psi;
                if (HERMITE_SRC) s_qx[at] = qx, s_qy[at] = qy;
            }
        }
    }
    const int x = x0 + 2 * lane, y = y0 + warp;
    const bool mine = warp < rows;
    if (mine) node(lane, warp, P);
    __syncthreads();
    if (wall_y && (y0 == 0 || y0 + rows == ny)) {   // the walls' colour field; their q u is zero
        for (int side = 0; side < 2; side++) {
            if (side == 0 ? y0 != 0 : y0 + rows != ny) continue;
            const float *f = s_psi + (side == 0 ? 1 : rows) * PITCH + 2;
            float *to = s_psi + (side == 0 ? 0 : rows + 1) * PITCH + 2;
            for (int c = tid - 1; c <= w; c += blockDim.x) {
                to[c] = wall_psi(p, x0 + c, [&](int X) { return f[X - x0]; });
                if (HERMITE_SRC) {
                    s_qx[(to - s_psi) + c] = 0.0f;
                    s_qy[(to - s_psi) + c] = 0.0f;
                }
            }
        }
        __syncthreads();
    }
    if (!mine || x >= nx) return;

    // 12 times the S2I4 gradient, in the strip kernel's order
    const f2 four = lit<f2, LIT_FOUR>();
    auto row_diff = [](f2 m, float west, float east) { return f2{m.y - west, east - m.x}; };
    const float *c = s_psi + (warp + 1) * PITCH + 2 * lane + 2, *s = c - PITCH, *n = c + PITCH;
    const f2 cC = pair_at(c), sC = pair_at(s), nC = pair_at(n);
    const float cW = c[-1], cE = c[2], sW = s[-1], sE = s[2], nW = n[-1], nE = n[2];
    f2 Fx = fmav(four, row_diff(cC, cW, cE), row_diff(nC, nW, nE) + row_diff(sC, sW, sE));
    const f2 dC = nC - sC;
    f2 Fy = fmav(four, dC, f2{dC.y + (nW - sW), (nE - sE) + dC.x});
    f2 dQx{0.0f, 0.0f}, dQy{0.0f, 0.0f};
    if (WET) {
        contact_angle_adjust(d.wet, p, y, Fx.x, Fy.x);
        contact_angle_adjust(d.wet, p, y, Fx.y, Fy.y);
    }
    if (HERMITE_SRC) {
        const float *qx = s_qx + (c - s_psi), *qy = s_qy + (c - s_psi);
        auto diff = [&](const float *q) { return f2{q[1] - q[-1], q[2] - q[0]}; };
        dQx = fmav(four, diff(qx), diff(qx + PITCH) + diff(qx - PITCH));
        const f2 dq = pair_at(qy + PITCH) - pair_at(qy - PITCH);
        dQy = fmav(four, dq, f2{dq.y + (qy[PITCH - 1] - qy[-PITCH - 1]), (qy[PITCH + 2] - qy[-PITCH + 2]) + dq.x});
    }
    Collided<f2> o;
    collide_of<CV, SPLIT, f2>(p, K, P, cC, Fx, Fy, dQx, dQy, o);
    store_pair<T, SPLIT>(d, true, x, x + 1 < nx,
                         reinterpret_cast<char *>(d.rho + bdst * d.rho_buf + (long long)y * d.rho_row + d.ghost + x),
                         reinterpret_cast<char *>(reinterpret_cast<T *>(d.dev) + bdst * d.dev_buf + (long long)y * d.dev_row +
                                                  d.ghost + x),
                         P.rr, P.rb, o);
}

// --------------------------------------------------------- two-pass kernels

// Pass 1: colour field, colour densities and q u of every node.
template <typename T, int CV>
__global__ void k_tp_moments(const SimDesc *__restrict__ dp, int step_offset, float *__restrict__ aux) {
    constexpr bool HERMITE = (CV & CV_HERMITE) != 0, HERMITE_SRC = HERMITE && (CV & CV_MRT);
    const SimDesc &d = *dp;
    const Phys p = d.ph;
    const long long t = d.t0 + step_offset;
    if (t >= d.t_end) return;   // this simulation has stopped
    const int nx = p.nx, ny = p.ny;
    const long long n = (long long)nx * ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(k % nx), y = (int)(k / nx);
        const RowLoader<T> L(d, (int)(t & 1), y);
        Pulled P;
        pull_node<HERMITE>(p, L, x, y, t, false, 0.0f, 0.0f, P);
        const NodeMoments m = node_moments(p, P);
        aux[k] = m.psi;
        aux[n + k] = m.rr;
        aux[2 * n + k] = m.rb;
        if (HERMITE_SRC) {
            const float q = p.q_r * m.rr + p.q_b * m.rb;
            aux[3 * n + k] = q * m.ux;
            aux[4 * n + k] = q * m.uy;
        }
    }
}

// Value of an aux field at lattice position (X, Y) next to the domain.
__device__ __forceinline__ float aux_at(const Phys &p, const float *f, int X, int Y, bool is_psi) {
    const int nx = p.nx, ny = p.ny;
    if (Y < 0 || Y >= ny) {
        if (p.bc_y == BC_WALL) {
            if (!is_psi) return 0.0f;
            const int Yn = Y < 0 ? 0 : ny - 1;
            return wall_psi(p, X, [&](int Xp) {
                const int xw = Xp < 0 ? Xp + nx : (Xp >= nx ? Xp - nx : Xp);
                return f[(long long)Yn * nx + xw];
            });
        }
        Y = Y < 0 ? Y + ny : Y - ny;
    }
    if (X < 0 || X >= nx) {
        if (p.bc_x == BC_PERIODIC) X = X < 0 ? X + nx : X - nx;
        else X = X < 0 ? 0 : nx - 1;
    }
    return f[(long long)Y * nx + X];
}

// Pass 2: gradient from the scratch field, collision, perturbation,
// recolouring and store of every node.
template <typename T, int CV>
__global__ void k_tp_collide(const SimDesc *__restrict__ dp, int step_offset, const float *__restrict__ aux) {
    constexpr bool HERMITE = (CV & CV_HERMITE) != 0, HERMITE_SRC = HERMITE && (CV & CV_MRT);
    const SimDesc &d = *dp;
    const Phys p = d.ph;
    const long long t = d.t0 + step_offset;
    if (t >= d.t_end) return;   // this simulation has stopped
    const int nx = p.nx, ny = p.ny;
    const long long n = (long long)nx * ny;
    const int bsrc = (int)(t & 1);
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(k % nx), y = (int)(k / nx);
        const RowLoader<T> L(d, (int)(t & 1), y);
        Pulled P;
        pull_node<HERMITE>(p, L, x, y, t, true, aux[n + k], aux[2 * n + k], P);
        float Fx, Fy, dQx = 0.0f, dQy = 0.0f;
        s2i4([&](int dx, int dy) { return aux_at(p, aux, x + dx, y + dy, true); }, Fx, Fy);
        contact_angle_adjust(d.wet, p, y, Fx, Fy);
        if (HERMITE_SRC) {
            float gx_, gy_;
            s2i4([&](int dx, int dy) { return aux_at(p, aux + 3 * n, x + dx, y + dy, false); }, dQx, gy_);
            s2i4([&](int dx, int dy) { return aux_at(p, aux + 4 * n, x + dx, y + dy, false); }, gx_, dQy);
        }
        float dr[9], db[9];
        float sm, sgx, sgy;
        collide_node<CV, SplitStore<T>::value>(p, P, aux[k], Fx, Fy, dQx, dQy, dr, db, sm, sgx, sgy);
        NodeStore<T>(d, p, bsrc ^ 1, x, y).put(P.rr, P.rb, dr, db, sm, sgx, sgy);
    }
}

// ------------------------------------------------------------ init / fields

// Equilibrium state from FP64 fields at t = 0.  The stored state is the one
// whose first pull yields N^k_i(x, 0) = N^{k(e)}_i(x): the slot (i, y) holds
// the equilibrium population of the node that will read it -- node y + c_i,
// or node y itself in direction opp(i) when that link is bounced by a wall.
// The stored colour density of y is the sum of its slots, the deviations are
// taken from it.
// With `pops` non-null the pre-collision populations N^k_i(x, 0) are given
// directly (layout [2][9][ny][nx]) instead of being the equilibria of the fields.
template <typename T>
__global__ void k_init(const SimDesc *__restrict__ dp, const double *__restrict__ rr,
                       const double *__restrict__ rb, const double *__restrict__ ux,
                       const double *__restrict__ uy, const double *__restrict__ pops) {
    const SimDesc &d = *dp;
    const Phys p = d.ph;
    const bool hermite = (d.variant & CV_HERMITE) != 0;
    const int nx = p.nx, ny = p.ny;
    const long long n = (long long)nx * ny;
    const double herm[2] = {p.herm_r, p.herm_b};
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(k % nx), y = (int)(k / nx);
        // equilibrium population i of colour kk at node (X, Y) (in the domain)
        auto feq = [&](int kk, int i, int X, int Y) {
            const long long m = (long long)Y * nx + X;
            if (pops) return pops[(long long)(kk * 9 + i) * n + m];
            const double vx = ux[m], vy = uy[m], usq = vx * vx + vy * vy;
            const double rho = kk == 0 ? rr[m] : rb[m];
            const double cu = CX(i) * vx + CY(i) * vy;
            double lin = 3.0 * cu;
            if (hermite) lin = 3.0 * cu * (1.0 + 0.5 * herm[kk] * (3.0 * C2(i) - 4.0));
            return rho * (double)phi_k(p, kk, C2(i)) + rho * WT(i) * (lin + 4.5 * cu * cu - 1.5 * usq);
        };
        double v[2][9];
#pragma unroll
        for (int i = 0; i < 9; i++) {
            int X = x + CX(i), Y = y + CY(i);
            // 0: read by node (X, Y), 1: bounced back to (x, y), 2: unread,
            // 3: sent on along a free-slip wall to node (X, y) in direction MIRY(i)
            int mode = 0;
            if (i != 0) {
                if (Y < 0 || Y >= ny) {
                    if (p.bc_y == BC_WALL) {
                        mode = 1;
                        if (d.wet.slip && (p.bc_x == BC_PERIODIC || (X >= 0 && X < nx))) {
                            mode = 3;
                            Y = y;
                            X = X < 0 ? X + nx : (X >= nx ? X - nx : X);
                        }
                    } else {
                        Y = Y < 0 ? Y + ny : Y - ny;
                    }
                }
                if (mode == 0 && (X < 0 || X >= nx)) {
                    if (p.bc_x == BC_PERIODIC) X = X < 0 ? X + nx : X - nx;
                    else mode = 2;
                }
            }
            for (int kk = 0; kk < 2; kk++) {
                if (mode == 0) v[kk][i] = feq(kk, i, X, Y);
                else if (mode == 3) v[kk][i] = feq(kk, MIRY(i), X, Y);
                else if (mode == 1) v[kk][i] = feq(kk, OPP(i), x, y);
                else v[kk][i] = pops ? pops[(long long)(kk * 9 + i) * n + k]
                                     : (double)phi_k(p, kk, C2(i)) * (kk == 0 ? rr[k] : rb[k]);
            }
        }
        float dr[9], db[9];
        double rs[2];
        for (int kk = 0; kk < 2; kk++) {
            double s = 0.0;
            for (int i = 0; i < 9; i++) s += v[kk][i];
            rs[kk] = s;
            for (int i = 1; i < 9; i++) {
                const float dv = (float)(v[kk][i] - (double)phi_k(p, kk, C2(i)) * s);
                if (kk == 0) dr[i] = dv; else db[i] = dv;
            }
        }
        dr[0] = db[0] = 0.0f;
        NodeStore<T>(d, p, 0, x, y).store((float)rs[0], (float)rs[1], dr, db);
    }
}

// Macroscopic fields of the state at time t (pre-collision moments).
template <typename T, bool HERMITE>
__global__ void k_fields(const SimDesc *__restrict__ dp, long long t, double *__restrict__ out) {
    const SimDesc &d = *dp;
    const Phys p = d.ph;
    const int nx = p.nx, ny = p.ny;
    const long long n = (long long)nx * ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(k % nx), y = (int)(k / nx);
        const RowLoader<T> L(d, (int)(t & 1), y);
        Pulled P;
        pull_node<HERMITE>(p, L, x, y, t, false, 0.0f, 0.0f, P);
        const NodeMoments m = node_moments(p, P);
        out[k] = m.rr;
        out[n + k] = m.rb;
        out[2 * n + k] = m.ux;
        out[3 * n + k] = m.uy;
        out[4 * n + k] = (double)m.rr * p.cs2_r + (double)m.rb * p.cs2_b;
    }
}

// Slug-train profile of the state at time t (the measurements of Sec. 5.1), in
// FP64: per column x the light-phase thickness g(x) = sum_y (1 - psi)/2, and the
// colour field psi_c(x) on the channel centreline (the middle row, or the mean
// of the two middle rows when ny is even).  out[0, nx) = g, out[nx, 2 nx) = psi_c.
// A block takes 32 columns, each warp every SLUG_WARPS-th row of them (neighbouring columns
// in a warp); the warps' sums are added in a fixed order.  Bound by the latency of the
// pulls, which a thread walking a whole column made one after another: diagnostics and
// profile of a 2048 x 128 lattice together took 842 us, now 119 (profile 50).
constexpr int SLUG_WARPS = 16;
template <typename T, bool HERMITE>
__global__ void __launch_bounds__(32 * SLUG_WARPS) k_slug_profile(const SimDesc *__restrict__ dp, long long t,
                                                                  double *__restrict__ out) {
    const SimDesc &d = *dp;
    const Phys p = d.ph;
    const int nx = p.nx, ny = p.ny;
    const int ya = (ny - 1) / 2, yb = ny / 2;   // the same row when ny is odd
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ double sh_g[SLUG_WARPS][32], sh_a[32], sh_b[32];
    for (int x0 = blockIdx.x * 32; x0 < nx; x0 += gridDim.x * 32) {
        const int x = x0 + lane;
        double g = 0.0;
        if (x < nx) {
            for (int y = warp; y < ny; y += SLUG_WARPS) {
                const RowLoader<T> L(d, (int)(t & 1), y);
                Pulled P;
                pull_node<HERMITE>(p, L, x, y, t, false, 0.0f, 0.0f, P);
                const double a = (double)P.rr * p.inv_gamma, b = (double)P.rb;
                const double psi = (a - b) / (a + b);     // Eq. (eq:color_field)
                g += 0.5 * (1.0 - psi);
                if (y == ya) sh_a[lane] = psi;
                if (y == yb) sh_b[lane] = psi;
            }
        }
        sh_g[warp][lane] = g;
        __syncthreads();
        if (warp == 0 && x < nx) {
            double sum = sh_g[0][lane];
#pragma unroll
            for (int k = 1; k < SLUG_WARPS; k++) sum += sh_g[k][lane];
            out[x] = sum;
            out[nx + x] = ya == yb ? sh_a[lane] : 0.5 * (sh_a[lane] + sh_b[lane]);
        }
        __syncthreads();
    }
}

// Pre-collision populations of every node at time t, layout [2][9][ny][nx].
template <typename T, bool HERMITE>
__global__ void k_read_pops(const SimDesc *__restrict__ dp, long long t, double *__restrict__ out) {
    const SimDesc &d = *dp;
    const Phys p = d.ph;
    const int nx = p.nx, ny = p.ny;
    const long long n = (long long)nx * ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(k % nx), y = (int)(k / nx);
        const RowLoader<T> L(d, (int)(t & 1), y);
        double nr[9], nb[9];
        pull_populations<HERMITE>(p, L, x, y, t, nr, nb);
#pragma unroll
        for (int i = 0; i < 9; i++) {
            out[i * n + k] = nr[i];
            out[(9 + i) * n + k] = nb[i];
        }
    }
}

// ---------------------------------------------------------------- diagnostics
constexpr int DIAG_NQ = 16;        // slots of a block's partial sums
constexpr int DIAG_SUMS = 2 * DIAG_NQ;   // of both passes
constexpr int DIAG_THREADS = 256;
constexpr int DIAG_BLOCKS = 152 * 2;   // at most: all resident at 128 registers a thread, one reduction each

// pass 0: mass_r, mass_b, mom_x, mom_y, area_b, max |u|^2 (slot 5), sum x w_b, sum y w_b,
//         sum ux w_b, sum ux w_r, sum w_r, nonfinite
// pass 1: sum p (r < r_eff / 2), count, sum p (r > r_eff + 8), count around the centre, from
//         pass 0's sums (and the caller's centre, if there is one) in device memory
// Every block reduces its nodes' values through shared memory into part[block]; the last
// block to finish adds the blocks in order (deterministic) into fin[pass].  FP64 runs at
// 2 operations per clock and SM, so a node's FP64 work is kept small (|u| is compared
// squared, distances are decided in FP32 unless they lie within rounding of a radius), and
// threads take several nodes before one reduction (a reduction per 256 nodes by shuffles
// cost more FP64 time than the sums).  lbm_diagnostics of a 2048 x 128 / 8192 x 256 lattice:
// 68 / 228 us with two resident blocks per SM, 91 / 254 with four.
template <typename T, bool HERMITE, int PASS>
__global__ void __launch_bounds__(DIAG_THREADS, 2) k_diag(const SimDesc *__restrict__ dp, long long t, bool has_center,
                                                       double cx, double cy, double *__restrict__ part,
                                                       double *__restrict__ fin, unsigned *__restrict__ ticket) {
    constexpr int NQ = PASS == 0 ? 12 : 4;
    const SimDesc &d = *dp;
    const Phys p = d.ph;
    const int nx = p.nx, ny = p.ny;
    const long long n = (long long)nx * ny;
    __shared__ double sh[NQ][DIAG_THREADS];
    __shared__ bool s_last;
    double acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; q++) acc[q] = 0.0;
    double r_in = 0.0, r_out = 0.0;
    float cxf = 0.0f, cyf = 0.0f, in2 = 0.0f, out2 = 0.0f;
    if (PASS == 1) {
        const double area = fin[4];
        if (!has_center) {
            cx = area > 0.0 ? fin[6] / area : 0.0;
            cy = area > 0.0 ? fin[7] / area : 0.0;
        }
        const double r_eff = sqrt(fmax(area, 0.0) / 3.14159265358979323846);
        r_in = r_eff / 2.0;
        r_out = r_eff + 8.0;
        cxf = (float)cx, cyf = (float)cy, in2 = (float)(r_in * r_in), out2 = (float)(r_out * r_out);
    }
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        int x, y;
        if (n <= 0x7fffffffLL) {
            y = (int)((unsigned)k / (unsigned)nx);
            x = (int)((unsigned)k - (unsigned)y * (unsigned)nx);
        } else {
            y = (int)(k / nx);
            x = (int)(k - (long long)y * nx);
        }
        const RowLoader<T> L(d, (int)(t & 1), y);
        Pulled P;
        pull_node<HERMITE>(p, L, x, y, t, false, 0.0f, 0.0f, P);
        if (PASS == 0) {
            const NodeMoments m = node_moments(p, P);
            const bool bad = !(isfinite(m.rr) && isfinite(m.rb) && isfinite(m.ux) && isfinite(m.uy));
            if (bad) { acc[NQ - 1] += 1.0; continue; }
            const double rho = (double)m.rr + m.rb, ux = m.ux, uy = m.uy;
            const double wb = 0.5 * (1.0 - m.psi), wr = 1.0 - wb;
            acc[0] += m.rr;
            acc[1] += m.rb;
            acc[2] += rho * ux;
            acc[3] += rho * uy;
            acc[NQ > 4 ? 4 : 0] += wb;
            acc[NQ > 5 ? 5 : 0] = fmax(acc[NQ > 5 ? 5 : 0], ux * ux + uy * uy);
            acc[NQ > 6 ? 6 : 0] += wb * x;
            acc[NQ > 7 ? 7 : 0] += wb * y;
            acc[NQ > 8 ? 8 : 0] += wb * ux;
            acc[NQ > 9 ? 9 : 0] += wr * ux;
            acc[NQ > 10 ? 10 : 0] += wr;
        } else {
            float fx = fabsf((float)x - cxf), fy = fabsf((float)y - cyf);
            if (p.bc_x == BC_PERIODIC) fx = fminf(fx, (float)nx - fx);
            if (p.bc_y == BC_PERIODIC) fy = fminf(fy, (float)ny - fy);
            const float f2 = fx * fx + fy * fy;
            bool inside = f2 < in2, outside = f2 > out2;
            // FP32 rounding of the coordinates and of the squares: 1e-5 of the lattice and of r^2
            const float slack = 1e-5f * f2 + 4e-6f * (float)(nx + ny) * (fabsf(fx) + fabsf(fy) + 1.0f);
            if (!(fabsf(f2 - in2) > slack && fabsf(f2 - out2) > slack)) {
                double dx = fabs(x - cx), dy = fabs(y - cy);
                if (p.bc_x == BC_PERIODIC) dx = fmin(dx, nx - dx);
                if (p.bc_y == BC_PERIODIC) dy = fmin(dy, ny - dy);
                const double r = sqrt(dx * dx + dy * dy);
                inside = r < r_in;
                outside = r > r_out;
            }
            if (inside || outside) {
                const double pr = (double)P.rr * p.cs2_r + (double)P.rb * p.cs2_b;
                if (inside) { acc[0] += pr; acc[1] += 1.0; }
                if (outside) { acc[2] += pr; acc[3] += 1.0; }
            }
        }
    }
    // 16 threads per quantity add 16 values each, then a shuffle tree over the 16
    auto is_max = [](int q) { return PASS == 0 && q == 5; };
    auto tree = [&](int q, double v) {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            const double w = __shfl_xor_sync(0xffffffffu, v, o);
            v = is_max(q) ? fmax(v, w) : v + w;
        }
        return v;
    };
    const int q = threadIdx.x >> 4, l = threadIdx.x & 15;
#pragma unroll
    for (int j = 0; j < NQ; j++) sh[j][threadIdx.x] = acc[j];
    __syncthreads();
    double v = 0.0;
    if (q < NQ) {
        for (int j = l; j < DIAG_THREADS; j += 16) v = is_max(q) ? fmax(v, sh[q][j]) : v + sh[q][j];
    }
    v = tree(q, v);
    if (q < NQ && l == 0) part[(long long)blockIdx.x * DIAG_NQ + q] = v;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;   // wraps to 0 for the next launch
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    v = 0.0;
    if (q < NQ) {
        for (int b = l; b < (int)gridDim.x; b += 16) {
            const double w = __ldcg(part + (long long)b * DIAG_NQ + q);
            v = is_max(q) ? fmax(v, w) : v + w;
        }
    }
    v = tree(q, v);
    if (q < NQ && l == 0) fin[PASS * DIAG_NQ + q] = v;
}

#ifndef LBM_DEVICE_HELPERS_ONLY   // non-template kernels: defined in one translation unit
// ------------------------------------------------------------------- time
__global__ void k_advance(SimDesc *descs, int n, long long k) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) descs[i].t0 += k;
}

// A descriptor's start time and stop time (a batch keeps its own copies of its
// members' descriptors, so both follow the member's logical time and stop here).
__global__ void k_set_times(SimDesc *desc, long long t0, long long t_end) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        desc->t0 = t0;
        desc->t_end = t_end;
    }
}

#endif

}  // namespace lbm
