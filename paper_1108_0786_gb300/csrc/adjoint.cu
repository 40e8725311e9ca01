// adjoint.cu -- reverse sweep of the coupled step: the transposed Jacobian of
// the rigid-body step (Algorithm 1 with Eq. FB1-FB3, osci_i, osci_j), of the
// momentum-exchange force (Eq. hydroF and its torque), of the LBGK collision
// with Guo's term (Eq. 2), of the refill of uncovered cells and of the stream
// with velocity-corrected bounce-back (Eq. 3, 4 and the moving-wall rule of
// Sec. 2.3).  The obstacle maps of the recorded forward run are held fixed.
//
// Reverse step n (forward step n maps G^{n-1}, S^{n-1}, S^n to G^n, S^{n+1}):
//   adj_integrate  Sh^{n+1} -> Sh^n (rigid-body part), Fh^n, Th^n, dJ/dtheta
//   adj cells      Ph^{n+1} (adjoint of the pre-collision populations of step
//                  n+1) -> Ah^n (adjoint of G^n: the transposed stream, the
//                  bounce-back and refill terms of step n+1 and the force
//                  terms of step n) -> Ph^n = collision^T Ah^n
// The cell part is a pull on the adjoint: cell x gathers Ph^{n+1}_a(x + e_a),
// the reverse of the forward pull.  Cells whose flags are zero in epochs n
// and n+1 (no obstacle in reach, no wall, not uncovered) take a pure gather
// (bulk kernel); the others (bodies' cubes, wall faces) the full rule, with
// the per-body adjoint sums reduced in a fixed order.
#include <algorithm>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "../../include/lbm.h"
#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr int ADJ_THREADS = 256;
// boundary blocks are small: the cube's few link cells carry nearly all of
// the work, and small blocks spread them over more SMs
constexpr int ADJ_BOUNDARY_THREADS = 64;

// flags of epoch n+1 that call for the full rule (a cell that is only F_LINK has
// no neighbour solid at n)
constexpr uint8_t F_FULL_RULE = F_SOLID | F_SOLID_PREV | F_NEAR | F_WALL;

// the collision's parameters in the adjoint's precision, rounded once on the host
// (an FP64 conversion a thread would take the FP64 pipe's 64 cycles a warp)
template <typename A> struct AdjParams;
template <> struct AdjParams<double> {
    __device__ static double omega(const Device &dv) { return dv.omega; }
    __device__ static double guo(const Device &dv) { return 1.0 - 0.5 * dv.omega; }
    __device__ static double half_g(const Device &dv, int i) { return 0.5 * dv.g[i]; }
    __device__ static double g3(const Device &dv, int i) { return 3.0 * dv.g[i]; }
    __device__ static double eg(const Device &dv, int b) { return ex(b) * dv.g[0] + ey(b) * dv.g[1] + ez(b) * dv.g[2]; }
};
template <> struct AdjParams<float> {
    __device__ static float omega(const Device &dv) { return dv.omega_f; }
    __device__ static float guo(const Device &dv) { return dv.guo_f; }
    __device__ static float half_g(const Device &dv, int i) { return dv.gh_f[i]; }
    __device__ static float g3(const Device &dv, int i) { return dv.g3_f[i]; }
    __device__ static float eg(const Device &dv, int b) { return dv.eg_f[b]; }
};

// acc + s v for a component s of a direction
template <typename A> __device__ __forceinline__ A plus(A acc, int s, A v) { return s > 0 ? acc + v : (s < 0 ? acc - v : acc); }

// density and velocity of step n from the post-collision deviations:
// rho = 1 + sum delta; the collision adds g to the momentum (Guo), so
// rho u = sum e delta - g / 2
template <typename A>
__device__ inline void moments_post(const A (&G)[Q], const Device &dv, A &rho, A (&u)[3]) {
    A r = 0, j0 = 0, j1 = 0, j2 = 0;
#pragma unroll
    for (int b = 0; b < Q; ++b) {
        r += G[b];
        j0 = plus(j0, ex(b), G[b]);
        j1 = plus(j1, ey(b), G[b]);
        j2 = plus(j2, ez(b), G[b]);
    }
    rho = (A)1 + r;
    const A ir = (A)1 / rho;
    u[0] = (j0 - AdjParams<A>::half_g(dv, 0)) * ir;
    u[1] = (j1 - AdjParams<A>::half_g(dv, 1)) * ir;
    u[2] = (j2 - AdjParams<A>::half_g(dv, 2)) * ir;
}

// Transposed Jacobian of the LBGK collision with Guo's forcing at one cell:
// a holds the adjoint of the post-collision populations on entry and that
// of the pre-collision ones on exit.
//   G_b = P_b - omega (P_b - feq_b(rho, u)) + (1 - omega / 2) w_b s_b(u)
//   rho = sum P, u = (sum e P + g / 2) / rho, d u_i / d P_a = (e_ai - u_i) / rho
// With t_b = w_b a_b the sums over b are t0 = sum t, sr = sum t feq / (w rho),
// s_i = sum t (c e_i - 3 u_i) with c = 3 + 9 e.u, and f_i of the forcing.
template <typename A>
__device__ inline void collide_adjoint(A (&a)[Q], A rho, const A (&u)[3], const Device &dv) {
    const A om = AdjParams<A>::omega(dv);
    const A uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const A rest = (A)1 - (A)1.5 * uu;
    A t0 = 0, sr = 0, s0 = 0, s1 = 0, s2 = 0, f0 = 0, f1 = 0, f2 = 0;
#pragma unroll
    for (int b = 0; b < Q; ++b) {
        const A eu = plus(plus(plus((A)0, ex(b), u[0]), ey(b), u[1]), ez(b), u[2]);
        const A t = (A)wgt(b) * a[b];
        t0 += t;
        sr += t * (eu * ((A)4.5 * eu + (A)3) + rest);
        const A tc = t * ((A)9 * eu + (A)3);
        s0 = plus(s0, ex(b), tc);
        s1 = plus(s1, ey(b), tc);
        s2 = plus(s2, ez(b), tc);
        if (dv.forced) {
            const A te = t * AdjParams<A>::eg(dv, b);
            f0 = plus(f0, ex(b), te);
            f1 = plus(f1, ey(b), te);
            f2 = plus(f2, ez(b), te);
        }
    }
    s0 -= (A)3 * u[0] * t0;
    s1 -= (A)3 * u[1] * t0;
    s2 -= (A)3 * u[2] * t0;
    const A kf = AdjParams<A>::guo(dv);
    const A ir = (A)1 / rho;
    A su0 = om * s0, su1 = om * s1, su2 = om * s2;          // om rho s / rho
    if (dv.forced) {
        su0 += kf * ((A)9 * f0 - AdjParams<A>::g3(dv, 0) * t0) * ir;
        su1 += kf * ((A)9 * f1 - AdjParams<A>::g3(dv, 1) * t0) * ir;
        su2 += kf * ((A)9 * f2 - AdjParams<A>::g3(dv, 2) * t0) * ir;
    }
    const A base = om * sr - (su0 * u[0] + su1 * u[1] + su2 * u[2]);
    const A om1 = (A)1 - om;
#pragma unroll
    for (int b = 0; b < Q; ++b)
        a[b] = plus(plus(plus(om1 * a[b] + base, ex(b), su0), ey(b), su1), ez(b), su2);
}

// adjoint of the body-surface velocity u_w(p) = V + W x (p - X) for the
// scalar uh . u_w: acc[0..2] += d/dX, acc[3..5] += d/dV, acc[6..8] += d/dW
// (terms formed in S, summed in Acc)
template <typename S, typename Acc>
__device__ inline void adj_surface(const S W[3], const S o[3], const S uh[3], Acc acc[9]) {
    acc[0] += (Acc)(W[1] * uh[2] - W[2] * uh[1]);
    acc[1] += (Acc)(W[2] * uh[0] - W[0] * uh[2]);
    acc[2] += (Acc)(W[0] * uh[1] - W[1] * uh[0]);
    acc[3] += (Acc)uh[0]; acc[4] += (Acc)uh[1]; acc[5] += (Acc)uh[2];
    acc[6] += (Acc)(o[1] * uh[2] - o[2] * uh[1]);
    acc[7] += (Acc)(o[2] * uh[0] - o[0] * uh[2]);
    acc[8] += (Acc)(o[0] * uh[1] - o[1] * uh[0]);
}

// ---- bulk cells: pure gather + transposed collision -------------------------
// block `blk` of z-plane z: the plane's cells in row order, ADJ_THREADS a block
template <typename A, typename T, bool FIRST>
__device__ __forceinline__ void adj_bulk_cells(const Device &dv, const AdjPtrs &ap, int blk, int z) {
    const Domain &d = dv.dom;
    const unsigned nx = (unsigned)d.nx, q = (unsigned)blk * ADJ_THREADS + threadIdx.x;
    if (q >= nx * (unsigned)d.ny) return;
    unsigned r = __umulhi(q, ap.row_recip), xr = q - r * nx;         // row_recip: q / nx
    if (xr >= nx) {
        xr -= nx;
        ++r;
    }
    const int x = (int)xr, y = (int)r;
    const long long C = d.C;
    const unsigned c = ((unsigned)z * d.ny + y) * nx + xr;
    const uint8_t fn = ap.flags_next[c], fc = ap.flags_cur[c];
    const A *__restrict__ ain = static_cast<const A *>(ap.ain);
    const T *__restrict__ G = static_cast<const T *>(ap.G);
    A a[Q], g[Q];
    // sources x + e (wrapped; a cell whose neighbour lies beyond a wall is not a bulk cell)
    const int xs[3] = {x == 0 ? d.nx - 1 : x - 1, x, x == d.nx - 1 ? 0 : x + 1};
    const int ys[3] = {y == 0 ? d.ny - 1 : y - 1, y, y == d.ny - 1 ? 0 : y + 1};
    const int zs[3] = {z == 0 ? d.nz - 1 : z - 1, z, z == d.nz - 1 ? 0 : z + 1};
#pragma unroll
    for (int b = 0; b < Q; ++b)
        a[b] = ain[b * C + (((unsigned)zs[1 + ez(b)] * d.ny + ys[1 + ey(b)]) * nx + xs[1 + ex(b)])];
    if constexpr (!FIRST) {
#pragma unroll
        for (int b = 0; b < Q; ++b) g[b] = (A)G[b * C + c];
    }
    if ((fn & F_FULL_RULE) || (fc & F_SOLID_PREV)) return;           // the cube or wall kernel's
    if constexpr (!FIRST) {
        A rho, u[3];
        moments_post<A>(g, dv, rho, u);
        collide_adjoint<A>(a, rho, u, dv);
    }
    A *__restrict__ aout = static_cast<A *>(ap.aout);
#pragma unroll
    for (int b = 0; b < Q; ++b) aout[b * C + c] = a[b];
}

// ---- wall-face cells: the full rule, a thread per cell -----------------------
// Block row blockIdx.y = wall face (axis * 2 + side) of a non-periodic axis.
// The body terms of the links of these cells are summed by adj_cube_kernel
// (a face cell next to a body lies in its cube); this kernel writes the
// adjoint of every face cell.  A cell in both is written twice with the
// same rule, this kernel's last.
template <typename A, typename T, bool FIRST>
__global__ void __launch_bounds__(ADJ_BOUNDARY_THREADS) adj_wall_kernel(const Device dv, const AdjPtrs ap) {
    const Domain d = dv.dom;
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    int x = 0, y = 0, z = 0;
    bool live = true;
    {
        const int axis = blockIdx.y >> 1, hi = blockIdx.y & 1;
        const int n3[3] = {d.nx, d.ny, d.nz}, per[3] = {d.px, d.py, d.pz};
        if (per[axis]) return;
        const int ua = axis == 0 ? 1 : 0, va = axis == 2 ? 1 : 2;
        if (l >= n3[ua] * n3[va]) return;
        int p[3];
        p[axis] = hi ? n3[axis] - 1 : 0;
        p[ua] = l % n3[ua];
        p[va] = l / n3[ua];
        x = p[0]; y = p[1]; z = p[2];
    }
    const long long C = d.C;
    const long long c = ((long long)z * d.ny + y) * d.nx + x;
    if (live) {
        const uint8_t fcur = ap.flags_cur[c], fnext = ap.flags_next[c];
        if (!(fnext & F_FULL_RULE) && !(fcur & F_SOLID_PREV)) live = false;     // a bulk cell
        else if (fcur & F_SOLID) {                                    // obstacle at n: no adjoint
            A *aout = static_cast<A *>(ap.aout);
#pragma unroll
            for (int b = 0; b < Q; ++b) aout[(long long)b * C + c] = (A)0;
            if constexpr (!FIRST) static_cast<A *>(ap.rout)[c] = (A)0;
            live = false;
        }
        if (live) {
            const A *__restrict__ ain = static_cast<const A *>(ap.ain);
            const A *__restrict__ rin = static_cast<const A *>(ap.rin);
            const T *__restrict__ G = static_cast<const T *>(ap.G);
            A rho, u[3], gv[Q];
#pragma unroll
            for (int b = 0; b < Q; ++b) gv[b] = (A)G[(long long)b * C + c];
            moments_post<A>(gv, dv, rho, u);
            const bool fluid_next = !(fnext & F_SOLID);
            A own[Q], a[Q];
#pragma unroll
            for (int b = 0; b < Q; ++b) own[b] = ain[(long long)b * C + c];
            a[0] = own[0];
            A cr = 0;
#pragma unroll
            for (int b = 1; b < Q; ++b) {
                const int zx = x + ex(b), zy = y + ey(b), zz = z + ez(b);
                const bool wall = (!d.px && (zx < 0 || zx >= d.nx)) || (!d.py && (zy < 0 || zy >= d.ny)) ||
                                  (!d.pz && (zz < 0 || zz >= d.nz));
                if (wall) {                      // Eq. 4 at step n+1
                    a[b] = own[opp(b)];
                    continue;
                }
                const long long zc = ((long long)wrap_axis(zz, d.nz) * d.ny + wrap_axis(zy, d.ny)) * d.nx +
                                     wrap_axis(zx, d.nx);
                const uint8_t fz = ap.flags_cur[zc];
                if (fz & F_SOLID) {
                    // link (x, b) of step n: moving bounce-back of step n+1 and
                    // the momentum exchange of step n share u_w(x + e_b; S^n).
                    // The offset from the body centre is taken in FP64, the
                    // link's terms in the adjoint's precision.
                    const int k = ap.bid_cur[zc];
                    const BodyState &sk = ap.body[k];
                    double od[3];
                    offset_from(d, sk, (double)zx, (double)zy, (double)zz, od);
                    const A o[3] = {(A)od[0], (A)od[1], (A)od[2]};
                    const A W[3] = {(A)sk.W[0], (A)sk.W[1], (A)sk.W[2]};
                    A uw[3];
                    uw[0] = (A)sk.V[0] + (W[1] * o[2] - W[2] * o[1]);
                    uw[1] = (A)sk.V[1] + (W[2] * o[0] - W[0] * o[2]);
                    uw[2] = (A)sk.V[2] + (W[0] * o[1] - W[1] * o[0]);
                    const A ua = -((A)ex(b) * uw[0] + (A)ey(b) * uw[1] + (A)ez(b) * uw[2]);   // e_-b . u_w
                    A mh = 0;
                    if constexpr (!FIRST) {
                        const double *fa = ap.fadj + 6 * k;
                        // (mid - X) x e_b, mid = x + e_b / 2 = (x + e_b) - e_b / 2
                        const A m[3] = {o[0] - (A)(0.5 * ex(b)), o[1] - (A)(0.5 * ey(b)), o[2] - (A)(0.5 * ez(b))};
                        const A t0 = m[1] * (A)ez(b) - m[2] * (A)ey(b), t1 = m[2] * (A)ex(b) - m[0] * (A)ez(b),
                                t2 = m[0] * (A)ey(b) - m[1] * (A)ex(b);
                        mh = (A)ex(b) * (A)fa[0] + (A)ey(b) * (A)fa[1] + (A)ez(b) * (A)fa[2] + t0 * (A)fa[3] +
                             t1 * (A)fa[4] + t2 * (A)fa[5];
                    }
                    const A wh = own[opp(b)];
                    a[b] = wh + (A)2 * mh;
                    cr += (A)(6.0 * wgt(b)) * ua * (wh + mh);
                    // z uncovered at n+1: x (fluid at n and n+1) fed its density
                    if (!(ap.flags_next[zc] & F_SOLID) && fluid_next) cr += rin[zc];
                } else {
                    a[b] = ain[(long long)b * C + zc];
                }
            }
#pragma unroll
            for (int b = 0; b < Q; ++b) a[b] += cr;
            A *__restrict__ aout = static_cast<A *>(ap.aout);
            if constexpr (FIRST) {
#pragma unroll
                for (int b = 0; b < Q; ++b) aout[(long long)b * C + c] = a[b];
            } else {
                collide_adjoint<A>(a, rho, u, dv);
#pragma unroll
                for (int b = 0; b < Q; ++b) aout[(long long)b * C + c] = a[b];
                A rh_out = 0;
                if (fcur & F_SOLID_PREV) {
                    // uncovered at n: P = f_eq(rho_avg, u_w(x; S^n)) of the body
                    // that covered x at n-1, rho_avg over the neighbours fluid
                    // in epochs n-1 and n (rho_avg = rho^n(x))
                    int cnt = 0;
#pragma unroll
                    for (int b = 1; b < Q; ++b) {
                        const int nx_ = x + ex(b), ny_ = y + ey(b), nz_ = z + ez(b);
                        const bool in = !((!d.px && (nx_ < 0 || nx_ >= d.nx)) || (!d.py && (ny_ < 0 || ny_ >= d.ny)) ||
                                          (!d.pz && (nz_ < 0 || nz_ >= d.nz)));
                        const long long nc = ((long long)wrap_axis(nz_, d.nz) * d.ny + wrap_axis(ny_, d.ny)) * d.nx +
                                             wrap_axis(nx_, d.nx);
                        if (in && !(ap.flags_cur[nc] & (F_SOLID | F_SOLID_PREV))) ++cnt;
                    }
                    const int k = ap.bid_prev[c];
                    if (k != NO_BODY) {
                        const BodyState sk = ap.body[k];
                        double o[3], uw[3];
                        offset_from(d, sk, (double)x, (double)y, (double)z, o);
                        uw[0] = sk.V[0] + (sk.W[1] * o[2] - sk.W[2] * o[1]);
                        uw[1] = sk.V[1] + (sk.W[2] * o[0] - sk.W[0] * o[2]);
                        uw[2] = sk.V[2] + (sk.W[0] * o[1] - sk.W[1] * o[0]);
                        const double uu = uw[0] * uw[0] + uw[1] * uw[1] + uw[2] * uw[2];
                        double rh = 0.0;
#pragma unroll
                        for (int b = 0; b < Q; ++b) {
                            const double eu = ex(b) * uw[0] + ey(b) * uw[1] + ez(b) * uw[2];
                            rh += (double)a[b] * wgt(b) * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu);
                        }
                        if (cnt) rh_out = (A)(rh / cnt);
                    }
                }
                static_cast<A *>(ap.rout)[c] = rh_out;
            }
        }
    }
}

// ---- boundary cells of the body cubes: a warp per cell -------------------------
// Block (blk, kb) classifies ADJ_BOUNDARY_THREADS cells of body kb's cube, every
// gridDim.x-th from blk (the full-rule cells are a shell, which consecutive cells
// would leave to a few blocks: 27.8 against 13.3 us a launch on the 96 x 48 x 48
// study) (cells whose flags are zero in epochs n and n+1 and that
// were not uncovered at n: adj_bulk_cells'; solid at n: zero adjoint; the
// others the full rule, as adj_wall_kernel applies it) and lists the full-rule cells
// in cube order.  Each warp then takes the listed cells w, w + 8, ... with
// lane b the direction b: the pull, wall and link terms of the 18
// directions in parallel, the cell's sums (the density terms, the
// transposed collision's moments, the refill sums, body kb's terms) by
// butterfly shuffles, so every lane holds the same sum and the order is
// fixed.  The block adds its warps' body sums in warp order into
// part[kb][blk] (the layout adj_integrate reads).
constexpr int ADJ_CUBE_WARPS = 8;

// the sums of v[0..3] over the warp, in every lane: halves exchange values (lane
// bit 4: the first or last two, bit 3: one of them), then three butterfly steps
template <typename V> __device__ __forceinline__ void warp_sum4(V (&v)[4]) {
    constexpr unsigned FULL = 0xffffffffu;
    const bool hi = threadIdx.x & 16, odd = threadIdx.x & 8;
    const V k0 = hi ? v[2] : v[0], k1 = hi ? v[3] : v[1], o0 = hi ? v[0] : v[2], o1 = hi ? v[1] : v[3];
    const V a0 = k0 + __shfl_xor_sync(FULL, o0, 16), a1 = k1 + __shfl_xor_sync(FULL, o1, 16);
    V a = (odd ? a1 : a0) + __shfl_xor_sync(FULL, odd ? a0 : a1, 8);
    a += __shfl_xor_sync(FULL, a, 4);
    a += __shfl_xor_sync(FULL, a, 2);
    a += __shfl_xor_sync(FULL, a, 1);
    v[0] = __shfl_sync(FULL, a, 0);
    v[1] = __shfl_sync(FULL, a, 8);
    v[2] = __shfl_sync(FULL, a, 16);
    v[3] = __shfl_sync(FULL, a, 24);
}

template <typename V> __device__ __forceinline__ V warp_sum(V v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// a centre's cell, wrapped into the domain on periodic axes, and its position
// within it, as a value in A and the rest
template <typename A>
__device__ __forceinline__ void centre_cell(const Domain &d, const double (&X)[3], int (&ci)[3], A (&cf)[3], A (&cr)[3]) {
    const int n3[3] = {d.nx, d.ny, d.nz}, per[3] = {d.px, d.py, d.pz};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double f = floor(X[i]);
        ci[i] = (int)f;
        if (per[i]) ci[i] = ((ci[i] % n3[i]) + n3[i]) % n3[i];
        const double in = X[i] - f;
        cf[i] = (A)in;
        cr[i] = (A)(in - (double)cf[i]);
    }
}

// i - (c + r) rounded once to A: the difference's own rounding error (TwoSum) joins the rest
template <typename A> __device__ __forceinline__ A cell_offset(int i, A c, A r) {
    if constexpr (sizeof(A) == 8) return (A)i - c;
    const A a = (A)i, s = a - c, t = s - a;
    return s + (((a - (s - t)) - (c + t)) - r);
}

template <typename A, typename T, bool FIRST>
__global__ void __launch_bounds__(32 * ADJ_CUBE_WARPS) adj_cube_kernel(const Device dv, const AdjPtrs ap) {
    const Domain d = dv.dom;
    const int kb = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long C = d.C;
    const int half = dv.props[kb].E + REMAP_MARGIN;
    const int side = 2 * half + 1;
    const BodyState &sb = ap.body[kb];
    const int fx = (int)floor(sb.X[0]), fy = (int)floor(sb.X[1]), fz = (int)floor(sb.X[2]);
    int ci[3];
    A cf[3], cr[3];
    centre_cell(d, sb.X, ci, cf, cr);
    // cube cell l -> lattice cell (x, y, z); false outside the cube or the domain
    auto cube_cell = [&](int l, int &x, int &y, int &z) {
        if (l >= side * side * side) return false;
        bool live = true;
        x = fx - half + l % side;
        y = fy - half + (l / side) % side;
        z = fz - half + l / (side * side);
        if (d.px) x = ((x % d.nx) + d.nx) % d.nx; else live = live && x >= 0 && x < d.nx;
        if (d.py) y = ((y % d.ny) + d.ny) % d.ny; else live = live && y >= 0 && y < d.ny;
        if (d.pz) z = ((z % d.nz) + d.nz) % d.nz; else live = live && z >= 0 && z < d.nz;
        return live;
    };
    __shared__ int list[ADJ_BOUNDARY_THREADS];
    __shared__ int wcount[ADJ_BOUNDARY_THREADS / 32];
    __shared__ double wacc[ADJ_CUBE_WARPS][9];
    A *__restrict__ aout = static_cast<A *>(ap.aout);
    // 1. classify this block's cells (the first ADJ_BOUNDARY_THREADS threads)
    bool listed = false;
    const int l = blockIdx.x + tid * gridDim.x;
    if (tid < ADJ_BOUNDARY_THREADS) {
        int x, y, z;
        if (cube_cell(l, x, y, z)) {
            const long long c = ((long long)z * d.ny + y) * d.nx + x;
            const uint8_t fcur = ap.flags_cur[c], fnext = ap.flags_next[c];
            if (!(fnext & F_FULL_RULE) && !(fcur & F_SOLID_PREV)) {
                // a bulk cell: adj_bulk_cells'
            } else if (fcur & F_SOLID) {            // obstacle at n: no adjoint
#pragma unroll
                for (int b = 0; b < Q; ++b) aout[(long long)b * C + c] = (A)0;
                if constexpr (!FIRST) static_cast<A *>(ap.rout)[c] = (A)0;
            } else {
                listed = true;
            }
        }
    }
    unsigned lm = 0;                                 // the warp's listed lanes
    if (warp < ADJ_BOUNDARY_THREADS / 32) {
        lm = __ballot_sync(0xffffffffu, listed);
        if (lane == 0) wcount[warp] = __popc(lm);
    }
    __syncthreads();
    if (listed) {
        int base = 0;
        for (int w = 0; w < warp; ++w) base += wcount[w];
        list[base + __popc(lm & ((1u << lane) - 1u))] = l;
    }
    int nlist = 0;
    for (int w = 0; w < ADJ_BOUNDARY_THREADS / 32; ++w) nlist += wcount[w];
    __syncthreads();
    // 2. a warp per listed cell, lane b = direction b
    const bool act = lane < Q;
    const int b = act ? lane : 0;
    const int bx = ex(b), by = ey(b), bz = ez(b), ob = opp(b);
    const A wb = (A)wgt(b);
    const A *__restrict__ ain = static_cast<const A *>(ap.ain);
    const A *__restrict__ rin = static_cast<const A *>(ap.rin);
    const T *__restrict__ G = static_cast<const T *>(ap.G);
    A acc[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};         // this lane's body-kb terms over the warp's cells
    // body kb's velocities and load adjoint in A, once a warp
    const A V0[3] = {(A)sb.V[0], (A)sb.V[1], (A)sb.V[2]}, W0[3] = {(A)sb.W[0], (A)sb.W[1], (A)sb.W[2]};
    A fa0[6] = {0, 0, 0, 0, 0, 0};
    if constexpr (!FIRST)
        for (int i = 0; i < 6; ++i) fa0[i] = (A)ap.fadj[6 * kb + i];
    const A eg = dv.forced ? AdjParams<A>::eg(dv, b) : (A)0;
    const A g30 = AdjParams<A>::g3(dv, 0), g31 = AdjParams<A>::g3(dv, 1), g32 = AdjParams<A>::g3(dv, 2);
    const A hg0 = AdjParams<A>::half_g(dv, 0), hg1 = AdjParams<A>::half_g(dv, 1), hg2 = AdjParams<A>::half_g(dv, 2);
    for (int e = warp; e < nlist; e += ADJ_CUBE_WARPS) {
        int x, y, z;
        cube_cell(list[e], x, y, z);
        const long long c = ((long long)z * d.ny + y) * d.nx + x;
        const uint8_t fcur = ap.flags_cur[c], fnext = ap.flags_next[c];
        const bool fluid_next = !(fnext & F_SOLID);
        // density and velocity of step n from the post-collision populations
        const A gv = act ? (A)G[(long long)b * C + c] : (A)0;
        A m[4] = {gv, (A)bx * gv, (A)by * gv, (A)bz * gv};
        warp_sum4(m);
        const A rho = (A)1 + m[0];
        const A ir = (A)1 / rho;
        const A u0 = (m[1] - hg0) * ir, u1 = (m[2] - hg1) * ir, u2 = (m[3] - hg2) * ir;
        const A own = act ? ain[(long long)b * C + c] : (A)0;
        const A own_opp = __shfl_sync(0xffffffffu, own, ob);
        A a = own, crb = 0;
        if (act && b > 0) {
            const int zx = x + bx, zy = y + by, zz = z + bz;
            const bool wall = (!d.px && (zx < 0 || zx >= d.nx)) || (!d.py && (zy < 0 || zy >= d.ny)) ||
                              (!d.pz && (zz < 0 || zz >= d.nz));
            if (wall) {                              // Eq. 4 at step n+1
                a = own_opp;
            } else {
                const long long zc = ((long long)wrap_axis(zz, d.nz) * d.ny + wrap_axis(zy, d.ny)) * d.nx +
                                     wrap_axis(zx, d.nx);
                const uint8_t fzc = ap.flags_cur[zc];
                const int k = ap.bid_cur[zc];
                const A pulled = ain[(long long)b * C + zc];
                if (fzc & F_SOLID) {
                    // link (x, b) of step n: moving bounce-back of step n+1 and
                    // the momentum exchange of step n share u_w(x + e_b; S^n);
                    // the offset from the centre is an integer difference of
                    // cells less the centre's position within its cell, rounded once (the same
                    // expression for every body: a cell in two cubes is written
                    // by both blocks), the terms in A
                    const BodyState &sk = ap.body[k];
                    int kc[3] = {ci[0], ci[1], ci[2]};
                    A kf[3] = {cf[0], cf[1], cf[2]}, kr[3] = {cr[0], cr[1], cr[2]};
                    if (k != kb) centre_cell(d, sk.X, kc, kf, kr);
                    A o[3];
                    const int zp[3] = {wrap_axis(zx, d.nx), wrap_axis(zy, d.ny), wrap_axis(zz, d.nz)};
                    const int n3[3] = {d.nx, d.ny, d.nz}, per[3] = {d.px, d.py, d.pz};
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        int io = zp[i] - kc[i];
                        if (per[i]) io = 2 * io > n3[i] ? io - n3[i] : (2 * io < -n3[i] ? io + n3[i] : io);
                        o[i] = cell_offset(io, kf[i], kr[i]);
                    }
                    A W[3] = {W0[0], W0[1], W0[2]}, V[3] = {V0[0], V0[1], V0[2]};
                    A fa[6] = {fa0[0], fa0[1], fa0[2], fa0[3], fa0[4], fa0[5]};
                    if (k != kb) {
                        for (int i = 0; i < 3; ++i) {
                            W[i] = (A)sk.W[i];
                            V[i] = (A)sk.V[i];
                        }
                        if constexpr (!FIRST)
                            for (int i = 0; i < 6; ++i) fa[i] = (A)ap.fadj[6 * k + i];
                    }
                    const A uw0 = V[0] + (W[1] * o[2] - W[2] * o[1]);
                    const A uw1 = V[1] + (W[2] * o[0] - W[0] * o[2]);
                    const A uw2 = V[2] + (W[0] * o[1] - W[1] * o[0]);
                    const A ua = -((A)bx * uw0 + (A)by * uw1 + (A)bz * uw2);     // e_-b . u_w
                    A mh = 0;
                    if constexpr (!FIRST) {
                        // (mid - X) x e_b, mid = x + e_b / 2 = (x + e_b) - e_b / 2
                        const A m0 = o[0] - (A)(0.5 * bx), m1 = o[1] - (A)(0.5 * by), m2 = o[2] - (A)(0.5 * bz);
                        const A t0 = m1 * (A)bz - m2 * (A)by, t1 = m2 * (A)bx - m0 * (A)bz, t2 = m0 * (A)by - m1 * (A)bx;
                        mh = (A)bx * fa[0] + (A)by * fa[1] + (A)bz * fa[2] + t0 * fa[3] + t1 * fa[4] + t2 * fa[5];
                    }
                    const A wh = own_opp;
                    a = wh + (A)2 * mh;
                    crb = (A)6 * wb * ua * (wh + mh);
                    if (k == kb) {
                        const A sc = (A)6 * wb * rho * (wh + mh);
                        const A uh[3] = {-(A)bx * sc, -(A)by * sc, -(A)bz * sc};
                        adj_surface<A, A>(W, o, uh, acc);
                    }
                    // z uncovered at n+1: x (fluid at n and n+1) fed its density
                    if (!(ap.flags_next[zc] & F_SOLID) && fluid_next) crb += rin[zc];
                } else {
                    a = pulled;
                }
            }
        }
        a += warp_sum(crb);
        if constexpr (FIRST) {
            if (act) aout[(long long)b * C + c] = a;
        } else {
            // the transposed collision (collide_adjoint), its sums over the lanes
            const A om = AdjParams<A>::omega(dv);
            const A uu = u0 * u0 + u1 * u1 + u2 * u2;
            const A eu = (A)bx * u0 + (A)by * u1 + (A)bz * u2;
            const A wa = act ? wb * a : (A)0;
            const A cc = (A)3 + (A)9 * eu;
            A t4[4] = {wa * ((A)1 + (A)3 * eu + (A)4.5 * eu * eu - (A)1.5 * uu), wa * (cc * (A)bx - (A)3 * u0),
                       wa * (cc * (A)by - (A)3 * u1), wa * (cc * (A)bz - (A)3 * u2)};
            warp_sum4(t4);
            const A sr = t4[0], s0 = t4[1], s1 = t4[2], s2 = t4[3];
            A f0 = 0, f1 = 0, f2 = 0;
            if (dv.forced) {
                A f4[4] = {wa * ((A)9 * (A)bx * eg - g30), wa * ((A)9 * (A)by * eg - g31), wa * ((A)9 * (A)bz * eg - g32), (A)0};
                warp_sum4(f4);
                f0 = f4[0]; f1 = f4[1]; f2 = f4[2];
            }
            const A kf = AdjParams<A>::guo(dv);
            const A su0 = (om * rho * s0 + kf * f0) * ir, su1 = (om * rho * s1 + kf * f1) * ir,
                    su2 = (om * rho * s2 + kf * f2) * ir;
            const A base = om * sr - (su0 * u0 + su1 * u1 + su2 * u2);
            a = ((A)1 - om) * a + base + (A)bx * su0 + (A)by * su1 + (A)bz * su2;
            if (act) aout[(long long)b * C + c] = a;
            A rh_out = 0;
            if (fcur & F_SOLID_PREV) {
                // uncovered at n: P = f_eq(rho_avg, u_w(x; S^n)) of the body
                // that covered x at n-1, rho_avg over the neighbours fluid in
                // epochs n-1 and n (rho_avg = rho^n(x))
                bool nf = false;
                if (act && b > 0) {
                    const int nx_ = x + bx, ny_ = y + by, nz_ = z + bz;
                    const bool in = !((!d.px && (nx_ < 0 || nx_ >= d.nx)) || (!d.py && (ny_ < 0 || ny_ >= d.ny)) ||
                                      (!d.pz && (nz_ < 0 || nz_ >= d.nz)));
                    const long long nc = ((long long)wrap_axis(nz_, d.nz) * d.ny + wrap_axis(ny_, d.ny)) * d.nx +
                                         wrap_axis(nx_, d.nx);
                    nf = in && !(ap.flags_cur[nc] & (F_SOLID | F_SOLID_PREV));
                }
                const int cnt = __popc(__ballot_sync(0xffffffffu, nf));
                const int k = ap.bid_prev[c];
                if (k != NO_BODY) {
                    const BodyState &sk = ap.body[k];
                    double o[3], uw[3];
                    offset_from(d, sk, (double)x, (double)y, (double)z, o);
                    uw[0] = sk.V[0] + (sk.W[1] * o[2] - sk.W[2] * o[1]);
                    uw[1] = sk.V[1] + (sk.W[2] * o[0] - sk.W[0] * o[2]);
                    uw[2] = sk.V[2] + (sk.W[0] * o[1] - sk.W[1] * o[0]);
                    const double uuw = uw[0] * uw[0] + uw[1] * uw[1] + uw[2] * uw[2];
                    const double rho_d = (double)rho;
                    const double euw = bx * uw[0] + by * uw[1] + bz * uw[2];
                    const double pa = act ? (double)a * wgt(b) : 0.0;
                    const double cw = rho_d * (3.0 + 9.0 * euw);
                    const double rh = warp_sum(pa * (1.0 + 3.0 * euw + 4.5 * euw * euw - 1.5 * uuw));
                    const double uh[3] = {warp_sum(pa * (cw * bx - 3.0 * rho_d * uw[0])),
                                          warp_sum(pa * (cw * by - 3.0 * rho_d * uw[1])),
                                          warp_sum(pa * (cw * bz - 3.0 * rho_d * uw[2]))};
                    if (cnt) rh_out = (A)(rh / cnt);
                    if (k == kb && lane == 0) adj_surface<double, A>(sk.W, o, uh, acc);
                }
            }
            if (lane == 0) static_cast<A *>(ap.rout)[c] = rh_out;
        }
    }
    // 3. the block's body-kb sums, warps in order
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const A v = warp_sum(acc[i]);
        if (lane == 0) wacc[warp][i] = (double)v;
    }
    __syncthreads();
    if (tid < 9) {
        double v = 0.0;
        for (int w = 0; w < ADJ_CUBE_WARPS; ++w) v += wacc[w][tid];
        ap.part[((long long)kb * ap.part_stride + blockIdx.x) * 9 + tid] = v;
    }
}

// ---- rigid-body step, reversed ------------------------------------------------
// Reverse of Algorithm 1 at step t with the state S^n and the hydrodynamic
// load fh^n of the tape:
//   V' = V + F / m, X' = X + V', W' = W + R diag(1/I) R^T T,
//   q' = normalise(q + (0, W') q / 2),
//   F = F_hydro + g vol + sum_d amp_d sin(omega_d t - phase_d) R a_d + springs.
// The terms that depend only on S^n and fh^n (R, F, R^T T, W', q', the drive
// sines, the spring geometry) are made for every step of a segment by
// adj_terms_kernel, a thread per body, drive term or spring and step; the
// serial kernel adj_integrate does the rest, linear in the adjoint.

// state-only terms of steps t0 .. t0 + L - 1: thread (j, i) with i < nb a
// body, then the drive terms, then the springs
__global__ void __launch_bounds__(ADJ_THREADS)
adj_terms_kernel(const Device dv, const BodyState *states, const double *fhs, long long t0, int L,
                 AdjBodyTerms *tb, AdjDriveTerms *td, AdjSpringTerms *ts) {
    const int per = dv.nb + dv.nd + dv.ns;
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (long long)L * per) return;
    const int j = (int)(id / per), i = (int)(id % per);
    const BodyState *S = states + (long long)j * dv.nb;
    const double tt = (double)(t0 + j);
    auto drive_value = [&](const DriveTerm &dt, double &sn_, double &cs) {
        sn_ = 0.0;
        cs = 0.0;
        if (tt < dt.t_on || tt >= dt.t_off) return 0.0;
        sincos(dt.omega * tt - dt.phase, &sn_, &cs);
        return dt.amp * sn_;
    };
    if (i < dv.nb) {
        const int b = i;
        const BodyProps pb = dv.props[b];
        const BodyState st = S[b];
        const double *fh = fhs + ((long long)j * dv.nb + b) * 6;
        double R[3][3];
        quat_to_matrix(st.q, R);
        // F: the hydrodynamic force, g times the volume, the body's drive
        // terms in term order and its springs in spring order (the order
        // of the forward's sums)
        double F[3];
        for (int a = 0; a < 3; ++a) F[a] = fh[a] + dv.g[a] * pb.volume;
        for (int k = pb.drive_first; k < pb.drive_first + pb.drive_count; ++k) {
            const DriveTerm dt = dv.drives[k];
            double sn_, cs;
            const double f = drive_value(dt, sn_, cs);
            for (int a = 0; a < 3; ++a)
                F[a] += f * (R[a][0] * dt.axis[0] + R[a][1] * dt.axis[1] + R[a][2] * dt.axis[2]);
        }
        for (int kk = pb.spring_first; kk < pb.spring_first + pb.spring_count; ++kk) {
            const int k = dv.spring_list[kk];
            const Spring sp_ = dv.springs[k];
            const BodyState si = S[sp_.i], sj = S[sp_.j];
            const double dd[3] = {si.X[0] - sj.X[0], si.X[1] - sj.X[1], si.X[2] - sj.X[2]};
            const double len = sqrt(dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2]);
            const double inv_len = len > 0 ? 1.0 / len : 0.0;
            for (int a = 0; a < 3; ++a) {
                const double f = -sp_.k * (len - sp_.rest) * (dd[a] * inv_len) - sp_.gamma * (si.V[a] - sj.V[a]);
                F[a] += sp_.i == b ? f : -f;
            }
        }
        const double *T = fh + 3;
        double beta[3], W1[3];
        for (int a = 0; a < 3; ++a) beta[a] = R[0][a] * T[0] + R[1][a] * T[1] + R[2][a] * T[2];
        for (int a = 0; a < 3; ++a)
            W1[a] = st.W[a] + (R[a][0] * beta[0] * pb.inv_inertia[0] + R[a][1] * beta[1] * pb.inv_inertia[1] +
                               R[a][2] * beta[2] * pb.inv_inertia[2]);
        const double w = st.q[0], v0 = st.q[1], v1 = st.q[2], v2 = st.q[3];
        const double c0 = W1[1] * v2 - W1[2] * v1, c1 = W1[2] * v0 - W1[0] * v2, c2 = W1[0] * v1 - W1[1] * v0;
        const double q4[4] = {w - 0.5 * (W1[0] * v0 + W1[1] * v1 + W1[2] * v2), v0 + 0.5 * (w * W1[0] + c0),
                              v1 + 0.5 * (w * W1[1] + c1), v2 + 0.5 * (w * W1[2] + c2)};
        const double inv_nn = rsqrt(q4[0] * q4[0] + q4[1] * q4[1] + q4[2] * q4[2] + q4[3] * q4[3]);
        AdjBodyTerms o;
        for (int r = 0; r < 3; ++r)
            for (int c = 0; c < 3; ++c) o.R[3 * r + c] = R[r][c];
        for (int a = 0; a < 3; ++a) {
            o.F[a] = F[a];
            o.beta[a] = beta[a];
            o.W1[a] = W1[a];
        }
        for (int a = 0; a < 4; ++a) o.q1[a] = q4[a] * inv_nn;
        o.inv_nn = inv_nn;
        tb[(long long)j * dv.nb + b] = o;
    } else if (i < dv.nb + dv.nd) {
        const int k = i - dv.nb;
        const DriveTerm dt = dv.drives[k];
        AdjDriveTerms o;
        o.f = drive_value(dt, o.sn, o.cs);
        double R[3][3];
        quat_to_matrix(S[dt.body].q, R);
        for (int a = 0; a < 3; ++a) o.aw[a] = R[a][0] * dt.axis[0] + R[a][1] * dt.axis[1] + R[a][2] * dt.axis[2];
        td[(long long)j * dv.nd + k] = o;
    } else {
        const int k = i - dv.nb - dv.nd;
        const Spring sp_ = dv.springs[k];
        const BodyState si = S[sp_.i], sj = S[sp_.j];
        const double dd[3] = {si.X[0] - sj.X[0], si.X[1] - sj.X[1], si.X[2] - sj.X[2]};
        const double len = sqrt(dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2]);
        AdjSpringTerms o;
        o.len = len;
        o.ratio = len > 0 ? (len - sp_.rest) / len : 0.0;
        for (int a = 0; a < 3; ++a) {
            o.dir[a] = len > 0 ? dd[a] / len : 0.0;
            o.dv[a] = si.V[a] - sj.V[a];
        }
        ts[(long long)j * dv.ns + k] = o;
    }
}

// Sh^{n+1} = sa_next + the cell sums of reverse step n+1 (part, a fixed order); then the reverse step with the state-only terms
// of step n.  Writes Sh^n (rigid-body part plus the lever-arm term Th x
// F_hydro of the torque sum) to sa_cur, (Fh, Th) to fadj and adds
// dJ/dtheta.  A warp a body with components on lanes (axes, quaternion and matrix
// entries): an FP64 warp instruction costs ~64 issue cycles whatever its lanes
// carry, and this kernel is on the sweep's serial chain (a thread a body
// took 19.8 us a launch for three bodies, this takes 11.4).  Past eight bodies the
// bodies are dealt to several blocks, and the last of them to finish (ab.done)
// does the drive terms and springs.  In one block the bodies' rounds of eight cost
// more than the thread-a-body form from about 100 bodies on; a reverse step of 100
// and 200 spheres of radius 3 (FP32, 96^3 and 120 x 96 x 96 cells) took 363 and
// 662 us so, 351 and 584 us with a thread a body, 266 and 454 us with blocks.
constexpr int ADJ_WARPS = ADJ_THREADS / 32;
constexpr int ADJ_AXIS_GROUPS = 32 / 3;     // bodies a warp takes side by side, three axes each
__host__ __device__ inline int adj_integrate_blocks(int nb) { return (nb + ADJ_WARPS - 1) / ADJ_WARPS; }
constexpr int ADJ_SUM_GROUPS = 3;           // records a warp's lanes take side by side, nine sums each

__device__ __forceinline__ void adj_integrate(const Device &dv, const AdjBody &ab, int blk, int blocks) {
    constexpr unsigned FULL = 0xffffffffu;
    const int nb = dv.nb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ double s_sum[ADJ_WARPS][9];
    __shared__ double s_F[LBM_MAX_BODIES_DEV][3];       // Fh of every body
    __shared__ int s_last;
    const int ax = lane < 3 ? lane : 0, i1 = (ax + 1) % 3, i2 = (ax + 2) % 3;
    auto at = [](double v, int l) { return __shfl_sync(FULL, v, l); };
    // warps that share a body's cell sums
    const int share = nb <= 2 ? 4 : (nb <= 4 ? 2 : 1);
    const int bodies = ADJ_WARPS / share;               // bodies in flight
    for (int b0 = blk * bodies; b0 < nb; b0 += blocks * bodies) {
        // 1. complete Sh^{n+1}: lane 9 g + c of each of the body's warps adds
        //    component c of every (share x groups)-th record
        const int b = b0 + warp % bodies, part = warp / bodies;
        if (b < nb) {
            double v = 0.0;
            if (lane < 9 * ADJ_SUM_GROUPS) {
                const double *p = ab.part + (long long)b * ab.part_stride * 9 + lane % 9;
                const int step = share * ADJ_SUM_GROUPS;
                int k = part * ADJ_SUM_GROUPS + lane / 9;
                for (; k + 3 * step < ab.part_count; k += 4 * step) {
                    const double q0 = p[9 * k], q1 = p[9 * (k + step)], q2 = p[9 * (k + 2 * step)],
                                 q3 = p[9 * (k + 3 * step)];
                    v += q0; v += q1; v += q2; v += q3;
                }
                for (; k < ab.part_count; k += step) v += p[9 * k];
            }
            const double w = v + at(v, lane + 9 < 32 ? lane + 9 : lane) + at(v, lane + 18 < 32 ? lane + 18 : lane);
            if (lane < 9) s_sum[warp][lane] = w;
        }
        __syncthreads();
        if (part == 0 && b < nb) {
            const BodyProps *pb = dv.props + b;
            const double *st = reinterpret_cast<const double *>(ab.state + b);
            const AdjBodyTerms *tm = ab.tb + b;
            const double *fh = ab.fh + 6 * b;
            // loads: the adjoint of state n + 1 (lane i < 13 component i), the terms
            double sn = lane < 13 ? ab.sa_next[13 * b + lane] : 0.0;
            const int c4 = lane < 4 ? lane : 0;
            const double q1 = tm->q1[c4], q4s = st[3 + c4], inv_nn = tm->inv_nn;
            const double W1 = tm->W1[ax], beta = tm->beta[ax], F = tm->F[ax], inv_I = pb->inv_inertia[ax];
            const double R0i = tm->R[ax], R1i = tm->R[3 + ax], R2i = tm->R[6 + ax];         // column ax
            const double Ri0 = tm->R[3 * ax], Ri1 = tm->R[3 * ax + 1], Ri2 = tm->R[3 * ax + 2];
            const double fhF = fh[ax], fhT = fh[3 + ax], inv_m = pb->inv_m, g = dv.g[ax];
            const int d0 = pb->drive_first, d1 = d0 + pb->drive_count;
            // the cell sums: X, V, W of components 0..2, 7..9, 10..12
            {
                const int c = lane < 3 ? lane : (lane >= 7 && lane < 13 ? lane - 4 : -1);
                if (c >= 0) {
                    double v = s_sum[warp][c];
                    for (int k = 1; k < share; ++k) v += s_sum[warp + k * bodies][c];
                    sn += v;
                    ab.sa_next[13 * b + lane] = sn;
                }
            }
            // quaternion: qh4 = (qh - q1 (q1 . qh)) / |q|
            const double qh = at(sn, 3 + c4);
            double dot = q1 * qh;
            dot += __shfl_xor_sync(FULL, dot, 1);
            dot += __shfl_xor_sync(FULL, dot, 2);
            const double qh4 = (qh - q1 * dot) * inv_nn;
            const double h0 = at(qh4, 0), hv0 = at(qh4, 1), hv1 = at(qh4, 2), hv2 = at(qh4, 3);
            auto hv = [&](int i) { return i == 0 ? hv0 : (i == 1 ? hv1 : hv2); };
            const double Wa = at(W1, 0), Wb = at(W1, 1), Wc = at(W1, 2);
            auto Wv = [&](int i) { return i == 0 ? Wa : (i == 1 ? Wb : Wc); };
            const double w = at(q4s, 0), va = at(q4s, 1), vb = at(q4s, 2), vc = at(q4s, 3);
            auto vv = [&](int i) { return i == 0 ? va : (i == 1 ? vb : vc); };
            // the adjoint of q_n through the update: lane 0 the scalar part,
            // lane 1 + i the vector component i
            double qout;
            {
                const int i = lane >= 1 && lane <= 3 ? lane - 1 : 0, j = (i + 1) % 3, k = (i + 2) % 3;
                const bool s0 = lane == 0;
                const double p1 = s0 ? hv(0) : -h0, r1 = s0 ? Wv(0) : Wv(i);
                const double p2 = s0 ? hv(1) : hv(j), r2 = s0 ? Wv(1) : Wv(k);
                const double p3 = s0 ? hv(2) : -hv(k), r3 = s0 ? Wv(2) : Wv(j);
                qout = (s0 ? h0 : hv(i)) + 0.5 * (p1 * r1 + p2 * r2 + p3 * r3);
            }
            // Omega: Wh1 = Wh + 1/2 (w qv - qh0 v + v x qv), lanes 0..2
            const double Wh1 = at(sn, 10 + ax) + 0.5 * (w * hv(ax) - h0 * vv(ax) + vv(i1) * hv(i2) - vv(i2) * hv(i1));
            const double w0 = at(Wh1, 0), w1 = at(Wh1, 1), w2 = at(Wh1, 2);
            const double alpha = R0i * w0 + R1i * w1 + R2i * w2;
            const double aI = alpha * inv_I;
            const double a0 = at(aI, 0), a1 = at(aI, 1), a2 = at(aI, 2);
            const double Th = Ri0 * a0 + Ri1 * a1 + Ri2 * a2;
            // translation
            const double snx = at(sn, ax), vh1 = at(sn, 7 + ax) + snx;
            const double Fh = vh1 * inv_m;
            double F2 = vh1 * F, gv = g * Fh;
            F2 = at(F2, 0) + at(F2, 1) + at(F2, 2);
            gv = at(gv, 0) + at(gv, 1) + at(gv, 2);
            // lever arm of the torque sum: T = sum (mid - X) x F_link
            const double xout = snx + (at(Th, i1) * at(fhF, i2) - at(Th, i2) * at(fhF, i1));
            // Rh_ij = Wh1_i beta_j / I_j + T_i alpha_j / I_j on lane 3 i + j, and the
            // drive terms (F = f R a: dF_i / dR_ij = f a_j)
            const int ri = lane < 9 ? lane / 3 : 0, rj = lane < 9 ? lane % 3 : 0;
            const double bI = beta * inv_I;
            double Rh = at(Wh1, ri) * at(bI, rj) + at(fhT, ri) * at(aI, rj);
            const double Fi = at(Fh, ri);
            for (int k = d0; k < d1; ++k) Rh += ab.td[k].f * Fi * dv.drives[k].axis[rj];     // f: zero outside the window
            // the adjoint of R(q): antisymmetric, symmetric and diagonal pairs of Rh
            // on lanes 0..2, 3..5, 6..8, then a component of q a lane
            const double c0 = at(Rh, lane == 0 ? 7 : lane == 1 ? 2 : lane == 2 ? 3 : lane == 3 ? 1 : lane == 4 ? 2 : lane == 5 ? 5
                                  : lane == 6 ? 4 : 0);
            const double c1 = at(Rh, lane == 0 ? 5 : lane == 1 ? 6 : lane == 2 ? 1 : lane == 3 ? 3 : lane == 4 ? 6 : lane == 5 ? 7
                                  : lane == 8 ? 4 : 8);
            const double pr = lane < 3 ? c0 - c1 : c0 + c1;
            const double A0 = at(pr, 0), A1 = at(pr, 1), A2 = at(pr, 2), S01 = at(pr, 3), S02 = at(pr, 4), S12 = at(pr, 5),
                         Dx = at(pr, 6), Dy = at(pr, 7), Dz = at(pr, 8);
            {
                const double p0 = lane == 0 ? A0 : lane == 1 ? S01 : lane == 2 ? S01 : S02;
                const double r0 = lane == 0 ? va : lane == 1 ? vb : va;
                const double p1 = lane == 0 ? A1 : lane == 1 ? S02 : S12;
                const double r1 = lane == 0 ? vb : lane == 3 ? vb : vc;
                const double p2 = lane == 0 ? A2 : lane == 1 ? A0 : lane == 2 ? A1 : A2;
                const double r2 = lane == 0 ? vc : w;
                const double p3 = lane == 0 ? 0.0 : lane == 1 ? Dx : lane == 2 ? Dy : Dz;
                const double r3 = lane == 1 ? va : lane == 2 ? vb : vc;
                qout += 2.0 * (p0 * r0 + p1 * r1 + p2 * r2 - 2.0 * p3 * r3);
            }
            double *sc = ab.sa_cur + 13 * b;
            if (lane < 3) {
                sc[lane] = xout;
                sc[7 + lane] = vh1;
                sc[10 + lane] = Wh1;
                ab.fadj[6 * b + lane] = Fh;
                ab.fadj[6 * b + 3 + lane] = Th;
                s_F[b][lane] = Fh;
                ab.grad_body[5 * b + 1 + lane] += -beta * alpha * inv_I * inv_I;
            }
            if (lane < 4) sc[3 + lane] = qout;
            if (lane == 0) {
                ab.grad_body[5 * b] += -F2 * inv_m * inv_m;
                ab.grad_body[5 * b + 4] += gv;
            }
        }
        __syncthreads();
    }
    if (blocks > 1) {
        if (threadIdx.x == 0) {
            __threadfence();
            s_last = atomicAdd(ab.done, 1u) == (unsigned)blocks - 1;
            if (s_last) *ab.done = 0u;
            __threadfence();
        }
        __syncthreads();
        if (!s_last) return;
        for (int i = threadIdx.x; i < 3 * nb; i += ADJ_THREADS) s_F[i / 3][i % 3] = __ldcg(ab.fadj + 6 * (i / 3) + i % 3);
        __syncthreads();
    }
    // 2. drive-term and spring gradients (one thread per term), and the spring
    //    terms of each body's adjoint (three lanes a body, an axis each, its
    //    springs in order)
    const double tt = (double)ab.t;
    for (int k = threadIdx.x; k < dv.nd; k += blockDim.x) {
        const DriveTerm dt = dv.drives[k];
        if (tt < dt.t_on || tt >= dt.t_off) continue;
        const AdjDriveTerms tdk = ab.td[k];
        const double *fa = s_F[dt.body];
        const double proj = fa[0] * tdk.aw[0] + fa[1] * tdk.aw[1] + fa[2] * tdk.aw[2];
        ab.grad_drive[2 * k] += tdk.sn * proj;
        ab.grad_drive[2 * k + 1] += -dt.amp * tdk.cs * proj;
    }
    for (int k = (int)threadIdx.x - 32; k < dv.ns; k += blockDim.x) {
        if (k < 0) continue;
        const Spring sp_ = dv.springs[k];
        const AdjSpringTerms tsk = ab.ts[k];
        double fh[3], dvv = 0.0, fd = 0.0;
        for (int i = 0; i < 3; ++i) {
            fh[i] = s_F[sp_.i][i] - s_F[sp_.j][i];
            dvv += fh[i] * tsk.dv[i];
        }
        ab.grad_spring[3 * k + 2] += -dvv;
        if (tsk.len > 0) {
            for (int i = 0; i < 3; ++i) fd += fh[i] * tsk.dir[i];
            ab.grad_spring[3 * k] += -(tsk.len - sp_.rest) * fd;
            ab.grad_spring[3 * k + 1] += sp_.k * fd;
        }
    }
    const int grp = lane / 3, axis = lane % 3;
    for (int b0 = (ADJ_WARPS - 1 - warp) * ADJ_AXIS_GROUPS; b0 < nb; b0 += ADJ_WARPS * ADJ_AXIS_GROUPS) {
        const int b = b0 + grp;
        const bool on = grp < ADJ_AXIS_GROUPS && b < nb;
        const BodyProps *pb = dv.props + (on ? b : 0);
        const int s0 = pb->spring_first, count = on ? pb->spring_count : 0;
        int most = count;
        for (int o = 16; o > 0; o >>= 1) most = max(most, __shfl_xor_sync(FULL, most, o));
        double *sc = ab.sa_cur + 13 * (on ? b : 0);
        double x = 0.0, v = 0.0;
        if (on) {
            x = __ldcg(sc + axis);
            v = __ldcg(sc + 7 + axis);
        }
        for (int i = 0; i < most; ++i) {
            const bool has = i < count;
            double sign = 0.0, fh = 0.0, dir = 0.0, k = 0.0, ratio = 0.0, gamma = 0.0, len = 0.0;
            if (has) {
                const int j = dv.spring_list[s0 + i];
                const Spring sp_ = dv.springs[j];
                const AdjSpringTerms *tsk = ab.ts + j;
                sign = sp_.i == b ? 1.0 : -1.0;
                fh = s_F[sp_.i][axis] - s_F[sp_.j][axis];
                dir = tsk->dir[axis];
                k = sp_.k;
                gamma = sp_.gamma;
                ratio = tsk->ratio;
                len = tsk->len;
            }
            const double prod = fh * dir;
            const double fd = at(prod, 3 * grp) + at(prod, 3 * grp + 1) + at(prod, 3 * grp + 2);
            if (has) {
                v += -sign * gamma * fh;
                if (len > 0) x += sign * (-k * (fd * dir + ratio * (fh - fd * dir)));
            }
        }
        if (on) {
            sc[axis] = x;
            sc[7 + axis] = v;
        }
    }
}

// The first launch of reverse step n: blocks (0, y) the rigid-body step, the others
// the bulk cells, which need neither its result nor each other's.  One launch
// instead of two on two streams with events between them (96 x 48 x 48 study: a
// launch takes 14.2 us, the rigid-body step alone 11.4 us).
template <typename A, typename T, bool FIRST>
__global__ void __launch_bounds__(ADJ_THREADS, sizeof(A) == 4 ? 3 : 2)
adj_step_kernel(const Device dv, const AdjPtrs ap, const AdjBody ab, int body) {
    int blk = blockIdx.x;
    if (body) {
        if (blk == 0) {
            const int blocks = min(adj_integrate_blocks(dv.nb), (int)gridDim.y);
            if ((int)blockIdx.y < blocks) adj_integrate(dv, ab, blockIdx.y, blocks);
            return;
        }
        --blk;
    }
    adj_bulk_cells<A, T, FIRST>(dv, ap, blk, blockIdx.y);
}

__global__ void __launch_bounds__(ADJ_THREADS) adj_integrate_kernel(const Device dv, const AdjBody ab) {
    adj_integrate(dv, ab, blockIdx.x, gridDim.x);
}

// sa[b] += the cell sums part[b][0..count) (the last reverse step)
__global__ void adj_reduce_kernel(int nb, const double *part, int stride, int count, double *sa) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    double *s = sa + 13 * b;
    for (int k = 0; k < count; ++k) {
        const double *p = part + ((long long)b * stride + k) * 9;
        for (int i = 0; i < 3; ++i) { s[i] += p[i]; s[7 + i] += p[3 + i]; s[10 + i] += p[6 + i]; }
    }
}

template <typename A, typename T, bool FIRST>
void launch_step_cells(const Device &dv, const AdjPtrs &ptrs, const AdjBody *ab, cudaStream_t s) {
    AdjPtrs ap = ptrs;
    ap.row_recip = row_recip(dv.dom.nx);
    const long long plane = (long long)dv.dom.nx * dv.dom.ny;
    const dim3 grid((unsigned)((plane + ADJ_THREADS - 1) / ADJ_THREADS) + (ab ? 1 : 0), dv.dom.nz);
    adj_step_kernel<A, T, FIRST><<<grid, ADJ_THREADS, 0, s>>>(dv, ap, ab ? *ab : AdjBody{}, ab ? 1 : 0);
}

template <typename A, typename T, bool FIRST>
void launch_boundary_cells(const Device &dv, const AdjPtrs &ap, cudaStream_t s) {
    if (dv.nb > 0)
        adj_cube_kernel<A, T, FIRST><<<dim3(ap.part_stride, dv.nb), 32 * ADJ_CUBE_WARPS, 0, s>>>(dv, ap);
    if (!(dv.dom.px && dv.dom.py && dv.dom.pz)) {
        const long long nx = dv.dom.nx, ny = dv.dom.ny, nz = dv.dom.nz;
        const long long area = std::max(ny * nz, std::max(nx * nz, nx * ny));
        adj_wall_kernel<A, T, FIRST>
            <<<dim3((unsigned)((area + ADJ_BOUNDARY_THREADS - 1) / ADJ_BOUNDARY_THREADS), 6), ADJ_BOUNDARY_THREADS, 0,
               s>>>(dv, ap);
    }
}

}  // namespace

int adjoint_part_stride(const Device &dv) {
    const long long side = dv.remap_side;
    return (int)((side * side * side + ADJ_BOUNDARY_THREADS - 1) / ADJ_BOUNDARY_THREADS);
}

void launch_adj_integrate(const Device &dv, const AdjBody &ab, cudaStream_t s) {
    adj_integrate_kernel<<<adj_integrate_blocks(dv.nb), ADJ_THREADS, 0, s>>>(dv, ab);
}

void launch_adj_terms(const Device &dv, const BodyState *states, const double *fh, long long t0, int L,
                      AdjBodyTerms *tb, AdjDriveTerms *td, AdjSpringTerms *ts, cudaStream_t s) {
    const long long n = (long long)L * (dv.nb + dv.nd + dv.ns);
    if (n > 0)
        adj_terms_kernel<<<(unsigned)((n + ADJ_THREADS - 1) / ADJ_THREADS), ADJ_THREADS, 0, s>>>(dv, states, fh, t0, L,
                                                                                                 tb, td, ts);
}

void launch_adj_step(const Device &dv, const AdjPtrs &ap, const AdjBody *ab, cudaStream_t s) {
    if (dv.precision == LBM_PREC_F64) {
        if (!ab) launch_step_cells<double, double, true>(dv, ap, ab, s);
        else launch_step_cells<double, double, false>(dv, ap, ab, s);
    } else {
        if (!ab) launch_step_cells<float, float, true>(dv, ap, ab, s);
        else launch_step_cells<float, float, false>(dv, ap, ab, s);
    }
}

void launch_adj_boundary(const Device &dv, const AdjPtrs &ap, bool first, cudaStream_t s) {
    if (dv.precision == LBM_PREC_F64) {
        if (first) launch_boundary_cells<double, double, true>(dv, ap, s);
        else launch_boundary_cells<double, double, false>(dv, ap, s);
    } else {
        if (first) launch_boundary_cells<float, float, true>(dv, ap, s);
        else launch_boundary_cells<float, float, false>(dv, ap, s);
    }
}

void launch_adj_reduce(const Device &dv, const double *part, int stride, int count, double *sa, cudaStream_t s) {
    if (dv.nb > 0) adj_reduce_kernel<<<(dv.nb + 127) / 128, 128, 0, s>>>(dv.nb, part, stride, count, sa);
}

}  // namespace lbm
