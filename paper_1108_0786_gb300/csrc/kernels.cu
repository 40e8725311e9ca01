// kernels.cu -- the per-body kernels of one coupled step and the field
// export / import kernels:
//   prep       per-body geometry records (remade only for states set from
//              outside) and, for more than REMAP_STAGED bodies, the batched
//              remap's candidate lists; steps of a single lattice and batched
//              steps of few bodies run it only after the host wrote a state
//   remap      map the bodies onto the lattice (Sec. 2.3), epoch flags, the
//              boundary kernel's cell list
//   links      per-body list of fluid->solid links (ballot + block scan)
//   loads      drive terms (Eq. FB1-FB3) and spring forces (Eq. osci_i,
//              osci_j) of the step
//   force      momentum-exchange force and torque (Eq. hydroF): FP64 with a
//              fixed-order reduction for FP64 storage, exact integer and
//              fixed-point sums for 32/16-bit storage (deterministic both);
//              the last block of each body runs its rigid-body time step
//              (Algorithm 1) in FP64 on two warps (translation, rotation)
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "../../include/lbm.h"
#include "lbm_internal.cuh"

namespace lbm {
namespace {

__device__ inline bool cell_inside(const Domain &d, const BodyProps &p, const BodyState &b, int x,
                                   int y, int z) {
    double o[3];
    offset_from(d, b, x, y, z, o);
    if (p.shape == 0) return o[0] * o[0] + o[1] * o[1] + o[2] * o[2] <= p.r * p.r;
    double R[3][3];
    quat_to_matrix(b.q, R);
    const double a0 = R[0][0], a1 = R[1][0], a2 = R[2][0];
    double s = o[0] * a0 + o[1] * a1 + o[2] * a2;
    const double h = 0.5 * p.l;
    s = s > h ? h : (s < -h ? -h : s);
    const double e0 = o[0] - s * a0, e1 = o[1] - s * a1, e2 = o[2] - s * a2;
    return e0 * e0 + e1 * e1 + e2 * e2 <= p.r * p.r;
}

// The inside test in FP32: the minimum-image offset as an integer difference
// of cells (wrapped by compares) minus the centre's offset within its cell,
// then the distance in FP32 from that small, nearly exact offset (a few ulps of
// r^2 off; an axis rounded once: growing with l r for long thin capsules).
// Outside the margin max(5e-5 max(r^2, 1), 2e-6 l max(r, 1)) of r^2, at least 14
// times the error found, the screen returns 1 (inside) or 0 (outside), within it
// -1 and the FP64 test decides: the map is the FP64 map bit for bit.
__device__ inline float body_distance2(const Domain &d, const BodyGeom *__restrict__ g, int x, int y, int z) {
    const int n3[3] = {d.nx, d.ny, d.nz}, per[3] = {d.px, d.py, d.pz}, q3[3] = {x, y, z};
    float o[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        int io = q3[i] - g->ci[i];
        if (per[i]) io = 2 * io > n3[i] ? io - n3[i] : (2 * io < -n3[i] ? io + n3[i] : io);
        o[i] = (float)io - g->cf[i];
    }
    const float o0 = o[0], o1 = o[1], o2 = o[2];
    if (g->shape == 0) return o0 * o0 + o1 * o1 + o2 * o2;
    const float h = g->h;
    float sp = o0 * g->ax[0] + o1 * g->ax[1] + o2 * g->ax[2];
    sp = sp > h ? h : (sp < -h ? -h : sp);
    const float e0 = o0 - sp * g->ax[0], e1 = o1 - sp * g->ax[1], e2 = o2 - sp * g->ax[2];
    return e0 * e0 + e1 * e1 + e2 * e2;
}
__device__ inline int inside_screen(const BodyGeom *__restrict__ g, float d2) {
    const float r2 = g->r2, margin = g->margin;
    return d2 < r2 - margin ? 1 : (d2 > r2 + margin ? 0 : -1);
}

__device__ inline uint8_t wall_bit(const Domain &d, int x, int y, int z) {
    const bool w = (!d.px && (x == 0 || x == d.nx - 1)) || (!d.py && (y == 0 || y == d.ny - 1)) ||
                   (!d.pz && (z == 0 || z == d.nz - 1));
    return w ? F_WALL : 0;
}

__global__ void init_flags_kernel(const Domain d, uint8_t *f0, uint8_t *f1, uint8_t *b0, uint8_t *b1) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.C) return;
    const int x = (int)(c % d.nx);
    const int y = (int)((c / d.nx) % d.ny);
    const int z = (int)(c / ((long long)d.nx * d.ny));
    const uint8_t w = wall_bit(d, x, y, z);
    f0[c] = w;
    f1[c] = w;
    b0[c] = NO_BODY;
    b1[c] = NO_BODY;
}

// A cell farther than this from a body's bounding box [floor(X - reach),
// floor(X + reach)] can hold no flag of that body in epochs n-2 .. n: solid
// cells of epoch n-3 lie within 1.5 cells of the current extent, NEAR adds a
// neighbour's 1.42 cells, and the floor of the upper bound loses up to one.
constexpr int STATIC_REACH = 4;

// Axis a of a body's geometry record from that axis' centre coordinate and
// velocity (geom_place), angular velocity and the body x axis' component
// (geom_turn).  Every FP64
// rounding is explicit, so a record made here and one made by the
// rigid-body step's warp agree bit for bit.
__device__ inline void geom_place(const Domain &d, const BodyProps &p, int a, double Xa, double Va, BodyGeom &g) {
    const int n = a == 0 ? d.nx : (a == 1 ? d.ny : d.nz);
    const int per = a == 0 ? d.px : (a == 1 ? d.py : d.pz);
    const double inv = a == 0 ? d.inx : (a == 1 ? d.iny : d.inz);
    const int half = p.E + REMAP_MARGIN;
    const double c = per ? __fma_rn(-(double)n, floor(__dmul_rn(Xa, inv)), Xa) : Xa;
    const double fc = floor(c);
    int o = (int)fc - half;
    if (per) o = ((o % n) + n) % n;
    g.origin[a] = o;
    g.ci[a] = (int)fc;
    g.cfd[a] = __dsub_rn(c, fc);
    g.cf[a] = (float)g.cfd[a];
    g.v[a] = (float)Va;
    const int lo = (int)floor(__dsub_rn(Xa, p.reach)), hi = (int)floor(__dadd_rn(Xa, p.reach));
    int elo = lo - STATIC_REACH, ewidth = hi - lo + 1 + 2 * STATIC_REACH;
    if (per) {
        elo %= n;
        if (elo < 0) elo += n;
        if (ewidth > n) ewidth = n;
    }
    // a body's cube holds its grown box, also where X + reach rounds up to a cell
    int ahead = elo - o;
    if (per && ahead < 0) ahead += n;
    ewidth = min(ewidth, 2 * half + 1 - ahead);
    g.ebox[a] = elo;
    g.ebox[3 + a] = ewidth;
}

__device__ inline void geom_turn(int a, double Wa, double axa, BodyGeom &g) {
    g.w[a] = (float)Wa;
    g.ax[a] = (float)axa;
}

__device__ inline void geom_scalars(const BodyProps &p, BodyGeom &g) {
    g.r2 = p.r2f;
    g.h = p.hf;
    g.margin = p.marginf;
    g.link2 = p.link2f;
    g.shape = p.shape;
    g.side = 2 * (p.E + REMAP_MARGIN) + 1;
}

// a body may not cross a wall: its extent along axis a (with the x axis'
// component axa of a capsule) beyond the wall planes
__device__ inline bool outside_walls(const Domain &d, const BodyProps &p, int a, double Xa, double axa) {
    const int per = a == 0 ? d.px : (a == 1 ? d.py : d.pz);
    if (per) return false;
    const int n = a == 0 ? d.nx : (a == 1 ? d.ny : d.nz);
    const double ext = p.r + (p.shape == 1 ? 0.5 * p.l * fabs(axa) : 0.0);
    return Xa - ext < -0.5 || Xa + ext > n - 0.5;
}

// the whole record of state s, one thread (prep_kernel's fallback)
__device__ void make_geom(const Domain &d, const BodyProps &p, const BodyState &s, BodyGeom &g, int *status) {
    const double w = s.q[0], qx = s.q[1], qy = s.q[2], qz = s.q[3];
    const double axv[3] = {__dsub_rn(1.0, __dmul_rn(2.0, __fma_rn(qy, qy, __dmul_rn(qz, qz)))),
                           __dmul_rn(2.0, __fma_rn(qx, qy, __dmul_rn(w, qz))),
                           __dmul_rn(2.0, __fma_rn(qx, qz, -__dmul_rn(w, qy)))};
    bool out = false;
    for (int a = 0; a < 3; ++a) {
        geom_place(d, p, a, s.X[a], s.V[a], g);
        geom_turn(a, s.W[a], axv[a], g);
        out = out || outside_walls(d, p, a, s.X[a], axv[a]);
    }
    geom_scalars(p, g);
    if (out) atomicOr(status, ST_OUTSIDE);
}

__device__ inline bool same_state(const BodyState &a, const BodyState &b) {
    const long long *x = reinterpret_cast<const long long *>(&a), *y = reinterpret_cast<const long long *>(&b);
    bool eq = true;
#pragma unroll
    for (int i = 0; i < 13; ++i) eq = eq && x[i] == y[i];
    return eq;
}

// Drive terms (Eq. FB1-FB3) and spring forces (Eq. osci_i, osci_j) of step
// n into scratch: they depend on state n only.  Thread `rank` of `count`
// takes drive terms rank, rank + count, ... and springs likewise.
__device__ void body_loads(const Device &dv, const StepPtrs &sp, int drive_rank, int spring_rank, int count) {
    const double t = (double)*dv.t_dev;
    for (int k = drive_rank; k < dv.nd; k += count) {
        const DriveTerm dt = dv.drives[k];
        double f = 0.0;
        if (!(t < dt.t_on || t >= dt.t_off)) f = dt.amp * sin(dt.omega * t - dt.phase);
        double R[3][3];                                 // the drive acts along R(q) axis
        quat_to_matrix(sp.body_cur[dt.body].q, R);
        for (int i = 0; i < 3; ++i)
            dv.drive_f[3 * k + i] = f * (R[i][0] * dt.axis[0] + R[i][1] * dt.axis[1] + R[i][2] * dt.axis[2]);
    }
    for (int k = spring_rank; k < dv.ns; k += count) {
        const Spring sp_ = dv.springs[k];
        const BodyState si = sp.body_cur[sp_.i], sj = sp.body_cur[sp_.j];
        const double dd[3] = {si.X[0] - sj.X[0], si.X[1] - sj.X[1], si.X[2] - sj.X[2]};
        const double len = sqrt(dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2]);
        const double inv_len = len > 0 ? 1.0 / len : 0.0;
        for (int i = 0; i < 3; ++i)
            dv.spring_f[3 * k + i] = -sp_.k * (len - sp_.rest) * (dd[i] * inv_len) - sp_.gamma * (si.V[i] - sj.V[i]);
    }
}

// the drive and spring loads of step n, two warps on two SM sub-partitions
// (an FP64 warp instruction occupies its sub-partition's FP64 pipe for the
// same time however many lanes it carries)
__device__ __forceinline__ void loads_body(const Device &dv, const StepPtrs &sp) {
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) body_loads(dv, sp, lane, dv.ns, 32);
    else body_loads(dv, sp, dv.nd, lane, 32);
}

__global__ void __launch_bounds__(64) loads_kernel(const Device dv, const StepPtrs sp) { loads_body(dv, sp); }

__global__ void __launch_bounds__(64) loads_batch(const Batch bt) {
    LBM_BATCH_MEMBER(bt);
    loads_body(sdv, ssp);
}

// does the cell span [b0, b0 + bw) meet the span [e0, e0 + ew) on an axis of
// n cells?  (On a periodic axis b0 and e0 are wrapped into [0, n).)
__device__ inline bool spans_meet(int b0, int bw, int e0, int ew, int n, int periodic) {
    if (!periodic) return b0 < e0 + ew && e0 < b0 + bw;
    if (bw >= n || ew >= n) return true;
    int o = b0 - e0;                // the start of [b0, ..) seen from e0, in [0, n)
    if (o < 0) o += n;
    return o < ew || o + bw > n;
}

// Body preparation, one block: the geometry records of states n and n-1
// (slots by body buffer: remade only when the slot's stamp differs from the
// state, i.e. when no rigid-body step produced that state), each body's
// remap candidates for the batched remap (the bodies, in order, whose grown
// box meets its remap cube; a warp a body, ballots over the candidates; a
// single lattice's remap finds its own), and the start of the boundary
// kernel's list.  A single lattice's steps whose states the rigid-body step
// made (and whose list the previous step's last block emptied) skip it.
constexpr int PREP_THREADS = 256;

__device__ __forceinline__ void prep_body(const Device &dv, const StepPtrs &sp) {
    const Domain d = dv.dom;
    const int n3[3] = {d.nx, d.ny, d.nz}, per[3] = {d.px, d.py, d.pz};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    BodyGeom *cur = dv.geom + sp.parity * dv.nb, *prev = dv.geom + (sp.parity ^ 1) * dv.nb;
    BodyState *scur = dv.gstamp + sp.parity * dv.nb, *sprev = dv.gstamp + (sp.parity ^ 1) * dv.nb;
    if (threadIdx.x == 0) *dv.bcount = 0;           // the remap refills the boundary kernel's list
    if (warp < 2) {
        BodyGeom *g = warp == 0 ? cur : prev;
        BodyState *st = warp == 0 ? scur : sprev;
        const BodyState *state = warp == 0 ? sp.body_cur : sp.body_prev;
        for (int k = lane; k < dv.nb; k += 32) {
            const BodyState sb = state[k];
            if (same_state(sb, st[k])) continue;
            make_geom(d, dv.props[k], sb, g[k], dv.status);
            st[k] = sb;
        }
    }
    __syncthreads();
    __shared__ int s_box[LBM_MAX_BODIES_DEV][8];        // ebox (6), then origin packed per axis below
    __shared__ int s_org[LBM_MAX_BODIES_DEV][4];
    for (int k = threadIdx.x; k < dv.nb; k += blockDim.x) {
        for (int i = 0; i < 6; ++i) s_box[k][i] = cur[k].ebox[i];
        for (int i = 0; i < 3; ++i) s_org[k][i] = cur[k].origin[i];
        s_org[k][3] = cur[k].side;
    }
    __syncthreads();
    for (int b = warp; b < dv.nb; b += PREP_THREADS / 32) {
        int cnt = 0;
        for (int k0 = 0; k0 < dv.nb; k0 += 32) {
            const int k = k0 + lane;
            bool meets = k < dv.nb;
            for (int a = 0; a < 3 && meets; ++a)
                meets = spans_meet(s_org[b][a], s_org[b][3], s_box[k][a], s_box[k][3 + a], n3[a], per[a]);
            const unsigned bal = __ballot_sync(0xffffffffu, meets);
            if (meets) dv.cand[b * dv.nb + cnt + __popc(bal & ((1u << lane) - 1u))] = (uint8_t)k;
            cnt += __popc(bal);
        }
        if (lane == 0) cur[b].ncand = cnt;
    }
}

__global__ void __launch_bounds__(PREP_THREADS) prep_kernel(const Device dv, const StepPtrs sp) { prep_body(dv, sp); }

__global__ void __launch_bounds__(PREP_THREADS) prep_batch(const Batch bt) {
    LBM_BATCH_MEMBER(bt);
    prep_body(sdv, ssp);
}


// a coordinate of the cube, o + l with o in [0, n) and l < side, wrapped
// into [0, n) on a periodic axis (one compare unless the cube exceeds the axis)
__device__ inline int wrap_up(int v, int n) { return v < n ? v : (v - n < n ? v - n : v % n); }

// Remap: block row blockIdx.y = body b; the cube of side 2 (E_b +
// REMAP_MARGIN) + 1 around floor(X_b) at state n is taken as one run of
// side^3 cells in (z, y, x) order, REMAP_CELLS consecutive cells a block and
// REMAP_R a thread (i and i + REMAP_THREADS: their flag loads are issued
// together, so a block's latency chain covers both).  No thread idles on a
// cube narrower than a warp, and the grid of the 24-capsule swarm (side 23)
// fits in one wave of resident blocks.  Every covered cell gets its epoch-n
// flags from the geometry of all bodies and the epoch-(n-1) buffer;
// overlapping cubes write identical values.  A cell tests only body b's
// candidates, in body order (integer boxes, the FP32 screen, and the FP64
// inside test only within the screen's margin).  Fluid cells flagged F_NEAR
// F_SOLID_PREV or F_LINK are appended to the boundary kernel's list, each once:
// by the block row of the lowest-numbered body whose grown box holds the cell
// (that body's cube covers it, and every cube that does has the body among its
// candidates), so the list never exceeds C.
constexpr int REMAP_THREADS = 256;
constexpr int REMAP_R = 2;
constexpr int REMAP_CELLS = REMAP_THREADS * REMAP_R;    // cube cells a block covers
constexpr int REMAP_STAGED = 8;

// blocks a body of remap-cube side `side` takes
inline int remap_blocks(int side) {
    const long long cells = (long long)side * side * side;
    return (int)((cells + REMAP_CELLS - 1) / REMAP_CELLS);
}
static_assert(sizeof(BodyGeom) % sizeof(int) == 0, "geometry records are copied as ints");

template <bool SELF_CAND>
__device__ __forceinline__ void remap_body(const Device &dv, const StepPtrs &sp, const Blk &bk, int init_mode) {
    const Domain d = dv.dom;
    const int b = bk.y;
    const BodyGeom *__restrict__ geo = dv.geom + sp.parity * dv.nb;    // state n
    // body b's candidates, the first REMAP_STAGED of them with their
    // records in shared memory
    __shared__ BodyGeom cg[REMAP_STAGED];
    __shared__ int cid[LBM_MAX_BODIES_DEV];
    __shared__ int s_ncand;
    const int n3[3] = {d.nx, d.ny, d.nz}, per[3] = {d.px, d.py, d.pz};
    const int side = geo[b].side;
    const int side2 = side * side, cells = side2 * side;
    const int i0 = bk.x * REMAP_CELLS;
    if (i0 >= cells) return;                  // the grid covers the largest body's cube
    // the step's index by parity (the force kernel advances the clock while the
    // bulk kernel may still read it); an overlapped step's is there already
    if (threadIdx.x == 0 && bk.x == 0 && b == 0 && !init_mode) {
        const long long t = *dv.t_dev;
        if (dv.tstep[sp.parity] != t) dv.tstep[sp.parity] = t;
    }
    // this block's share of the boundary kernel's list, gathered in shared
    // memory and appended with one atomic at the end
    __shared__ uint32_t lbuf[REMAP_CELLS];
    __shared__ int lcount, lbase;
    const int org[3] = {geo[b].origin[0], geo[b].origin[1], geo[b].origin[2]};
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    if (tid == 0) lcount = 0;
    // the candidates: the bodies, in body order, whose grown box (the cells
    // their flags of epochs n-3 .. n can reach) meets b's cube.  A single
    // lattice's block finds them (the first warp, ballots over 32 bodies at
    // a time); the batched remap takes the preparation kernel's list.  The
    // first REMAP_STAGED records are staged in shared memory.
    // With at most REMAP_STAGED bodies every body is a candidate (the cells' box
    // tests sort them out): one round of loads less in a block's latency chain
    // (0.9 us of a 128 x 64 x 64 channel step).
    const bool all = dv.nb <= REMAP_STAGED;
    if (all) {
        if (tid < dv.nb) cid[tid] = tid;
    } else if constexpr (SELF_CAND) {
        if (tid < 32) {
            int cnt = 0;
            for (int k0 = 0; k0 < dv.nb; k0 += 32) {
                const int k = k0 + tid;
                bool meets = k < dv.nb;
                int e[6];
                for (int i = 0; i < 6; ++i) e[i] = geo[min(k, dv.nb - 1)].ebox[i];
                for (int a = 0; a < 3; ++a) meets = meets && spans_meet(org[a], side, e[a], e[3 + a], n3[a], per[a]);
                const unsigned bal = __ballot_sync(0xffffffffu, meets);
                if (meets) cid[cnt + __popc(bal & ((1u << tid) - 1u))] = k;
                cnt += __popc(bal);
            }
            if (tid == 0) s_ncand = cnt;
        }
    } else {
        const int nc = geo[b].ncand;
        for (int i = tid; i < nc; i += REMAP_THREADS) cid[i] = dv.cand[b * dv.nb + i];
        if (tid == 0) s_ncand = nc;
    }
    if (!all) __syncthreads();
    const int ncand = all ? dv.nb : s_ncand;
    {
        constexpr int W = (int)(sizeof(BodyGeom) / sizeof(int));
        const int staged = min(ncand, REMAP_STAGED);
        for (int i = tid; i < staged * W; i += REMAP_THREADS)
            reinterpret_cast<int *>(cg)[i] = reinterpret_cast<const int *>(geo + (all ? i / W : cid[i / W]))[i % W];
    }
    __syncthreads();

    // every lane runs each of its cells, so the ballots below see whole warps
        {
            int xr[REMAP_R], yr[REMAP_R], zr[REMAP_R], idr[REMAP_R];
            bool linkr[REMAP_R], minr[REMAP_R];
            long long cr[REMAP_R];
            bool liver[REMAP_R];
#pragma unroll
            for (int r = 0; r < REMAP_R; ++r) {
                const int ci = i0 + r * REMAP_THREADS + tid;
                bool live = ci < cells;
                const int lz = ci / side2, rem = ci - lz * side2;
                const int ly = rem / side, lx = rem - ly * side;
                int x = org[0] + lx, y = org[1] + ly, z = org[2] + lz;
                if (d.px) x = wrap_up(x, d.nx); else live = live && x >= 0 && x < d.nx;
                if (d.py) y = wrap_up(y, d.ny); else live = live && y >= 0 && y < d.ny;
                if (d.pz) z = wrap_up(z, d.nz); else live = live && z >= 0 && z < d.nz;
                const int p3[3] = {x, y, z};
                int id = NO_BODY;
                bool reached = false;           // within STATIC_REACH cells of some body's box
                bool mine = false;              // and of no lower-numbered body's than b: this block lists it
                bool link = false;
                for (int i = 0; i < ncand && live; ++i) {
                    const int kb = cid[i];
                    const BodyGeom *g = i < REMAP_STAGED ? cg + i : geo + kb;
                    bool in = true;
                    for (int a = 0; a < 3 && in; ++a) {
                        int o = p3[a] - g->ebox[a];
                        if (per[a] && o < 0) o += n3[a];
                        in = o >= 0 && o < g->ebox[3 + a];
                    }
                    if (!in) continue;
                    if (!reached) mine = kb == b;
                    reached = true;
                    // the squared distance to the centre or axis in FP32: cells
                    // that may hold links, and the inside screen (cells within
                    // its margin of the surface take the FP64 test)
                    const float d2 = body_distance2(d, g, x, y, z);
                    link = link || d2 < g->link2;
                    const int screen = inside_screen(g, d2);
                    if (screen == 0 || (screen < 0 && !cell_inside(d, dv.props[kb], sp.body_cur[kb], x, y, z)))
                        continue;
                    if (id != NO_BODY) atomicOr(dv.status, ST_OVERLAP);
                    id = kb;
                }
                // farther than STATIC_REACH from every body's box: the cell holds
                // its static flags in both epoch buffers already (nothing within
                // reach was solid in the last three steps, at most 0.5 cells of
                // motion per step)
                xr[r] = x;
                yr[r] = y;
                zr[r] = z;
                idr[r] = id;
                linkr[r] = link;
                minr[r] = mine;
                cr[r] = ((long long)z * d.ny + y) * d.nx + x;
                liver[r] = live && reached;
            }
            // the epoch-(n-1) flags and body id of every row's cell and whether
            // any pull source x - e_a held an obstacle of step n-1 (sources
            // beyond a wall do not count): all loads before any use
            uint8_t prevr[REMAP_R], nearr[REMAP_R], bidr[REMAP_R];
#pragma unroll
            for (int r = 0; r < REMAP_R; ++r) {
                prevr[r] = 0;
                nearr[r] = 0;
                bidr[r] = NO_BODY;
                if (!liver[r] || init_mode) continue;
                const long long c = cr[r];
                const int x = xr[r], y = yr[r], z = zr[r];
                prevr[r] = sp.flags_prev[c];
                bidr[r] = sp.bid_prev[c];
                uint8_t near = 0;
                const long long sy = d.nx, sz = (long long)d.nx * d.ny;
                if (x > 0 && x < d.nx - 1 && y > 0 && y < d.ny - 1 && z > 0 && z < d.nz - 1) {
#pragma unroll
                    for (int a = 1; a < Q; ++a) near |= sp.flags_prev[c - ex(a) - ey(a) * sy - ez(a) * sz];
                } else {
#pragma unroll
                    for (int a = 1; a < Q; ++a) {
                        const int sx_ = x - ex(a), sy_ = y - ey(a), sz_ = z - ez(a);
                        const bool in = !((!d.px && (sx_ < 0 || sx_ >= d.nx)) || (!d.py && (sy_ < 0 || sy_ >= d.ny)) ||
                                          (!d.pz && (sz_ < 0 || sz_ >= d.nz)));
                        const uint8_t v = sp.flags_prev[((long long)wrap_axis(sz_, d.nz) * d.ny + wrap_axis(sy_, d.ny)) * d.nx +
                                                        wrap_axis(sx_, d.nx)];
                        near |= in ? v : 0;
                    }
                }
                nearr[r] = near;
            }
#pragma unroll
            for (int r = 0; r < REMAP_R; ++r) {
                const bool live = liver[r];
                const int id = idr[r];
                const long long c = cr[r];
                uint8_t flags = 0;
                if (live) {
                    const uint8_t solid = id != NO_BODY ? F_SOLID : 0;
                    flags = solid | wall_bit(d, xr[r], yr[r], zr[r]);
                    if (!init_mode) {
                        if (linkr[r]) flags |= F_LINK;
                        const uint8_t prev = prevr[r] & F_SOLID;
                        if (prev) flags |= F_SOLID_PREV;
                        if (nearr[r] & F_SOLID) flags |= F_NEAR;
                        if ((solid != 0) != (prev != 0) || (solid && bidr[r] != id)) dv.changed[sp.parity] = 1;
                    }
                    sp.flags_cur[c] = flags;
                    sp.bid_cur[c] = (uint8_t)id;
                }
                // the boundary kernel's cells: a shared-memory atomic per warp
                const bool mine = live && minr[r] && !init_mode && !(flags & F_SOLID) && (flags & F_LISTED);
                const unsigned mb = __ballot_sync(0xffffffffu, mine);
                if (mb) {
                    const int leader = __ffs(mb) - 1;
                    int base = 0;
                    if (lane == leader) base = atomicAdd(&lcount, __popc(mb));
                    base = __shfl_sync(0xffffffffu, base, leader);
                    if (mine) lbuf[base + __popc(mb & ((1u << lane) - 1u))] = (uint32_t)c;
                }
            }
        }
    __syncthreads();
    if (tid == 0) lbase = lcount ? atomicAdd(dv.bcount, lcount) : 0;
    __syncthreads();
    const int nl = lcount;
    for (int i = tid; i < nl; i += REMAP_THREADS) {
        if (lbase + i < dv.blist_cap) dv.blist[lbase + i] = lbuf[i];
        else atomicOr(dv.status, ST_LINKS);
    }
}

__global__ void __launch_bounds__(REMAP_THREADS, 4) remap_kernel(const Device dv, const StepPtrs sp, int init_mode) {
    pdl_enter();
    remap_body<true>(dv, sp, launch_blk(), init_mode);
}

__global__ void __launch_bounds__(REMAP_THREADS, 4) remap_batch(const Batch bt) {
    LBM_BATCH_MEMBER(bt);
    remap_body<false>(sdv, ssp, sbk, 0);
}

// Links: block (k, b) scans z-plane k of the cube of side 2 E_b + 3 around
// floor(X_b) and stores the links (x_f, a) with x_f fluid and x_f + e_a a
// cell of body b, in (y, x, a) order, into segment (b, k).  Runs only when
// the remap changed a flag; otherwise the previous lists stand.
__device__ __forceinline__ void links_body(const Device &dv, const StepPtrs &sp, const Blk &bk) {
    if (dv.changed[sp.parity] == 0) return;
    const Domain d = dv.dom;
    const int b = bk.y, k = bk.x;
    const BodyProps pb = dv.props[b];
    const int half = pb.E + 1;
    const int side = 2 * half + 1;
    int *count = dv.seg_count + (long long)b * dv.link_side + k;
    if (k >= side) {
        if (threadIdx.x == 0) *count = 0;
        return;
    }
    const BodyState sb = sp.body_cur[b];
    Link *seg = dv.links + ((long long)b * dv.link_side + k) * dv.seg_cap;
    const int ox = (int)floor(sb.X[0]) - half, oy = (int)floor(sb.X[1]) - half;
    int z = (int)floor(sb.X[2]) - half + k;
    bool zok = true;
    if (d.pz) z = ((z % d.nz) + d.nz) % d.nz; else zok = z >= 0 && z < d.nz;

    __shared__ int warp_tot[32];
    __shared__ int base;
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int area = side * side;
    for (int start = 0; start < area; start += blockDim.x) {
        const int l = start + threadIdx.x;
        unsigned mask = 0;
        long long c = 0;
        if (zok && l < area) {
            int x = ox + l % side, y = oy + l / side;
            bool ok = true;
            if (d.px) x = ((x % d.nx) + d.nx) % d.nx; else ok = ok && x >= 0 && x < d.nx;
            if (d.py) y = ((y % d.ny) + d.ny) % d.ny; else ok = ok && y >= 0 && y < d.ny;
            if (ok) {
                c = ((long long)z * d.ny + y) * d.nx + x;
                if (!(sp.flags_cur[c] & F_SOLID)) {
                    for (int a = 1; a < Q; ++a) {
                        int nx_ = x + ex(a), ny_ = y + ey(a), nz_ = z + ez(a);
                        if ((!d.px && (nx_ < 0 || nx_ >= d.nx)) || (!d.py && (ny_ < 0 || ny_ >= d.ny)) ||
                            (!d.pz && (nz_ < 0 || nz_ >= d.nz)))
                            continue;
                        nx_ = wrap_axis(nx_, d.nx); ny_ = wrap_axis(ny_, d.ny); nz_ = wrap_axis(nz_, d.nz);
                        const long long n = ((long long)nz_ * d.ny + ny_) * d.nx + nx_;
                        if ((sp.flags_cur[n] & F_SOLID) && sp.bid_cur[n] == b) mask |= 1u << a;
                    }
                }
            }
        }
        // block-wide exclusive scan of the per-thread link counts
        const int cnt = __popc(mask);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) warp_tot[warp] = incl;
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < nwarps; ++w) {
            if (w < warp) before += warp_tot[w];
            total += warp_tot[w];
        }
        int pos = base + before + incl - cnt;
        while (mask) {
            const int a = __ffs(mask) - 1;
            mask &= mask - 1;
            if (pos < dv.seg_cap) seg[pos] = Link{(uint32_t)c, (uint32_t)a};
            else atomicOr(dv.status, ST_LINKS);
            ++pos;
        }
        __syncthreads();
        if (threadIdx.x == 0) base += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) *count = base;
}

__global__ void __launch_bounds__(256) links_kernel(const Device dv, const StepPtrs sp) { links_body(dv, sp, launch_blk()); }

__global__ void __launch_bounds__(256) links_batch(const Batch bt) {
    // nearly always there is nothing to rebuild: look before fetching the member
    if (bt.dv[bt.member[blockIdx.x]].changed[bt.parity] == 0) return;
    LBM_BATCH_MEMBER(bt);
    links_body(sdv, ssp, sbk);
}

// a stored deviation in FP32 (exact for FP32, FP16 times its power-of-two
// scale, BF16), without a trip through FP64
template <typename T> __device__ inline float load_dev_f(const T *p, float inv_scale);
template <> __device__ inline float load_dev_f<float>(const float *p, float) { return *p; }
template <> __device__ inline float load_dev_f<__half>(const __half *p, float s) { return __half2float(*p) * s; }
template <> __device__ inline float load_dev_f<__nv_bfloat16>(const __nv_bfloat16 *p, float) {
    return __bfloat162float(*p);
}

template <typename T> __device__ inline double load_dev(const T *p, float inv_scale);
template <> __device__ inline double load_dev<double>(const double *p, float) { return *p; }
template <> __device__ inline double load_dev<float>(const float *p, float) { return (double)*p; }
template <> __device__ inline double load_dev<__half>(const __half *p, float s) {
    return (double)(__half2float(*p) * s);
}
template <> __device__ inline double load_dev<__nv_bfloat16>(const __nv_bfloat16 *p, float) {
    return (double)__bfloat162float(*p);
}

constexpr int FORCE_THREADS = 256;                  // link threads of a force block ...
constexpr int FORCE_BLOCK = FORCE_THREADS + 64;     // ... and the two warps of the rigid-body step

// barrier of the link threads
__device__ __forceinline__ void link_sync() { asm volatile("bar.sync 1, %0;" ::"n"(FORCE_THREADS) : "memory"); }
constexpr int MAX_SEGMENTS = 1024;

// minimum image of a cell difference o (|o| < n + 1) by integer compares
__device__ inline int near_cell_k(int o, int n, int periodic) {
    if (!periodic) return o;
    return 2 * o > n ? o - n : (2 * o < -n ? o + n : o);
}

// periodic minimum image of d for |d| < 3n/2 (two compares, no FP64 floor)
__device__ inline double wrap_near(double d, int n, int periodic) {
    if (!periodic) return d;
    const double h = 0.5 * n;
    return d > h ? d - n : (d < -h ? d + n : d);
}

// Rigid-body step (Algorithm 1, Eq. totalFSwimmer) of body b by two warps, the
// translation by one and the rotation by the other.  An FP64 warp instruction
// occupies its sub-partition for the same ~64 cycles however many lanes it
// carries, so lanes hold components (six load components, three axes, nine
// rotation-matrix entries, four quaternion components) and the two halves sit on
// different sub-partitions.  Per axis it adds, in order, the momentum-exchange
// sum, g times the volume, the body's drive terms in term order and its springs
// in spring order (body_loads' scratch), then advances by semi-implicit Euler
// (dt = 1) in FP64.  Both halves write their part of the geometry record of the
// new state into that state's slot, with its stamp, and check the new state
// (walls, finite, at most MAX_STEP per step).
//
// `wait()` separates what depends on the state of step n alone (loads, the
// external force, R(q): done while the link sums are formed) from what needs the
// hydrodynamic load; it returns false in a block that does not finish the body.
// (128 x 64 x 64 channel, a step: 40.1 us with one warp doing it all after the
// sums, 34.6 us so.)

// the hydrodynamic load of step n: lane i < 6 component i of force and torque
__device__ __forceinline__ double hydro_load(const Device &dv, const StepPtrs &sp, int b, int with_fluid,
                                             const double (&c)[3]) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    double hyd = 0.0;
    if (with_fluid && dv.precision == 0) {
        if (lane < 6) {
            double v[FORCE_BLOCKS];
#pragma unroll
            for (int k = 0; k < FORCE_BLOCKS; ++k) v[k] = __ldcg(dv.fpart + ((long long)b * FORCE_BLOCKS + k) * 6 + lane);
#pragma unroll
            for (int k = 0; k < FORCE_BLOCKS; ++k) hyd += v[k];
        }
    } else if (with_fluid) {
        // F = S1 / 36 + Fv, T = S2 / 36 + Tv - c x F with c the centre's
        // position within its cell (the force kernel's terms)
        if (lane < 6) {
            const long long fx = __ldcg(dv.fx + b * 6 + lane);
            const int si = __ldcg(dv.fi + b * 6 + lane);
            hyd = fma((double)si, 1.0 / 36.0, (double)fx * (1.0 / (double)(1LL << FIX_BITS)));
        }
        const int i = lane % 3, j = (i + 1) % 3, k = (i + 2) % 3;
        const double fj = __shfl_sync(FULL, hyd, j), fk = __shfl_sync(FULL, hyd, k);
        const double cj = j == 0 ? c[0] : (j == 1 ? c[1] : c[2]), ck = k == 0 ? c[0] : (k == 1 ? c[1] : c[2]);
        if (lane >= 3) hyd = fma(ck, fj, fma(-cj, fk, hyd));
    }
    return hyd;
}

// external force on axis ax: g times the volume, then the body's drive terms in
// term order and its springs in spring order
__device__ __forceinline__ double external_force(const Device &dv, const BodyProps *pb, int b, int ax) {
    double F = dv.g[ax] * pb->volume;
    const int d0 = pb->drive_first, d1 = d0 + pb->drive_count, s0 = pb->spring_first, s1 = s0 + pb->spring_count;
    // the springs' chains of dependent loads start first
    constexpr int AHEAD = 4;
    double fs[AHEAD];
#pragma unroll
    for (int i = 0; i < AHEAD; ++i) {
        fs[i] = 0.0;
        if (s0 + i < s1) {
            const int k = dv.spring_list[s0 + i];
            const double f = dv.spring_f[3 * k + ax];
            fs[i] = dv.springs[k].i == b ? f : -f;
        }
    }
    for (int k = d0; k < d1; ++k) F += dv.drive_f[3 * k + ax];
#pragma unroll
    for (int i = 0; i < AHEAD; ++i)
        if (s0 + i < s1) F += fs[i];
    for (int kk = s0 + AHEAD; kk < s1; ++kk) {
        const int k = dv.spring_list[kk];
        const double f = dv.spring_f[3 * k + ax];
        F += dv.springs[k].i == b ? f : -f;
    }
    return F;
}

// entries [o, o + n) of the 13 of a state, lane i < n entry o + i, into the new
// state, its stamp and its tape and history entries
__device__ __forceinline__ void put_state(const Device &dv, const StepPtrs &sp, int b, long long tstep,
                                          const TapeCtl &tc, int o, int n, double v) {
    const int lane = threadIdx.x & 31;
    if (lane >= n) return;
    reinterpret_cast<double *>(sp.body_next + b)[o + lane] = v;
    reinterpret_cast<double *>(dv.gstamp + (sp.parity ^ 1) * dv.nb + b)[o + lane] = v;
    const long long j = tstep - tc.t0;
    if (tc.on && j >= 0 && j < tc.cap) tc.state[((j + 2) * dv.nb + b) * 13 + o + lane] = v;
    if (dv.hist) dv.hist[((tstep % dv.hist_cap) * dv.nb + b) * 13 + o + lane] = v;
}

template <typename Wait>
__device__ __forceinline__ void integrate_translation(const Device &dv, const StepPtrs &sp, int b, int with_fluid,
                                                      Wait wait) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, ax = lane < 3 ? lane : 0;
    const BodyProps *pb = dv.props + b;
    const double *st = reinterpret_cast<const double *>(sp.body_cur + b);       // X q V W
    const double X = st[ax], V = st[7 + ax], inv_m = pb->inv_m;
    const long long tstep = *dv.t_dev;
    const double prev = lane < 6 ? dv.fh[b * 6 + lane] : 0.0;
    const TapeCtl tc = dv.tape ? *dv.tape : TapeCtl{};
    const double Fext = external_force(dv, pb, b, ax);
    const double *cg = dv.geom[sp.parity * dv.nb + b].cfd;
    const double c[3] = {cg[0], cg[1], cg[2]};
    if (!wait()) return;
    const double hyd = hydro_load(dv, sp, b, with_fluid, c);
    double v = hyd;
    if (lane < 6) {
        dv.fh[b * 6 + lane] = hyd;
        if (dv.avg_force && tstep > 0) v = 0.5 * (hyd + prev);
    }
    const double Vn = V + (v + Fext) * inv_m;
    const double Xn = X + Vn;
    put_state(dv, sp, b, tstep, tc, 0, 3, Xn);
    put_state(dv, sp, b, tstep, tc, 7, 3, Vn);
    if (lane < 6) {
        const long long j = tstep - tc.t0;
        if (tc.on && j >= 0 && j < tc.cap) tc.force[(j * dv.nb + b) * 6 + lane] = hyd;
    }
    BodyGeom *g = dv.geom + (sp.parity ^ 1) * dv.nb + b;
    if (lane < 3) geom_place(dv.dom, *pb, ax, Xn, Vn, *g);
    if (lane == 0) geom_scalars(*pb, *g);
    const bool finite = __all_sync(FULL, lane >= 3 || (isfinite(Xn) && isfinite(Vn)));
    const bool fast = __any_sync(FULL, lane < 3 && fabs(Vn) > MAX_STEP);
    if (lane == 0 && (!finite || fast)) atomicOr(dv.status, !finite ? ST_NAN : ST_UNSTABLE);
}

template <typename Wait>
__device__ __forceinline__ void integrate_rotation(const Device &dv, const StepPtrs &sp, int b, int with_fluid,
                                                   Wait wait) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, ax = lane < 3 ? lane : 0;
    const BodyProps *pb = dv.props + b;
    const double *st = reinterpret_cast<const double *>(sp.body_cur + b);       // X q V W
    const double W = st[10 + ax], inv_I = pb->inv_inertia[ax];
    const long long tstep = *dv.t_dev;
    const double prev = lane < 6 ? dv.fh[b * 6 + lane] : 0.0;
    const TapeCtl tc = dv.tape ? *dv.tape : TapeCtl{};
    const double *cg = dv.geom[sp.parity * dv.nb + b].cfd;
    const double c[3] = {cg[0], cg[1], cg[2]};
    // with walls: the new position again, for the wall check of a capsule's ends
    const bool walls = !(dv.dom.px && dv.dom.py && dv.dom.pz);
    double X = 0.0, V = 0.0, inv_m = 0.0, Fext = 0.0;
    if (walls) {
        X = st[ax];
        V = st[7 + ax];
        inv_m = pb->inv_m;
        Fext = external_force(dv, pb, b, ax);
    }
    // R(q) of state n, entry (r, c) on lane 3 r + c < 9: 1 - 2 (a^2 + b^2)
    // on the diagonal, 2 (p q +- w u) off it
    const double qw = st[3], qv[3] = {st[4], st[5], st[6]};
    double Rrc;
    {
        const int r = lane < 9 ? lane / 3 : 0, cc = lane < 9 ? lane % 3 : 0;
        double A, Bq, Cq, D, base;
        if (r == cc) {
            A = -qv[(r + 1) % 3]; Bq = qv[(r + 1) % 3];
            Cq = -qv[(r + 2) % 3]; D = qv[(r + 2) % 3];
            base = 1.0;
        } else {
            const bool plus = (r == 1 && cc == 0) || (r == 0 && cc == 2) || (r == 2 && cc == 1);
            A = qv[min(r, cc)]; Bq = qv[max(r, cc)];
            Cq = plus ? qw : -qw; D = qv[3 - r - cc];
            base = 0.0;
        }
        Rrc = base + 2.0 * (A * Bq + Cq * D);
    }
    const double R0i = __shfl_sync(FULL, Rrc, ax), R1i = __shfl_sync(FULL, Rrc, 3 + ax),
                 R2i = __shfl_sync(FULL, Rrc, 6 + ax);
    const double Ri0 = __shfl_sync(FULL, Rrc, 3 * ax), Ri1 = __shfl_sync(FULL, Rrc, 3 * ax + 1),
                 Ri2 = __shfl_sync(FULL, Rrc, 3 * ax + 2);
    if (!wait()) return;
    const double hyd = hydro_load(dv, sp, b, with_fluid, c);
    double v = hyd;
    if (dv.avg_force && tstep > 0) v = 0.5 * (hyd + prev);
    // Omega += R diag(1/I) R^T T, lanes 0..2
    const double T0 = __shfl_sync(FULL, v, 3), T1 = __shfl_sync(FULL, v, 4), T2 = __shfl_sync(FULL, v, 5);
    const double Tb = (R0i * T0 + R1i * T1 + R2i * T2) * inv_I;
    const double Tb0 = __shfl_sync(FULL, Tb, 0), Tb1 = __shfl_sync(FULL, Tb, 1), Tb2 = __shfl_sync(FULL, Tb, 2);
    const double Wn = W + (Ri0 * Tb0 + Ri1 * Tb1 + Ri2 * Tb2);

    // q += 1/2 (0, Omega) (x) q, renormalised; lane 0 the scalar part,
    // lane 1 + i the vector component i
    const double W0 = __shfl_sync(FULL, Wn, 0), W1 = __shfl_sync(FULL, Wn, 1), W2 = __shfl_sync(FULL, Wn, 2);
    const double Wv[3] = {W0, W1, W2};
    double q4;
    {
        // lane 0: w - 1/2 (W . v); lane 1 + i: v_i + 1/2 (w W_i + (W x v)_i),
        // one expression with the operands chosen per lane (no divergence)
        const int i = lane >= 1 && lane <= 3 ? lane - 1 : 0, i1 = (i + 1) % 3, i2 = (i + 2) % 3;
        const bool s0 = lane == 0;
        const double base = s0 ? qw : qv[i];
        const double p1 = s0 ? -W0 : qw, r1 = s0 ? qv[0] : Wv[i];
        const double p2 = s0 ? -W1 : Wv[i1], r2 = s0 ? qv[1] : qv[i2];
        const double p3 = s0 ? -W2 : -Wv[i2], r3 = s0 ? qv[2] : qv[i1];
        q4 = base + 0.5 * (p1 * r1 + p2 * r2 + p3 * r3);
    }
    double sq = lane < 4 ? q4 * q4 : 0.0;
    sq += __shfl_xor_sync(FULL, sq, 1);
    sq += __shfl_xor_sync(FULL, sq, 2);
    const double qn = q4 * rsqrt(sq);
    put_state(dv, sp, b, tstep, tc, 3, 4, qn);
    put_state(dv, sp, b, tstep, tc, 10, 3, Wn);

    // the rotational part of the new state's geometry record; the body x axis is
    // column 0 of R(q_{n+1})
    const double nw = __shfl_sync(FULL, qn, 0), nq[3] = {__shfl_sync(FULL, qn, 1), __shfl_sync(FULL, qn, 2),
                                                         __shfl_sync(FULL, qn, 3)};
    // column 0 of R: 1 - 2 (y^2 + z^2), 2 (x y + w z), 2 (x z - w y), one
    // expression base + 2 (A B + C D) with the operands chosen per lane
    double axa;
    {
        const double A = ax == 0 ? -nq[1] : nq[0], B = ax == 0 ? nq[1] : (ax == 1 ? nq[1] : nq[2]);
        const double Cq = ax == 0 ? -nq[2] : (ax == 1 ? nw : -nw), D = ax == 0 ? nq[2] : (ax == 1 ? nq[2] : nq[1]);
        axa = (ax == 0 ? 1.0 : 0.0) + 2.0 * (A * B + Cq * D);
    }
    BodyGeom *g = dv.geom + (sp.parity ^ 1) * dv.nb + b;
    if (lane < 3) geom_turn(ax, Wn, axa, *g);
    const bool finite = __all_sync(FULL, lane >= 3 || isfinite(Wn));
    if (lane == 0 && !finite) atomicOr(dv.status, ST_NAN);
    if (walls) {
        const double Xn = X + (V + (v + Fext) * inv_m);
        const bool any_out = __any_sync(FULL, lane < 3 && outside_walls(dv.dom, *pb, ax, Xn, axa));
        if (lane == 0 && any_out) atomicOr(dv.status, ST_OUTSIDE);
    }
}

// after every body's step: the clock advances and the next epoch's change
// flag starts clear
__device__ inline void finish_step(const Device &dv, const StepPtrs &sp) {
    *dv.t_dev = *dv.t_dev + 1;
    dv.changed[sp.parity ^ 1] = 0;
    if (dv.bcount) *dv.bcount = 0;          // the next remap refills the boundary kernel's list
}

// round(v 2^FIX_BITS) to the nearest integer, ties away from zero, from the
// bits of v in integer operations (a 64-bit conversion would take the slow
// FP64 pipe); |v| < 2^(62 - FIX_BITS) is the caller's to ensure
__device__ inline long long to_fixed(float v) {
    const unsigned u = __float_as_uint(v);
    const int e = (int)((u >> 23) & 0xffu);
    if (e == 0 || e == 0xff) return 0;
    const long long m = (long long)((u & 0x7fffffu) | 0x800000u);     // v = m 2^(e - 150)
    const int sh = e - 150 + FIX_BITS;
    long long r;
    if (sh >= 0) r = m << sh;
    else if (sh > -25) r = (m + (1LL << (-sh - 1))) >> (-sh);
    else r = 0;
    return (u >> 31) ? -r : r;
}

// Momentum exchange (Eq. hydroF): blocks (k, b), k < FORCE_BLOCKS, split the
// links of body b into contiguous chunks and sum
//   F = sum e_a [2 f~_a(x_f) + 6 w_a rho(x_f) e_-a . u_w(x_f + e_a)],
//   T = sum (x_f + e_a / 2 - X) x F_link
// with f~ of step n (dst) and the body state of step n.  The last of body
// b's blocks to finish runs body b's rigid-body step on the two warps past its
// link warps; the last body to finish ends the step (clock, change flag).
//
// FP64 storage: every term in FP64; each block reduces with warp shuffles
// in a fixed order and writes its partial sums, which the rigid-body step
// adds in block order (deterministic).
//
// 32/16-bit storage: f~_a = w_a + delta_a splits each link term into a
// constant part 2 w_a e_a and a small variable part v e_a with
// v = 2 delta_a + 6 w_a rho e_-a . u_w.  With the fluid cell at integer
// offset i from the centre's cell and c the centre's position within it
// (x_f - X = i - c), the sums are
//   F = S1 / 36 + Fv,  T = (S2 - c x S1) / 36 + Tv - c x Fv,
//   S1 = sum 72 w_a e_a,  S2 = sum i x 72 w_a e_a   (exact integers),
//   Fv = sum v e_a,  Tv = sum v (i x e_a)           (FP32 terms, each rounded
// to 2^-FIX_BITS and added as 64-bit integers),
// since e_a x e_a = 0.  The large, cancelling constant part never meets a
// rounding, the variable part is ~1e-3 of a term, and integer sums make
// the result independent of the order of the blocks' atomic additions.
template <typename T>
__device__ __forceinline__ void force_body(const Device &dv, const StepPtrs &sp, const Blk &bk) {
    const Domain d = dv.dom;
    const int b = bk.y, kb = bk.x;
    const BodyProps pb = dv.props[b];
    const int side = 2 * (pb.E + 1) + 1;
    const int *counts = dv.seg_count + (long long)b * dv.link_side;
    const Link *links = dv.links + (long long)b * dv.link_side * dv.seg_cap;
    const T *pop = static_cast<const T *>(sp.dst);
    const long long C = d.C;
    const float s = dv.f16_inv_scale;

    // the two warps past the link warps integrate the body in the block that
    // finishes it; what they need of the state is loaded and formed meanwhile
    __shared__ int last_of_body;
    if (threadIdx.x >= FORCE_THREADS) {
        auto wait = [&] {
            __syncthreads();
            return last_of_body != 0;
        };
        if (threadIdx.x < FORCE_THREADS + 32) integrate_translation(dv, sp, b, 1, wait);
        else integrate_rotation(dv, sp, b, 1, wait);
        if (!last_of_body) return;
        asm volatile("bar.sync 2, 64;" ::: "memory");
        if (threadIdx.x < FORCE_THREADS + 32) {
            // the sums start the next step at zero
            const int ln = threadIdx.x & 31;
            if (sizeof(T) != 8 && ln < 6) {
                dv.fx[b * 6 + ln] = 0;
                dv.fi[b * 6 + ln] = 0;
            }
            if (ln == 0) {
                dv.body_done[b] = 0u;
                __threadfence();
                if (atomicAdd(dv.blocks_done, 1u) == (unsigned)bk.gy - 1) {
                    *dv.blocks_done = 0u;
                    finish_step(dv, sp);
                }
            }
        }
        return;
    }

    // exclusive prefix of the segment counts: thread t holds segments
    // [t per, (t+1) per), per <= 4 (side <= MAX_SEGMENTS), block scan
    __shared__ int prefix[MAX_SEGMENTS + 1];
    __shared__ int seg_warp[FORCE_THREADS / 32];
    {
        const int per = (side + FORCE_THREADS - 1) / FORCE_THREADS;
        const int k0 = threadIdx.x * per;
        int loc[MAX_SEGMENTS / FORCE_THREADS], sum = 0;
#pragma unroll
        for (int i = 0; i < MAX_SEGMENTS / FORCE_THREADS; ++i) {
            const int k = k0 + i;
            loc[i] = (i < per && k < side) ? counts[k] : 0;
            sum += loc[i];
        }
        const int ln = threadIdx.x & 31, wp = threadIdx.x >> 5;
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (ln >= o) incl += v;
        }
        if (ln == 31) seg_warp[wp] = incl;
        link_sync();
        int acc = incl - sum;
        for (int w = 0; w < wp; ++w) acc += seg_warp[w];
#pragma unroll
        for (int i = 0; i < MAX_SEGMENTS / FORCE_THREADS; ++i) {
            const int k = k0 + i;
            if (i < per && k < side) prefix[k] = acc;
            acc += loc[i];
        }
        if (threadIdx.x == FORCE_THREADS - 1) prefix[side] = acc;
    }
    link_sync();
    const int total = prefix[side];
    // FP64 partial sums are added in block order: the split is fixed.  The fixed-
    // point sums of the other types take any number of blocks.
    const int blocks = sizeof(T) == 8 ? FORCE_BLOCKS : bk.gx;
    const int chunk = (total + blocks - 1) / blocks;
    const int j0 = kb * chunk, j1 = min(total, j0 + chunk);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    if constexpr (sizeof(T) == 8) {
        const BodyState sb = sp.body_cur[b];
        // body centre wrapped into the domain (once per block)
        const double xw[3] = {d.px ? sb.X[0] - d.nx * floor(sb.X[0] * d.inx) : sb.X[0],
                              d.py ? sb.X[1] - d.ny * floor(sb.X[1] * d.iny) : sb.X[1],
                              d.pz ? sb.X[2] - d.nz * floor(sb.X[2] * d.inz) : sb.X[2]};
        double acc[6] = {0, 0, 0, 0, 0, 0};
        for (int j = j0 + threadIdx.x; j < j1; j += FORCE_THREADS) {
            int lo = 0, hi = side - 1;       // segment k with prefix[k] <= j < prefix[k+1]
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (prefix[mid] <= j) lo = mid; else hi = mid - 1;
            }
            const Link lk = links[(long long)lo * dv.seg_cap + (j - prefix[lo])];
            const long long c = lk.cell;
            const int a = (int)lk.dir;
            // cells are 32-bit indices (C < 2^31): 32-bit division
            const unsigned cu = lk.cell, nxu = (unsigned)d.nx, nyu = (unsigned)d.ny;
            const int x = (int)(cu % nxu), y = (int)((cu / nxu) % nyu), z = (int)(cu / (nxu * nyu));
            double rho = 1.0;
            for (int q = 0; q < Q; ++q) rho += load_dev<T>(pop + q * C + c, s);
            const double g_a = wgt(a) + load_dev<T>(pop + a * C + c, s);
            // offsets of the fluid cell, of the link end and of the link midpoint
            const double o0 = wrap_near(x - xw[0], d.nx, d.px);
            const double o1 = wrap_near(y - xw[1], d.ny, d.py);
            const double o2 = wrap_near(z - xw[2], d.nz, d.pz);
            const double e0 = o0 + ex(a), e1 = o1 + ey(a), e2 = o2 + ez(a);
            const double u0 = sb.V[0] + (sb.W[1] * e2 - sb.W[2] * e1);
            const double u1 = sb.V[1] + (sb.W[2] * e0 - sb.W[0] * e2);
            const double u2 = sb.V[2] + (sb.W[0] * e1 - sb.W[1] * e0);
            const double eu = -(ex(a) * u0 + ey(a) * u1 + ez(a) * u2);   // e_-a . u_w
            const double mag = 2.0 * g_a + 6.0 * wgt(a) * rho * eu;
            const double fl[3] = {ex(a) * mag, ey(a) * mag, ez(a) * mag};
            const double m0 = o0 + 0.5 * ex(a), m1 = o1 + 0.5 * ey(a), m2 = o2 + 0.5 * ez(a);
            acc[0] += fl[0]; acc[1] += fl[1]; acc[2] += fl[2];
            acc[3] += m1 * fl[2] - m2 * fl[1];
            acc[4] += m2 * fl[0] - m0 * fl[2];
            acc[5] += m0 * fl[1] - m1 * fl[0];
        }
        __shared__ double part[FORCE_THREADS / 32][6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            double v = acc[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) part[warp][i] = v;
        }
        link_sync();
        if (warp == 0) {
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                double v = lane < FORCE_THREADS / 32 ? part[lane][i] : 0.0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                if (lane == 0) dv.fpart[((long long)b * FORCE_BLOCKS + kb) * 6 + i] = v;
            }
        }
    } else {
        const BodyGeom *g = dv.geom + sp.parity * dv.nb + b;       // state n
        const int ci[3] = {g->ci[0], g->ci[1], g->ci[2]};
        const float cf[3] = {g->cf[0], g->cf[1], g->cf[2]};
        const float vf[3] = {g->v[0], g->v[1], g->v[2]}, wf[3] = {g->w[0], g->w[1], g->w[2]};
        long long accx[6] = {0, 0, 0, 0, 0, 0};
        int acci[6] = {0, 0, 0, 0, 0, 0};
        int bad = 0;
        for (int j = j0 + threadIdx.x; j < j1; j += FORCE_THREADS) {
            int lo = 0, hi = side - 1;       // segment k with prefix[k] <= j < prefix[k+1]
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (prefix[mid] <= j) lo = mid; else hi = mid - 1;
            }
            const Link lk = links[(long long)lo * dv.seg_cap + (j - prefix[lo])];
            const long long c = lk.cell;
            const int a = (int)lk.dir;
            const unsigned cu = lk.cell, nxu = (unsigned)d.nx, nyu = (unsigned)d.ny;
            const int x = (int)(cu % nxu), y = (int)((cu / nxu) % nyu), z = (int)(cu / (nxu * nyu));
            // rho - 1 of the fluid cell: the boundary kernel's record (every
            // link cell is listed, F_LINK)
            const float drho = __ldcg(dv.rho_near + c);
            const float rho = 1.0f + drho;
            const float da = load_dev_f<T>(pop + a * C + c, s);
            const int i0 = near_cell_k(x - ci[0], d.nx, d.px);
            const int i1 = near_cell_k(y - ci[1], d.ny, d.py);
            const int i2 = near_cell_k(z - ci[2], d.nz, d.pz);
            // u_w at the link end x_f + e_a
            const float e0 = ((float)i0 - cf[0]) + ex(a), e1 = ((float)i1 - cf[1]) + ey(a),
                        e2 = ((float)i2 - cf[2]) + ez(a);
            const float u0 = vf[0] + (wf[1] * e2 - wf[2] * e1);
            const float u1 = vf[1] + (wf[2] * e0 - wf[0] * e2);
            const float u2 = vf[2] + (wf[0] * e1 - wf[1] * e0);
            const float eu = -(ex(a) * u0 + ey(a) * u1 + ez(a) * u2);
            const float w6 = a < 7 ? 1.0f / 3.0f : 1.0f / 6.0f;    // 6 w_a (a > 0)
            const float v = 2.0f * da + w6 * rho * eu;
            // |delta| >= 2 is no fluid state; the bound keeps every sum in range
            if (!(fabsf(v) < 4.0f)) bad |= v != v ? ST_NAN : ST_UNSTABLE;
            const long long vx = to_fixed(v);
            accx[0] += ex(a) * vx;
            accx[1] += ey(a) * vx;
            accx[2] += ez(a) * vx;
            const int c0 = i1 * ez(a) - i2 * ey(a), c1 = i2 * ex(a) - i0 * ez(a), c2 = i0 * ey(a) - i1 * ex(a);
            accx[3] += to_fixed((float)c0 * v);
            accx[4] += to_fixed((float)c1 * v);
            accx[5] += to_fixed((float)c2 * v);
            const int K = a < 7 ? 4 : 2;          // 72 w_a
            acci[0] += K * ex(a);
            acci[1] += K * ey(a);
            acci[2] += K * ez(a);
            acci[3] += K * c0;
            acci[4] += K * c1;
            acci[5] += K * c2;
        }
        if (bad) atomicOr(dv.status, bad);
        __shared__ long long px_[FORCE_THREADS / 32][6];
        __shared__ int pi_[FORCE_THREADS / 32][6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            long long v = accx[i];
            int w = acci[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                v += __shfl_down_sync(0xffffffffu, v, o);
                w += __shfl_down_sync(0xffffffffu, w, o);
            }
            if (lane == 0) {
                px_[warp][i] = v;
                pi_[warp][i] = w;
            }
        }
        link_sync();
        if (threadIdx.x < 6) {
            const int i = threadIdx.x;
            long long v = 0;
            int w = 0;
            for (int k = 0; k < FORCE_THREADS / 32; ++k) {
                v += px_[k][i];
                w += pi_[k][i];
            }
            if (v) atomicAdd(reinterpret_cast<unsigned long long *>(dv.fx + b * 6 + i), (unsigned long long)v);
            if (w) atomicAdd(dv.fi + b * 6 + i, w);
        }
    }
    // the last of body b's blocks lets its integrating warps go on; the last body
    // ends the step
    link_sync();
    if (threadIdx.x == 0) {
        __threadfence();
        last_of_body = atomicAdd(dv.body_done + b, 1u) == (unsigned)bk.gx - 1;
        __threadfence();
    }
    __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(FORCE_BLOCK) force_kernel(const Device dv, const StepPtrs sp) {
    pdl_enter();
    force_body<T>(dv, sp, launch_blk());
}

template <typename T>
__global__ void __launch_bounds__(FORCE_BLOCK) force_batch(const Batch bt) {
    LBM_BATCH_MEMBER(bt);
    force_body<T>(sdv, ssp, sbk);
}

// the end of a step of a lattice without bodies: the step counter advances
// (BF16 storage draws its rounding bits from it) and the next epoch's change
// flag starts clear
__global__ void tick_kernel(const Device dv, const StepPtrs sp) {
    if (threadIdx.x == 0) finish_step(dv, sp);
}

// The near tiles of the step of parity q (one block): the marks of that
// parity's previous list are cleared, then every TILE_X-cell tile of an
// x-row that meets the remap cube of a body in `states` grown by one cell is
// marked and listed once.  The cube is the remap's: half-width
// E + REMAP_MARGIN around floor(X).  Also stores the step's index.
__global__ void __launch_bounds__(512) near_tiles_kernel(const Device dv, const BodyState *states, int q,
                                                         int step_offset) {
    const Domain d = dv.dom;
    unsigned *mask = dv.near_mask[q];
    int *list = dv.near_list[q];
    const int old = min(dv.near_count[q], dv.near_cap);
    for (int i = threadIdx.x; i < old; i += blockDim.x) mask[list[i]] = 0u;
    __syncthreads();
    if (threadIdx.x == 0) {
        dv.near_count[q] = 0;
        dv.tstep[q] = *dv.t_dev + step_offset;
    }
    __syncthreads();
    const int ntx = (d.nx + TILE_X - 1) / TILE_X;
    const int n3[3] = {d.nx, d.ny, d.nz}, per[3] = {d.px, d.py, d.pz};
    for (int b = 0; b < dv.nb; ++b) {
        const int half = dv.props[b].E + REMAP_MARGIN + 1;
        const int side = 2 * half + 1;
        int o[3];
        for (int a = 0; a < 3; ++a) o[a] = (int)floor(states[b].X[a]) - half;
        for (int r = threadIdx.x; r < side * side; r += blockDim.x) {
            int y = o[1] + r % side, z = o[2] + r / side;
            if (per[1]) y = ((y % n3[1]) + n3[1]) % n3[1]; else if (y < 0 || y >= n3[1]) continue;
            if (per[2]) z = ((z % n3[2]) + n3[2]) % n3[2]; else if (z < 0 || z >= n3[2]) continue;
            // the row's x range as up to two unwrapped pieces [lo, hi]
            int lo[2], hi[2], pieces = 1;
            if (!per[0]) {
                lo[0] = max(o[0], 0);
                hi[0] = min(o[0] + side - 1, n3[0] - 1);
            } else if (side >= n3[0]) {
                lo[0] = 0;
                hi[0] = n3[0] - 1;
            } else {
                const int x0 = ((o[0] % n3[0]) + n3[0]) % n3[0];
                lo[0] = x0;
                hi[0] = min(x0 + side - 1, n3[0] - 1);
                if (x0 + side - 1 >= n3[0]) {
                    lo[1] = 0;
                    hi[1] = x0 + side - 1 - n3[0];
                    pieces = 2;
                }
            }
            const long long rowt = ((long long)z * n3[1] + y) * ntx;
            for (int k = 0; k < pieces; ++k)
                for (int cx = lo[k] / TILE_X; lo[k] <= hi[k] && cx <= hi[k] / TILE_X; ++cx) {
                    const int t = (int)(rowt + cx);
                    if (atomicExch(mask + t, 1u) == 0u) {
                        const int i = atomicAdd(dv.near_count + q, 1);
                        if (i < dv.near_cap) list[i] = t;
                        else atomicOr(dv.status, ST_LINKS);
                    }
                }
        }
    }
}

// the rigid-body step alone (bodies without fluid): the loads (each block all of
// them, the same values), then two warps a body, INTEGRATE_BODIES of them a block.
// Bound by the FP64 pipe, so many bodies in one block wait for one SM's (254
// bodies: 179 us a step with a warp a body and 186 us with two in one block, 6.0
// us in blocks of four bodies); the last block to finish ends the step.
constexpr int INTEGRATE_BODIES = 4;
__global__ void __launch_bounds__(64 * INTEGRATE_BODIES) integrate_kernel(const Device dv, const StepPtrs sp, int with_fluid) {
    body_loads(dv, sp, threadIdx.x, threadIdx.x, blockDim.x);
    __syncthreads();
    auto go = [] { return true; };
    const int i = blockIdx.x * 2 * INTEGRATE_BODIES + (threadIdx.x >> 5);
    if (i < 2 * dv.nb) {
        if (i & 1) integrate_rotation(dv, sp, i >> 1, with_fluid, go);
        else integrate_translation(dv, sp, i >> 1, with_fluid, go);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (gridDim.x > 1) {
            __threadfence();
            if (atomicAdd(dv.blocks_done, 1u) != gridDim.x - 1) return;
            *dv.blocks_done = 0u;
        }
        finish_step(dv, sp);
    }
}

// ---- field export / import -----------------------------------------------

// The rounding error of s = a + b: TwoSum (Knuth; Moller), so that a + b = s + e exactly.
// Infinities and NaN do not survive it (inf - inf): callers check the result.
__device__ __forceinline__ float sum_error(float a, float b, float s) {
    const float t = s - a;
    return (a - (s - t)) + (b - t);
}

// Sums of 19 FP32 values as float expansions, without the FP64 pipe (2 results a
// cycle an SM here, against 128 FP32 ones).  FloatSum (hi + lo) is off by at most
// 190 2^-48 of the values' absolute sum S, enough beside 1 in a density; FloatSum3
// by less than 2^-60 S, which also leaves a small difference of large values its digits.
struct FloatSum {
    float hi, lo;
    __device__ __forceinline__ void add(float v) {
        const float s = hi + v;
        lo += sum_error(hi, v, s);
        hi = s;
    }
};
struct FloatSum3 {
    float a, b, c;
    __device__ __forceinline__ void add_low(float v) {      // a value of the size of a's rounding errors
        const float s = b + v;
        c += sum_error(b, v, s);
        b = s;
    }
    __device__ __forceinline__ void add(float v) {
        const float s = a + v;
        add_low(sum_error(a, v, s));
        a = s;
    }
    // the sum as hi + lo, lo at most half an ulp of hi (to 2^-48 of the sum)
    __device__ __forceinline__ FloatSum two() const {
        const float h = a + b, l = sum_error(a, b, h);
        const float l2 = l + c, m = sum_error(l, c, l2);
        const float g = h + l2;
        return FloatSum{g, sum_error(h, l2, g) + m};
    }
};

// w_a + delta as stored in O.  FP32 output of 32/16-bit storage adds the two
// parts of w_a (FP32 value and remainder) with one TwoSum: the FP64 sum rounded
// to FP32, but within 2^-23 of an ulp of a tie, where the rounding of the
// remainders decides (a branch to FP64 there costs what FP64 for all does).
template <typename O, typename T>
__device__ __forceinline__ O pop_value(double w, float wh, float wl, const T *v, float scale) {
    if constexpr (sizeof(O) == 4 && sizeof(T) <= 4) {
        const float x = load_dev_f<T>(v, scale);
        const float s = wh + x;
        return fabsf(s) < INFINITY ? s + (sum_error(wh, x, s) + wl) : s;
    } else {
        return (O)(w + load_dev<T>(v, scale));
    }
}

// Populations: a plain stream of V-wide vectors, EXPORT_U of them a thread in
// flight, direction blockIdx.y.  Bound by HBM: 33.5 M cells from FP32 to FP32
// (5.1 GB) take 0.72 ms; a thread a cell with FP64 sums took 3.38 ms, bound by
// the FP64 pipe's conversions and additions.
constexpr int EXPORT_THREADS = 256;
constexpr int EXPORT_U = 4;

template <int BYTES> struct Chunk;
template <> struct Chunk<2> { using type = unsigned short; };
template <> struct Chunk<4> { using type = unsigned; };
template <> struct Chunk<8> { using type = uint2; };
template <> struct Chunk<16> { using type = uint4; };

// V consecutive values to `p` in pieces of at most 16 bytes
template <typename O, int V>
__device__ __forceinline__ void put_values(O *p, const O (&o)[V]) {
    constexpr int B = V * (int)sizeof(O) < 16 ? V * (int)sizeof(O) : 16, PER = B / (int)sizeof(O);
    using R = typename Chunk<B>::type;
#pragma unroll
    for (int k = 0; k < V / PER; ++k) {
        R r;
        memcpy(&r, o + k * PER, B);
        *reinterpret_cast<R *>(p + k * PER) = r;
    }
}

template <typename T, typename O, int V>
__global__ void __launch_bounds__(EXPORT_THREADS)
export_pop_kernel(const T *__restrict__ pop, long long C, float scale, O *__restrict__ out) {
    using R = typename Chunk<V * (int)sizeof(T)>::type;
    const int a = blockIdx.y;
    const double w = wgt(a);
    const float wh = (float)w, wl = (float)(w - (double)wh);
    const T *__restrict__ src = pop + a * C;
    O *__restrict__ dst = out + a * C;
    const long long groups = C / V, i0 = (long long)blockIdx.x * (EXPORT_THREADS * EXPORT_U) + threadIdx.x;
    R r[EXPORT_U];
#pragma unroll
    for (int u = 0; u < EXPORT_U; ++u) {
        const long long i = i0 + u * EXPORT_THREADS;
        if (i < groups) r[u] = __ldg(reinterpret_cast<const R *>(src) + i);
    }
#pragma unroll
    for (int u = 0; u < EXPORT_U; ++u) {
        const long long i = i0 + u * EXPORT_THREADS;
        if (i >= groups) break;
        T v[V];
        memcpy(&v, &r[u], sizeof(R));
        O o[V];
#pragma unroll
        for (int k = 0; k < V; ++k) o[k] = pop_value<O, T>(w, wh, wl, v + k, scale);
        put_values<O, V>(dst + i * V, o);
    }
}

// density deviation and momentum of one cell's deviations, in FP64, in
// direction order
template <typename T>
__device__ __forceinline__ void moments_f64(const T (&v)[Q], float scale, double &drho, double (&j)[3]) {
    drho = j[0] = j[1] = j[2] = 0.0;
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        const double x = load_dev<T>(&v[a], scale);
        drho += x;
        if (ex(a)) j[0] += ex(a) > 0 ? x : -x;
        if (ey(a)) j[1] += ey(a) > 0 ? x : -x;
        if (ez(a)) j[2] += ez(a) > 0 ? x : -x;
    }
}

// Density (U = false) or velocity (U = true) of each cell, one thread a cell,
// all 19 loads issued before the sums.  FP32 output of 32/16-bit storage sums in
// float expansions and divides with one correction step: the exact value rounded
// once, to 2^-20 of an ulp, as from FP64 sums (one FP32 remainder of a two-part
// momentum was up to 7e-4 of an ulp further off where forces cancel it).  FP64
// storage and FP64 output sum in FP64, as does a cell whose sums are not finite.
// (128^3 cells from FP32, velocity: 48 us, FP64 sums 480 us, two-part sums 41 us.)
template <typename T, typename O, bool U>
__global__ void __launch_bounds__(EXPORT_THREADS)
export_moments_kernel(const Device dv, const T *__restrict__ pop, const uint8_t *__restrict__ flags, int mask_solid,
                      O *__restrict__ out) {
    const long long C = dv.dom.C;
    const long long c = (long long)blockIdx.x * EXPORT_THREADS + threadIdx.x;
    if (c >= C) return;
    const float scale = dv.f16_inv_scale;
    const bool solid = mask_solid && (flags[c] & F_SOLID);
    T v[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) v[a] = pop[a * C + c];
    if (solid) {
        if constexpr (U) {
            for (int i = 0; i < 3; ++i) out[i * C + c] = (O)0;
        } else {
            out[c] = (O)1;
        }
        return;
    }
    if constexpr (sizeof(O) == 4 && sizeof(T) <= 4) {
        float x[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) x[a] = load_dev_f<T>(&v[a], scale);
        FloatSum s{x[0], 0.0f};
#pragma unroll
        for (int a = 1; a < Q; ++a) s.add(x[a]);
        FloatSum rho{1.0f, s.lo};
        rho.add(s.hi);
        if constexpr (!U) {
            const float r = rho.hi + rho.lo;
            if (fabsf(r) < INFINITY) {
                out[c] = r;
                return;
            }
        } else {
            // momentum by pairs of opposite directions: x_a - x_a+1 = dh + dl
            FloatSum3 j[3];
#pragma unroll
            for (int p = 0; p < Q / 2; ++p) {
                const int a = 2 * p + 1;
                const float dh = x[a] - x[a + 1], dl = sum_error(x[a], -x[a + 1], dh);
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const int e = i == 0 ? ex(a) : (i == 1 ? ey(a) : ez(a));
                    if (e == 0) continue;
                    if (p == i) {
                        j[i] = FloatSum3{dh, dl, 0.0f};
                    } else {
                        j[i].add(e > 0 ? dh : -dh);
                        j[i].add_low(e > 0 ? dl : -dl);
                    }
                }
            }
            const float inv = 1.0f / rho.hi;
            float q[3];
            bool finite = true;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const float gh = dv.gh_f[i];            // g / 2 in three parts
                j[i].add(-gh);
                j[i].add_low(-dv.gl_f[i]);
                j[i].c -= dv.gr_f[i];
                // scaled, so that the remainders of the smallest momenta do not underflow
                FloatSum n = j[i].two();
                n.hi *= 0x1p48f;
                n.lo *= 0x1p48f;
                const float q0 = n.hi * inv;
                q[i] = fmaf(fmaf(-q0, rho.hi, n.hi) + fmaf(-q0, rho.lo, n.lo), inv, q0);
                finite = finite && fabsf(q[i]) < INFINITY;
            }
            if (finite) {
                for (int i = 0; i < 3; ++i) out[i * C + c] = q[i] * 0x1p-48f;
                return;
            }
        }
    }
    double drho, j[3];
    moments_f64<T>(v, scale, drho, j);
    const double rho = 1.0 + drho;
    if constexpr (U) {
        for (int i = 0; i < 3; ++i) out[i * C + c] = (O)((j[i] - 0.5 * dv.g[i]) / rho);
    } else {
        out[c] = (O)rho;
    }
}

__global__ void export_flags_kernel(const uint8_t *flags, const uint8_t *bid, long long C, int mask_solid, uint8_t *out) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < C) out[c] = mask_solid && (flags[c] & F_SOLID) ? (uint8_t)(bid[c] + 1) : 0;
}

// Running time average of the velocity (Sec. 6, the flow fields averaged
// over swimming cycles): each step adds the velocity of the populations it
// wrote, u = (sum e f~ - g/2) / rho (0 in obstacle cells, the value the U
// field reports), to an FP64 sum per cell and component.  The moments are
// FP64 for FP64 storage and FP32 otherwise (FP64 arithmetic is slow on this
// part); the sum is FP64 so that long windows keep their digits.
template <typename T>
__global__ void __launch_bounds__(256) average_kernel(const Device dv, const StepPtrs sp) {
    const long long C = dv.dom.C;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    double u[3] = {0.0, 0.0, 0.0};
    if (!(sp.flags_cur[c] & F_SOLID)) {
        const T *pop = static_cast<const T *>(sp.dst);
        if constexpr (sizeof(T) == 8) {
            double drho = 0.0, j[3] = {0.0, 0.0, 0.0};
            for (int a = 0; a < Q; ++a) {
                const double v = pop[a * C + c];
                drho += v;
                j[0] += ex(a) * v; j[1] += ey(a) * v; j[2] += ez(a) * v;
            }
            for (int i = 0; i < 3; ++i) u[i] = (j[i] - 0.5 * dv.g[i]) / (1.0 + drho);
        } else {
            float drho = 0.0f, j[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                const float v = load_dev_f<T>(pop + a * C + c, dv.f16_inv_scale);
                drho += v;
                if (ex(a)) j[0] += ex(a) > 0 ? v : -v;
                if (ey(a)) j[1] += ey(a) > 0 ? v : -v;
                if (ez(a)) j[2] += ez(a) > 0 ? v : -v;
            }
            const float inv = 1.0f / (1.0f + drho);
            for (int i = 0; i < 3; ++i) u[i] = (double)((j[i] - 0.5f * dv.g_f[i]) * inv);
        }
    }
    for (int i = 0; i < 3; ++i) dv.avg_u[i * C + c] += u[i];
    if (c == 0) *dv.avg_n += 1;
}

template <typename T>
__global__ void import_kernel(const Device dv, T *pop, const double *in) {
    const long long C = dv.dom.C;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    for (int a = 0; a < Q; ++a) {
        const double delta = in[a * C + c] - wgt(a);
        if constexpr (sizeof(T) == 8) pop[a * C + c] = delta;
        else if constexpr (sizeof(T) == 4) pop[a * C + c] = (float)delta;
        else if constexpr (std::is_same<T, __half>::value) pop[a * C + c] = __float2half_rn((float)delta * dv.f16_scale);
        else pop[a * C + c] = __float2bfloat16_rn((float)delta);
    }
}

unsigned blocks_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

}  // namespace

void launch_init_flags(const Device &dv, uint8_t *flags0, uint8_t *flags1, uint8_t *bid0, uint8_t *bid1,
                       cudaStream_t s) {
    init_flags_kernel<<<blocks_for(dv.dom.C, 256), 256, 0, s>>>(dv.dom, flags0, flags1, bid0, bid1);
}

void launch_prep(const Device &dv, const StepPtrs &sp, cudaStream_t s) {
    prep_kernel<<<1, PREP_THREADS, 0, s>>>(dv, sp);
}

void launch_remap(const Device &dv, const StepPtrs &sp, int init_mode, cudaStream_t s, bool prep) {
    if (prep) launch_prep(dv, sp, s);
    const int side = dv.remap_side;
    launch_kernel(dv.pdl != 0, remap_kernel, dim3((unsigned)remap_blocks(side), dv.nb), dim3(REMAP_THREADS), 0, s,
                  dv, sp, init_mode);
}

void launch_links(const Device &dv, const StepPtrs &sp, cudaStream_t s) {
    links_kernel<<<dim3(dv.link_side, dv.nb), 256, 0, s>>>(dv, sp);
}

void launch_loads(const Device &dv, const StepPtrs &sp, cudaStream_t s) { loads_kernel<<<1, 64, 0, s>>>(dv, sp); }

void launch_force(const Device &dv, const StepPtrs &sp, cudaStream_t s) {
    const dim3 grid(FORCE_BLOCKS, dv.nb), block(FORCE_BLOCK);
    const bool pdl = dv.pdl != 0;
    switch (dv.precision) {
    case 0: launch_kernel(pdl, force_kernel<double>, grid, block, 0, s, dv, sp); break;
    case 1: launch_kernel(pdl, force_kernel<float>, grid, block, 0, s, dv, sp); break;
    case 2: launch_kernel(pdl, force_kernel<__half>, grid, block, 0, s, dv, sp); break;
    default: launch_kernel(pdl, force_kernel<__nv_bfloat16>, grid, block, 0, s, dv, sp); break;
    }
}

void launch_integrate(const Device &dv, const StepPtrs &sp, int with_fluid, cudaStream_t s) {
    integrate_kernel<<<(dv.nb + INTEGRATE_BODIES - 1) / INTEGRATE_BODIES, 64 * INTEGRATE_BODIES, 0, s>>>(dv, sp, with_fluid);
}

void launch_tick(const Device &dv, const StepPtrs &sp, cudaStream_t s) { tick_kernel<<<1, 32, 0, s>>>(dv, sp); }

void launch_near_tiles(const Device &dv, const BodyState *states, int q, int step_offset, cudaStream_t s) {
    near_tiles_kernel<<<1, 512, 0, s>>>(dv, states, q, step_offset);
}

long long near_tile_count(const Device &dv) {
    return (long long)((dv.dom.nx + TILE_X - 1) / TILE_X) * dv.dom.ny * dv.dom.nz;
}

int near_tile_cap(const Device &dv, int emax) {
    const long long side = 2LL * (emax + REMAP_MARGIN + 1) + 1;
    const long long per_body = side * side * ((side + TILE_X - 1) / TILE_X + 1);
    return (int)std::min<long long>((long long)dv.nb * per_body, near_tile_count(dv));
}

// Force blocks a body in a batched launch over `members` lattices like dv: with
// many bodies a block's member lookup and reductions cost more than its further
// rounds of links, also for large bodies (FP32, a step with this rule and with 8
// blocks a body: 48 boxes of three spheres of radius 3 193 and 213 us, 8 boxes of
// 27 of radius 5 192 and 211, 24 boxes of three of radius 10 648 and 655, 12 of
// three of radius 12 506 and 508, 70 boxes of one of radius 12 394 and 401 us).
// FP64 keeps its split, which the sums' order depends on.
static int force_batch_blocks(const Device &dv, int members) {
    const int bodies = members * dv.nb;
    return dv.precision == 0 || bodies < 16 ? FORCE_BLOCKS : (bodies < 64 ? 2 : 1);
}

// the grids of launch_remap, launch_links and launch_force for one lattice of a
// batched launch over `members` of them
void batch_grid_small(const Device &dv, int k, int members, int g[3]) {
    g[0] = g[1] = g[2] = 0;
    if (dv.nb == 0) return;
    const int side = dv.remap_side;
    switch (k) {
    // few bodies are all remap candidates, and states the host wrote are prepared
    // before a batched run: nothing to prepare in its steps
    case BK_PREP: g[0] = g[1] = g[2] = dv.nb > REMAP_STAGED ? 1 : 0; break;
    case BK_LOADS: g[0] = g[1] = g[2] = 1; break;
    case BK_REMAP:
        g[0] = remap_blocks(side);
        g[1] = dv.nb; g[2] = 1;
        break;
    case BK_LINKS: g[0] = dv.link_side; g[1] = dv.nb; g[2] = 1; break;
    case BK_FORCE: g[0] = force_batch_blocks(dv, members); g[1] = dv.nb; g[2] = 1; break;
    default: break;
    }
}

void launch_batch_small(int k, const Batch &bt, unsigned blocks, int precision, cudaStream_t s) {
    if (blocks == 0) return;
    switch (k) {
    case BK_PREP: prep_batch<<<blocks, PREP_THREADS, 0, s>>>(bt); break;
    case BK_REMAP: remap_batch<<<blocks, REMAP_THREADS, 0, s>>>(bt); break;
    case BK_LINKS: links_batch<<<blocks, 256, 0, s>>>(bt); break;
    case BK_LOADS: loads_batch<<<blocks, 64, 0, s>>>(bt); break;
    case BK_FORCE:
        switch (precision) {
        case 0: force_batch<double><<<blocks, FORCE_BLOCK, 0, s>>>(bt); break;
        case 1: force_batch<float><<<blocks, FORCE_BLOCK, 0, s>>>(bt); break;
        case 2: force_batch<__half><<<blocks, FORCE_BLOCK, 0, s>>>(bt); break;
        default: force_batch<__nv_bfloat16><<<blocks, FORCE_BLOCK, 0, s>>>(bt); break;
        }
        break;
    default: break;
    }
}

template <typename T, typename O, int V>
static void export_pop(const Device &dv, const T *pop, O *out, cudaStream_t s) {
    const long long groups = dv.dom.C / V;
    const dim3 grid(blocks_for(groups, EXPORT_THREADS * EXPORT_U), Q);
    export_pop_kernel<T, O, V><<<grid, EXPORT_THREADS, 0, s>>>(pop, dv.dom.C, dv.f16_inv_scale, out);
}

template <typename T, typename O>
static void export_typed(const Device &dv, const void *pop_, const uint8_t *flags, int what, int mask_solid, O *out,
                         cudaStream_t s) {
    const T *pop = static_cast<const T *>(pop_);
    const unsigned bl = blocks_for(dv.dom.C, EXPORT_THREADS);
    if (what == LBM_FIELD_RHO) {
        export_moments_kernel<T, O, false><<<bl, EXPORT_THREADS, 0, s>>>(dv, pop, flags, mask_solid, out);
    } else if (what == LBM_FIELD_U) {
        export_moments_kernel<T, O, true><<<bl, EXPORT_THREADS, 0, s>>>(dv, pop, flags, mask_solid, out);
    } else {
        // 16-byte loads where every direction's run of cells and the caller's
        // buffer allow them; the planes themselves are aligned (the handle's
        // allocation), an odd cell count or an offset buffer takes single values
        constexpr int V = 16 / (int)sizeof(T);
        constexpr int A = V * (int)sizeof(O) < 16 ? V * (int)sizeof(O) : 16;
        if (dv.dom.C % V == 0 && reinterpret_cast<uintptr_t>(out) % A == 0 &&
            reinterpret_cast<uintptr_t>(pop_) % 16 == 0)
            export_pop<T, O, V>(dv, pop, out, s);
        else
            export_pop<T, O, 1>(dv, pop, out, s);
    }
}

template <typename O>
static void export_as(const Device &dv, const void *pop, const uint8_t *flags, int what, int mask_solid, O *out,
                      cudaStream_t s) {
    switch (dv.precision) {
    case 0: export_typed<double, O>(dv, pop, flags, what, mask_solid, out, s); break;
    case 1: export_typed<float, O>(dv, pop, flags, what, mask_solid, out, s); break;
    case 2: export_typed<__half, O>(dv, pop, flags, what, mask_solid, out, s); break;
    default: export_typed<__nv_bfloat16, O>(dv, pop, flags, what, mask_solid, out, s); break;
    }
}

void launch_export(const Device &dv, const void *pop, const uint8_t *flags, const uint8_t *bid, int what,
                   int mask_solid, void *out, int dtype, cudaStream_t s) {
    if (what == LBM_FIELD_FLAGS)
        export_flags_kernel<<<blocks_for(dv.dom.C, 256), 256, 0, s>>>(flags, bid, dv.dom.C, mask_solid,
                                                                      static_cast<uint8_t *>(out));
    else if (dtype == LBM_DTYPE_F32)
        export_as<float>(dv, pop, flags, what, mask_solid, static_cast<float *>(out), s);
    else
        export_as<double>(dv, pop, flags, what, mask_solid, static_cast<double *>(out), s);
}

void launch_average(const Device &dv, const StepPtrs &sp, cudaStream_t s) {
    const unsigned bl = blocks_for(dv.dom.C, 256);
    switch (dv.precision) {
    case 0: average_kernel<double><<<bl, 256, 0, s>>>(dv, sp); break;
    case 1: average_kernel<float><<<bl, 256, 0, s>>>(dv, sp); break;
    case 2: average_kernel<__half><<<bl, 256, 0, s>>>(dv, sp); break;
    default: average_kernel<__nv_bfloat16><<<bl, 256, 0, s>>>(dv, sp); break;
    }
}

void launch_import_pop(const Device &dv, void *pop, const double *in, cudaStream_t s) {
    const unsigned bl = blocks_for(dv.dom.C, 256);
    switch (dv.precision) {
    case 0: import_kernel<double><<<bl, 256, 0, s>>>(dv, (double *)pop, in); break;
    case 1: import_kernel<float><<<bl, 256, 0, s>>>(dv, (float *)pop, in); break;
    case 2: import_kernel<__half><<<bl, 256, 0, s>>>(dv, (__half *)pop, in); break;
    default: import_kernel<__nv_bfloat16><<<bl, 256, 0, s>>>(dv, (__nv_bfloat16 *)pop, in); break;
    }
}

}  // namespace lbm
