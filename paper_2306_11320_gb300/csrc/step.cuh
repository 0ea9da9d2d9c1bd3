// The fused time step of the three coupled LBEs (arXiv 2306.11320, Sec. 3-4):
// a general tile routine (every boundary rule, thread loads) and a persistent
// kernel that stages interior tiles in shared memory with TMA, double buffered.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lattice.cuh"

namespace tpf {

// FP16 storage keeps the scaled deviation s_k (q_i - r_i) of each population from a
// reference r_i built from a record that the population's writer leaves for the next
// step:
//   f: r_i = w_i (phi + c_i . J_f / cs2)      h: r_i = w_i (T + c_i . J_h / cs2)
//   g: r_i = wg_i p / cs2 + w_i c_i . J_g / cs2   (wg_0 = w_0 - 1, wg_i = w_i)
// with phi, T, p the writer's moments and J_f, J_g, J_h the first moments of its
// post-collision f, g, h, i.e. the rest equilibrium plus the first-order Hermite term
// of what it emitted, so that only the higher-order non-equilibrium part is
// quantised.  The writer of population i at y is the node it streamed from, y - c_i
// (wrapped when periodic), except where y - c_i lies outside the fluid: a population
// reflected at a wall or at the inlet (and g reflected at the outflow) was written by
// y itself, and f, h entering through the outflow are the copies that the last
// column's node y - c_iy (same column) made of its own populations.  A record is one
// 8-byte word per LBE and node: the zeroth moment in float32 and J / cs2 as two
// halves; the writer encodes against the rounded record, so encoder and decoder see
// the same reference bit for bit.
template <class S>
constexpr bool kRef = S::kRecords;

using RefT = uint2;  // one reference record: float32 zeroth moment, half2 first moment / cs2
constexpr int kRecF = 0, kRecG = 1, kRecH = 2;  // record planes

struct RefVals {
    float m0, jx, jy;
};
__device__ __forceinline__ RefVals ref_unpack(RefT q)
{
    const float2 j = __half22float2(*reinterpret_cast<const __half2*>(&q.y));
    return {__uint_as_float(q.x), j.x, j.y};
}
// keeps m0, rounds (jx, jy) to halves; r receives the values the decoder will see
__device__ __forceinline__ RefT ref_pack(float m0, float jx, float jy, RefVals& r)
{
    const __half2 j = __floats2half2_rn(jx, jy);
    const float2 fj = __half22float2(j);
    r = {m0, fj.x, fj.y};
    RefT q;
    q.x = __float_as_uint(m0);
    q.y = *reinterpret_cast<const uint32_t*>(&j);
    return q;
}

// c_i . (vx, vy) for a moving direction i, adding only its nonzero components (after
// unrolling, i is a constant and the selects fold away)
__device__ __forceinline__ float cdot(int i, float vx, float vy)
{
    const float a = cx(i) > 0 ? vx : -vx, b = cy(i) > 0 ? vy : -vy;
    return cx(i) == 0 ? b : (cy(i) == 0 ? a : a + b);
}
// reference of population i of f or h from its writer's record
__device__ __forceinline__ float ref_pop(int i, const RefVals& r)
{
    return i == 0 ? wq(0) * r.m0 : wq(i) * (r.m0 + cdot(i, r.jx, r.jy));
}
// reference of population i of g (r.m0 = p / cs2)
__device__ __forceinline__ float ref_g(int i, const RefVals& r)
{
    return i == 0 ? wg(0) * r.m0 : fmaf(wg(i), r.m0, wq(i) * cdot(i, r.jx, r.jy));
}

// deviations v - ref_pop and v - ref_g with the reference's product in the same rounding
// (the encoder's side)
__device__ __forceinline__ float dev_pop(int i, const RefVals& r, float v)
{
    return i == 0 ? fmaf(-wq(0), r.m0, v) : fmaf(-wq(i), r.m0 + cdot(i, r.jx, r.jy), v);
}
__device__ __forceinline__ float dev_g(int i, const RefVals& r, float v)
{
    return i == 0 ? fmaf(-wg(0), r.m0, v) : v - ref_g(i, r);
}

// node that wrote population i at (x, y), whose record is its FP16 reference (for the
// g LBE when g_lbe: the outflow reflects g at the node itself)
__device__ __forceinline__ int ref_source(const DevParams& P, int x, int y, int i, bool g_lbe)
{
    int sx = x - cx(i), sy = y - cy(i);
    if (P.bc_x == 0) sx = wrap(sx, P.nx);
    if (P.bc_y == 1) sy = wrap(sy, P.ny);
    if (sy < 0 || sy >= P.ny || sx < 0 || (sx >= P.nx && g_lbe)) return y * P.nx + x;
    if (sx >= P.nx) return sy * P.nx + (P.nx - 1);  // outflow copy made by (nx - 1, sy)
    return sy * P.nx + sx;
}

// ref_source for a node of a TMA tile: the writer's slot in the tile's record box
// (origin x0 - 4, y0 - 2, RW x RH; columns beyond a periodic x seam hold the wrapped nodes'
// records).  Every writer lies in the box; the clamps only keep the slot inside it when P
// itself is not to be trusted (a batched tile whose copies, parameters included, timed out).
template <bool SEAM>
__device__ __forceinline__ int ref_slot_box(const DevParams& P, int x, int y, int i, bool g_lbe, int x0, int y0,
                                            int RW, int RH)
{
    int sx = x - cx(i), sy = y - cy(i);
    const bool open = !SEAM || P.bc_x != 0;  // x ends at an inlet and an outflow
    if (sy < 0 || sy >= P.ny || (open && (sx < 0 || (sx >= P.nx && g_lbe)))) {
        sx = x;
        sy = y;
    } else if (open && sx >= P.nx) {
        sx = P.nx - 1;
    }
    const int c = min(max(sx - x0 + 4, 0), RW - 1), r = min(max(sy - y0 + 2, 0), RH - 1);
    return r * RW + c;
}

// Decoded populations of node (x, y) read from global memory (general path).
template <class S, bool WANT_G = true>
__device__ __forceinline__ void load_node(const DevParams& P, const typename S::elem* __restrict__ A,
                                          const RefT* __restrict__ ref, int x, int y, float* f, float* g,
                                          float* h)
{
    const long long pl = P.plane;
    const int n = y * P.nx + x;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        float rf = 0.f, rg = 0.f, rh = 0.f;
        if constexpr (kRef<S>) {
            const int s = ref_source(P, x, y, i, false);
            rf = ref_pop(i, ref_unpack(ref[kRecF * pl + s]));
            rh = ref_pop(i, ref_unpack(ref[kRecH * pl + s]));
            if constexpr (WANT_G) rg = ref_g(i, ref_unpack(ref[kRecG * pl + ref_source(P, x, y, i, true)]));
        }
        f[i] = S::ld(A + i * pl, n, P.is_f, rf);
        if constexpr (WANT_G) g[i] = S::ld(A + (9 + i) * pl, n, P.is_g, rg);
        h[i] = S::ld(A + (18 + i) * pl, n, P.is_h, rh);
    }
}

// Shared staging of phi, T, 1/(rho c_p) and pre-collision h for a tile and its ring.
template <int BX, int BY>
struct RingSmem {
    static constexpr int SX = BX + 2, SY = BY + 2, SN = SX * SY;
    float phi[SN];
    float T[SN];
    float irc[SN];
    float h[9][SN];
};

// What lies one c_i away from node (x, y): the wall, the inlet, the outflow or node d.
enum Link { kNode, kWall, kInlet, kOutflow };
__device__ __forceinline__ Link link_of(const DevParams& P, int x, int y, int i, int& d)
{
    int dx = x + cx(i), dy = y + cy(i);
    if (P.bc_x == 0) dx = wrap(dx, P.nx);
    if (P.bc_y == 1) dy = wrap(dy, P.ny);
    d = dy * P.nx + dx;
    if (dy < 0 || dy >= P.ny) return kWall;
    return dx < 0 ? kInlet : (dx >= P.nx ? kOutflow : kNode);
}
// temperature of the wall, and speed of the inlet, where link i of node (x, y) crosses it
__device__ __forceinline__ float link_T_wall(const DevParams& P, int x, int i)
{
    const float xc = (float)x + 0.5f * cx(i);
    return (cy(i) < 0) ? T_wall_bottom(P, xc) : T_wall_top(P, xc);
}
__device__ __forceinline__ float link_u_inlet(const DevParams& P, int y, int i)
{
    return u_inlet(P, (float)y + 0.5f + 0.5f * cy(i));
}
// the outflow's ghost column feeds node (x, y + c_iy) of the last column
__device__ __forceinline__ bool link_copies(const DevParams& P, int x, int y, int i)
{
    return P.bc_x == 1 && x == P.nx - 1 && cx(i) < 0 && y + cy(i) >= 0 && y + cy(i) < P.ny;
}
// What the boundary sends back along link i as population o = opp(i): f and g, and h before
// its Eq. 28 update.
//   wall: halfway bounce-back of f and g; anti-bounce-back of h with the wall temperature
__device__ __forceinline__ void wall_rule(int i, float Tw, float h, float& hin)
{
    hin = -h + 2.f * wq(opp(i)) * Tw;
}
//   velocity inlet: bounce-back carrying the inlet momentum and phi_in
__device__ __forceinline__ void inlet_rule(const DevParams& P, int i, float u_in, float rho, float& f, float& g, float h,
                                           float& hin)
{
    const int o = opp(i);
    const float cu = cx(o) * u_in;
    hin = -h + 2.f * wq(o) * P.T_in;
    f = f + 2.f * wq(o) * P.phi_in * cu * kInvCs2;
    g = g + 2.f * wq(o) * rho * cu * kInvCs2;
}
//   outflow: pressure anti-bounce-back of g (f and h arrive by the copy)
__device__ __forceinline__ float outflow_rule(const DevParams& P, int i, const Macro& m, float g)
{
    const int o = opp(i);
    const float cu = cx(o) * m.ux + cy(o) * m.uy;
    const float sym = P.p_out * kInvCs2 +
                      m.rho * (0.5f * cu * cu * kInvCs2 * kInvCs2 - 0.5f * (m.ux * m.ux + m.uy * m.uy) * kInvCs2);
    return -g + 2.f * wq(o) * sym;
}

// The first-moment records of what a node emits (post-collision f, g, h; FP16), as the
// decoder sees them; out(k, record) takes each.
struct NodeRecords {
    RefVals f{0.f, 0.f, 0.f}, g{0.f, 0.f, 0.f}, h{0.f, 0.f, 0.f};
};
template <class OUT>
__device__ __forceinline__ void node_records(const Macro& m, const float* f, const float* g, const float* h,
                                             NodeRecords& r, OUT out)
{
    float jfx, jfy, jgx, jgy, jhx, jhy;
    dq9_moment1(f, jfx, jfy);
    dq9_moment1(g, jgx, jgy);
    dq9_moment1(h, jhx, jhy);
    out(kRecF, ref_pack(m.phi, jfx * kInvCs2, jfy * kInvCs2, r.f));
    out(kRecG, ref_pack(m.p * kInvCs2, jgx * kInvCs2, jgy * kInvCs2, r.g));
    out(kRecH, ref_pack(m.T, jhx * kInvCs2, jhy * kInvCs2, r.h));
}

// Whether every link of node (x, y) leads to a node, and the periodic x wrap of its neighbours'
// indices.  The nodes of a boundary tile that pass push like those of any other tile; with
// rows as warps, the rest of a tile at a wall or at a seam does (wraps in y go the long way).
struct Wrap {
    int l = 0, r = 0;
};
__device__ __forceinline__ bool plain_node(const DevParams& P, int x, int y, Wrap& wr)
{
    if (P.bc_x == 0) {
        wr.l = x == 0 ? P.nx : 0;
        wr.r = x == P.nx - 1 ? -P.nx : 0;
    } else if (x == 0 || x == P.nx - 1) {
        return false;
    }
    return y > 0 && y < P.ny - 1;
}

// Collide the node's populations and push them to their destinations, with every
// boundary rule; for FP16 also leave the node's reference records in refB (every
// population this node writes is encoded against them).  hold(i, k) and irc(k) give
// the pre-collision h_i and 1/(rho c_p) of the node in ring slot k.  plain: every link of the
// node leads to a node (plain_node); wr: what the wrap of a periodic x adds to the index of a
// neighbour to the left and to the right.
template <class S, int SX, class HOLD, class IRC>
__device__ __forceinline__ void collide_push(const DevParams& P, typename S::elem* __restrict__ B,
                                             RefT* __restrict__ refB, int x, int y, int kown, bool plain, Wrap wr,
                                             const Macro& m, float* f, float* g, float* h, HOLD hold, IRC irc)
{
    const long long pl = P.plane;
    const int n = y * P.nx + x;
    node_collide(P, m, f, g, h);
    NodeRecords r;
    if constexpr (kRef<S>) node_records(m, f, g, h, r, [&](int k, RefT q) { refB[k * pl + n] = q; });
    auto put_f = [&](int i, int d, float v) { S::st_dev(B + i * pl, d, v, dev_pop(i, r.f, v), P.s_f); };
    auto put_g = [&](int i, int d, float v) { S::st_dev(B + (9 + i) * pl, d, v, dev_g(i, r.g, v), P.s_g); };
    auto put_h = [&](int i, int d, float v) { S::st_dev(B + (18 + i) * pl, d, v, dev_pop(i, r.h, v), P.s_h); };
    if (plain) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int d = n + cy(i) * P.nx + cx(i) + (cx(i) < 0 ? wr.l : cx(i) > 0 ? wr.r : 0);
            const int kd = kown + cy(i) * SX + cx(i);
            put_f(i, d, f[i]);
            put_g(i, d, g[i]);
            const float ho = hold(i, kd);
            put_h(i, d, fmaf(h[i] - ho, irc(kd), ho));
        }
        return;
    }
    const float irc_own = irc(kown);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int o = opp(i);
        int d;
        const Link link = link_of(P, x, y, i, d);
        if (link == kWall || link == kInlet) {
            float fo = f[i], go = g[i], hin;
            if (link == kWall) wall_rule(i, link_T_wall(P, x, i), h[i], hin);
            else inlet_rule(P, i, link_u_inlet(P, y, i), m.rho, fo, go, h[i], hin);
            put_f(o, n, fo);
            put_g(o, n, go);
            const float ho = hold(o, kown);
            put_h(o, n, fmaf(hin - ho, irc_own, ho));
        } else if (link == kOutflow) {
            put_g(o, n, outflow_rule(P, i, m, g[i]));
        } else {
            const int kd = kown + cy(i) * SX + cx(i);
            put_f(i, d, f[i]);
            put_g(i, d, g[i]);
            const float ho = hold(i, kd);
            put_h(i, d, fmaf(h[i] - ho, irc(kd), ho));
        }
        // zero-gradient outflow of f and h: the ghost column beyond x = nx-1 carries the
        // post-collision populations of the last column (this node wrote them, so they
        // are encoded against its own records).
        if (link_copies(P, x, y, i)) {
            const int dc = n + cy(i) * P.nx;
            const int kd = kown + cy(i) * SX;
            put_f(i, dc, f[i]);
            const float ho = hold(i, kd);
            put_h(i, dc, fmaf(h[i] - ho, irc(kd), ho));
        }
    }
}

// One tile through the general path: thread loads, ghost values and every boundary
// rule.  Used for lattices whose rows do not meet TMA alignment or that are periodic in x and at
// most one tile wide, by the batched ensemble, and in the TMA kernel for the tiles next to a
// periodic y seam.  The tile covers nodes [x0, x0 + w) x [y0, y0 + h), 1 <= w <= BX, 1 <= h <= BY.
//
// One thread per ring node issues that node's loads together with its own node's, so the
// tile waits on one round trip to memory whatever its extent; ghost ring nodes take
// their mirror's values from shared memory once those are in.
//
// NODES: each node of a boundary tile that can pushes like an interior one (256-lattice
// ensemble, FP32 0.403 -> 0.386 ms per step, FP16 0.82 -> 0.67); without it a tile that touches
// the boundary pushes by the rules as a whole, which is the better code inside the TMA kernel
// (both axes periodic, us per step without / with: 1024 x 1024 FP16 70.8 / 74.0, 2048 x 64 FP16
// 13.8 / 14.5, FP32 9.4 / 9.8, 256 x 1024 FP32 18.6 / 18.9, all before the CTAs with such tiles
// took fewer others).
template <int BX, int BY, class S, bool NODES>
__device__ __forceinline__ void step_tile_general(const DevParams& P, const typename S::elem* __restrict__ A,
                                                  typename S::elem* __restrict__ B, float* __restrict__ phiu,
                                                  const RefT* __restrict__ refA, RefT* __restrict__ refB,
                                                  RingSmem<BX, BY>& sm, int x0, int y0, int w, int h_)
{
    constexpr int SX = RingSmem<BX, BY>::SX;
    const int tx = threadIdx.x % BX, ty = threadIdx.x / BX;
    const int x = x0 + tx, y = y0 + ty;
    const bool active = tx < w && ty < h_;
    const long long pl = P.plane;
    const int n = y * P.nx + x;
    const int kown = (ty + 1) * SX + tx + 1;

    constexpr int kRing = 2 * (BX + BY) + 4;
    static_assert(kRing <= BX * BY, "one thread per ring node");
    // slot (rx, ry) of this thread's ring node (worked out again where it is needed: nothing
    // of it stays in registers while the loads are out)
    auto ring_slot = [&](int& rx, int& ry) {
        const int r = threadIdx.x, sx = w + 2;
        if (r < sx) { rx = r; ry = 0; }
        else if (r < 2 * sx) { rx = r - sx; ry = h_ + 1; }
        else if (r < 2 * sx + h_) { rx = 0; ry = r - 2 * sx + 1; }
        else { rx = w + 1; ry = r - 2 * sx - h_ + 1; }
    };
    int kr = 0;
    bool rload = false, rghost = false;
    float ra[9], rc[9];
    if ((int)threadIdx.x < 2 * (w + h_) + 4) {
        int rx, ry;
        ring_slot(rx, ry);
        kr = ry * SX + rx;
        int wx = x0 + rx - 1, wy = y0 + ry - 1;
        if (P.bc_x == 0) wx = wrap(wx, P.nx);
        if (P.bc_y == 1) wy = wrap(wy, P.ny);
        rload = wx >= 0 && wx < P.nx && wy >= 0 && wy < P.ny;
        rghost = !rload;
        if (rload) load_node<S, false>(P, A, refA, wx, wy, ra, nullptr, rc);
    }

    float f[9], g[9], h[9];
    if (active) {
        load_node<S>(P, A, refA, x, y, f, g, h);
        float sf = 0.f, sh = 0.f;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            sf += f[i];
            sh += h[i];
        }
        sm.phi[kown] = sf;
        sm.T[kown] = sh;
        sm.irc[kown] = __frcp_rn(fmaf(P.rcp_b, clamp1(sf), P.rcp_a));
#pragma unroll
        for (int i = 0; i < 9; ++i) sm.h[i][kown] = h[i];
    }
    if (rload) {
        float sf = 0.f, sh = 0.f;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            sf += ra[i];
            sh += rc[i];
            sm.h[i][kr] = rc[i];
        }
        sm.phi[kr] = sf;
        sm.T[kr] = sh;
        sm.irc[kr] = __frcp_rn(fmaf(P.rcp_b, clamp1(sf), P.rcp_a));
    }
    // ghost ring nodes beyond walls, inlet and outflow (as phiT_at): phi mirrored,
    // T by the boundary's rule; the mirror is the adjacent slot inside the lattice
    if (__syncthreads_or(rghost) && rghost) {
        int rx, ry;
        ring_slot(rx, ry);
        const int gx = x0 + rx - 1, gy = y0 + ry - 1;
        const int wx = P.bc_x == 0 ? wrap(gx, P.nx) : gx, wy = P.bc_y == 1 ? wrap(gy, P.ny) : gy;
        const int mx = min(max(wx, 0), P.nx - 1), my = min(max(wy, 0), P.ny - 1);
        const int km = kr + (my - wy) * SX + mx - wx;
        const float tm = sm.T[km];
        const float tg = (wx < 0) ? 2.f * P.T_in - tm : tm;
        const bool oy = wy < 0 || wy >= P.ny;
        sm.phi[kr] = sm.phi[km];
        sm.T[kr] = oy ? 2.f * (wy < 0 ? T_wall_bottom(P, (float)gx) : T_wall_top(P, (float)gx)) - tg : tg;
        sm.irc[kr] = 0.f;
    }
    __syncthreads();
    if (active) {
        float phin[9], Tn[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int k = kown + cy(i) * SX + cx(i);
            phin[i] = sm.phi[k];
            Tn[i] = sm.T[k];
        }
        const Macro m = node_macro(P, f, g, h, phin, Tn, phiu[n], phiu[pl + n]);
        phiu[n] = m.phi * m.ux;
        phiu[pl + n] = m.phi * m.uy;
        Wrap wr;
        const bool plain = NODES ? plain_node(P, x, y, wr)
                                 : x0 >= 1 && x0 + w <= P.nx - 1 && y0 >= 1 && y0 + h_ <= P.ny - 1;
        collide_push<S, SX>(
            P, B, refB, x, y, kown, plain, wr, m, f, g, h, [&](int i, int k) { return sm.h[i][k]; },
            [&](int k) { return sm.irc[k]; });
    }
    __syncthreads();  // the caller may reuse sm for the next tile
}
// Tile b of an axis of n nodes: start and extent.  Whole tiles of B nodes first, the
// ragged one last (tile_whole), or nt = ceil(n / B) tiles of nearly equal extent (tile_even:
// the many-step kernel, whose step takes as long as its fullest tile; where tiles come in
// waves, whole ones are faster: 1702 x 226 51.5 us per step against 54.9).
__device__ __forceinline__ void tile_whole(int n, int B, int b, int& x0, int& w)
{
    x0 = b * B;
    w = min(B, n - x0);
}
__device__ __forceinline__ void tile_even(int n, int nt, int b, int& x0, int& w)
{
    x0 = (int)((long long)b * n / nt);
    w = (int)((long long)(b + 1) * n / nt) - x0;
}

template <int BX, int BY, class S>
__global__ void __launch_bounds__(BX * BY, 3)
k_step_general(const DevParams P, const typename S::elem* __restrict__ A, typename S::elem* __restrict__ B,
               float* __restrict__ phiu, const RefT* __restrict__ refA, RefT* __restrict__ refB)
{
    __shared__ RingSmem<BX, BY> sm;
    int x0, y0, w, h;
    tile_whole(P.nx, BX, blockIdx.x, x0, w);
    tile_whole(P.ny, BY, blockIdx.y, y0, h);
    step_tile_general<BX, BY, S, true>(P, A, B, phiu, refA, refB, sm, x0, y0, w, h);
}

// ------------------------------------------------------- many steps per launch
//
// Lattices small enough that every tile has a CTA of its own on the GPU at once advance
// many steps in one cooperative launch.  A step of such a lattice is latency: one launch
// per step pays the kernel boundary and the kernel's start on top of the memory round trip
// and the arithmetic.  Here each CTA keeps its tile's populations in shared memory from
// the first step, which reads the population buffer A, to the last, which writes B; (phi u)
// stays in registers.  B is the other buffer after an odd number of steps, and A itself
// after an even one, as one launch per step would leave them: whoever reads a slot in the
// first step has done so before the slot's writer gets through its second.
//
// What the tiles exchange goes through L2 as self-validating words: the populations i of
// the three LBEs that arrive at a node (f_i, g_i, h_i) and the number of the step that
// they begin, 16 bytes read and written as one.  A reader polls the word itself until the
// number is right, so a step has no fence, no flag and no second round trip.  Words exist
// for the nodes on the rim of each tile (slots of two sets of 9 planes, used in turn):
// whoever pushes to such a node writes the word, its tile reads the ones that came from
// outside, and the tiles that have the node in their ring read all nine, for its phi, T
// and h_i.  A slot is written again two steps later by a tile that has by then received
// a push of the step between from every tile that reads the slot (they lie within two
// nodes of the writer), so it has been read.
//
// FP16 storage: a population is rounded through its code as it is emitted and travels
// decoded (the writer knows the reference), so that a step gives the very values that the
// one-step kernels store, without records in between.
//
// What a step costs (512 x 128, in cycles of a CTA): the words' way through L2 and the
// slowest neighbour 3,700, the moments 900, the macroscopic state 1,000, collisions and
// pushes 2,200; it is bound by this chain, not by bandwidth (about 5 MB of words per step).
// Measured against one launch per step (us/step, same process): 128 x 32 5.4 -> 2.6, 512 x
// 128 6.7 -> 3.6, 160 x 320 6.4 -> 3.5, 331 x 117 5.5 -> 3.4; FP16 7.8 -> 3.0, 10.3 -> 4.1,
// 10.6 -> 4.2, 12.7 -> 4.1.  Tried: step counters per tile with release/acquire and the
// populations in L2 (4.3 and 5.3 at 128 x 32 and 512 x 128); 32 x 4 tiles (3.8, 5.6: each
// thread then reads twice the words); 16 x 8 tiles (2.5, 4.1) and 16 x 16 (2.9, 4.2); testing
// the kind of each link in turn instead of masks (3.4, 4.1).
//
// The waits are bounded: a CTA that gives up raises err and returns, and so do the
// others, which look at err now and then; with err up no later launch starts.

__device__ __forceinline__ uint4 ld_word(const uint4* p)
{
    unsigned long long lo, hi;
    asm volatile("{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}\n"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p));
    return make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
}
// (predicated in the instruction: nine of them follow one another in every node's push, and a
// branch around each costs more than the store)
__device__ __forceinline__ void st_word(uint4* p, float f, float g, float h, uint32_t tag, bool on = true)
{
    const unsigned long long lo = ((unsigned long long)__float_as_uint(g) << 32) | __float_as_uint(f);
    const unsigned long long hi = ((unsigned long long)tag << 32) | __float_as_uint(h);
    asm volatile(
        "{\n .reg .b128 t;\n .reg .pred q;\n setp.ne.b32 q, %3, 0;\n mov.b128 t, {%1, %2};\n"
        " @q st.relaxed.gpu.global.b128 [%0], t;\n}\n" ::"l"(p),
        "l"(lo), "l"(hi), "r"((uint32_t)on));
}

constexpr uint32_t kWordWaitLimit = 1u << 22;  // polls, about half a microsecond each

// Shared memory of one tile: the populations of its nodes and its ring (of the ring
// nodes f and h), their phi, T and 1/(rho c_p), the list of words it reads, and per node
// what its links need: the slots of the words it writes, wall temperatures (by c_ix) and
// inlet velocities (by c_iy) at the crossing points.
template <int BX, int BY>
struct ManySmem {
    static constexpr int SX = BX + 2, SN = (BX + 2) * (BY + 2), NT = BX * BY;
    static constexpr int kRing = 2 * (BX + BY) + 4;
    static constexpr int kWords = 9 * kRing + 6 * (BX + BY);
    float f[9][SN], g[9][SN], h[9][SN];
    float phi[SN], T[SN], irc[SN];
    uint2 word[kWords];  // x: slot in a word set; y: i * SN + ring slot, bit 31: g_i is used too
    uint32_t slot[9][NT];
    float Tw[3][NT], uin[3][NT];
    int nwords;
};

// A node's links, worked out once per launch: bit i of each mask.
struct TileMasks {
    uint32_t wall, inlet, outflow, copies;
    uint32_t inside;  // what lies one c_i away is a node of the tile
    uint32_t rim;     // it is a node on the rim of its tile
};

// Collide a node and push its populations: into the tile's shared memory, and as words of
// step `tag` into set `out` for nodes on a rim.  The slot of population i at a node is read
// (as h_i before the step) and written by the one node that pushes to it.
template <class S, class SM>
__device__ __forceinline__ void tile_push(const DevParams& P, const TileMasks& M, SM& sm, uint4* out, uint32_t tag,
                                          int kown, const Macro& m, float* f, float* g, float* h)
{
    const int tid = threadIdx.x;
    node_collide(P, m, f, g, h);
    NodeRecords r;
    if constexpr (kRef<S>) node_records(m, f, g, h, r, [](int, RefT) {});
    auto thru_f = [&](int i, float v) { return S::through(v, dev_pop(i, r.f, v), P.s_f, P.is_f, ref_pop(i, r.f)); };
    auto thru_g = [&](int i, float v) { return S::through(v, dev_g(i, r.g, v), P.s_g, P.is_g, ref_g(i, r.g)); };
    auto thru_h = [&](int i, float v) { return S::through(v, dev_pop(i, r.h, v), P.s_h, P.is_h, ref_pop(i, r.h)); };
    auto word = [&](int i, int j, float vf, float vg, float vh) {
        st_word(out + (uint32_t)(i * (int)P.plane) + sm.slot[j][tid], vf, vg, vh, tag);
    };
    if (M.wall | M.inlet | M.outflow) {
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            const int o = opp(i);
            if ((M.wall | M.inlet) >> i & 1) {
                float vf = f[i], vg = g[i], hin;
                if (M.wall >> i & 1) wall_rule(i, sm.Tw[cx(i) + 1][tid], h[i], hin);
                else inlet_rule(P, i, sm.uin[cy(i) + 1][tid], m.rho, vf, vg, h[i], hin);
                const float hold = sm.h[o][kown];
                vf = thru_f(o, vf);
                vg = thru_g(o, vg);
                const float vh = thru_h(o, fmaf(hin - hold, sm.irc[kown], hold));
                sm.f[o][kown] = vf;
                sm.g[o][kown] = vg;
                sm.h[o][kown] = vh;
                if (M.rim & 1) word(o, 0, vf, vg, vh);
            } else if (M.outflow >> i & 1) {
                sm.g[o][kown] = thru_g(o, outflow_rule(P, i, m, g[i]));
            }
            if (cx(i) < 0 && M.copies >> i & 1) {
                const int j = cy(i) == 0 ? 0 : (cy(i) > 0 ? 2 : 4);  // the copy's destination: a node of the column
                const int kd = kown + cy(i) * SM::SX;
                const float hold = sm.h[i][kd];
                const float vf = thru_f(i, f[i]), vh = thru_h(i, fmaf(h[i] - hold, sm.irc[kd], hold));
                if (M.inside >> j & 1) {
                    sm.f[i][kd] = vf;
                    sm.h[i][kd] = vh;
                }
                if (M.rim >> j & 1) word(i, j, vf, 0.f, vh);
            }
        }
    }
    // links to nodes: everything is read before anything is written (the compiler cannot
    // tell the slots apart), and the words, which other tiles wait for, go first
    float ho[9], ic[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int kd = kown + cy(i) * SM::SX + cx(i);
        ho[i] = sm.h[i][kd];
        ic[i] = sm.irc[kd];
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        f[i] = thru_f(i, f[i]);
        g[i] = thru_g(i, g[i]);
        h[i] = thru_h(i, fmaf(h[i] - ho[i], ic[i], ho[i]));
    }
    if (M.rim) {
        uint32_t slot[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) slot[i] = sm.slot[i][tid];
#pragma unroll
        for (int i = 0; i < 9; ++i)
            st_word(out + (uint32_t)(i * (int)P.plane) + slot[i], f[i], g[i], h[i], tag, M.rim >> i & 1);
    }
    // (without a test: what goes to a ring slot is replaced by the words of the next step before
    // anything reads it, what goes to a ghost slot is never read)
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int kd = kown + cy(i) * SM::SX + cx(i);
        sm.f[i][kd] = f[i];
        sm.g[i][kd] = g[i];
        sm.h[i][kd] = h[i];
    }
}

template <int BX, int BY, class S>
__global__ void __launch_bounds__(BX * BY, 512 / (BX * BY))
k_step_many(const DevParams P, const typename S::elem* A, typename S::elem* B, float* phiu, const RefT* refA, RefT* refB,
            uint4* words, uint32_t* count, int ntx, int nty, int nsteps, int* err)
{
    using SM = ManySmem<BX, BY>;
    constexpr int SX = SM::SX, SN = SM::SN, NT = BX * BY;
    constexpr int kPerThread = (SM::kWords + NT - 1) / NT;
    static_assert(2 * SM::kRing <= NT, "one thread per ring moment");
    extern __shared__ __align__(128) unsigned char dsm[];
    SM& sm = *reinterpret_cast<SM*>(dsm);
    const int tid = threadIdx.x;
    int x0, y0, w, h_;
    tile_even(P.nx, ntx, blockIdx.x % ntx, x0, w);
    tile_even(P.ny, nty, blockIdx.x / ntx, y0, h_);
    const long long pl = P.plane;
    // steps this tile has done, ever (the same for all tiles between launches): the
    // numbers of this launch's words start after it
    const uint32_t base = count[blockIdx.x];
    const int e0 = *(volatile int*)err;
    if (tid == 0) sm.nwords = 0;
    if (__syncthreads_or(e0)) return;

    const int tx = tid % BX, ty = tid / BX;
    const int x = x0 + tx, y = y0 + ty;
    const bool active = tx < w && ty < h_;
    const int n = y * P.nx + x;
    const int kown = (ty + 1) * SX + tx + 1;
    const int nring = 2 * (w + h_) + 4;
    // slot (rx, ry) of ring node r; true when it lies inside the lattice, at (wx, wy)
    auto ring_node = [&](int r, int& rx, int& ry, int& wx, int& wy) {
        const int sx = w + 2;
        if (r < sx) { rx = r; ry = 0; }
        else if (r < 2 * sx) { rx = r - sx; ry = h_ + 1; }
        else if (r < 2 * sx + h_) { rx = 0; ry = r - 2 * sx + 1; }
        else { rx = w + 1; ry = r - 2 * sx - h_ + 1; }
        wx = x0 + rx - 1;
        wy = y0 + ry - 1;
        if (P.bc_x == 0) wx = wrap(wx, P.nx);
        if (P.bc_y == 1) wy = wrap(wy, P.ny);
        return wx >= 0 && wx < P.nx && wy >= 0 && wy < P.ny;
    };
    // this thread's moment of the ring: thread r takes phi (and 1/(rho c_p)), thread
    // kRing + r takes T, of ring slot kr.  Ghost nodes beyond walls, inlet and outflow sum
    // their mirror's populations (the adjacent slot inside the lattice, km) and follow
    // phiT_at: phi is mirrored; T is 2 T_wall - T at a wall, 2 T_in - T at the inlet.
    const bool ring_h = tid >= SM::kRing;
    const int ring = ring_h ? tid - SM::kRing : tid;
    int kr = -1, km = 0;
    bool ghost = false, g_in = false, g_wall = false;
    float gT2 = 0.f;  // twice the wall's temperature
    if (ring < nring) {
        int rx, ry, wx, wy;
        ghost = !ring_node(ring, rx, ry, wx, wy);
        kr = km = ry * SX + rx;
        if (ghost) {
            const int mx = min(max(wx, 0), P.nx - 1), my = min(max(wy, 0), P.ny - 1);
            km = (ry + my - wy) * SX + rx + mx - wx;
            g_in = wx < 0;
            g_wall = wy < 0 || wy >= P.ny;
            const int gx = x0 + rx - 1;
            if (g_wall) gT2 = 2.f * (wy < 0 ? T_wall_bottom(P, (float)gx) : T_wall_top(P, (float)gx));
        }
    }

    // the words this tile reads: all nine of each ring node, and of its own nodes those
    // that arrive from outside the tile (at the outflow, f and h of the last column come
    // from the column's other nodes)
    {
        auto append = [&](bool take, uint2 v) {
            const unsigned m = __ballot_sync(0xffffffffu, take);
            int at = 0;
            if ((tid & 31) == 0 && m) at = atomicAdd(&sm.nwords, __popc(m));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (take) sm.word[at + __popc(m & ((1u << (tid & 31)) - 1u))] = v;
        };
        const int rr = (9 * nring + NT - 1) / NT;
        for (int j = 0; j < rr; ++j) {
            const int idx = tid + j * NT, i = idx / nring;
            int rx = 0, ry = 0, wx = 0, wy = 0;
            bool take = i < 9 && ring_node(idx - i * nring, rx, ry, wx, wy);
            append(take, make_uint2((uint32_t)(i * pl + (long long)wy * P.nx + wx), (uint32_t)(i * SN + ry * SX + rx)));
        }
        for (int i = 1; i < 9; ++i) {
            const int lx = tx - cx(i), ly = ty - cy(i);  // the source, in the tile's coordinates
            int sx = x - cx(i), sy = y - cy(i);
            if (P.bc_x == 0) sx = wrap(sx, P.nx);
            if (P.bc_y == 1) sy = wrap(sy, P.ny);
            const bool in_y = sy >= 0 && sy < P.ny;
            const bool out_tile = lx < 0 || lx >= w || ly < 0 || ly >= h_;
            const bool copied = sx >= P.nx;  // outflow: written by (nx - 1, sy)
            const bool take = active && in_y && sx >= 0 && (copied ? (ly < 0 || ly >= h_) : out_tile);
            append(take, make_uint2((uint32_t)(i * pl + n), (uint32_t)(i * SN + kown) | (copied ? 0u : 1u << 31)));
        }
    }
    TileMasks M{0, 0, 0, 0, 0, 0};
    if (active) {
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const int lx = tx + cx(j), ly = ty + cy(j);
            const bool in = lx >= 0 && lx < w && ly >= 0 && ly < h_;
            int d;
            const Link link = link_of(P, x, y, j, d);
            M.wall |= (uint32_t)(link == kWall) << j;
            M.inlet |= (uint32_t)(link == kInlet) << j;
            M.outflow |= (uint32_t)(link == kOutflow) << j;
            M.copies |= (uint32_t)link_copies(P, x, y, j) << j;
            M.inside |= (uint32_t)(link == kNode && in) << j;
            M.rim |= (uint32_t)(link == kNode && (!in || lx == 0 || lx == w - 1 || ly == 0 || ly == h_ - 1)) << j;
            sm.slot[j][tid] = (uint32_t)d;
            if (link == kWall) sm.Tw[cx(j) + 1][tid] = link_T_wall(P, x, j);
            if (link == kInlet) sm.uin[cy(j) + 1][tid] = link_u_inlet(P, y, j);
        }
    }

    float pu_x = 0.f, pu_y = 0.f;
    if (active) {
        pu_x = phiu[n];
        pu_y = phiu[pl + n];
    }
    // first step: the populations from the buffer
    int rx, ry, wx, wy;
    if (tid < nring && ring_node(tid, rx, ry, wx, wy)) {
        float ra[9], rc[9];
        load_node<typename S::Once, false>(P, A, refA, wx, wy, ra, nullptr, rc);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            sm.f[i][kr] = ra[i];
            sm.h[i][kr] = rc[i];
        }
    }
    if (active) {
        float f[9], g[9], h[9];
        load_node<typename S::Once>(P, A, refA, x, y, f, g, h);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            sm.f[i][kown] = f[i];
            sm.g[i][kown] = g[i];
            sm.h[i][kown] = h[i];
        }
    }
    __syncthreads();
    const int nwords = sm.nwords;
    uint2 rd[kPerThread];  // the words this thread reads
#pragma unroll
    for (int j = 0; j < kPerThread; ++j)
        rd[j] = tid + j * NT < nwords ? sm.word[tid + j * NT] : make_uint2(0, 0);

    for (int s = 0; s < nsteps; ++s) {
        if (s > 0) {
            bool ok = true;
            // the words of this step, written by the tiles around during the last one
            const uint32_t tag = base + (uint32_t)s;
            const uint4* in = words + (size_t)(tag & 1) * 9 * pl;
            uint4 v[kPerThread];
            bool all = true;
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) v[j].w = tag - 1;
            for (uint32_t it = 1;; ++it) {
#pragma unroll
                for (int j = 0; j < kPerThread; ++j)
                    if (tid + j * NT < nwords && v[j].w != tag) v[j] = ld_word(in + rd[j].x);
                all = true;
#pragma unroll
                for (int j = 0; j < kPerThread; ++j) all = all && (tid + j * NT >= nwords || v[j].w == tag);
                if (all) break;
                if (it >= kWordWaitLimit || ((it & 1023) == 0 && *(volatile int*)err)) {
                    ok = false;
                    break;
                }
            }
#pragma unroll
            for (int j = 0; j < kPerThread; ++j) {
                if (tid + j * NT >= nwords) continue;
                const uint32_t at = rd[j].y & 0x7fffffffu;
                (&sm.f[0][0])[at] = __uint_as_float(v[j].x);
                if (rd[j].y >> 31) (&sm.g[0][0])[at] = __uint_as_float(v[j].y);
                (&sm.h[0][0])[at] = __uint_as_float(v[j].z);
            }
            if (__syncthreads_or(!ok)) {
                if (tid == 0) atomicExch(err, 1);
                return;
            }
        }
        float f[9], g[9], h[9], sf = 0.f, sh = 0.f, sr = 0.f;
        {
            const float(*rq)[SN] = ring_h ? sm.h : sm.f;
            float q[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                f[i] = sm.f[i][kown];
                g[i] = sm.g[i][kown];
                h[i] = sm.h[i][kown];
                q[i] = kr >= 0 ? rq[i][km] : 0.f;
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                sf += f[i];
                sh += h[i];
                sr += q[i];
            }
        }
        if (active) {
            sm.phi[kown] = sf;
            sm.T[kown] = sh;
            sm.irc[kown] = __frcp_rn(fmaf(P.rcp_b, clamp1(sf), P.rcp_a));
        }
        if (kr >= 0) {
            if (!ring_h) {
                sm.phi[kr] = sr;
                sm.irc[kr] = ghost ? 0.f : __frcp_rn(fmaf(P.rcp_b, clamp1(sr), P.rcp_a));
            } else {
                if (g_in) sr = 2.f * P.T_in - sr;
                if (g_wall) sr = gT2 - sr;
                sm.T[kr] = sr;
            }
        }
        __syncthreads();
        if (active) {
            float phin[9], Tn[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const int k = kown + cy(i) * SX + cx(i);
                phin[i] = sm.phi[k];
                Tn[i] = sm.T[k];
            }
            const Macro m = node_macro(P, f, g, h, phin, Tn, pu_x, pu_y);
            pu_x = m.phi * m.ux;
            pu_y = m.phi * m.uy;
            if (s + 1 < nsteps) {
                const uint32_t tag = base + (uint32_t)s + 1;
                tile_push<S>(P, M, sm, words + (size_t)(tag & 1) * 9 * pl, tag, kown, m, f, g, h);
            } else {
                Wrap wr;
                const bool plain = plain_node(P, x, y, wr);
                collide_push<S, SX>(
                    P, B, refB, x, y, kown, plain, wr, m, f, g, h, [&](int i, int k) { return sm.h[i][k]; },
                    [&](int k) { return sm.irc[k]; });
            }
        }
        __syncthreads();
    }
    if (active) {
        phiu[n] = pu_x;
        phiu[pl + n] = pu_y;
    }
    if (tid == 0) count[blockIdx.x] = base + (uint32_t)nsteps;
}

// ------------------------------------------------------------ TMA kernel
//
// Persistent CTAs walk a tile list: first the TMA tiles, then the remaining tiles
// through the general path.  TMA tiles are, along a walled or inlet/outflow axis, all tiles, the
// ragged last one too: there the box reaches past the lattice, the copy fills it with zeros, and
// the tile takes its ghost ring nodes and its boundary nodes' FP16 records by the boundary
// rules instead; along a periodic x axis of two tiles and more, all tiles too (see seam_side); along
// a periodic y axis, the tiles whose halo lies inside the lattice (y0 >= 2, y0 + BY + 2 <= ny).
// For a TMA tile one elected thread issues 3D bulk
// tensor copies (cp.async.bulk.tensor) of the 9 f planes and the 9 h planes over the
// tile plus a one-node ring (widened to XP columns each side for the 16-byte rule),
// the 9 g planes and the 2 (phi u) planes over the tile, and for FP16 the 3 planes of
// reference records over the tile plus a two-node ring, all completing on one mbarrier.  While a
// tile is computed, the next tile's copies are in flight into the other stage.

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
            smem_u32(dst)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// bounded wait: false after `limit` polls (about 2^22 in the step kernels; each
// try_wait suspends for a while)
constexpr uint32_t kWaitLimit = 1u << 22;
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint32_t limit = kWaitLimit)
{
    for (uint32_t it = 0; it < limit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

template <int BX, int BY, class S>
struct TmaLayout {
    using E = typename S::elem;
    static constexpr int XP = 16 / (int)sizeof(E);           // column pad for 16-byte aligned boxes
    static constexpr int FW = BX + 2 * XP, FH = BY + 2;     // f/h box (tile + ring, widened)
    static constexpr int RW = BX + 8, RH = BY + 4;          // reference box (tile + 2-ring, widened)
    static constexpr int rnd(int b) { return (b + 127) / 128 * 128; }
    static constexpr int F_BYTES = 9 * FH * FW * (int)sizeof(E);
    static constexpr int G_BYTES = 9 * BY * BX * (int)sizeof(E);
    static constexpr int U_BYTES = 2 * BY * BX * 4;
    static constexpr int R_BYTES = kRef<S> ? 3 * RH * RW * (int)sizeof(RefT) : 0;
    static constexpr int OFF_F = 0, OFF_H = rnd(F_BYTES), OFF_G = OFF_H + rnd(F_BYTES), OFF_U = OFF_G + rnd(G_BYTES),
                         OFF_R = OFF_U + rnd(U_BYTES), OFF_C = OFF_R + rnd(R_BYTES);
    // the wrapped ring column of f and of h of a seam tile, boxes of CW columns, and for FP16
    // the two wrapped columns of the records
    static constexpr int CW = 16 / (int)sizeof(E), C_BYTES = 9 * FH * CW * (int)sizeof(E);
    static constexpr int CR_BYTES = kRef<S> ? 3 * RH * 2 * (int)sizeof(RefT) : 0;
    static constexpr int OFF_CH = OFF_C + rnd(C_BYTES), OFF_CR = OFF_CH + rnd(C_BYTES), STAGE = OFF_CR + rnd(CR_BYTES);
    static constexpr int stage(bool seam) { return seam ? STAGE : OFF_C; }  // bytes in use
    static constexpr uint32_t TX_BYTES = 2 * F_BYTES + G_BYTES + U_BYTES + R_BYTES;
};

// Which side of a periodic x seam a TMA tile sits on: -1 its left ring column wraps to
// x = nx - 1, +1 its right one to x = 0, 0 neither.  Seam tiles are staged by TMA in lattices
// more than a tile wide (so no tile has both sides).
template <int BX>
__device__ __forceinline__ int seam_side(const DevParams& P, int x0)
{
    if (P.bc_x != 0) return 0;
    return x0 == 0 ? -1 : (x0 + BX >= P.nx ? 1 : 0);
}

struct TmaMaps {
    CUtensorMap popF;  // populations, box FW x FH x 9 (used for f at z = 0 and h at z = 18)
    CUtensorMap popG;  // populations, box BX x BY x 9 (g at z = 9)
    CUtensorMap phiu;  // (phi u) planes, box BX x BY x 2
    CUtensorMap ref;   // FP16 reference records (8-byte elements), box RW x RH x 3
};

struct SeamMaps {     // the wrapped columns at a periodic x seam
    CUtensorMap pop;  // populations, box CW x FH x 9
    CUtensorMap ref;  // FP16 reference records, box 2 x RH x 3
};

// The copies of one TMA tile into stage st, completing on bar (one elected thread).  seam: see
// seam_side; nx is needed at a left seam only.
template <int BX, int BY, class S>
__device__ __forceinline__ void tma_issue_tile(const TmaMaps& M, const SeamMaps& C, unsigned char* st, uint64_t* bar, int x0, int y0,
                                               int seam, int nx)
{
    using L = TmaLayout<BX, BY, S>;
    fence_proxy_async();
    mbar_expect_tx(bar, L::TX_BYTES + (seam ? 2 * L::C_BYTES + L::CR_BYTES : 0));
    if (seam) {
        const int cx0 = seam < 0 ? nx - L::CW : 0;
        tma_load_3d(st + L::OFF_C, &C.pop, bar, cx0, y0 - 1, 0);
        tma_load_3d(st + L::OFF_CH, &C.pop, bar, cx0, y0 - 1, 18);
        if constexpr (kRef<S>) tma_load_3d(st + L::OFF_CR, &C.ref, bar, seam < 0 ? nx - 2 : 0, y0 - 2, 0);
    }
    tma_load_3d(st + L::OFF_F, &M.popF, bar, x0 - L::XP, y0 - 1, 0);
    tma_load_3d(st + L::OFF_H, &M.popF, bar, x0 - L::XP, y0 - 1, 18);
    tma_load_3d(st + L::OFF_G, &M.popG, bar, x0, y0, 9);
    tma_load_3d(st + L::OFF_U, &M.phiu, bar, x0, y0, 0);
    if constexpr (kRef<S>) tma_load_3d(st + L::OFF_R, &M.ref, bar, x0 - 4, y0 - 2, 0);
}

// phi, T and 1/(rho c_p) of a TMA tile and its ring
template <int BX, int BY>
struct PhiSmem {
    static constexpr int SN = (BX + 2) * (BY + 2);
    float phi[SN];
    float T[SN];
    float irc[SN];
};

// Periodic x seam: the wrapped ring column of f and h, and for FP16 the wrapped columns of the
// records, into the boxes, where the copies left zeros, from the columns staged beside them,
// before anything decodes them (rows beyond a wall are zero on both sides).  Fetching the columns
// here, out of global memory, cost every seam tile a memory round trip (256 x 1024 FP32, a
// quarter of whose tiles are seam tiles: 13.6 us per step against 13.1).  Ends with a block
// barrier.
template <int BX, int BY, class S>
__device__ __forceinline__ void seam_patch(unsigned char* st, int seam, int w)
{
    using L = TmaLayout<BX, BY, S>;
    using E = typename S::elem;
    const int k = threadIdx.x;
    constexpr int kCol = 9 * L::FH, kRec = kRef<S> ? 3 * L::RH * 2 : 0;
    static_assert(2 * kCol + kRec <= BX * BY, "one value per thread");
    if (k < 2 * kCol) {
        const int fc = seam < 0 ? L::XP - 1 : L::XP + w, cc = seam < 0 ? L::CW - 1 : 0;
        const bool hh = k >= kCol;
        const int q = hh ? k - kCol : k;
        E* box = (E*)(st + (hh ? L::OFF_H : L::OFF_F));
        const E* col = (const E*)(st + (hh ? L::OFF_CH : L::OFF_C));
        box[q * L::FW + fc] = col[q * L::CW + cc];
    } else if (k < 2 * kCol + kRec) {
        // record row q / 2 (of 3 RH), column q % 2 of the two beyond the seam: x = -2, -1 or
        // x0 + w, x0 + w + 1, in a box that starts at x0 - 4
        const int q = k - 2 * kCol, c0 = seam < 0 ? 2 : w + 4;
        RefT* box = (RefT*)(st + L::OFF_R);
        const RefT* col = (const RefT*)(st + L::OFF_CR);
        box[(q >> 1) * L::RW + c0 + (q & 1)] = col[q];
    }
    __syncthreads();
}

// The body of one TMA tile, shared by the single-lattice and the batched kernels: decode
// the staged populations of the tile (stage st, landed unless ok is false) and its
// ring, phi / T / 1/(rho c_p) into sm, one block barrier (which also votes on ok:
// on_abort() runs on every thread and the tile returns true when any wait ran out),
// after_ring() on every thread, then per node the macroscopic state, the collisions
// and the push to B.  EDGE: the tile touches the lattice boundary (ghost ring nodes,
// boundary records, boundary-aware push for every node); RAGGED: it covers w x h_ nodes (BX x BY
// otherwise); seam (seam_side; SEAM: it may be set): the wrapped
// column of a periodic x seam is put into the box first.  EDGE, seam, w and h_ must be the
// same on every thread and must not come from a staged P (it is not to be trusted
// before the vote).
template <int BX, int BY, class S, bool EDGE, bool RAGGED, bool SEAM, bool PRELOAD, class OnAbort, class AfterRing>
__device__ __forceinline__ bool tma_tile(const DevParams& P, typename S::elem* __restrict__ B,
                                         float* __restrict__ phiu, RefT* __restrict__ refB, unsigned char* st, PhiSmem<BX, BY>& sm, int x0, int y0, int w_, int h__,
                                         int seam, bool ok, OnAbort on_abort, AfterRing after_ring)
{
    // (constants where the tile cannot be ragged)
    const int w = RAGGED ? w_ : BX, h_ = RAGGED ? h__ : BY;
    using L = TmaLayout<BX, BY, S>;
    using E = typename S::elem;
    constexpr int SX = BX + 2;
    constexpr int kRing = 2 * (BX + BY) + 4;
    static_assert(2 * kRing <= BX * BY, "one thread per ring moment");
    const int tid = threadIdx.x;
    const long long pl = P.plane;
    const E* sF = (const E*)(st + L::OFF_F);
    const E* sH = (const E*)(st + L::OFF_H);
    const E* sG = (const E*)(st + L::OFF_G);
    const float* sU = (const float*)(st + L::OFF_U);
    const RefT* sR = (const RefT*)(st + L::OFF_R);
    (void)sR;
    constexpr bool edge = EDGE;
    // nodes on a walled, inlet or outflow boundary (a periodic one has none), and ring
    // nodes beyond one.  Without SEAM the TMA tiles keep one node clear of every periodic
    // edge, where the plain tests agree.
    auto on_boundary = [&](int gx, int gy) {
        return ((!SEAM || P.bc_x != 0) && (gx == 0 || gx == P.nx - 1)) || gy == 0 || gy == P.ny - 1;
    };
    auto is_ghost = [&](int gx, int gy) {
        return ((!SEAM || P.bc_x != 0) && (gx < 0 || gx >= P.nx)) || gy < 0 || gy >= P.ny;
    };
    if constexpr (edge) {
        if constexpr (SEAM) {
            if (seam) seam_patch<BX, BY, S>(st, seam, w);
        }
    }

    // decoded population i of ring slot (lx, ly) from the f (or h) box
    auto decF = [&](const E* box, float is, int rplane, int i, int lx, int ly, bool bnode) {
        float r = 0.f;
        if constexpr (kRef<S>) {
            const int k = bnode ? ref_slot_box<SEAM>(P, x0 + lx - 1, y0 + ly - 1, i, false, x0, y0, L::RW, L::RH)
                                : (ly + 1 - cy(i)) * L::RW + lx + 3 - cx(i);
            r = ref_pop(i, ref_unpack(sR[rplane * L::RH * L::RW + k]));
        }
        return S::lds(box, (i * L::FH + ly) * L::FW + lx - 1 + L::XP, is, r);
    };

    // own node: decoded populations, phi, T, 1/(rho c_p)
    const int tx = tid % BX, ty = tid / BX;
    const int lx = tx + 1, ly = ty + 1, kown = ly * SX + lx;
    const int x = x0 + tx, y = y0 + ty;
    const int n = y * P.nx + x;
    const bool active = !RAGGED || (tx < w && ty < h_);
    const bool bnode = edge && on_boundary(x, y);
    float f[9], g[9], h[9], phin[9], Tn[9];
    {
        float sf = 0.f, sh = 0.f;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            float rf = 0.f, rg = 0.f, rh = 0.f;
            if constexpr (kRef<S>) {
                int k = (ly + 1 - cy(i)) * L::RW + lx + 3 - cx(i), kg = k;
                if (bnode) {
                    k = ref_slot_box<SEAM>(P, x, y, i, false, x0, y0, L::RW, L::RH);
                    kg = ref_slot_box<SEAM>(P, x, y, i, true, x0, y0, L::RW, L::RH);
                }
                rf = ref_pop(i, ref_unpack(sR[kRecF * L::RH * L::RW + k]));
                rg = ref_g(i, ref_unpack(sR[kRecG * L::RH * L::RW + kg]));
                rh = ref_pop(i, ref_unpack(sR[kRecH * L::RH * L::RW + k]));
            }
            f[i] = S::lds(sF, (i * L::FH + ly) * L::FW + lx - 1 + L::XP, P.is_f, rf);
            h[i] = S::lds(sH, (i * L::FH + ly) * L::FW + lx - 1 + L::XP, P.is_h, rh);
            g[i] = S::lds(sG, (i * BY + ty) * BX + tx, P.is_g, rg);
            sf += f[i];
            sh += h[i];
        }
        if (active) {
            sm.phi[kown] = sf;
            sm.T[kown] = sh;
            sm.irc[kown] = __frcp_rn(fmaf(P.rcp_b, clamp1(sf), P.rcp_a));
        }
    }
    // PRELOAD (tiles without boundary nodes): the rest of the tile's reads of the stage,
    // done before the ring barrier so that the stage is free after it: the destinations'
    // pre-collision h_i for the push (each came from this node, so for FP16 its
    // reference is this node's record) and the previous (phi u)
    constexpr bool kPre = PRELOAD && !EDGE;
    float hold_r[9], pu_x = 0.f, pu_y = 0.f;
    RefVals rown_h{0.f, 0.f, 0.f};
    (void)hold_r;
    if constexpr (kPre) {
        if constexpr (kRef<S>) rown_h = ref_unpack(sR[(kRecH * L::RH + ly + 1) * L::RW + lx + 3]);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int kd = kown + cy(i) * SX + cx(i);
            float r = 0.f;
            if constexpr (kRef<S>) r = ref_pop(i, rown_h);
            hold_r[i] = S::lds(sH, (i * L::FH + kd / SX) * L::FW + kd % SX - 1 + L::XP, P.is_h, r);
        }
        pu_x = sU[ty * BX + tx];
        pu_y = sU[(BY + ty) * BX + tx];
    }
    // ring: 2 (w + h_) + 4 nodes, one zeroth moment (f or h) per thread
    auto ring_slot = [&](int r, int& rx, int& ry) {
        const int sx = w + 2;
        if (r < sx) { rx = r; ry = 0; }
        else if (r < 2 * sx) { rx = r - sx; ry = h_ + 1; }
        else if (r < 2 * sx + h_) { rx = 0; ry = r - 2 * sx + 1; }
        else { rx = w + 1; ry = r - 2 * sx - h_ + 1; }
    };
    const int nring = 2 * (w + h_) + 4;  // <= kRing
    if (tid < 2 * nring) {
        const bool ring_f = tid < nring;
        int rx, ry;
        ring_slot(ring_f ? tid : tid - nring, rx, ry);
        const int k = ry * SX + rx;
        const int gx = x0 + rx - 1, gy = y0 + ry - 1;
        const bool ghost = edge && is_ghost(gx, gy);
        const bool rb = edge && on_boundary(gx, gy);
        float s = 0.f;
        if (ghost) {
            // filled below from the node it mirrors
        } else if (ring_f) {
#pragma unroll
            for (int i = 0; i < 9; ++i) s += decF(sF, P.is_f, kRecF, i, rx, ry, rb);
            sm.phi[k] = s;
            sm.irc[k] = __frcp_rn(fmaf(P.rcp_b, clamp1(s), P.rcp_a));
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) s += decF(sH, P.is_h, kRecH, i, rx, ry, rb);
            sm.T[k] = s;
        }
    }
    if constexpr (edge) {
        // ghost ring nodes beyond walls, inlet and outflow: phi mirrored, T by the
        // boundary's rule (as phiT_at does for the general path)
        __syncthreads();
        if (tid < nring) {
            int rx, ry;
            ring_slot(tid, rx, ry);
            const int gx = x0 + rx - 1, gy = y0 + ry - 1;
            const bool ox = (!SEAM || P.bc_x != 0) && (gx < 0 || gx >= P.nx), oy = gy < 0 || gy >= P.ny;
            if (ox || oy) {
                const int mx = ox ? (gx < 0 ? 0 : P.nx - 1) : gx;
                const int my = oy ? (gy < 0 ? 0 : P.ny - 1) : gy;
                // (the clamp only matters when P is not to be trusted, as above)
                const int km = min(max((my - y0 + 1) * SX + mx - x0 + 1, 0), PhiSmem<BX, BY>::SN - 1);
                const float tm = sm.T[km];
                const float tx = (ox && gx < 0) ? 2.f * P.T_in - tm : tm;
                const int k = ry * SX + rx;
                sm.phi[k] = sm.phi[km];
                sm.T[k] = oy ? 2.f * (gy < 0 ? T_wall_bottom(P, (float)gx) : T_wall_top(P, (float)gx)) - tx : tx;
                sm.irc[k] = 0.f;
            }
        }
    }
    if (__syncthreads_or(!ok)) {
        on_abort();
        return true;
    }
    after_ring();
    if (!active) return false;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int k = kown + cy(i) * SX + cx(i);
        phin[i] = sm.phi[k];
        Tn[i] = sm.T[k];
    }
    if constexpr (!kPre) {
        pu_x = sU[ty * BX + tx];
        pu_y = sU[(BY + ty) * BX + tx];
    }
    const Macro m = node_macro(P, f, g, h, phin, Tn, pu_x, pu_y);
    phiu[n] = m.phi * m.ux;
    phiu[pl + n] = m.phi * m.uy;
    if constexpr (kRef<S> && !kPre) rown_h = ref_unpack(sR[(kRecH * L::RH + ly + 1) * L::RW + lx + 3]);
    collide_push<S, SX>(
        P, B, refB, x, y, kown, !edge, Wrap{}, m, f, g, h,
        [&](int i, int kd) {
            if constexpr (kPre) {
                return hold_r[i];  // interior tiles push only to kd = own + c_i
            } else {
                // h_i of destination kd came from this node: its reference is this node's record
                float r = 0.f;
                if constexpr (kRef<S>) r = ref_pop(i, rown_h);
                return S::lds(sH, (i * L::FH + kd / SX) * L::FW + kd % SX - 1 + L::XP, P.is_h, r);
            }
        },
        [&](int kd) { return sm.irc[kd]; });
    return false;
}

// CTAs per SM the TMA kernel is built for (shared memory allows up to 2 for FP32 and
// 3 for FP16; more CTAs means fewer registers per thread).
#ifndef TPF_TMA_BLOCKS_F32
#define TPF_TMA_BLOCKS_F32 2
#endif
#ifndef TPF_TMA_BLOCKS_F16
#define TPF_TMA_BLOCKS_F16 2
#endif
template <class S>
constexpr int kTmaMinBlocks = kRef<S> ? TPF_TMA_BLOCKS_F16 : TPF_TMA_BLOCKS_F32;

// RAGGED: the lattice has ragged TMA tiles (a body with constant extents is 1% faster on 256 x
// 1024, a quarter of whose tiles are boundary tiles).
// SEAM: x is periodic, so the lattice has seam tiles (the 2048 x 512 inlet/outflow channel, which
// has none, takes 44.9 us per step with FP32 without their code and 45.2 with it).
// REST: with the general path, for the tiles that a periodic y leaves to it (the 2048 x 512 channel,
// which has none, takes 50.7 us per step with FP16 without that code and 51.3 with it).
template <int BX, int BY, class S, bool RAGGED, bool SEAM, bool REST>
__global__ void __launch_bounds__(BX * BY, kTmaMinBlocks<S>)
k_step_tma(const DevParams P, const __grid_constant__ TmaMaps maps, const typename S::elem* __restrict__ A,
           typename S::elem* __restrict__ B, float* __restrict__ phiu, const RefT* __restrict__ refA,
           RefT* __restrict__ refB, const int2* __restrict__ tiles, int bx0, int by0, int ntbx, int ntby,
           int* __restrict__ err, const __grid_constant__ SeamMaps smaps, int lead)
{
    using L = TmaLayout<BX, BY, S>;
    constexpr int kStage = SEAM ? L::STAGE : L::OFF_C;  // = L::stage(SEAM)
    static_assert(sizeof(RingSmem<BX, BY>) <= 2 * kStage, "general-path tiles reuse the stages");
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) uint64_t bar[2];
    // Where a tile's copies are issued: tile t + 2 (this CTA's after next) goes into the
    // stage of tile t as soon as tile t no longer reads it.  Tiles without boundary
    // nodes read everything they need from the stage before their ring barrier
    // (PRELOAD), so their stage is refilled right after it and the tile ends without a
    // block barrier; boundary tiles end with one and refill after it.  phi, T and
    // 1/(rho c_p) are double buffered: a warp may start the next tile while others still
    // push (it cannot get two tiles ahead: the next ring barrier waits for them).
    __shared__ PhiSmem<BX, BY> smb[2];

    const int ntma = ntbx * ntby;  // TMA tiles: bx in [bx0, bx0 + ntbx), by in [by0, by0 + ntby)
    const int tilesx = (P.nx + BX - 1) / BX, tilesy = (P.ny + BY - 1) / BY;
    const int nall = tilesx * tilesy;
    const int nedge = nall - ntma;
    const int tid = threadIdx.x;

    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();

    auto tile_of = [&](int t, int k, int& x0, int& y0) {
        const int2 v = __ldg(tiles + t);
        x0 = v.x;
        y0 = v.y;
    };

    auto issue = [&](int t, int k, int s) {
        int x0, y0;
        tile_of(t, k, x0, y0);
        tma_issue_tile<BX, BY, S>(maps, smaps, dsm + s * kStage, &bar[s], x0, y0, SEAM ? seam_side<BX>(P, x0) : 0, P.nx);
    };

    // This CTA's tiles: t, next(t), ...  With REST, the first `more` CTAs have one general tile more
    // than the others and sit out the first `lead` rounds of the TMA tiles (tma_lead).
    const int grid = gridDim.x, more = REST && lead > 0 ? nedge % grid : 0, early = lead * (grid - more);
    auto next = [&](int t) {
        if (REST && more > 0 && t < early) return t + grid - more < early ? t + grid - more : early + (int)blockIdx.x;
        return t + grid;
    };
    int it = 0;
    int t = blockIdx.x;
    if (REST && more > 0) t = t < more ? early + t : t - more;
    if (tid == 0) {
        if (t < ntma) issue(t, 0, 0);
        if (next(t) < ntma) issue(next(t), 1, 1);
    }
    for (; t < ntma; t = next(t), ++it) {
        const int s = it & 1;
        const int tn = next(t), t2 = next(tn);
        PhiSmem<BX, BY>& sm = smb[s];
        // every thread waits for the stage itself; a thread whose wait ran out reads
        // stale (in-bounds) shared memory until the block votes at the next barrier
        const bool ok = mbar_wait_bounded(&bar[s], (it >> 1) & 1);
        int x0, y0;
        tile_of(t, it, x0, y0);
        // the tile body is compiled twice: for tiles touching the lattice boundary and
        // for all others, which keep the plain interior code
        auto on_abort = [&]() {
            if (tid == 0) {
                atomicExch(err, 1);
                // let this CTA's copies in flight land (bounded) before leaving
                mbar_wait_bounded(&bar[s], (it >> 1) & 1);
                if (tn < ntma) mbar_wait_bounded(&bar[s ^ 1], ((it + 1) >> 1) & 1);
            }
        };
        auto refill = [&]() {
            if (t2 < ntma && tid == 0) issue(t2, it + 2, s);
        };
        auto no_refill = [&]() {};
        unsigned char* st = dsm + s * kStage;
        const bool edge_tile = x0 <= 1 || x0 + BX >= P.nx - 1 || y0 <= 1 || y0 + BY >= P.ny - 1;
        const int seam = SEAM ? seam_side<BX>(P, x0) : 0;
        // interior tiles first: with the two bodies the other way round 512 x 512 takes 13.3 us per
        // step with FP32 and 18.8 with FP16, so 13.05 and 18.55
        if (!edge_tile) {
            if (tma_tile<BX, BY, S, false, false, false, true>(P, B, phiu, refB, st, sm, x0, y0, BX, BY, 0, ok,
                                                               on_abort, refill))
                return;
        } else {
            if (tma_tile<BX, BY, S, true, RAGGED, SEAM, false>(P, B, phiu, refB, st, sm, x0, y0, min(BX, P.nx - x0),
                                                               min(BY, P.ny - y0), seam, ok, on_abort, no_refill))
                return;
            __syncthreads();  // every warp is done with stage s
            refill();
        }
    }
    // the tiles outside the TMA rectangle (next to a periodic y seam) through the general path; their
    // ring lives in the stages, which the last TMA tile may still be reading
    if constexpr (REST) {
        if ((int)blockIdx.x < nedge) __syncthreads();
        for (int e = blockIdx.x; e < nedge; e += grid) {
            // map edge index e to the e-th tile outside the TMA rectangle
            int idx = e, bx = 0, by = 0;
            {
                // tiles in row-major order, skipping the TMA rectangle
                int row = 0;
                for (row = 0; row < tilesy; ++row) {
                    const bool inner = row >= by0 && row < by0 + ntby;
                    const int cnt = inner ? tilesx - ntbx : tilesx;
                    if (idx < cnt) break;
                    idx -= cnt;
                }
                by = row;
                const bool inner = by >= by0 && by < by0 + ntby;
                bx = (inner && idx >= bx0) ? idx + ntbx : idx;
            }
            int x0, y0, w, h;
            tile_whole(P.nx, BX, bx, x0, w);
            tile_whole(P.ny, BY, by, y0, h);
            step_tile_general<BX, BY, S, false>(P, A, B, phiu, refA, refB, *reinterpret_cast<RingSmem<BX, BY>*>(dsm), x0, y0,
                                                w, h);
        }
    }
}

}  // namespace tpf
