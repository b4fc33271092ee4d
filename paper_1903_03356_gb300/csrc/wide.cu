// Two-kernel step for contexts of few capsules on lattices that stay in L2 (Coclite et al.,
// arXiv:1903.03356, Section 2.3.2 and 2.4): one kernel updates the vertices of step n and
// spreads the forces of step n + 1, one updates the lattice with those forces.
//
// With few capsules a step is a chain of dependent round trips, not a matter of bandwidth:
// one tiled CTA spends 17 k cycles on the spread of 16 vertices (9.6 k of them in the
// compare-and-swap loops of shared float atomics and in double instructions, each of which
// holds a warp for 64 cycles on GB300) and 19 k on their update. These kernels shorten the
// chain instead of sharing work:
//   - nine lanes per interpolation point, one per support node: each pulls its own node's
//     nine populations (one round trip), and the weighted sums are shuffles. No tile.
//   - the spread is one double reduction per lane straight into the force field in L2.
//   - everything that does not depend on the lattice (the staged ring, membrane terms,
//     probe places, shape functions) is done before griddepcontrol.wait, beside the lattice
//     kernel (programmatic dependent launch).
// Per step, tiled kernels against these: 100 x 100 shear box, 64 vertices, Kinematic, FP64
// 42.8 -> 18.0 us; 360 x 120 open channel, 586 vertices, Dynamic, FP32 27.4 -> 16.4 us.
#include <cooperative_groups.h>

#include <algorithm>
#include <initializer_list>
#include <map>
#include <mutex>
#include <utility>

#include "ring.cuh"

namespace cg = cooperative_groups;

namespace lbmib {
namespace {

template <typename C>
struct V2 {
    C x, y;
};

// What one traction probe leaves in shared memory: density and rho nu (G + G^T) n.
template <typename C>
struct Probe9 {
    C rho, tx, ty;
};

// Programmatic dependent launch. Every kernel here waits before it reads what the kernel
// before it wrote, and lets the next one start only after that wait: what a kernel reads
// before its own wait was therefore written two kernels earlier at least, and is complete.
// What is read after the wait was written while the kernel was already resident: plain
// loads only (pull_all with NC = false, no __restrict__ const pointers), since the read-only
// path may hold lines from before.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// A lane's place among the three nine-lane groups of its warp (lanes 27-31 repeat lane 26).
struct Lane9 {
    int grp, base, k, a, b;
    bool on;
    __device__ __forceinline__ Lane9() {
        const int lane = threadIdx.x & 31;
        on = lane < 27;
        grp = on ? lane / 9 : 2;
        base = 9 * grp;
        k = on ? lane - base : 8;
        a = k % 3;
        b = k / 3;
    }
};

template <typename T>
__device__ __forceinline__ T get9(T v, int lane) {
    return __shfl_sync(0xffffffffu, v, lane);
}

// Sum over a group, valid in its lane k = 0.
template <typename T>
__device__ __forceinline__ T sum9(T v) {
    v += __shfl_down_sync(0xffffffffu, v, 1) + __shfl_down_sync(0xffffffffu, v, 2);
    return v + (__shfl_down_sync(0xffffffffu, v, 3) + __shfl_down_sync(0xffffffffu, v, 6));
}

// The lane's share of the MLS fit (Eq. 8-9) at a point whose centre node lies at the offset
// (dx, dy) from it. Whole warp. Per axis, with offsets d_j, weights w_j, S = sum w, mean
// offset m and V = sum w (d - m)^2: q = w/S, g = w (d - m)/V, h = q - m g, and the value
// weight of the lane's node is h_x q_y + q_x h_y - q_x q_y, its slope weights g_x q_y and
// q_x g_y (the diagonal moment matrix of mls_weights, per axis). One exponential per lane
// (in FP64 some twenty instructions of 64 cycles): lanes 0-2 of a group do the x axis, 3-5
// the y axis; the sums are shuffles. Single precision: every lane takes the tiled kernels' fit
// (its weights bit for bit, so that a ring at rest, whose forces are all rounding, spreads the
// same ones) and picks its node's.
template <typename C>
struct Fit9 {
    C phi, gx, gy;
    __device__ __forceinline__ Fit9(const Lane9& l, C dx, C dy) {
        if constexpr (sizeof(C) == 4) {
            const MlsW<C> m = mls_weights<C>(0, 0, dx, dy, true);
            auto pick = [](const C (&v)[3], int i) { return i == 0 ? v[0] : (i == 1 ? v[1] : v[2]); };
            const C px = pick(m.dxp, l.a), py = pick(m.dyp, l.b), w = pick(m.wx, l.a) * pick(m.wy, l.b);
            phi = w * (m.k0 + m.kx * px + m.ky * py);
            gx = m.gx * (w * px);
            gy = m.gy * (w * py);
            return;
        }
        const int j = l.a, ax = l.base + (l.k < 3 ? 0 : 3);   // own index, first lane of the own axis
        const C d0 = l.k < 3 ? dx : dy, d = d0 + C(j - 1);
        const C w = exp(-d * d * C(kMlsInvLen2));
        const C w0 = get9(w, ax), w1 = get9(w, ax + 1), w2 = get9(w, ax + 2);
        const C is = rcp_bounded(w0 + w1 + w2);
        const C t = (w2 - w0) * is;                           // m = d0 + t
        const C dm = C(j - 1) - t;
        const C iV = rcp_bounded(w0 * (C(1) + t) * (C(1) + t) + w1 * t * t + w2 * (C(1) - t) * (C(1) - t));
        const C q = w * is, g = w * dm * iV, h = q - (d0 + t) * g;
        const int lx = l.base + l.a, ly = l.base + 3 + l.b;
        const C qx = get9(q, lx), hx = get9(h, lx), sx = get9(g, lx);
        const C qy = get9(q, ly), hy = get9(h, ly), sy = get9(g, ly);
        phi = hx * qy + qx * hy - qx * qy;
        gx = sx * qy;
        gy = qx * sy;
    }
    // velocity at the point, in every lane of the group
    __device__ __forceinline__ V2<C> velocity(const Lane9& l, const Mom<C>& f) const {
        return V2<C>{get9(sum9<C>(phi * f.ux), l.base), get9(sum9<C>(phi * f.uy), l.base)};
    }
    // the probe's values in lane k = 0: linear in the slopes, contracted with n before the sum
    __device__ __forceinline__ Probe9<C> probe(const Mom<C>& f, C nx, C ny, C nu) const {
        const C dux = gx * f.ux, duy = gy * f.ux, dvx = gx * f.uy, dvy = gy * f.uy;
        const C rho = C(1) + sum9<C>(phi * f.drho), m = rho * nu;
        return Probe9<C>{rho, m * sum9<C>(C(2) * dux * nx + (duy + dvx) * ny),
                         m * sum9<C>((duy + dvx) * nx + C(2) * dvy * ny)};
    }
};

// Own vertices of CTA `rank`: [v0, v0 + m) of a split of the ring into chunks; they are
// staged in slots kHalo .. kHalo + m - 1 with kHalo neighbours on each side.
struct Part {
    int cap, rank, arcs, n, off, v0, m, chunk;
    __device__ __forceinline__ int node(int li) const { return off + (v0 - kHalo + li + 2 * n) % n; }
    __device__ __forceinline__ int first(int r) const { return r * chunk; }
    __device__ __forceinline__ int owner(int v) const { return v / chunk; }   // the CTA that owns vertex v
};

// What a launch works on besides the lattice and the vertices.
struct WideIO {
    const double* fib_n;   // Kinematic: the force of the step whose update this is
    double* fib;           // force buffer of the next step's spread
    int* list;             // its node list: entry 9 g + k is support node k of vertex g
    int* count;            // its length (set to nine entries per vertex, or to 0 without a spread)
    unsigned* status;
    double2* tape;         // optional: X^{n+1} of every vertex
};

// Shared arrays besides CapSmem's: X^{n+1} (or its float increment), the support frames
// (centre node, offset of the centre node from the vertex; a NaN offset marks a position that
// was not sane), the elements' probes and tractions, the next vertex velocity, the lengths.
template <typename C>
struct WideSmem {
    double2* X1;
    int2* fc;
    V2<C>* fd;
    Probe9<C>* pv;   // [2 li + side]
    V2<C>* ext;
    V2<C>* uv;
    V2<C>* inc;
    C* len;
    static size_t bytes(int slots) {
        return (size_t)slots * (sizeof(double2) + sizeof(int2) + 4 * sizeof(V2<C>) + 2 * sizeof(Probe9<C>) + sizeof(C)) + 16;
    }
    __device__ __forceinline__ WideSmem(unsigned char* p, int slots) {
        X1 = reinterpret_cast<double2*>(p);
        fc = reinterpret_cast<int2*>(X1 + slots);
        fd = reinterpret_cast<V2<C>*>(fc + slots);
        ext = fd + slots;
        uv = ext + slots;
        inc = uv + slots;
        pv = reinterpret_cast<Probe9<C>*>(inc + slots);
        len = reinterpret_cast<C*>(pv + 2 * slots);
    }
};

__device__ __forceinline__ bool wide_part(const Nodes& nd, int max_n, int arcs, CapsuleParams& P, Part& p,
                                          unsigned* status) {
    p.arcs = arcs;
    p.cap = blockIdx.x / arcs;
    p.rank = blockIdx.x - p.cap * arcs;
    P = nd.caps[p.cap];
    if (P.n < 3 || P.n > max_n || P.off < 0 || P.off + P.n > nd.count) {
        pdl_wait();   // the kernel must not finish before the one it waits for
        if (threadIdx.x == 0) atomicOr(status, kStatRing);
        return false;
    }
    p.n = P.n;
    p.off = P.off;
    p.chunk = (P.n + arcs - 1) / arcs;
    p.v0 = p.first(p.rank);
    p.m = max(0, min(P.n - p.v0, p.chunk));
    return true;
}

// Support frame of the position X in slot li.
template <typename C>
__device__ __forceinline__ void set_frame(const Lat& L, const WideSmem<C>& ws, int li, double2 X) {
    int cx, cy;
    bool sane;
    support_centre(L, X.x, X.y, cx, cy, &sane);
    ws.fc[li] = make_int2(cx, cy);
    ws.fd[li] = V2<C>{sane ? C((double)cx - X.x) : C(__int_as_float(0x7fc00000)), C((double)cy - X.y)};
}

// Support frame at X^{n+1} = X^n + inc from the frame at X^n in single precision: the centre
// node in float, the offset as the exact double difference (as in the tiled kernels).
__device__ __forceinline__ void move_frame(const WideSmem<float>& ws, int li, float ix, float iy, double2 Xn) {
    int2 c = ws.fc[li];
    V2<float> d = ws.fd[li];
    const float px = ix - d.x, py = iy - d.y;
    if (fabsf(px) < 1024.0f && fabsf(py) < 1024.0f) {   // false for NaN too
        c.x += (int)floorf(px + 0.5f);
        c.y += (int)floorf(py + 0.5f);
        d.x = (float)((double)c.x - Xn.x);
        d.y = (float)((double)c.y - Xn.y);
    } else {
        d.x = __int_as_float(0x7fc00000);
    }
    ws.fc[li] = c;
    ws.fd[li] = d;
}

// Point of the nine-lane interpolation: centre node and its offset from the point.
template <typename C>
struct Point9 {
    int cx, cy;
    C dx, dy;
    bool ok;
};

// The point of slot li's own frame.
template <typename C>
__device__ __forceinline__ Point9<C> point_at(const Lat& L, const WideSmem<C>& ws, int li) {
    const int2 c = ws.fc[li];
    const V2<C> d = ws.fd[li];
    const bool sane = !isnan(d.x);
    Point9<C> p{sane ? c.x : 0, sane ? c.y : 0, sane ? d.x : C(0), sane ? d.y : C(0), false};
    p.ok = sane && support_inside(L, p.cx, p.cy);
    return p;
}

// The point at the offset (ox, oy) from slot li's position.
template <typename C>
__device__ __forceinline__ Point9<C> point_near(const Lat& L, const WideSmem<C>& ws, int li, C ox, C oy) {
    const Point9<C> v = point_at<C>(L, ws, li);
    C px = ox - v.dx, py = oy - v.dy;
    const bool sane = fabs(px) < C(1024) && fabs(py) < C(1024);   // false for NaN too
    if (!sane) px = py = C(0);
    const C kx = floor(px + C(0.5)), ky = floor(py + C(0.5));
    Point9<C> p{v.cx + (int)kx, v.cy + (int)ky, kx - px, ky - py, false};
    p.ok = v.ok && sane && support_inside(L, p.cx, p.cy);
    return p;
}

__device__ __forceinline__ void support_node(const Lat& L, const Lane9& l, int cx, int cy, int& x, int& y) {
    x = wrapi(cx + l.a - 1, L.nx);
    y = support_row(L, cy + l.b - 1);
}

// The lane's share of the spread of F (times c_l, already in F) with its value weight w: one
// double reduction per lane and component into the force field in L2.
template <typename C>
__device__ __forceinline__ void spread9(const Lat& L, const Lane9& l, const WideIO& io, int x, int y, int g, C w,
                                        C Fx, C Fy) {
    const long long N = (long long)L.nx * L.ny;
    const int cell = y * L.nx + x;
    atomicAdd(io.fib + cell, (double)(w * Fx));
    atomicAdd(io.fib + N + cell, (double)(w * Fy));
    io.list[9LL * g + l.k] = cell;
}

// Twice the enclosed area of the capsule (Eq. 14), needed only with an area constant.
// Collective over the cluster.
template <typename C>
__device__ __forceinline__ double area2_of(const CapSmem& sm, const Part& p, double2 X0, double* part) {
    double v[1] = {0.0};
    for (int k = threadIdx.x; k < p.m; k += blockDim.x) {
        const int li = kHalo + k;
        if constexpr (sizeof(C) == 4) {
            const double2 X = sm.X[li];
            const float2 e = ring_f(sm)[li].e;
            v[0] += (double)((float)(X.x - X0.x) * e.y - (float)(X.y - X0.y) * e.x);
        } else {
            v[0] += area_term(X0, sm.X[li], sm.X[li + 1]);
        }
    }
    block_reduce<1, false>(v, sm.red);
    if (p.arcs == 1) return v[0];
    cg::cluster_group cl = cg::this_cluster();
    if (threadIdx.x == 0) *part = v[0];
    cl.sync();
    double t = 0.0;
    for (int r = 0; r < p.arcs; r++) t += *cl.map_shared_rank(part, r);   // in rank order: the same bits everywhere
    cl.sync();
    return t;
}

// Membrane terms of the own slots and one on each side.
template <typename C>
__device__ __forceinline__ void terms9(const CapSmem& sm, const CapsuleParams& P, const Nodes& nd, const Part& p) {
    for (int k = threadIdx.x; k < (p.m > 0 ? p.m + 2 : 0); k += blockDim.x) {
        const int li = kHalo - 1 + k;
        if constexpr (sizeof(C) == 4) vertex_terms_f(sm, P, nd, li - 1, li, li + 1, p.node(li));
        else vertex_terms(sm, P, nd, li - 1, li, li + 1, p.node(li));
    }
}

// CTA sizes: single precision up to 768 threads (85 registers), double 384.
template <typename S>
constexpr int wide_threads() {
    return sizeof(typename St<S>::C) == 4 ? 768 : 384;
}

// ---------------------------------------------------------------------------------
// Dynamic scheme. UPD: steps 7-8 of step n (probe tractions on the lattice state after the
// fluid update, membrane forces at X^n, Eq. 23-24). SPR: steps 1-3 of step n + 1 (U at
// X^{n+1} on the same state, F = u_v - U, spread with c_l). A capsule's `arcs` CTAs are a
// cluster: its barrier orders every read of X^n before any write of X^{n+1}, and the
// neighbours' increments are read from distributed shared memory.
// ---------------------------------------------------------------------------------
template <typename S, bool UPD, bool SPR>
__global__ void __launch_bounds__(wide_threads<S>()) k_wide_dyn(const S* pops, Lat L, Nodes nd,
                                                                int max_n, int arcs, WideIO io) {
    using C = typename St<S>::C;
    constexpr bool F32 = sizeof(C) == 4;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double s_part;
    const int slots = arc_slots(max_n, arcs) + 1;
    const CapSmem sm = carve(smem, slots);
    const WideSmem<C> ws(sm.tile, slots);
    CapsuleParams P;
    Part p;
    if (!wide_part(nd, max_n, arcs, P, p, io.status)) return;
    const int m = p.m, nw = blockDim.x >> 5, warp = threadIdx.x >> 5;
    const Lane9 l;
    bool ok = true, waited = false;
    // before the wait: the staged ring, its membrane terms and support frames
    for (int li = threadIdx.x; li < (m > 0 ? m + 2 * kHalo : 0); li += blockDim.x) sm.X[li] = nd.X[p.node(li)];
    if (UPD)
        for (int k = threadIdx.x; k < m; k += blockDim.x) {   // X^{n-1} and the tentative velocity U
            const int g = p.node(kHalo + k);
            sm.ext[kHalo + k] = nd.Xm1[g];
            if constexpr (F32) xd_f(sm)[kHalo + k] = u_f(nd)[g];
            else sm.xd[kHalo + k] = nd.U[g];
        }
    __syncthreads();
    if (UPD) terms9<C>(sm, P, nd, p);
    // frames of the own slots and (for the element before them) of the slot before, on the
    // CTA's last warps: beside the terms
    for (int k = (int)blockDim.x - 1 - (int)threadIdx.x; k < (m > 0 ? m + 1 : 0); k += blockDim.x)
        set_frame<C>(L, ws, kHalo - 1 + k, sm.X[kHalo - 1 + k]);
    __syncthreads();
    double A2 = 0.0;
    if (UPD && P.ka != 0.0) A2 = area2_of<C>(sm, p, nd.X[p.off], &s_part);
    if (UPD && arcs > 1) asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");   // X^n is read
    if (UPD) {
        // tractions (Eq. 15-16) of the own elements and the one before them: probe `side` of
        // element li at its centroid +/- 1.2 n+
        const int ns = m > 0 ? 2 * (m + 1) : 0;
        const C nu = C(L.nu);
        for (int s0 = 3 * warp; s0 < ns; s0 += 3 * nw) {
            const int s = min(s0 + l.grp, ns - 1), li = kHalo - 1 + (s >> 1);
            C ex_, ey_;
            if constexpr (F32) {
                ex_ = ring_f(sm)[li].e.x;
                ey_ = ring_f(sm)[li].e.y;
            } else {
                ex_ = sm.X[li + 1].x - sm.X[li].x;
                ey_ = sm.X[li + 1].y - sm.X[li].y;
            }
            const C e2 = ex_ * ex_ + ey_ * ey_, rl = rsqrt(e2);
            const C nx = ey_ * rl, ny = -ex_ * rl, sg = (s & 1) ? C(-1) : C(1);
            const Point9<C> q = point_near<C>(L, ws, li, C(0.5) * ex_ + sg * C(1.2) * nx, C(0.5) * ey_ + sg * C(1.2) * ny);
            const Fit9<C> w(l, q.dx, q.dy);
            int x, y;
            support_node(L, l, q.cx, q.cy, x, y);
            if (!waited) {
                pdl_wait();
                waited = true;
            }
            const Mom<C> f = node_moments<S, false>(pops, L, nullptr, x, y);
            const Probe9<C> pv = w.probe(f, nx, ny, nu);
            if (l.on && l.k == 0 && s0 + l.grp < ns) ws.pv[2 * li + (s & 1)] = pv;
            ok &= q.ok;
        }
    }
    if (!waited && !(SPR && !UPD)) pdl_wait();
    if (UPD) pdl_launch();
    __syncthreads();
    if (UPD && arcs > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    if (UPD) {
        // Eq. 15-16: the two probes' difference times the element's length
        for (int k = threadIdx.x; k < (m > 0 ? m + 1 : 0); k += blockDim.x) {
            const int li = kHalo - 1 + k;
            C ex_, ey_;
            if constexpr (F32) {
                ex_ = ring_f(sm)[li].e.x;
                ey_ = ring_f(sm)[li].e.y;
            } else {
                ex_ = sm.X[li + 1].x - sm.X[li].x;
                ey_ = sm.X[li + 1].y - sm.X[li].y;
            }
            const C e2 = ex_ * ex_ + ey_ * ey_, rl = rsqrt(e2), len = e2 * rl;
            const Probe9<C> op = ws.pv[2 * li], om = ws.pv[2 * li + 1];
            // the pressures' difference with one product rounded, as the tiled kernels' is compiled:
            // in single precision that rounding is all the traction there is in a fluid at rest
            const C third = C(1.0 / 3.0), dp = fma(op.rho, third, -(om.rho * third));
            ws.ext[li] = V2<C>{(-dp * (ey_ * rl) + (op.tx - om.tx)) * len, (dp * (ex_ * rl) + (op.ty - om.ty)) * len};
        }
        __syncthreads();
        // Eq. 22-24 of the own vertices
        const float fa = F32 ? (float)P.ka * ((float)(P.A0 - 0.5 * A2) / (6.0f * (float)P.A0)) : 0.0f;
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
            const int li = kHalo + k, g = p.node(li);
            const double2 Xv = sm.X[li], Xm = sm.ext[li];
            const V2<C> f0 = ws.ext[li], f1 = ws.ext[li - 1];   // half of each element's traction
            C Fex = C(0.5) * (f0.x + f1.x), Fey = C(0.5) * (f0.y + f1.y);
            if (nd.Fpp) {   // Eq. 27, part of the total force (step 7)
                const double2 f = nd.Fpp[g];
                Fex += C(f.x);
                Fey += C(f.y);
            }
            double2 Xn, Fi2;
            V2<C> uvn;
            if constexpr (F32) {
                const float2 Fi = internal_force_f(sm, li - 1, li, li + 1, fa);
                const float hm = 0.5f / (float)P.m;
                const float2 U = xd_f(sm)[li];
                const float ix = U.x + hm * (Fi.x + Fex), iy = U.y + hm * (Fi.y + Fey);
                Xn = make_double2(Xv.x + (double)ix, Xv.y + (double)iy);
                uvn = V2<C>{1.5f * ix - 0.5f * (float)(Xv.x - Xm.x), 1.5f * iy - 0.5f * (float)(Xv.y - Xm.y)};
                ws.inc[li] = V2<C>{ix, iy};
                Fi2 = make_double2(Fi.x, Fi.y);
                if (SPR) move_frame(ws, li, ix, iy, Xn);
            } else {
                Fi2 = internal_force(sm, P, li - 1, li, li + 1, 0.5 * A2);
                const double hm = 0.5 / P.m;
                const double2 U = sm.xd[li];
                Xn = make_double2(Xv.x + U.x + hm * (Fi2.x + Fex), Xv.y + U.y + hm * (Fi2.y + Fey));
                uvn = V2<C>{1.5 * Xn.x - 2.0 * Xv.x + 0.5 * Xm.x, 1.5 * Xn.y - 2.0 * Xv.y + 0.5 * Xm.y};
                ws.X1[li] = Xn;
                if (SPR) set_frame<C>(L, ws, li, Xn);
            }
            ws.uv[li] = uvn;
            nd.X[g] = Xn;
            nd.Xm1[g] = Xv;
            nd.uv[g] = make_double2((double)uvn.x, (double)uvn.y);
            if (!SPR) {   // the forces a call ends with
                nd.Fint[g] = Fi2;
                nd.Fext[g] = make_double2((double)Fex, (double)Fey);
            }
            if (io.tape) io.tape[g] = Xn;
            nd.age[g] += 1;
        }
        if (SPR && m > 0) {
            // increments (single precision) or positions of the two neighbours at X^{n+1}
            if (arcs > 1) cg::this_cluster().sync();
            else __syncthreads();
            if (threadIdx.x < 2) {
                const int v = threadIdx.x == 0 ? (p.v0 + p.n - 1) % p.n : (p.v0 + m) % p.n;
                const int r = p.owner(v), from = kHalo + v - p.first(r), to = threadIdx.x == 0 ? kHalo - 1 : kHalo + m;
                if constexpr (F32) {
                    V2<C>* src = arcs > 1 ? cg::this_cluster().map_shared_rank(ws.inc, r) : ws.inc;
                    ws.inc[to] = src[from];
                } else {
                    double2* src = arcs > 1 ? cg::this_cluster().map_shared_rank(ws.X1, r) : ws.X1;
                    ws.X1[to] = src[from];
                }
            }
        } else if (SPR && arcs > 1) {
            cg::this_cluster().sync();
        }
        __syncthreads();
    }
    if (SPR) {
        // lengths of the elements on both sides of every own vertex at the new positions
        for (int k = threadIdx.x; k < (m > 0 ? m + 1 : 0); k += blockDim.x) {
            const int li = kHalo - 1 + k;
            C dx, dy;
            if constexpr (UPD && F32) {   // the edges at X^n and the float increments, off the FP64 pipe
                const float2 e = ring_f(sm)[li].e;
                dx = e.x + (ws.inc[li + 1].x - ws.inc[li].x);
                dy = e.y + (ws.inc[li + 1].y - ws.inc[li].y);
            } else {
                const double2* X = UPD ? ws.X1 : sm.X;
                const double2 d = X[li + 1] - X[li];
                dx = C(d.x);
                dy = C(d.y);
            }
            ws.len[li] = sqrt(dx * dx + dy * dy);
        }
        __syncthreads();
        for (int s0 = 3 * warp; s0 < m; s0 += 3 * nw) {
            const int s = min(s0 + l.grp, m - 1), li = kHalo + s, g = p.node(li);
            const Point9<C> q = point_at<C>(L, ws, li);
            const Fit9<C> w(l, q.dx, q.dy);
            int x, y;
            support_node(L, l, q.cx, q.cy, x, y);
            if (!UPD && !waited) {
                pdl_wait();
                waited = true;
            }
            const Mom<C> f = node_moments<S, false>(pops, L, nullptr, x, y);
            const V2<C> U = w.velocity(l, f);
            const C Ux = U.x, Uy = U.y;
            V2<C> uv;
            const bool act = l.on && s0 + l.grp < m, lead = act && l.k == 0;
            if (UPD) {
                uv = ws.uv[li];
            } else {
                const bool first = nd.age[g] == 0;   // a vertex's first step: u_v = U, X^{-1} = X^0 - U
                const double2 u = nd.uv[g];
                uv = first ? V2<C>{Ux, Uy} : V2<C>{C(u.x), C(u.y)};
                if (lead && first) {
                    nd.uv[g] = make_double2((double)Ux, (double)Uy);
                    nd.Xm1[g] = make_double2(sm.X[li].x - (double)Ux, sm.X[li].y - (double)Uy);
                }
            }
            const C cl = C(0.5) * (ws.len[li - 1] + ws.len[li]);
            const C Fx = cl * (uv.x - Ux), Fy = cl * (uv.y - Uy);
            if (lead) {
                if constexpr (F32) u_f(nd)[g] = make_float2(Ux, Uy);
                else nd.U[g] = make_double2(Ux, Uy);
                if (nd.Flc) nd.Flc[g] = make_double2((double)Fx, (double)Fy);
            }
            if (act) spread9<C>(L, l, io, x, y, g, w.phi, Fx, Fy);
            ok &= q.ok;
        }
        if (!UPD && !waited) pdl_wait();
        if (!UPD) pdl_launch();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *io.count = SPR ? 9 * nd.count : 0;
    if (!ok) atomicOr(io.status, kStatSupport);
    // no CTA leaves while another still reads its positions
    if (UPD && SPR && arcs > 1) cg::this_cluster().sync();
}

// ---------------------------------------------------------------------------------
// Kinematic scheme. UPD: steps vii-viii of step n (u at X^n with half the spread force,
// Eq. 25). SPR: steps i-iii of step n + 1 (membrane forces at X^{n+1} and their spread, with
// the repulsion when it is on).
// ---------------------------------------------------------------------------------
template <typename S, bool UPD, bool SPR>
__global__ void __launch_bounds__(wide_threads<S>()) k_wide_kin(const S* pops, Lat L, Nodes nd,
                                                                int max_n, int arcs, WideIO io) {
    using C = typename St<S>::C;
    constexpr bool F32 = sizeof(C) == 4;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double s_part;
    const int slots = arc_slots(max_n, arcs) + 1;
    const CapSmem sm = carve(smem, slots);
    const WideSmem<C> ws(sm.tile, slots);
    CapsuleParams P;
    Part p;
    if (!wide_part(nd, max_n, arcs, P, p, io.status)) return;
    const int m = p.m, nw = blockDim.x >> 5, warp = threadIdx.x >> 5;
    const Lane9 l;
    bool ok = true, waited = false;
    const int lo = UPD ? kHalo : 0, hi = m == 0 ? lo : (UPD ? kHalo + m : m + 2 * kHalo);
    for (int li = lo + threadIdx.x; li < hi; li += blockDim.x) sm.X[li] = nd.X[p.node(li)];
    if (UPD)
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
            const int g = p.node(kHalo + k);
            // Eq. 25 and the forward Euler of a first step as c0 X + c1 X^{n-1} + c2 u
            sm.ext[kHalo + k] = nd.Xm1[g];
            ws.len[kHalo + k] = nd.age[g] == 0 ? C(1) : C(0);
        }
    __syncthreads();
    for (int k = threadIdx.x; k < m; k += blockDim.x) set_frame<C>(L, ws, kHalo + k, sm.X[kHalo + k]);
    __syncthreads();
    if (UPD) {
        for (int s0 = 3 * warp; s0 < m; s0 += 3 * nw) {
            const int s = min(s0 + l.grp, m - 1), li = kHalo + s, g = p.node(li);
            const Point9<C> q = point_at<C>(L, ws, li);
            const Fit9<C> w(l, q.dx, q.dy);
            int x, y;
            support_node(L, l, q.cx, q.cy, x, y);
            if (!waited) {
                pdl_wait();
                waited = true;
            }
            const Mom<C> f = node_moments<S, false>(pops, L, io.fib_n, x, y);
            const V2<C> U = w.velocity(l, f);
            if (l.on && l.k == 0 && s0 + l.grp < m) {
                const double2 Xv = sm.X[li], Xm = sm.ext[li];
                const double ux = (double)U.x, uy = (double)U.y;
                double2 Xn;
                if (ws.len[li] != C(0)) Xn = make_double2(Xv.x + ux, Xv.y + uy);
                else Xn = make_double2((2.0 / 3.0) * (2.0 * Xv.x - 0.5 * Xm.x + ux),
                                       (2.0 / 3.0) * (2.0 * Xv.y - 0.5 * Xm.y + uy));
                ws.X1[li] = Xn;
                nd.Xm1[g] = Xv;
                nd.X[g] = Xn;
                nd.uv[g] = make_double2(ux, uy);
                if (io.tape) io.tape[g] = Xn;
                nd.age[g] += 1;
            }
            ok &= q.ok;
        }
    }
    if (!waited) pdl_wait();
    pdl_launch();
    if (UPD && SPR) {
        if (arcs > 1) cg::this_cluster().sync();
        else __syncthreads();
        // the own positions and kHalo neighbours on each side at X^{n+1}
        for (int li = threadIdx.x; li < (m > 0 ? m + 2 * kHalo : 0); li += blockDim.x) {
            const int v = (p.v0 - kHalo + li + 2 * p.n) % p.n, r = p.owner(v), from = kHalo + v - p.first(r);
            const double2* src = arcs > 1 ? cg::this_cluster().map_shared_rank(ws.X1, r) : ws.X1;
            sm.X[li] = src[from];
        }
        __syncthreads();
    }
    if (SPR) {
        terms9<C>(sm, P, nd, p);
        if (UPD)
            for (int k = (int)blockDim.x - 1 - (int)threadIdx.x; k < m; k += blockDim.x)
                set_frame<C>(L, ws, kHalo + k, sm.X[kHalo + k]);
        __syncthreads();
        double A2 = 0.0;
        if (P.ka != 0.0) {
            double2 X0;   // the capsule's first vertex, wherever it is staged
            if (UPD) X0 = arcs > 1 ? cg::this_cluster().map_shared_rank(ws.X1, p.owner(0))[kHalo] : ws.X1[kHalo];
            else X0 = nd.X[p.off];
            A2 = area2_of<C>(sm, p, X0, &s_part);
        }
        const float fa = F32 ? (float)P.ka * ((float)(P.A0 - 0.5 * A2) / (6.0f * (float)P.A0)) : 0.0f;
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
            const int li = kHalo + k, g = p.node(li);
            double2 F;
            if constexpr (F32) {
                const float2 f = internal_force_f(sm, li - 1, li, li + 1, fa);
                F = make_double2(f.x, f.y);
            } else {
                F = internal_force(sm, P, li - 1, li, li + 1, 0.5 * A2);
            }
            nd.Fint[g] = F;
            nd.Fext[g] = make_double2(0.0, 0.0);
            const double2 r = nd.Fpp ? nd.Fpp[g] : make_double2(0.0, 0.0);   // Eq. 27
            ws.uv[li] = V2<C>{C(F.x + r.x), C(F.y + r.y)};
        }
        __syncthreads();
        for (int s0 = 3 * warp; s0 < m; s0 += 3 * nw) {
            const int s = min(s0 + l.grp, m - 1), li = kHalo + s, g = p.node(li);
            const Point9<C> q = point_at<C>(L, ws, li);
            const Fit9<C> w(l, q.dx, q.dy);
            int x, y;
            support_node(L, l, q.cx, q.cy, x, y);
            const V2<C> F = ws.uv[li];
            if (l.on && s0 + l.grp < m) spread9<C>(L, l, io, x, y, g, w.phi, F.x, F.y);
            ok &= q.ok;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *io.count = SPR ? 9 * nd.count : 0;
    if (!ok) atomicOr(io.status, kStatSupport);
    if (UPD && SPR && arcs > 1) cg::this_cluster().sync();   // no CTA leaves while another reads its X^{n+1}
}

// ---------------------------------------------------------------------------------
// Lattice update with the force field read in place (Eq. 1-5), one node per thread: on a
// lattice that stays in L2 the sixteen bytes of force per node cost less than the patch's
// launch and list. A warp without forced nodes takes the uniform force (the test is on the
// bits: a double conversion would hold the warp for 64 cycles). Also clears the last step's
// force at its listed nodes; on an open channel the thread of an inlet or outlet node closes
// its own populations. One node per thread and 64-thread CTAs spread a small FP64 lattice
// over every SM's FP64 pipe.
// ---------------------------------------------------------------------------------
template <typename S>
__global__ void __launch_bounds__(128) k_collide_forced(const S* src, S* dst, Lat L,
                                                        OpenBC ob, const double* fib, double* fib_p,
                                                        const int* list_p, const int* count_p, int capacity,
                                                        CollideD kd, unsigned* status) {
    using C = typename St<S>::C;
    const long long N = (long long)L.nx * L.ny;
    const int node = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = node / L.nx, x = node - y * L.nx;
    pdl_wait();
    pdl_launch();
    bool bad = false;
    if (node < N) {
        C s[9];
        const long long bx = reinterpret_cast<const long long*>(fib)[node];
        const long long by = reinterpret_cast<const long long*>(fib)[N + node];
        pull_all<S, false>(src, L, x, y, s, &ob);
        C Fx = lat_c<C>(L.gx, L.gxf), Fy = lat_c<C>(L.gy, L.gyf);
        if (((bx | by) << 1) != 0) {
            Fx = C(L.gx + __longlong_as_double(bx));
            Fy = C(L.gy + __longlong_as_double(by));
        }
        C usq;
        if constexpr (sizeof(C) == 8) {   // the uniform force's constants come from the host
            CollideD k = kd;
            if (((bx | by) << 1) != 0) k = CollideD(Fx, Fy, L.omega);
            usq = collide_d(s, k);
        } else {
            usq = collide<C>(s, Fx, Fy, L.omegaf);
        }
        bad = !(usq < C(0.09));   // |u| > 0.3 or NaN
        S* o = dst + (long long)y * L.pitch + x;
#pragma unroll
        for (int i = 0; i < 9; i++) St<S>::st(o + (long long)i * L.plane, s[i], L);
    }
    if (bad) atomicOr(status, kStatUnstable);
    const int np = min(*count_p, capacity);
    for (int k = node; k < np; k += gridDim.x * blockDim.x) {
        const int cell = list_p[k];
        if (cell < 0 || cell >= N) {
            atomicOr(status, kStatCell);
            continue;
        }
        fib_p[cell] = 0.0;
        fib_p[N + cell] = 0.0;
    }
}

template <typename C>
size_t wide_smem(int max_n, int arcs) {
    const int slots = arc_slots(max_n, arcs) + 1;
    return ring_smem_bytes(slots) + WideSmem<C>::bytes(slots);
}

// Launch with programmatic stream serialisation (`pdl`) and the capsule's arcs as a cluster.
template <typename... P, typename... A>
void launch_pdl(void (*k)(P...), dim3 grid, int threads, size_t smem, int cluster, bool pdl, cudaStream_t s,
                A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    unsigned na = 0;
    if (cluster > 1) {
        at[na].id = cudaLaunchAttributeClusterDimension;
        at[na].val.clusterDim.x = (unsigned)cluster;
        at[na].val.clusterDim.y = 1;
        at[na].val.clusterDim.z = 1;
        na++;
    }
    if (pdl) {
        at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[na].val.programmaticStreamSerializationAllowed = 1;
        na++;
    }
    cfg.attrs = at;
    cfg.numAttrs = na;
    cudaLaunchKernelEx(&cfg, k, std::forward<A>(args)...);
}

}  // namespace

int wide_arcs(int max_n, int ncaps, int sms) {
    // about 16 vertices per CTA, while the CTAs number at most two per multiprocessor
    return std::max(1, std::min({kMaxArcs, (max_n + 15) / 16, 2 * sms / std::max(ncaps, 1)}));
}

// FP64 interpolations: two CTAs on one multiprocessor share its FP64 pipe and take twice as
// long, and beside the lattice kernel's last CTAs the scheduler does put two clusters onto the
// same multiprocessors while others are idle (8 rings of 512 vertices, Dynamic 183 us per step,
// alone 110; 2 rings with the repulsion 184 and 105). Asking for more than half of the shared
// memory keeps a CTA alone. Only while all find a place: fifteen clusters of eight do, with
// sixteen a second round follows (16 x 128 vertices 64 us, sharing 56).
constexpr size_t kAloneBytes = 116 * 1024;

bool wide_fits(int max_n, int arcs) { return wide_smem<double>(max_n, arcs) <= 200 * 1024; }

// As set_capsule_smem_limits: raised, never lowered, for the largest rings seen; per device,
// since every launch with FP64 interpolations that asks for kAloneBytes needs it.
void set_wide_smem_limits(int max_n, int arcs) {
    if (!wide_fits(max_n, arcs)) return;
    static std::mutex mu;
    static std::map<int, std::pair<size_t, size_t>> limits;   // device: single, double
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    std::lock_guard<std::mutex> lock(mu);
    auto& cur = limits.emplace(dev, std::make_pair(size_t(48 * 1024), size_t(48 * 1024))).first->second;
    auto raise = [&](size_t& have, size_t bytes, std::initializer_list<const void*> kernels) {
        if (bytes <= have) return;
        bool all = true;
        for (const void* k : kernels)
            all &= cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
        if (all) have = bytes;
    };
#define LBMIB_WIDE(S)                                                                                            \
    (const void*)k_wide_dyn<S, true, true>, (const void*)k_wide_dyn<S, true, false>,                             \
        (const void*)k_wide_dyn<S, false, true>, (const void*)k_wide_kin<S, true, true>,                         \
        (const void*)k_wide_kin<S, true, false>, (const void*)k_wide_kin<S, false, true>
    raise(cur.first, wide_smem<float>(max_n, arcs), {LBMIB_WIDE(float)});
    raise(cur.second, std::max(wide_smem<double>(max_n, arcs), kAloneBytes), {LBMIB_WIDE(double), LBMIB_WIDE(f32w)});
#undef LBMIB_WIDE
}

template <typename S>
void launch_wide(bool dynamic, bool upd, bool spr, const void* pops, const Lat& L, Nodes nd, int ncaps, int max_n,
                 int arcs, const double* fib_n, double* fib, int* list, int* count, unsigned* status, double2* tape,
                 bool pdl, cudaStream_t s) {
    using C = typename St<S>::C;
    const WideIO io{fib_n, fib, list, count, status, tape};
    size_t sh = wide_smem<C>(max_n, arcs);
    if (sizeof(C) == 8 && ncaps * arcs <= kWideAlone) sh = std::max(sh, kAloneBytes);
    // a warp for every three points of the larger sampling pass
    const int m = (max_n + arcs - 1) / arcs, pts = dynamic && upd ? 2 * (m + 1) : m;
    const int threads = std::max(128, std::min(wide_threads<S>(), (pts + 2) / 3 * 32));
    auto go = [&](auto* k) {
        launch_pdl(k, dim3((unsigned)(ncaps * arcs)), threads, sh, arcs, pdl, s, (const S*)pops, L, nd, max_n, arcs, io);
    };
    if (dynamic) {
        if (upd && spr) go(&k_wide_dyn<S, true, true>);
        else if (upd) go(&k_wide_dyn<S, true, false>);
        else go(&k_wide_dyn<S, false, true>);
    } else {
        if (upd && spr) go(&k_wide_kin<S, true, true>);
        else if (upd) go(&k_wide_kin<S, true, false>);
        else go(&k_wide_kin<S, false, true>);
    }
}

template <typename S>
void launch_collide_forced(const void* src, void* dst, const Lat& L, const OpenBC& ob, const double* fib,
                           double* fib_p, const int* list_p, const int* count_p, int capacity, unsigned* status,
                           bool pdl, cudaStream_t s) {
    const long long N = (long long)L.nx * L.ny;
    const int bs = sizeof(typename St<S>::C) == 8 ? 64 : 128;
    launch_pdl(&k_collide_forced<S>, dim3((unsigned)((N + bs - 1) / bs)), bs, 0, 1, pdl, s, (const S*)src, (S*)dst, L,
               ob, fib, fib_p, list_p, count_p, capacity, CollideD(L.gx, L.gy, L.omega), status);
}

#define LBMIB_INSTANTIATE_WIDE(S)                                                                              \
    template void launch_wide<S>(bool, bool, bool, const void*, const Lat&, Nodes, int, int, int, const double*, \
                                 double*, int*, int*, unsigned*, double2*, bool, cudaStream_t);
LBMIB_INSTANTIATE_WIDE(double)
LBMIB_INSTANTIATE_WIDE(float)
LBMIB_INSTANTIATE_WIDE(f32w)
#define LBMIB_INSTANTIATE_FORCED(S)                                                                            \
    template void launch_collide_forced<S>(const void*, void*, const Lat&, const OpenBC&, const double*, double*, \
                                           const int*, const int*, int, unsigned*, bool, cudaStream_t);
LBMIB_INSTANTIATE_FORCED(double)
LBMIB_INSTANTIATE_FORCED(float)

}  // namespace lbmib
