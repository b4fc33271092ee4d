// Capsule-capsule repulsion (Section 3.4, Eq. 27): on vertex 1 of a capsule, from every
// vertex 2 of another capsule closer than the cut-off r_c,
//   F_1 += 1e-4 / (8 sqrt 2) sqrt(dx / d_12^5) n_1^-   (dx = 1),
// with n_1^- the inward normal at vertex 1: the negated, normalised sum of the outward
// normals (dy, -dx)/l of the two elements that meet there. Distances along periodic
// axes are minimum images (x is not periodic in an open channel).
//
// Broad phase: each capsule's bounding box, and its coarse cell (side >= largest capsule
// extent + r_c, so interacting capsules sit in neighbouring cells), hashed into
// fixed-capacity buckets. Narrow phase: one warp per 32 vertices of an arc; for each capsule
// of the 3 x 3 neighbouring cells whose box comes within r_c of theirs it tests the boxes of
// that ring's 32-vertex chunks (one lane each), and the vertices of the chunks that pass. A
// capsule is accepted only from its own cell, so hash collisions cannot count it twice.
//
// A double instruction holds a warp for 64 cycles on GB300, so every test is made in float,
// on positions rounded to float, with a reach that covers the rounding; only a pair that
// passes is decided and evaluated in double, and only a vertex with a force forms its normal.
// (In double throughout, the two kernels took 55 of the 83 us of a step with 16 rings of
// 1000 vertices on 1200 x 450; the step now takes 62.)
#include "ring.cuh"

namespace lbmib {
namespace {

__device__ __forceinline__ double min_image(double d, double P) {
    return P > 0.0 ? d - P * floor(d / P + 0.5) : d;
}

__device__ __forceinline__ int bucket_of(int ix, int iy, int nb) {
    unsigned h = (unsigned)ix * 73856093u ^ (unsigned)iy * 19349663u;
    return (int)(h & (unsigned)(nb - 1));
}

__device__ __forceinline__ float warp_min(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_max(float v) { return -warp_min(-v); }

// A ring that has drifted far through a periodic axis is rounded to float after whole periods
// have been taken off, so that its float positions stay as fine as at home: at 5e8 they would
// be rounded to multiples of 32, the ring's coarse cell could come out two cells off and its
// partners not be found, or its box be reported as outgrown. The pair tests take minimum images
// anyway. far_out: |x| >= 2^16, from the bits (a double comparison would hold the warp);
// whole_periods out of line, for the same reason, and NaN beyond the positions that are sane.
__device__ __forceinline__ bool far_out(double x) { return (__double2hiint(x) & 0x7fffffff) >= 0x40f00000; }
__device__ __noinline__ double2 whole_periods(int nx, int ny, bool px, bool py, double x, double y) {
    if (!(fabs(x) < 1e9 && fabs(y) < 1e9)) return make_double2(__longlong_as_double(-1), 0.0);
    return make_double2(px ? nx * floor(x / nx) : 0.0, py ? ny * floor(y / ny) : 0.0);
}

// First chunk box of a capsule: chunks of different capsules never share a slot.
__device__ __forceinline__ int first_chunk(int cap, int off) { return off / 32 + cap; }

// Float positions, chunk boxes, bounding box, coarse cell and bucket entry of every capsule
// (one CTA per capsule, one warp per chunk).
__global__ void __launch_bounds__(128) k_rep_bin(Lat L, Nodes nd, int max_n, RepGrid g, unsigned* status) {
    __shared__ float4 part[4];
    const int c = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const CapsuleParams P = nd.caps[c];
    if (P.n < 3 || P.n > max_n) return;
    const int first = first_chunk(c, P.off);
    const double2 X0 = nd.X[P.off];
    const float inf = __int_as_float(0x7f800000);
    float4 b = make_float4(inf, inf, -inf, -inf);   // min x, min y, max x, max y
    auto bin = [&](double2 shift, bool shifted) {
        for (int v0 = 32 * warp; v0 < P.n; v0 += 128) {
            const int v = v0 + lane;
            double2 X = nd.X[P.off + (v < P.n ? v : v0)];
            if (shifted) X = X - shift;
            const float2 f = make_float2((float)X.x, (float)X.y);
            if (v < P.n) g.xf[P.off + v] = f;
            const float4 q = make_float4(warp_min(f.x), warp_min(f.y), warp_max(f.x), warp_max(f.y));
            if (lane == 0) g.cbox[first + v0 / 32] = q;
            b = make_float4(fminf(b.x, q.x), fminf(b.y, q.y), fmaxf(b.z, q.z), fmaxf(b.w, q.w));
        }
    };
    bin(X0, false);
    if (far_out(X0.x) || far_out(X0.y)) {   // again (the test before would be a round trip for every ring)
        b = make_float4(inf, inf, -inf, -inf);
        bin(whole_periods(L.nx, L.ny, !L.inflow, !L.walls, X0.x, X0.y), true);
    }
    if (lane == 0) part[warp] = b;
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < 4; w++) {
        const float4 q = part[w];
        b = make_float4(fminf(b.x, q.x), fminf(b.y, q.y), fmaxf(b.z, q.z), fmaxf(b.w, q.w));
    }
    g.box[c] = b;
    // NaN positions are passed over by fminf and fmaxf: an all-NaN ring keeps the empty box
    const bool sane = fabsf(b.x) < 1e9f && fabsf(b.y) < 1e9f && fabsf(b.z) < 1e9f && fabsf(b.w) < 1e9f;
    const double cx = sane ? 0.5 * ((double)b.x + b.z) : 0.0, cy = sane ? 0.5 * ((double)b.y + b.w) : 0.0;
    if (!sane || (double)b.z - b.x > g.cellx - g.rc || (double)b.w - b.y > g.celly - g.rc) atomicOr(status, kStatGrid);
    int ix = (int)floor(cx / g.cellx) % g.ncx;
    if (ix < 0) ix += g.ncx;
    int iy = (int)floor(cy / g.celly);
    if (L.walls) iy = iy < 0 ? 0 : (iy >= g.ncy ? g.ncy - 1 : iy);
    else {
        iy %= g.ncy;
        if (iy < 0) iy += g.ncy;
    }
    g.cellof[c] = iy * g.ncx + ix;
    const int h = bucket_of(ix, iy, g.nbuckets);
    const int k = atomicAdd(&g.count[h], 1);
    if (k < kRepSlots) g.slot[(size_t)h * kRepSlots + k] = c;
    else atomicOr(status, kStatGrid);
}

// Gap between two intervals along one axis, through the periodic images when P > 0.
__device__ __forceinline__ float gap_f(float lo0, float hi0, float lo1, float hi1, float P, float iP) {
    float d = 0.5f * ((lo0 + hi0) - (lo1 + hi1));
    d -= P * rintf(d * iP);
    return fabsf(d) - 0.5f * ((hi0 - lo0) + (hi1 - lo1));
}

__device__ __forceinline__ float abs_max(const float4& b) {
    return fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fmaxf(fabsf(b.z), fabsf(b.w)));
}

// Eq. 27 forces on the vertices of one arc of a ring: CTA blockIdx.x = c * arcs + rank
// owns the same share of capsule c's ring as in the immersed-boundary kernels. The last CTA
// to finish empties the buckets for the next step.
__global__ void __launch_bounds__(128) k_repulsion(Lat L, Nodes nd, int max_n, int arcs, RepGrid g) {
    const int c = blockIdx.x / arcs, rank = blockIdx.x - c * arcs;
    const CapsuleParams P = nd.caps[c];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool good = P.n >= 3 && P.n <= max_n;
    const int n = P.n, chunk = good ? (n + arcs - 1) / arcs : 0, v0 = rank * chunk, m = good ? min(n - v0, chunk) : 0;
    const double px = L.inflow ? 0.0 : (double)L.nx, py = L.walls ? 0.0 : (double)L.ny;
    const float pxf = (float)px, pyf = (float)py, ipx = px > 0.0 ? 1.0f / pxf : 0.0f, ipy = py > 0.0 ? 1.0f / pyf : 0.0f;
    const int cell = g.cellof[c], ix = cell % g.ncx, iy = cell / g.ncx;
    const int nxs = g.ncx < 3 ? g.ncx : 3, nys = (!L.walls && g.ncy < 3) ? g.ncy : 3;
    for (int s0 = 32 * warp; s0 < m; s0 += 128) {
        const int k = s0 + lane, v = v0 + min(k, m - 1), gi = P.off + v;
        const float2 xf = g.xf[gi];
        const double2 X = nd.X[gi];
        const float4 wb = make_float4(warp_min(xf.x), warp_min(xf.y), warp_max(xf.x), warp_max(xf.y));
        double f = 0.0;
        for (int sy = 0; sy < nys; sy++) {
            int jy = iy + sy - (nys == 3 ? 1 : 0);
            if (L.walls && (jy < 0 || jy >= g.ncy)) continue;
            if (!L.walls) jy = ((jy % g.ncy) + g.ncy) % g.ncy;
            for (int sx = 0; sx < nxs; sx++) {
                const int jx = ((ix + sx - (nxs == 3 ? 1 : 0)) % g.ncx + g.ncx) % g.ncx;
                const int h = bucket_of(jx, jy, g.nbuckets);
                const int cnt = min(g.count[h], kRepSlots);
                for (int e = 0; e < cnt; e++) {
                    const int o = g.slot[(size_t)h * kRepSlots + e];
                    if (o == c || g.cellof[o] != jy * g.ncx + jx) continue;   // self, or another cell's entry
                    const float4 ob = g.box[o];
                    // the reach covers the rounding of the float positions, periods and boxes: a
                    // test may keep a pair that the double one then drops, never the reverse
                    const float big = fmaxf(fmaxf(abs_max(wb), abs_max(ob)), fmaxf(pxf, pyf));
                    const float reach = (float)g.rc + 1e-6f + 2e-6f * big;
                    if (gap_f(wb.x, wb.z, ob.x, ob.z, pxf, ipx) >= reach ||
                        gap_f(wb.y, wb.w, ob.y, ob.w, pyf, ipy) >= reach)
                        continue;
                    const CapsuleParams Q = nd.caps[o];
                    if (Q.n < 3 || Q.n > max_n) continue;
                    const int nch = (Q.n + 31) / 32, first = first_chunk(o, Q.off);
                    for (int c0 = 0; c0 < nch; c0 += 32) {
                        bool near = false;
                        if (c0 + lane < nch) {
                            const float4 cb = g.cbox[first + c0 + lane];
                            near = gap_f(wb.x, wb.z, cb.x, cb.z, pxf, ipx) < reach &&
                                   gap_f(wb.y, wb.w, cb.y, cb.w, pyf, ipy) < reach;
                        }
                        for (unsigned hit = __ballot_sync(0xffffffffu, near); hit; hit &= hit - 1) {
                            const int w0 = 32 * (c0 + __ffs((int)hit) - 1), nw = min(32, Q.n - w0);
                            const float2 of = g.xf[Q.off + w0 + min(lane, nw - 1)];
                            unsigned cand = 0;
                            for (int j = 0; j < nw; j++) {
                                float dx = xf.x - __shfl_sync(0xffffffffu, of.x, j);
                                float dy = xf.y - __shfl_sync(0xffffffffu, of.y, j);
                                dx -= pxf * rintf(dx * ipx);
                                dy -= pyf * rintf(dy * ipy);
                                if (dx * dx + dy * dy < reach * reach) cand |= 1u << j;
                            }
                            for (cand = k < m ? cand : 0u; cand; cand &= cand - 1) {
                                const double2 Y = nd.X[Q.off + w0 + __ffs((int)cand) - 1];
                                const double dx = min_image(X.x - Y.x, px), dy = min_image(X.y - Y.y, py);
                                const double d2 = dx * dx + dy * dy;
                                if (d2 < g.rc * g.rc) f += g.coeff * rsqrt(d2 * d2 * sqrt(d2));   // coeff d^{-5/2}
                            }
                            __syncwarp();
                        }
                    }
                }
            }
        }
        if (k < m) {
            double2 F = make_double2(0.0, 0.0);
            if (f != 0.0) {
                const double2 Xl = nd.X[P.off + (v + n - 1) % n], Xr = nd.X[P.off + (v + 1) % n];
                const double ax = X.x - Xl.x, ay = X.y - Xl.y, bx = Xr.x - X.x, by = Xr.y - X.y;
                const double la = sqrt(ax * ax + ay * ay), lb = sqrt(bx * bx + by * by);
                const double nx = ay / la + by / lb, ny = -ax / la - bx / lb;
                const double ln = sqrt(nx * nx + ny * ny);
                F = make_double2(f * (-nx / ln), f * (-ny / ln));
            }
            nd.Fpp[gi] = F;
        }
    }
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&g.count[g.nbuckets], 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (last)
        for (int h = threadIdx.x; h <= g.nbuckets; h += blockDim.x) g.count[h] = 0;
}

}  // namespace

void launch_repulsion(const Lat& L, Nodes nd, int ncaps, int max_n, int arcs, RepGrid g, unsigned* status,
                      cudaStream_t s) {
    k_rep_bin<<<ncaps, 128, 0, s>>>(L, nd, max_n, g, status);
    k_repulsion<<<ncaps * arcs, 128, 0, s>>>(L, nd, max_n, arcs, g);
}

}  // namespace lbmib
