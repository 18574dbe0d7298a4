// Force and flow update of a time step.
//
// Force: J = curl b by isotropic differences on the flow lattice,
//   J = sum_i 3 w_i c_i x b(x + c_i),
// F = F_body(t) e_axis + J x (B^ext + b).
//
// Flow (single step, Sec. III.E, or the macroscopic scheme's density, Sec. V.G):
// with f~_i = f_i^eq - w_i = w_i (drho + q_i + drho q_i),
// q_i = 3 c_i.u + 4.5 (c_i.u)^2 - 1.5 u.u (squares over gamma),
//   drho* = 2 f~_0(x) - drho(x) + sum_j [ 0.5 f~_j(y) + 1.5 f~_jbar(y) ]
//   m*    = sum_j c_j [ (tau - 1) f~_j(y) - tau f~_jbar(y) ] - 2 (tau - 1) rho u(x)
//           - (tau/2) sum_j c_j [ F_j(y) + F_jbar(y) ] + F(x),   y = x + c_j
// (macroscopic: drho* = f~_0(x) + sum_j f~_jbar(y)), the GZS terms
// F_j + F_jbar = (1 - 1/2tau) w_j (-6 u.F + 18 (c_j.u)(c_j.F)).  This uses
// sum_i f_i^eq(x) = rho and sum_i c_i f_i^eq(x) = rho u, exact on the lattice.
// With a = c_j.u and E = drho + rho (4.5 a^2 - 1.5 u.u) the pair of opposite
// equilibria is w (E +- 3 rho a), so a direction adds w (2 E - 3 rho a) to drho*
// (w (E - 3 rho a) in the macroscopic scheme) and w [(2 tau - 1) 3 rho a - E + (tau/2)
// (GZS)] c_j to m*: about 12 operations from seven values of the neighbour, of which
// what does not depend on the direction (FlowVals) is formed once per node.
//
// The sums run over the planes z - 1, z, z + 1 in turn (flow_plane), so that a CTA
// can march through z with three targets' sums in registers; the gathering form
// (flow_gather: 2-D, batched planes) adds in the same order.  Every rounding is
// spelled out: the two forms agree to the bit.  The node's own part of m*, its largest
// term, is added last, so that the others' sum is not rounded at its size.  For the same
// reason the z momentum that plane z - 1 hands to drho* and plane z + 1 takes back, half of
// rho u_z, stays out of both: each direction's part counts from that of the node below
// (ref; the weights cancel it).  FP32, one step against binary64: rms error of drho 0.4 of
// what the sum with opposite directions side by side has, 1.5 with the planes' parts whole
// (macroscopic scheme 0.7 and 2.5).
#pragma once

#include "qslbm_kernels.cuh"

namespace qslbm {

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }

// Weight of a direction with |c| nonzero components c0.
template <int Q>
__device__ __forceinline__ constexpr double flow_weight(int nonzero) {
    if (Q == 27) return nonzero == 0 ? 8.0 / 27.0 : (nonzero == 1 ? 2.0 / 27.0 : (nonzero == 2 ? 1.0 / 54.0 : 1.0 / 216.0));
    if (Q == 19) return nonzero == 0 ? 1.0 / 3.0 : (nonzero == 1 ? 1.0 / 18.0 : (nonzero == 2 ? 1.0 / 36.0 : 0.0));
    return nonzero == 0 ? 4.0 / 9.0 : (nonzero == 1 ? 1.0 / 9.0 : (nonzero == 2 ? 1.0 / 36.0 : 0.0));
}

// The in-plane neighbours in the order of the sums: the node itself, the axes, the
// diagonals.
__device__ __forceinline__ constexpr int flow_px(int i) {
    return i == 1 || i == 5 || i == 8 ? -1 : (i == 2 || i == 6 || i == 7 ? 1 : 0);
}
__device__ __forceinline__ constexpr int flow_py(int i) {
    return i == 3 || i == 5 || i == 7 ? -1 : (i == 4 || i == 6 || i == 8 ? 1 : 0);
}

// c . v, one rounding (c of at most three nonzero components: two).
template <typename T>
__device__ __forceinline__ T flow_dot(int cx, int cy, int cz, T x, T y, T z) {
    T a = T(0);
    bool any = false;
    if (cx) a = cx > 0 ? x : -x, any = true;
    if (cy) a = any ? add_rn(a, cy > 0 ? y : -y) : (cy > 0 ? y : -y), any = true;
    if (cz) a = any ? add_rn(a, cz > 0 ? z : -z) : (cz > 0 ? z : -z);
    return a;
}

template <typename T>
struct FlowConst {
    T kappa, h, kf6, kf18, ig05, ig15, ig, two_tm1;
    int mac;
    __device__ __forceinline__ explicit FlowConst(const FlowCoef<T>& c) {
        const T kf = T(0.5) * c.tau * c.kforce * c.ig2;
        kappa = c.mac ? T(1) : T(2);
        h = T(2) * c.tau - T(1);
        kf6 = T(6) * kf;
        kf18 = T(18) * kf;
        ig05 = T(0.5) * c.ig;
        ig15 = T(1.5) * c.ig;
        ig = c.ig;
        two_tm1 = T(2) * (c.tau - T(1));
        mac = c.mac;
    }
};

// What a node gives to its neighbours' sums: u, F scaled by 9 tau (1 - 1/2tau)
// / gamma^2, K = drho - 1.5 rho u.u / gamma, M = 3 tau (1 - 1/2tau) u.F / gamma^2 - K,
// 3 rho.
template <typename T>
struct FlowVals {
    T u[3], f[3], K, M, r3;
};
template <typename T>
__device__ __forceinline__ FlowVals<T> flow_vals(T dr, const T u[3], const T F[3], const FlowConst<T>& c) {
    FlowVals<T> v;
    const T uu = fma_rn(u[2], u[2], fma_rn(u[1], u[1], mul_rn(u[0], u[0])));
    const T uF = fma_rn(u[2], F[2], fma_rn(u[1], F[1], mul_rn(u[0], F[0])));
    v.r3 = fma_rn(T(3), dr, T(3));
    v.K = fma_rn(-mul_rn(c.ig05, v.r3), uu, dr);
    v.M = fma_rn(c.kf6, uF, -v.K);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        v.u[a] = u[a];
        v.f[a] = mul_rn(c.kf18, F[a]);
    }
    return v;
}

// 3 rho u_z of a node, the reference of the target above it.
template <typename T>
__device__ __forceinline__ T flow_ref(const FlowVals<T>& v) {
    return mul_rn(v.r3, v.u[2]);
}

// s = (drho*, m*): the neighbour at x + (cx, cy, cz), whose values are v; ref: the
// target's reference.
template <typename T, int Q>
__device__ __forceinline__ void flow_add(T s[4], int cx, int cy, int cz, const FlowVals<T>& v, T ref,
                                         const FlowConst<T>& c) {
    const T w = (T)flow_weight<Q>((cx != 0) + (cy != 0) + (cz != 0));
    const T a = flow_dot<T>(cx, cy, cz, v.u[0], v.u[1], v.u[2]);
    const T cf = flow_dot<T>(cx, cy, cz, v.f[0], v.f[1], v.f[2]);
    const T t = mul_rn(mul_rn(c.ig15, v.r3), a);
    const T p = mul_rn(v.r3, a);
    const T E = fma_rn(t, a, v.K);
    const T g = fma_rn(c.h, p, fma_rn(-a, add_rn(t, cf), v.M));
    const T q = cz == 0 ? p : add_rn(p, cz > 0 ? -ref : ref);
    s[0] = fma_rn(w, fma_rn(c.kappa, E, -q), s[0]);
    if (cx) s[1] = fma_rn(cx > 0 ? w : -w, g, s[1]);
    if (cy) s[2] = fma_rn(cy > 0 ? w : -w, g, s[2]);
    if (cz) s[3] = fma_rn(cz > 0 ? w : -w, g, s[3]);
}
// The node itself: its own values v and (drho, u, F); own: its part of m*.
template <typename T, int Q>
__device__ __forceinline__ void flow_own(T s[4], T own[3], const FlowVals<T>& v, T dr, const T F[3],
                                         const FlowConst<T>& c) {
    const T w0 = (T)flow_weight<Q>(0);
    s[0] = fma_rn(c.kappa * w0, v.K, s[0]);
    if (!c.mac) s[0] = add_rn(s[0], -dr);
    const T k = mul_rn(c.two_tm1, add_rn(T(1), dr));
#pragma unroll
    for (int a = 0; a < 3; ++a) own[a] = fma_rn(c.ig, F[a], -mul_rn(k, v.u[a]));
}
// Neighbour i of a plane (its place in-plane: flow_px, flow_py), for the target in
// the plane above it (cz = -1), its own (0), below it (+1).
template <typename T, int Q>
__device__ __forceinline__ void flow_place(T s[4], T own[3], int i, int cz, const FlowVals<T>& v, T ref, T dr,
                                           const T F[3], const FlowConst<T>& c) {
    const int cx = flow_px(i), cy = flow_py(i);
    if (i == 0 && cz == 0)
        flow_own<T, Q>(s, own, v, dr, F, c);
    else if (flow_weight<Q>((cx != 0) + (cy != 0) + (cz != 0)) != 0.0)
        flow_add<T, Q>(s, cx, cy, cz, v, ref, c);
}

// The update of one node, gathered from its neighbours.
template <typename T, int DIM, int Q>
__device__ __forceinline__ void flow_gather(const T* __restrict__ drho, const T* __restrict__ u,
                                            const T* __restrict__ F, T* __restrict__ drho_out, T* uout, long long n,
                                            int nx, int ny, int nz, int x, int y, int z, long long k,
                                            const FlowConst<T>& c) {
    T s[4] = {T(0), T(0), T(0), T(0)}, own[3] = {T(0), T(0), T(0)}, ref = T(0);
#pragma unroll
    for (int cz = (DIM == 3 ? -1 : 0); cz <= (DIM == 3 ? 1 : 0); ++cz)
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int cx = flow_px(i), cy = flow_py(i);
            if (flow_weight<Q>((cx != 0) + (cy != 0) + (cz != 0)) != 0.0) {
                const int q = (wrapi(z + cz, nz) * ny + wrapi(y + cy, ny)) * nx + wrapi(x + cx, nx);
                const T uq[3] = {u[q], u[q + n], u[q + 2 * n]};
                const T Fq[3] = {F[q], F[q + n], F[q + 2 * n]};
                const T dr = drho[q];
                const FlowVals<T> v = flow_vals<T>(dr, uq, Fq, c);
                if (cz == -1 && i == 0) ref = flow_ref(v);  // (the first neighbour of the sum)
                flow_place<T, Q>(s, own, i, cz, v, ref, dr, Fq, c);
            }
        }
    const T inv = T(1) / add_rn(T(1), s[0]);
    drho_out[k] = s[0];
#pragma unroll
    for (int a = 0; a < 3; ++a) uout[k + a * n] = mul_rn(add_rn(s[1 + a], own[a]), inv);
}

// J += 3 w c x b for neighbour i of a plane.
template <typename T, int Q>
__device__ __forceinline__ void curl_place(T J[3], int i, int cz, const T b[3]) {
    const int cx = flow_px(i), cy = flow_py(i);
    const double wd = 3.0 * flow_weight<Q>((cx != 0) + (cy != 0) + (cz != 0));
    if (wd == 0.0) return;
    const T w = (T)wd;
    const int c[3] = {cx, cy, cz};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int p = (a + 1) % 3, q = (a + 2) % 3;
        if (c[p]) J[a] = fma_rn(c[p] > 0 ? w : -w, b[q], J[a]);
        if (c[q]) J[a] = fma_rn(c[q] > 0 ? -w : w, b[p], J[a]);
    }
}

template <typename T>
__device__ __forceinline__ T body_force_at(const ForceCoef<T>& c, long long t) {
    const double fb_d = c.amp != 0.0 ? c.F0 * (1.0 + c.amp * sin(c.omega * (double)t)) : c.F0;
    return (T)fb_d;
}

// F of in-plane node p of plane z from J and b there.
template <typename T>
__device__ __forceinline__ void force_write(T* __restrict__ F, long long n, int P, int z, int p, const T J[3],
                                            const T b[3], const ForceCoef<T>& c, T fb) {
    T Be[3];
    bext_at(c.bext_z, c.be, z, Be);
    bext_add_xy(c.bext_xy, P, p, Be);
    const T B[3] = {add_rn(Be[0], b[0]), add_rn(Be[1], b[1]), add_rn(Be[2], b[2])};
    T L[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int p1 = (a + 1) % 3, p2 = (a + 2) % 3;
        L[a] = fma_rn(J[p1], B[p2], -mul_rn(J[p2], B[p1]));
        if (c.axis == a) L[a] = add_rn(L[a], fb);
        F[(long long)z * P + p + a * n] = L[a];
    }
}

template <typename T, int DIM, int Q>
__device__ __forceinline__ void force_gather(const T* __restrict__ b, T* __restrict__ F, long long n, int nx, int ny,
                                             int nz, int x, int y, int z, const ForceCoef<T>& c, T fb) {
    T J[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int cz = (DIM == 3 ? -1 : 0); cz <= (DIM == 3 ? 1 : 0); ++cz)
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int cx = flow_px(i), cy = flow_py(i);
            if ((i > 0 || cz != 0) && flow_weight<Q>((cx != 0) + (cy != 0) + (cz != 0)) != 0.0) {
                const int q = (wrapi(z + cz, nz) * ny + wrapi(y + cy, ny)) * nx + wrapi(x + cx, nx);
                const T bq[3] = {b[q], b[q + n], b[q + 2 * n]};
                curl_place<T, Q>(J, i, cz, bq);
            }
        }
    const int p = y * nx + x;
    const long long k = (long long)z * nx * ny + p;
    const T bk[3] = {b[k], b[k + n], b[k + 2 * n]};
    force_write<T>(F, n, nx * ny, z, p, J, bk, c, fb);
}

// Node-parallel forms (2-D): enough CTAs for a plane of a few thousand nodes.  One
// CTA for the whole plane, as the 3-D planes have it in a batch, left the 64x32 FP64
// channel with one SM's FP64 rate: force, flow and the IB on u 265 us a step, now 9.5.
constexpr int kFlowNodeThreads = 64;
template <typename T, int Q>
__global__ void __launch_bounds__(kFlowNodeThreads) k_force_nodes(Geo g, const T* __restrict__ b, T* __restrict__ F,
                                                                  ForceCoef<T> c, const long long* __restrict__ tstep) {
    const int p = blockIdx.x * kFlowNodeThreads + threadIdx.x;
    if (p >= g.nx * g.ny) return;
    force_gather<T, 2, Q>(b, F, g.n, g.nx, g.ny, 1, p % g.nx, p / g.nx, 0, c, body_force_at(c, *tstep));
}
template <typename T, int Q>
__global__ void __launch_bounds__(kFlowNodeThreads) k_flow_nodes(Geo g, const T* __restrict__ drho,
                                                                 const T* __restrict__ u, const T* __restrict__ F,
                                                                 T* __restrict__ drho_out, T* uout, FlowCoef<T> c,
                                                                 long long* tstep) {
    const int p = blockIdx.x * kFlowNodeThreads + threadIdx.x;
    if (p == 0) *tstep += 1;
    if (p >= g.nx * g.ny) return;
    flow_gather<T, 2, Q>(drho, u, F, drho_out, uout, g.n, g.nx, g.ny, 1, p % g.nx, p / g.nx, 0, p, FlowConst<T>(c));
}

// Marching forms (3-D): a CTA owns a tile of 32 x TY columns and walks a chunk of z
// planes.  A plane's values are staged once in shared memory (double buffered, one
// barrier a plane; loads one plane ahead), every neighbour of it is read once and
// added to the three targets above, in and below the plane, whose sums a thread
// keeps in registers: 56 shared-memory reads a node where the gathering form makes
// 126 loads through L1, and a third of its arithmetic.  Force, flow and the IB on u
// of a step, with one CTA per plane gathering from L1 / now: 96x96x512 289 / 131 us
// (the fields alone are 320 MB, 47 us at the measured copy rate), 40x40x192 51 / 22,
// 64x64x128 42 / 26, in FP64 about 760 / 200.  On small domains, where a step of few
// sweeps is a handful of launches, force, flow and the IB on u each start as the kernel
// before them ends (early): 16^3 at one sweep 18.9 us a step without, 16.9 with, 24x24x96
// at four 32.8 and 31.2.
constexpr int kFlowTX = 32;
template <typename T>
constexpr int kFlowTY = sizeof(T) == 4 ? 8 : 4;  // (the staged planes fit static shared memory)
template <typename T>
constexpr int kFlowThreads = kFlowTX * kFlowTY<T>;

// The tile and z chunk of this CTA: one grid dimension counts them all (tiles along x,
// then y, then chunks), since the other two hold 65535 CTAs and a long thin domain has
// more rows or planes than that many tiles.
struct FlowTile {
    int x0, y0, z0, z1;
};
template <typename T>
__device__ __forceinline__ FlowTile flow_tile(int nx, int ny, int nz, int chunk) {
    const unsigned tx = (unsigned)(nx + kFlowTX - 1) / kFlowTX, ty = (unsigned)(ny + kFlowTY<T> - 1) / kFlowTY<T>;
    const unsigned row = blockIdx.x / tx, layer = row / ty;
    const int z0 = (int)layer * chunk;
    return {(int)(blockIdx.x - row * tx) * kFlowTX, (int)(row - layer * ty) * kFlowTY<T>, z0, min(z0 + chunk, nz)};
}

// Halo cell h of a tile: rows above and below (with the corners), columns left and
// right.  cell: its offset in a staged plane; node: in-plane index (periodic image).
template <int TY>
__device__ __forceinline__ void flow_halo(int h, int x0, int y0, int nx, int ny, int& cell, int& node) {
    constexpr int W = kFlowTX + 2;
    int r, c;
    if (h < 2 * W) {
        r = h < W ? 0 : TY + 1;
        c = h < W ? h : h - W;
    } else {
        const int j = h - 2 * W;
        r = 1 + (j >> 1);
        c = (j & 1) ? kFlowTX + 1 : 0;
    }
    cell = r * W + c;
    node = ((y0 + r - 1 + ny) % ny) * nx + (x0 + c - 1 + nx) % nx;
}

template <typename T, int Q>
__global__ void __launch_bounds__(kFlowThreads<T>) k_force_march(Geo g, const T* __restrict__ b, T* __restrict__ F,
                                                                 ForceCoef<T> c, const long long* __restrict__ tstep,
                                                                 int chunk, bool early) {
    if (early) pdl_trigger();
    pdl_wait();
    constexpr int TY = kFlowTY<T>, W = kFlowTX + 2, CELLS = W * (TY + 2), HALO = 2 * W + 2 * TY;
    __shared__ T sm[2][3][CELLS];
    static_assert(HALO <= kFlowThreads<T>, "one halo cell a thread");
    const int nx = g.nx, ny = g.ny, nz = g.nz, P = nx * ny;
    const int n = (int)g.n;
    const int tx = threadIdx.x % kFlowTX, ty = threadIdx.x / kFlowTX;
    const FlowTile ft = flow_tile<T>(nx, ny, nz, chunk);
    const int x0 = ft.x0, y0 = ft.y0, z0 = ft.z0, z1 = ft.z1, x = x0 + tx, y = y0 + ty;
    const bool active = x < nx && y < ny;
    const int p = (y % ny) * nx + x % nx;
    const int cell = (ty + 1) * W + tx + 1;
    int hcell = -1, hp = 0;
    if (threadIdx.x < HALO) flow_halo<TY>(threadIdx.x, x0, y0, nx, ny, hcell, hp);
    const T fb = body_force_at(c, *tstep);
    T cur[3], halo[3] = {}, last[3] = {};
    T Jm[3] = {}, J0[3] = {}, Jp[3] = {};
    auto load = [&](int z, int q, T v[3]) {
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = b[z * P + q + a * n];
    };
    int zz = z0 == 0 ? nz - 1 : z0 - 1;  // the plane at hand (periodic image)
    load(zz, p, cur);
    if (hcell >= 0) load(zz, hp, halo);
    for (int s = z0 - 1; s <= z1; ++s) {
        T(*t)[CELLS] = sm[s & 1];
#pragma unroll
        for (int a = 0; a < 3; ++a) t[a][cell] = cur[a];
        if (hcell >= 0)
#pragma unroll
            for (int a = 0; a < 3; ++a) t[a][hcell] = halo[a];
        const T own[3] = {cur[0], cur[1], cur[2]};
        const int zn = wrap_inc(zz, nz);
        if (s < z1) {
            load(zn, p, cur);
            if (hcell >= 0) load(zn, hp, halo);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int o = cell + flow_py(i) * W + flow_px(i);
            const T v[3] = {t[0][o], t[1][o], t[2][o]};
            if (s > z0) curl_place<T, Q>(Jm, i, 1, v);
            if (s >= z0 && s < z1 && i > 0) curl_place<T, Q>(J0, i, 0, v);
            if (s < z1 - 1) curl_place<T, Q>(Jp, i, -1, v);
        }
        if (s > z0 && active) force_write<T>(F, n, P, s - 1, p, Jm, last, c, fb);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            Jm[a] = J0[a];
            J0[a] = Jp[a];
            Jp[a] = T(0);
            last[a] = own[a];
        }
        zz = zn;
    }
}

template <typename T, int Q>
__global__ void __launch_bounds__(kFlowThreads<T>) k_flow_march(Geo g, const T* __restrict__ drho,
                                                                const T* __restrict__ u, const T* __restrict__ F,
                                                                T* __restrict__ drho_out, T* uout, FlowCoef<T> fc,
                                                                long long* tstep, int chunk, bool early) {
    if (early) pdl_trigger();
    pdl_wait();
    constexpr int TY = kFlowTY<T>, W = kFlowTX + 2, CELLS = W * (TY + 2), HALO = 2 * W + 2 * TY;
    __shared__ T sm[2][9][CELLS];
    const int nx = g.nx, ny = g.ny, nz = g.nz, P = nx * ny;
    const int n = (int)g.n;
    const FlowConst<T> c(fc);
    const int tx = threadIdx.x % kFlowTX, ty = threadIdx.x / kFlowTX;
    const FlowTile ft = flow_tile<T>(nx, ny, nz, chunk);
    const int x0 = ft.x0, y0 = ft.y0, z0 = ft.z0, z1 = ft.z1, x = x0 + tx, y = y0 + ty;
    const bool active = x < nx && y < ny;
    const int p = (y % ny) * nx + x % nx;
    const int cell = (ty + 1) * W + tx + 1;
    int hcell = -1, hp = 0;
    if (threadIdx.x < HALO) flow_halo<TY>(threadIdx.x, x0, y0, nx, ny, hcell, hp);
    T cur[7], halo[7] = {};  // drho, u, F
    T sM[4] = {}, s0[4] = {}, sP[4] = {}, oM[3] = {}, o0[3] = {};  // the targets' sums and own parts
    T rM = T(0), r0 = T(0);                                        // their references
    auto load = [&](int z, int q, T v[7]) {
        const int k = z * P + q;
        v[0] = drho[k];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            v[1 + a] = u[k + a * n];
            v[4 + a] = F[k + a * n];
        }
    };
    auto stage = [&](T(*t)[CELLS], int at, const FlowVals<T>& v) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            t[a][at] = v.u[a];
            t[3 + a][at] = v.f[a];
        }
        t[6][at] = v.K;
        t[7][at] = v.M;
        t[8][at] = v.r3;
    };
    int zz = z0 == 0 ? nz - 1 : z0 - 1;  // the plane at hand (periodic image)
    load(zz, p, cur);
    if (hcell >= 0) load(zz, hp, halo);
    for (int s = z0 - 1; s <= z1; ++s) {
        T(*t)[CELLS] = sm[s & 1];
        const FlowVals<T> own = flow_vals<T>(cur[0], cur + 1, cur + 4, c);
        stage(t, cell, own);
        if (hcell >= 0) stage(t, hcell, flow_vals<T>(halo[0], halo + 1, halo + 4, c));
        const T dr = cur[0], Fk[3] = {cur[4], cur[5], cur[6]}, rP = flow_ref(own);
        const int zn = wrap_inc(zz, nz);
        if (s < z1) {
            load(zn, p, cur);
            if (hcell >= 0) load(zn, hp, halo);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            FlowVals<T> v = own;
            if (i > 0) {
                const int o = cell + flow_py(i) * W + flow_px(i);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    v.u[a] = t[a][o];
                    v.f[a] = t[3 + a][o];
                }
                v.K = t[6][o];
                v.M = t[7][o];
                v.r3 = t[8][o];
            }
            if (s > z0) flow_place<T, Q>(sM, oM, i, 1, v, rM, dr, Fk, c);
            if (s >= z0 && s < z1) flow_place<T, Q>(s0, o0, i, 0, v, r0, dr, Fk, c);
            if (s < z1 - 1) flow_place<T, Q>(sP, o0, i, -1, v, rP, dr, Fk, c);
        }
        if (s > z0 && active) {
            const int k = (s - 1) * P + p;
            const T inv = T(1) / add_rn(T(1), sM[0]);
            drho_out[k] = sM[0];
#pragma unroll
            for (int a = 0; a < 3; ++a) uout[k + a * n] = mul_rn(add_rn(sM[1 + a], oM[a]), inv);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            sM[a] = s0[a];
            s0[a] = sP[a];
            sP[a] = T(0);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) oM[a] = o0[a];
        rM = r0;
        r0 = rP;
        zz = zn;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *tstep += 1;
}

}  // namespace qslbm
