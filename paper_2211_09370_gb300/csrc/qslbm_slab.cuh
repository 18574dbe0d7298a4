// Resident magnetic sub-iteration of a single FP32 handle: one cooperative
// launch runs all N_mag sweeps (Sec. V.G) with the IB on b after each (Sec. V.D,
// V.F); each CTA holds a slab of G consecutive z planes on chip for the whole
// launch.
//
// What bounds it: for small slabs the latency of a sweep's phases and of handing
// the end planes to the neighbouring CTAs; for large ones shared-memory
// wavefronts (about 2.4 a node and sweep) and the sectors written to the
// exchange (one a clock per SM).  Hence:
//  - (b, u) per node in shared memory, packed FP32 arithmetic on x-adjacent node
//    pairs (one instruction for two nodes).  A component's even and odd columns
//    are separate halves: a warp's accesses to either node of its pairs and to
//    their x neighbours are consecutive words (pairs stored side by side made
//    every x neighbour a two-way bank conflict).  The strides between halves and
//    components are compile-time constants, immediates of one address.
//  - A thread owns K consecutive rows of one pair column for the whole launch
//    and slides a window of rows through registers, so that the rows above and
//    below are read once per K rows; its new values wait in registers until
//    every thread has read the old ones (no second buffer: 24 B a node).
//  - Slabs of up to two rows per thread hand their end planes over as 16-byte
//    messages that hold three values and the sweep's sequence number, and poll
//    the messages themselves: a fence, a flag and a second round trip per sweep
//    are gone, and nodes off the wall shell go out before the IB.  (40x40x150:
//    4.2 us a sweep against 6.5 with counters.)  A message holds the node's
//    complete share of the neighbour's update.  Larger slabs, whose messages
//    would saturate the writes, publish b with bulk copies and a counter.
//  - The applied field's flux does not change during the sweeps: its share S of
//    the update is formed once, from differences of u and B^ext, and a sweep
//    forms only that of b.  The large terms u B^ext are not rounded every sweep.
//
// Per sweep:
//   1. new b of the own nodes into registers, from shared memory and, for the
//      end planes, the neighbours' exchange                           | barrier
//   2. b of the own nodes to shared memory (messages: end-plane nodes off the
//      shell to the neighbours)                                       | barrier
//   3. IB: delta_j = -s_j D b* of every (plane, marker, component)    | barrier
//   4. IB: b = b* + D^T delta on the shell (messages: end-plane shell nodes to
//      the neighbours)                                                | barrier
// A slot of the exchange is written again two sweeps later: by then its writer
// has received the neighbour's data of the sweep between, which the neighbour
// sent after the barrier that ends its reads.
//
// Measured, us per sweep with the IB, this kernel against the other route there:
// 24x24x96 2.0 / 3.6 (one plane per CTA, k_sweeps_resident); against the marching pair
// sweep and its IB launches 24x24x300 2.9 / 6.5, 40x40x192 7.6 / 9.3, 57x57x304 16.5 /
// 17.8, 61x61x120 9.2 / 11.0, 64x64x128 with an in-plane field 7.1 / 12.7.
#pragma once

#include "qslbm_kernels.cuh"
#include "qslbm_resident.cuh"

namespace qslbm {

constexpr int kSlabThreads = 768;
// end planes travel as messages up to this many rows per thread (57x56x150, three
// rows: 7.6 us a sweep with messages, 7.1 with counters)
constexpr int kSlabMsgK = 2;
constexpr int kSlabMaxK = 5;  // rows per thread, at most (5 rows x 2 nodes x 768 threads = 7680 nodes a CTA)

// Rows per thread for a slab of G planes: the fewest at which the slab's pair
// columns fit the CTA's threads; 0 when none does.
__host__ __device__ inline int slab_rows(int nx, int ny, int G) {
    for (int K = 1; K <= kSlabMaxK; ++K)
        if ((long long)G * ((nx + 1) / 2) * ((ny + K - 1) / K) <= kSlabThreads) return K;
    return 0;
}
// Floats between a component's even and odd columns, and between components: a
// node of every thread's rows (and, for up to two rows, a quarter more, room for
// padded rows), then half a row of banks, and eight banks between components, so
// that neighbouring columns, and one node's components, fall into different banks.
__host__ __device__ constexpr int slab_half(int K) { return (K <= 2 ? kSlabThreads * 5 / 4 : kSlabThreads) * K + 48; }
__host__ __device__ constexpr int slab_stride(int K) { return 2 * slab_half(K) + 8; }
__host__ __device__ inline int slab_pairs(int nx) { return (nx + 1) / 2; }
// Pairs between rows: padded, when the slab has room, so that the block of rows
// K further continues the banks where a row ends (lanes of one warp cover
// several such blocks; without, 36x36x300 took 7.3 us a sweep, with it 5.7).
__host__ __device__ inline int slab_row_stride(int nx, int ny, int G, int K) {
    const int XP = slab_pairs(nx);
    for (int q = XP; q < XP + 32 && G * ((ny * q + 3) / 4 * 4) <= slab_half(K) - 48; ++q)
        if ((K * q - XP) % 32 == 0) return q;
    return XP;
}
// Floats between planes in a half: a multiple of four (16-byte bulk copies).
__host__ __device__ inline int slab_plane_stride(int nx, int ny, int G, int K) {
    return (ny * slab_row_stride(nx, ny, G, K) + 3) / 4 * 4;
}
// S is kept in shared memory for up to three rows per thread (36 B a node of at
// most 4608); beyond, it is read from L2.
__host__ __device__ inline bool slab_third(int K) { return K <= 3; }
// Messages of one direction and parity (a plane's even, then odd columns), and
// the floats of one CTA's exchange, 2 directions x 2 parities, of 16-byte
// messages or of a plane's b.
__host__ __device__ inline int slab_msgs(int nx, int ny) { return 2 * ny * slab_pairs(nx); }
__host__ __device__ inline int slab_dir_floats(int nx, int ny, int G, int K) {
    const int a = 8 * slab_msgs(nx, ny), b = 12 * slab_plane_stride(nx, ny, G, K);
    return ((a > b ? a : b) + 3) / 4 * 4;
}
inline long long slab_msg_floats(int nx, int ny, int G, int K) { return 2LL * slab_dir_floats(nx, ny, G, K); }

// One CTA's slab, in shared memory: the phases of a sweep read what they need
// of it as they begin.  (Held in registers over the whole loop, its pointers and
// strides spilled to local memory, and the L1 that the shared memory leaves is
// too small to hold spills: 12.7 against 7.1 us per sweep on 64x64x128.)
struct SlabJob {
    int nx, ny, nz, n;   // the instance's box
    int z0, G;           // planes z0 .. z0 + G - 1
    int nsweeps;
    int whole;           // the slab holds every plane: no exchange
    int zm, zp;          // the planes below and above it
    const float* b_in;
    float* b_out;
    const float* u;
    float* S;            // [3][n] scratch for S (slab_direct, more than three rows per thread)
    int more;            // list entries past a shell node's fourth, all of a plane (slab_direct)
    float *up, *down;    // own end planes for the next / previous slab: [parity][4 slab_msgs]
    const float *from_prev, *from_next;
    unsigned *count;     // end planes published so far
    const unsigned *count_prev, *count_next;
    int* err;            // set to 1 when a wait gives up
    // derived by slab_job_init
    int P, XP, XPS, PS, MS, MH;  // nodes of a plane, pairs of a row, strides (in shared memory, of messages)
    int XS;                      // floats of one half of a component of a plane in the exchange
    int R, S_;                   // markers and shell nodes of a ring
    unsigned mR, mS, base;
    float w0, w1, w1k, sq;
    float be[3];
    const float *bext_z, *bext_xy;
};
__device__ __forceinline__ float2 slab_mul(float2 a, float2 b) { return mul2(a, b); }
__device__ __forceinline__ float2 slab_sub(float2 a, float2 b) { return sub2(a, b); }
__device__ __forceinline__ float2 slab_fma(float2 a, float2 b, float2 c) { return fma2(a, b, c); }
__device__ __forceinline__ float slab_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float slab_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float slab_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
// c - a b
__device__ __forceinline__ float2 nfma2(float2 a, float2 b, float2 c) { return __ffma2_rn(f2(-a.x, -a.y), b, c); }

// bytes (a multiple of 16) of shared memory to global memory, both 16-byte
// aligned, by the bulk copy engine.
__device__ __forceinline__ void slab_bulk_store(float* dst, const float* src, unsigned bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
                 "r"((unsigned)__cvta_generic_to_shared(src)), "r"(bytes)
                 : "memory");
}

// Thread 0: what follows from the slab's own fields, its coefficients and tables.
__device__ __forceinline__ void slab_job_init(SlabJob& J, const SweepCoef<float>& c, const IBView<float>& ib, int K, int Gmax) {
    J.zm = J.z0 == 0 ? J.nz - 1 : J.z0 - 1;
    J.zp = J.z0 + J.G == J.nz ? 0 : J.z0 + J.G;
    J.P = J.nx * J.ny;
    J.XP = slab_pairs(J.nx);
    J.XPS = slab_row_stride(J.nx, J.ny, Gmax, K);
    J.PS = J.XS = slab_plane_stride(J.nx, J.ny, Gmax, K);
    J.MS = slab_msgs(J.nx, J.ny);
    J.MH = J.MS / 2;
    J.R = ib.ring_off[1] - ib.ring_off[0];
    J.S_ = ib.shell_off[1] - ib.shell_off[0];
    J.mR = magic_of((unsigned)J.R);
    J.mS = magic_of((unsigned)J.S_);
    J.base = *J.count;
    J.w0 = c.w0;
    J.w1 = c.w1;
    J.w1k = c.w1 * c.kappa;
    J.sq = c.sq;
    for (int a = 0; a < 3; ++a) J.be[a] = c.be[a];
    J.bext_z = c.bext_z;
    J.bext_xy = c.bext_xy;
}
// B^ext of plane row t of a slab (0: the plane below, G + 1: the one above), component a.
__device__ __forceinline__ float slab_bext(const SlabJob& J, int t, int a) {
    const int G = J.G, z = t == 0 ? J.zm : (t == G + 1 ? J.zp : J.z0 + t - 1);
    const float* bz = J.bext_z;
    return bz ? bz[3 * z + a] : J.be[a];
}

// Shared memory in bytes of a single handle's slab: b, w1 kappa u, S (slab_third)
// and the IB tables.
inline size_t slab_direct_smem_bytes(int nx, int ny, int G, int R, int S, int more) {
    const int K = slab_rows(nx, ny, G);
    size_t b = (size_t)slab_stride(K) * 4 * (slab_third(K) ? 9 : 6);
    b += (size_t)32 * S + (size_t)16 * G * R + (size_t)60 * R + (size_t)8 * more;
    return (b + 15) / 16 * 16;
}

// A node's share in the update of its z neighbours, from its b and v = w1 kappa
// u: w1 b + Phi for the node above it (up), w1 b - Phi for the one below.
template <bool UP, typename V>
__device__ __forceinline__ void z_share(V o[3], V w1, const V b[3], const V v[3]) {
    const V p0 = slab_mul(v[2], b[0]), q0 = slab_mul(v[0], b[2]), p1 = slab_mul(v[2], b[1]), q1 = slab_mul(v[1], b[2]);
    o[0] = slab_fma(w1, b[0], UP ? slab_sub(p0, q0) : slab_sub(q0, p0));
    o[1] = slab_fma(w1, b[1], UP ? slab_sub(p1, q1) : slab_sub(q1, p1));
    o[2] = slab_mul(w1, b[2]);
}

// The sweeps of a single handle.  The flux of b is formed from the neighbours'
// (b, u) as it is used (u scaled by w1 kappa once), without e in shared memory:
// more operations, but nothing to store or redo besides b, and less rounding;
// the applied field's share S comes in as the start of the sum.
template <int K>
__device__ __forceinline__ void slab_direct(const SlabJob& J, const IBView<float>& ib, unsigned char* smem, int* s_abort,
                                            int* s_more) {
    constexpr bool SSH = K <= 3;  // S in shared memory, else in global memory
    constexpr bool MSG = K <= kSlabMsgK;  // end planes as messages, else published by counters
    constexpr int HS = slab_half(K), CS = slab_stride(K);
    const int tid = threadIdx.x, NT = blockDim.x;
    float* const sb = reinterpret_cast<float*>(smem);  // [3][CS] b
    float* const su = sb + 3 * CS;                     // [3][CS] w1 kappa u
    float* const sS = su + 3 * CS;                     // [3][CS] S (SSH)
    // IB tables, from plane 0's: per shell node the first four list weights and
    // a record (markers 0 | 1 << 16, 2 | 3 << 16, offset | exchange place << 16,
    // first further entry | count << 16); deltas [G][R]; per marker ten floats
    // (nine weights, the scaling); further list entries (weight, marker); per
    // marker ten 16-bit support offsets
    auto t_sw = [&] { return reinterpret_cast<float4*>(SSH ? sS + 3 * CS : sS); };
    auto t_sm = [&] { return reinterpret_cast<uint4*>(t_sw() + J.S_); };
    auto t_d = [&] { return reinterpret_cast<float4*>(t_sm() + J.S_); };
    auto t_w = [&] { return reinterpret_cast<float2*>(t_d() + J.G * J.R); };
    auto t_more = [&] { return reinterpret_cast<uint2*>(t_w() + 5 * J.R); };
    auto t_q = [&] { return reinterpret_cast<unsigned*>(t_more() + J.more); };

    int xp, y0, g, gp, dl, dr, rows;
    bool two, mm, mp;  // the pair has a second node; z - 1 / z + 1 are in another CTA
    unsigned first_bits = 0, send_bits;  // the own nodes; those that go out before the IB
    {
        const int nx = J.nx, ny = J.ny, P = J.P, XP = J.XP, XPS = J.XPS, PS = J.PS, R = J.R, S = J.S_, G = J.G;
        const int MH = J.MH, n = J.n, z0 = J.z0, nz = J.nz;
        const int m0 = ib.ring_off[0], s0 = ib.shell_off[0];
        const float w1k_all = J.w1k, w1k = J.sq == 0.f ? 0.f : w1k_all;  // strict QS: the flux has no b part
        const float *b_in = J.b_in, *u = J.u;
        auto at = [&](int x, int y) { return (x & 1) * HS + y * XPS + (x >> 1); };
        // ---- tables
        float2* tw = t_w();
        unsigned* tq = t_q();
        float4* tsw = t_sw();
        uint4* tsm = t_sm();
        uint2* more = t_more();
        for (int i = tid; i < R; i += NT) {
            float w[10];
            unsigned q[10];
#pragma unroll
            for (int j = 0; j < 9; ++j) {
                w[j] = ib.mk_w[9 * (m0 + i) + j];
                const int p = ib.mk_q[9 * (m0 + i) + j], y = p / nx;
                q[j] = (unsigned)at(p - y * nx, y);
            }
            w[9] = ib.mk_s[m0 + i];
            q[9] = 0;
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                tw[5 * i + j] = f2(w[2 * j], w[2 * j + 1]);
                tq[5 * i + j] = q[2 * j] | (q[2 * j + 1] << 16);
            }
        }
        for (int i = tid; i < S; i += NT) {
            const int p = ib.shell_xy[s0 + i], y = p / nx, x = p - y * nx;
            const int ea = ib.csr_off[s0 + i], ne = ib.csr_off[s0 + i + 1] - ea;
            float w[4] = {0.f, 0.f, 0.f, 0.f};
            unsigned m[4] = {0, 0, 0, 0};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < ne) {
                    w[j] = ib.csr_w[ea + j];
                    m[j] = (unsigned)ib.csr_m[ea + j];
                }
            unsigned far = 0;
            if (ne > 4) {  // where in `more` does not matter
                const int k = atomicAdd(s_more, ne - 4);
                for (int j = 4; j < ne; ++j)
                    more[k + j - 4] = make_uint2(__float_as_uint(ib.csr_w[ea + j]), (unsigned)ib.csr_m[ea + j]);
                far = (unsigned)k | ((unsigned)(ne - 4) << 16);
            }
            tsw[i] = make_float4(w[0], w[1], w[2], w[3]);
            tsm[i] = make_uint4(m[0] | (m[1] << 16), m[2] | (m[3] << 16),
                                (unsigned)at(x, y) | ((unsigned)((x & 1) * MH + y * XP + (x >> 1)) << 16), far);
        }
        for (int i = tid; i < CS; i += NT) sb[i] = 0.f;  // marks of the shell nodes, below
        __syncthreads();
        for (int i = tid; i < S; i += NT) sb[tsm[i].z & 0xffffu] = 1.f;
        __syncthreads();

        // ---- this thread's nodes: rows y0 .. y0 + K - 1 of pair column xp, plane g
        const int YB = (ny + K - 1) / K;
        const bool active = tid < G * XP * YB;
        const int item = active ? tid : 0;
        xp = item % XP;
        y0 = (item / XP) % YB * K;
        g = item / (XP * YB);
        two = 2 * xp + 1 < nx;
        rows = active ? min(K, ny - y0) : 0;
        gp = g * PS + xp;  // offset of the pair in row 0 of its plane
        // x neighbours outside the pair, relative to it: the node before the even
        // one, the node after the odd one
        dl = xp > 0 ? HS - 1 : ((nx & 1) ? XP - 1 : HS + XP - 1);
        dr = xp + 1 < XP ? 1 : -xp;
        mm = active && !J.whole && g == 0;
        mp = active && !J.whole && g == G - 1;
        for (int k = 0; k < rows; ++k) first_bits |= (two ? 3u : 1u) << (2 * k);
        send_bits = first_bits;
        for (int k = 0; k < rows; ++k) {
            const int o = xp + (y0 + k) * XPS;
            if (sb[o] != 0.f) send_bits &= ~(1u << (2 * k));
            if (sb[o + HS] != 0.f) send_bits &= ~(2u << (2 * k));
        }
        __syncthreads();

        // ---- fields
        for (int i = tid; i < G * P; i += NT) {
            const int gg = i / P, p = i - gg * P, y = p / nx, x = p - y * nx;
            const int o = gg * PS + at(x, y), q = z0 * P + i;
            // the padding column of an odd row holds column 0: the last pair's right neighbour
            const bool pad = (nx & 1) && x == 0;
            const int op = gg * PS + at(nx, y);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float b = b_in[a * n + q], v = w1k * u[a * n + q];
                sb[a * CS + o] = b;
                su[a * CS + o] = v;
                if (pad) {
                    sb[a * CS + op] = b;
                    su[a * CS + op] = v;
                }
            }
        }

        // ---- S of the own nodes, from the differences of u and of B^ext
        const float* bxy = J.bext_xy;
        auto uat = [&](int zz, int y, int x, float v[3]) {
#pragma unroll
            for (int a = 0; a < 3; ++a) v[a] = __ldg(u + a * n + zz * P + y * nx + x);
        };
        auto bat = [&](int t, int y, int x, float v[3]) {
#pragma unroll
            for (int a = 0; a < 3; ++a) v[a] = slab_bext(J, t, a);
            bext_add_xy(bxy, P, y * nx + x, v);
        };
        auto cr = [](const float* v, const float* B, int a, int b) { return __fmaf_rn(v[a], B[b], -__fmul_rn(v[b], B[a])); };
        // u_a B_b - u_b B_a at place p less at place m
        auto dif = [&](const float* vp, const float* Bp, const float* vm, const float* Bm, int a, int b) {
            const float dv[3] = {vp[0] - vm[0], vp[1] - vm[1], vp[2] - vm[2]};
            const float dB[3] = {Bp[0] - Bm[0], Bp[1] - Bm[1], Bp[2] - Bm[2]};
            return cr(dv, Bp, a, b) + cr(vm, dB, a, b);
        };
#pragma unroll 1
        for (int i = tid; i < G * P; i += NT) {
            const int gg = i / P, p = i - gg * P, y = p / nx, x = p - y * nx, z = z0 + gg;
            const int za = z == 0 ? nz - 1 : z - 1, zb = z == nz - 1 ? 0 : z + 1;
            const int x_l = x == 0 ? nx - 1 : x - 1, x_r = x == nx - 1 ? 0 : x + 1;
            const int y_u = y == 0 ? ny - 1 : y - 1, y_d = y == ny - 1 ? 0 : y + 1;
            float s3[3], vp[3], vm[3], Bp[3], Bm[3];
            uat(z, y, x_l, vp);
            uat(z, y, x_r, vm);
            bat(gg + 1, y, x_l, Bp);
            bat(gg + 1, y, x_r, Bm);
            s3[1] = dif(vp, Bp, vm, Bm, 0, 1);
            s3[2] = dif(vp, Bp, vm, Bm, 0, 2);
            uat(z, y_u, x, vp);
            uat(z, y_d, x, vm);
            bat(gg + 1, y_u, x, Bp);
            bat(gg + 1, y_d, x, Bm);
            s3[0] = -dif(vp, Bp, vm, Bm, 0, 1);
            s3[2] += dif(vp, Bp, vm, Bm, 1, 2);
            uat(zb, y, x, vp);
            uat(za, y, x, vm);
            bat(gg + 2, y, x, Bp);
            bat(gg, y, x, Bm);
            s3[0] += dif(vp, Bp, vm, Bm, 0, 2);
            s3[1] += dif(vp, Bp, vm, Bm, 1, 2);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if constexpr (SSH)
                    sS[a * CS + gg * PS + at(x, y)] = s3[a] * w1k_all;
                else
                    J.S[a * n + z0 * P + i] = s3[a] * w1k_all;
            }
        }
    }
    __syncthreads();

    auto ld = [&](const float* q) { return f2(q[0], q[HS]); };  // a pair
    // messages: the nodes `out` of the own row k, their shares in the neighbours'
    // updates
    auto send_row = [&](int k, const float2 b[3], int par, unsigned seq, unsigned out) {
        const int MS = J.MS, MH = J.MH, m = par * MS + (y0 + k) * J.XP + xp;
        const unsigned go = out >> (2 * k), seq2 = msg_seq2(seq);
        const float w1 = J.w1;
        const float* q = su + gp + (y0 + k) * J.XPS;
        const float2 v[3] = {ld(q), ld(q + CS), ld(q + 2 * CS)};
        float2 o[3];
        if (mp) {
            z_share<true>(o, f2(w1, w1), b, v);
            uint4* x = reinterpret_cast<uint4*>(J.up) + m;
            msg_store(go & 1u, x, o[0].x, o[1].x, o[2].x, seq2);
            msg_store(go & 2u, x + MH, o[0].y, o[1].y, o[2].y, seq2);
        }
        if (mm) {
            z_share<false>(o, f2(w1, w1), b, v);
            uint4* x = reinterpret_cast<uint4*>(J.down) + m;
            msg_store(go & 1u, x, o[0].x, o[1].x, o[2].x, seq2);
            msg_store(go & 2u, x + MH, o[0].y, o[1].y, o[2].y, seq2);
        }
    };
    // counters: b of the end planes to the exchange by bulk copies, then the
    // count (thread 0, after a barrier that follows the writes of b)
    auto publish = [&](int par, unsigned n) {
        if (tid == 0) {
            const int XS = J.XS, PS = J.PS, G = J.G;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            for (int a = 0; a < 6; ++a) {  // component, half
                const float* q = sb + (a >> 1) * CS + (a & 1) * HS;
                slab_bulk_store(J.up + (6 * par + a) * XS, q + (G - 1) * PS, 4u * (unsigned)XS);
                if (G > 1) slab_bulk_store(J.down + (6 * par + a) * XS, q, 4u * (unsigned)XS);
            }
            asm volatile("cp.async.bulk.commit_group;\n\tcp.async.bulk.wait_group 0;\n\tfence.proxy.async;" ::: "memory");
            __threadfence();
            st_release_u32(J.count, n);
        }
    };
    if constexpr (MSG) {
        if (mm || mp)
            for (int k = 0; k < rows; ++k) {
                float2 b[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) b[a] = ld(sb + gp + (y0 + k) * J.XPS + a * CS);
                send_row(k, b, 0, J.base + 1u, first_bits);
            }
    } else {
        publish(0, J.base + 1u);
    }

    int s = 0;
#pragma unroll 1
    for (; s < J.nsweeps; ++s) {
        // 1. new b of the own nodes: the part from the slab first, which leaves
        // the exchange time to arrive.  Rows past the domain's end are computed
        // from row 0 and not stored.
        float2 nv[K][3];
        if (rows > 0) {
            const int ny = J.ny, XPS = J.XPS;
            const float w0 = J.w0, w1 = J.w1;
            const float2 w02 = f2(w0, w0), w12 = f2(w1, w1);
            {
                float2 ub[3], uv[3], cb[3], cv[3];  // (b, u) of the row above, the current row
                int oc = gp + y0 * XPS;
                const float* pu = sb + (y0 == 0 ? gp + (ny - 1) * XPS : oc - XPS);
                // S is read a row ahead
                const float* Sg = SSH ? sS + oc : J.S + (J.z0 + g) * J.P + y0 * J.nx + 2 * xp;
                const int nS = SSH ? CS : J.n, nxS = SSH ? XPS : J.nx, h2 = SSH ? HS : (two ? 1 : 0);
                float2 Sn[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) Sn[a] = f2(Sg[a * nS], Sg[a * nS + h2]);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    ub[a] = ld(pu + a * CS);
                    uv[a] = ld(pu + (3 + a) * CS);
                    cb[a] = ld(sb + oc + a * CS);
                    cv[a] = ld(sb + oc + (3 + a) * CS);
                }
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const int on = y0 + k + 1 < ny ? oc + XPS : gp;
                    const float *pd = sb + on, *pl = sb + oc + dl, *pr = sb + oc + dr;
                    // t: S plus the in-plane Phi_ab = u_b b_a - u_a b_b, + at x -
                    // e_b, - at x + e_b
                    float2 t[3], db[3], dv[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) t[a] = Sn[a];
                    if (k + 1 < K) {
                        if (k + 1 < rows) Sg += nxS;
#pragma unroll
                        for (int a = 0; a < 3; ++a) Sn[a] = f2(Sg[a * nS], Sg[a * nS + h2]);
                    }
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        db[a] = ld(pd + a * CS);
                        dv[a] = ld(pd + (3 + a) * CS);
                    }
                    t[0] = fma2(uv[1], ub[0], nfma2(uv[0], ub[1], t[0]));
                    t[0] = fma2(dv[0], db[1], nfma2(dv[1], db[0], t[0]));
                    t[2] = fma2(uv[1], ub[2], nfma2(uv[2], ub[1], t[2]));
                    t[2] = fma2(dv[2], db[1], nfma2(dv[1], db[2], t[2]));
#pragma unroll
                    for (int a = 0; a < 3; ++a) ub[a] = add2(ub[a], db[a]);
                    {
                        float2 lb[3], lv[3];
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            lb[a] = f2(pl[a * CS], cb[a].x);
                            lv[a] = f2(pl[(3 + a) * CS], cv[a].x);
                        }
                        t[1] = fma2(lv[0], lb[1], nfma2(lv[1], lb[0], t[1]));
                        t[2] = fma2(lv[0], lb[2], nfma2(lv[2], lb[0], t[2]));
#pragma unroll
                        for (int a = 0; a < 3; ++a) nv[k][a] = lb[a];
                    }
                    {
                        float2 rb[3], rv[3];
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            rb[a] = f2(cb[a].y, pr[a * CS]);
                            rv[a] = f2(cv[a].y, pr[(3 + a) * CS]);
                        }
                        t[1] = fma2(rv[1], rb[0], nfma2(rv[0], rb[1], t[1]));
                        t[2] = fma2(rv[2], rb[0], nfma2(rv[0], rb[2], t[2]));
#pragma unroll
                        for (int a = 0; a < 3; ++a)
                            nv[k][a] = fma2(w02, cb[a], fma2(w12, add2(add2(nv[k][a], rb[a]), ub[a]), t[a]));
                    }
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        ub[a] = cb[a];
                        uv[a] = cv[a];
                        cb[a] = db[a];
                        cv[a] = dv[a];
                    }
                    oc = on;
                }
            }
            if (!mm || !mp) {  // z neighbours in the slab
                const int G = J.G, PS = J.PS;
                const int ozm = (g > 0 ? -PS : (G - 1) * PS), ozp = g < G - 1 ? PS : (1 - G) * PS;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const int oc = gp + (k < rows ? y0 + k : 0) * XPS;
                    float2 b[3], v[3], o[3];
                    if (!mm) {
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            b[a] = ld(sb + oc + ozm + a * CS);
                            v[a] = ld(sb + oc + ozm + (3 + a) * CS);
                        }
                        z_share<true>(o, w12, b, v);
#pragma unroll
                        for (int a = 0; a < 3; ++a) nv[k][a] = add2(nv[k][a], o[a]);
                    }
                    if (!mp) {
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            b[a] = ld(sb + oc + ozp + a * CS);
                            v[a] = ld(sb + oc + ozp + (3 + a) * CS);
                        }
                        z_share<false>(o, w12, b, v);
#pragma unroll
                        for (int a = 0; a < 3; ++a) nv[k][a] = add2(nv[k][a], o[a]);
                    }
                }
            }
        }
        if constexpr (!MSG) {
            // the neighbours' end planes of the sweep before; after the barrier
            // no thread reads shared b of this sweep again
            if (!J.whole && tid == NT - 1 &&
                !wait_counters(J.count_prev, J.count_next, J.base + 1u + (unsigned)s, kWaitTimeoutNs)) {
                atomicExch(J.err, 1);
                *s_abort = 1;
            }
            __syncthreads();
            if (*(volatile int*)s_abort) break;  // uniform
        }
        if (mm || mp) {
            const int h2 = two ? J.MH : 0, XP = J.XP, MS = J.MS;
            if constexpr (MSG) {
                const unsigned seq = msg_seq2(J.base + 1u + (unsigned)s);
                const uint4 *qm = reinterpret_cast<const uint4*>(J.from_prev), *qp = reinterpret_cast<const uint4*>(J.from_next);
                unsigned polls = 0;
                unsigned long long t0 = 0;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const int o = (s & 1) * MS + (k < rows ? y0 + k : y0) * XP + xp;
                    Msg m[4];
                    for (;;) {
                        bool bad = false;
                        if (mm) m[0] = msg_load(qm + o), m[1] = msg_load(qm + o + h2);
                        if (mp) m[2] = msg_load(qp + o), m[3] = msg_load(qp + o + h2);
                        if (mm) bad = msg_stale(m[0], seq) || msg_stale(m[1], seq);
                        if (mp) bad = bad || msg_stale(m[2], seq) || msg_stale(m[3], seq);
                        if (!bad || msg_give_up(polls, t0, s_abort, J.err)) break;
                    }
                    float2 o3[3];
                    if (mm) {
                        msg_values(m[0], o3[0].x, o3[1].x, o3[2].x);
                        msg_values(m[1], o3[0].y, o3[1].y, o3[2].y);
#pragma unroll
                        for (int a = 0; a < 3; ++a) nv[k][a] = add2(nv[k][a], o3[a]);
                    }
                    if (mp) {
                        msg_values(m[2], o3[0].x, o3[1].x, o3[2].x);
                        msg_values(m[3], o3[0].y, o3[1].y, o3[2].y);
#pragma unroll
                        for (int a = 0; a < 3; ++a) nv[k][a] = add2(nv[k][a], o3[a]);
                    }
                }
            } else {
                const int XS = J.XS, XPS = J.XPS, nx = J.nx, n = J.n, h2u = two ? 1 : 0;
                const float w1 = J.w1, w1k = J.sq == 0.f ? 0.f : J.w1k;
                auto take = [&](const float* q, const float* u, auto above) {
                    q += 6 * (s & 1) * XS + xp;
                    u += 2 * xp;
                    constexpr int MB = K < 4 ? K : 2;  // rows in flight
#pragma unroll
                    for (int kb = 0; kb < K; kb += MB) {
                        float2 b[MB][3], v[MB][3], o[3];
#pragma unroll
                        for (int k = 0; k < MB && kb + k < K; ++k) {
                            const int y = kb + k < rows ? y0 + kb + k : y0;
                            const float *x = q + y * XPS, *w = u + y * nx;
#pragma unroll
                            for (int a = 0; a < 3; ++a) {
                                b[k][a] = f2(__ldcg(x + 2 * a * XS), __ldcg(x + (2 * a + 1) * XS));
                                v[k][a] = f2(__ldg(w + a * n), __ldg(w + a * n + h2u));
                            }
                        }
#pragma unroll
                        for (int k = 0; k < MB && kb + k < K; ++k) {
#pragma unroll
                            for (int a = 0; a < 3; ++a) v[k][a] = mul2(f2(w1k, w1k), v[k][a]);
                            z_share<!decltype(above)::value>(o, f2(w1, w1), b[k], v[k]);
#pragma unroll
                            for (int a = 0; a < 3; ++a) nv[kb + k][a] = add2(nv[kb + k][a], o[a]);
                        }
                    }
                };
                if (mm) take(J.from_prev, J.u + J.zm * J.P, std::false_type());
                if (mp) take(J.from_next, J.u + J.zp * J.P, std::true_type());
            }
        }
        if constexpr (MSG) {
            __syncthreads();
            if (*(volatile int*)s_abort) break;  // uniform: set only before the barrier above
        }
        // 2. to shared memory, and out
        const bool more_sweeps = s + 1 < J.nsweeps;
        const int par = (s + 1) & 1;
        const unsigned seq = J.base + 2u + (unsigned)s;
        {
            const int XPS = J.XPS, XP = J.XP;
            const bool pad = (J.nx & 1) && xp == 0;
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < rows) {
                    float* qb = sb + gp + (y0 + k) * XPS;
                    // an odd row's last pair has one node: the slot after it is the
                    // copy of column 0, which that column's owner writes
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        qb[a * CS] = nv[k][a].x;
                        if (two) qb[a * CS + HS] = nv[k][a].y;
                    }
                    if (pad)
#pragma unroll
                        for (int a = 0; a < 3; ++a) qb[a * CS + HS + XP - 1] = nv[k][a].x;
                    if (MSG && more_sweeps && (mm || mp)) send_row(k, nv[k], par, seq, send_bits);
                }
        }
        __syncthreads();
        if (J.R > 0) {
            // 3. deltas, a thread per (plane, marker, component)
            {
                const int R = J.R, PS = J.PS, n3 = 3 * J.G * R;
                const unsigned mR = J.mR;
                const float2* tw = t_w();
                const unsigned* tq = t_q();
                float4* td = t_d();
                for (int t = tid; t < n3; t += NT) {
                    const int gm = t / 3, a = t - 3 * gm;
                    const int pg = magic_div(gm, R, mR), m = gm - pg * R;
                    const float* f = sb + a * CS + pg * PS;
                    const float2* w = tw + 5 * m;
                    const unsigned* q = tq + 5 * m;
                    float v = 0.f;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float2 ww = w[j];
                        const unsigned qq = q[j];
                        v = __fmaf_rn(ww.x, f[qq & 0xffffu], v);
                        v = __fmaf_rn(ww.y, f[qq >> 16], v);
                    }
                    const float2 wl = w[4];
                    v = __fmaf_rn(wl.x, f[q[4] & 0xffffu], v);
                    reinterpret_cast<float*>(td + gm)[a] = -wl.y * v;
                }
            }
            __syncthreads();
            // 4. shell nodes
            {
                const int R = J.R, S = J.S_, PS = J.PS, G = J.G, nS = G * S, MS = J.MS, MH = J.MH, XP = J.XP;
                const unsigned mS = J.mS;
                const bool odd = J.nx & 1, out = MSG && more_sweeps && !J.whole;
                const float4 *td = t_d(), *tsw = t_sw();
                const uint4* tsm = t_sm();
                float *up = J.up, *down = J.down;
                const float w1 = J.w1;
                for (int t = tid; t < nS; t += NT) {
                    const int pg = magic_div(t, S, mS), i = t - pg * S;
                    const float4* dl4 = td + pg * R;
                    const float4 w = tsw[i];
                    const uint4 q = tsm[i];
                    float* qb = sb + pg * PS + (q.z & 0xffffu);
                    const float4 d0 = dl4[q.x & 0xffffu], d1 = dl4[q.x >> 16], d2 = dl4[q.y & 0xffffu], d3 = dl4[q.y >> 16];
                    float c0 = w.x * d0.x, c1 = w.x * d0.y, c2 = w.x * d0.z;
                    c0 = __fmaf_rn(w.y, d1.x, c0), c1 = __fmaf_rn(w.y, d1.y, c1), c2 = __fmaf_rn(w.y, d1.z, c2);
                    c0 = __fmaf_rn(w.z, d2.x, c0), c1 = __fmaf_rn(w.z, d2.y, c1), c2 = __fmaf_rn(w.z, d2.z, c2);
                    c0 = __fmaf_rn(w.w, d3.x, c0), c1 = __fmaf_rn(w.w, d3.y, c1), c2 = __fmaf_rn(w.w, d3.z, c2);
                    if (q.w) {
                        const uint2* more = t_more();
                        for (unsigned e = q.w & 0xffffu, ne = e + (q.w >> 16); e < ne; ++e) {
                            const uint2 l = more[e];
                            const float4 d = dl4[l.y];
                            const float x = __uint_as_float(l.x);
                            c0 = __fmaf_rn(x, d.x, c0), c1 = __fmaf_rn(x, d.y, c1), c2 = __fmaf_rn(x, d.z, c2);
                        }
                    }
                    c0 += qb[0], c1 += qb[CS], c2 += qb[2 * CS];
                    qb[0] = c0, qb[CS] = c1, qb[2 * CS] = c2;
                    const unsigned mi = q.z >> 16;
                    if (odd && mi < (unsigned)MH && mi % (unsigned)XP == 0) {  // column 0
                        float* qp = qb + HS + XP - 1;
                        qp[0] = c0, qp[CS] = c1, qp[2 * CS] = c2;
                    }
                    if (out && (pg == 0 || pg == G - 1)) {
                        const float *qv = qb + 3 * CS, b3[3] = {c0, c1, c2}, v3[3] = {qv[0], qv[CS], qv[2 * CS]};
                        auto put = [&](float* x, const float o[3]) {
                            msg_store(true, reinterpret_cast<uint4*>(x) + par * MS + mi, o[0], o[1], o[2], msg_seq2(seq));
                        };
                        float o[3];
                        if (pg == G - 1) {
                            z_share<true>(o, w1, b3, v3);
                            put(up, o);
                        }
                        if (pg == 0) {
                            z_share<false>(o, w1, b3, v3);
                            put(down, o);
                        }
                    }
                }
            }
            __syncthreads();
        }
        if (!MSG && more_sweeps) publish(par, seq);
    }
    // messages: the slots of the other parity, read for the last time before the
    // neighbour sent what the last sweep received: a sequence no launch will wait
    // for next (a launch of few sweeps leaves them as they are for long, and the 16
    // bits wrap)
    if (MSG && (mm || mp))
        for (int k = 0; k < rows; ++k) {
            const float2 none[3] = {};
            send_row(k, none, J.nsweeps & 1, J.base + (unsigned)J.nsweeps - 1u, first_bits);
        }
    {
        const int nx = J.nx, P = J.P, XPS = J.XPS, PS = J.PS, n = J.n, z0 = J.z0;
        float* b_out = J.b_out;
        for (int i = tid; i < J.G * P; i += NT) {
            const int pg = i / P, p = i - pg * P, y = p / nx, x = p - y * nx;
            const int o = pg * PS + (x & 1) * HS + y * XPS + (x >> 1);
#pragma unroll
            for (int a = 0; a < 3; ++a) b_out[a * n + z0 * P + i] = sb[a * CS + o];
        }
    }
    // (counters have it already, unless the sweeps were given up)
    if (tid == 0 && (MSG || s < J.nsweeps)) *J.count = J.base + (unsigned)J.nsweeps;
}

// A single handle: CTA j of gridDim.x holds the j-th slab of the balanced split
// of its planes.  msg: slab_msg_floats per CTA; counts: one per CTA.
template <int K>
__global__ void __launch_bounds__(kSlabThreads, 1)
    k_sweeps_slab(Geo g, const float* __restrict__ b_in, float* __restrict__ b_out, const float* __restrict__ u,
                  SweepCoef<float> c, IBView<float> ib, float* S, float* msg, ResidentSync* sync, int nsweeps,
                  int more) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_abort, s_more;
    __shared__ SlabJob s_job;
    if (threadIdx.x == 0) {
        s_abort = s_more = 0;
        const int ng = gridDim.x, j = blockIdx.x, q = g.nz / ng, r = g.nz % ng;
        const int Gmax = q + (r > 0), DF = slab_dir_floats(g.nx, g.ny, Gmax, K), jn = j == ng - 1 ? 0 : j + 1;
        auto planes = [&](int k) { return q + (k < r ? 1 : 0); };
        SlabJob& J = s_job;
        J.nx = g.nx;
        J.ny = g.ny;
        J.nz = g.nz;
        J.n = (int)g.n;
        J.z0 = j * q + min(j, r);
        J.G = planes(j);
        J.nsweeps = nsweeps;
        J.whole = ng == 1;
        J.b_in = b_in;
        J.b_out = b_out;
        J.u = u;
        J.S = S;
        J.more = more;
        const int jp = j == 0 ? ng - 1 : j - 1;
        auto slots = [&](int k) { return msg + (size_t)k * 2 * DF; };  // [direction][parity]
        J.up = slots(j);
        J.down = slots(j) + DF;
        J.from_prev = slots(jp);
        J.from_next = slots(jn) + (planes(jn) == 1 && K > kSlabMsgK ? 0 : DF);  // one plane is published once
        J.count = &sync->flags[j];
        J.count_prev = &sync->flags[jp];
        J.count_next = &sync->flags[jn];
        J.err = &sync->err;
        slab_job_init(J, c, ib, K, Gmax);
    }
    __syncthreads();
    slab_direct<K>(s_job, ib, smem_raw, &s_abort, &s_more);
}

}  // namespace qslbm
