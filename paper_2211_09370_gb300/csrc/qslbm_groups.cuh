// Resident sub-iteration for a batch of small instances (FP32): one
// cooperative launch per flow step runs all N_mag sweeps (Sec. V.G) with the
// IB on b after each (Sec. V.D, V.F) for every instance whose planes are
// small, each CTA holding a group of consecutive z planes of one instance in
// shared memory for the whole launch.
//
// A group is G planes of an instance (G P <= the stride of a field component in
// shared memory).  Per sweep the CTA forms every node's (e1, e2, e3) (the EMF form
// of k_sweep_march_pair; u comes from L2, loaded ahead of its use: it does not
// change during the sweeps), writes the new b of its nodes into the second of two
// b buffers (z neighbours inside the group from shared memory, those across its
// ends from the neighbouring groups) and applies the plane-local IB to each of its
// planes.  Neighbouring groups exchange their end planes as messages: 16 bytes a
// node, its three b values and the sweep's sequence number, which the reader polls
// for (with a limit of one second of the GPU's global timer, after which it raises
// an error flag and the sweeps end early).  A node off the wall's shell is sent
// where its new b is formed, a shell node after its IB correction.  Two sets of
// messages alternate: a thread sends sweep s + 2's only after it has received the
// neighbour's of sweep s + 1, sent after the neighbour read sweep s's.  All groups
// of one instance do the same number of sweeps, so their sequence numbers stay
// equal between launches.  The arithmetic is that of the split path (march_tile's
// EMF form, the staged IB's sums in the same order).
//
// What bounds it: the chain of a sweep (e, exchange, walk, markers, shell, with a
// barrier between each) and shared-memory wavefronts (about 3.3 a node and sweep).  Twelve
// pipes of 24^2 to 28^2 nodes, 151 groups of up to eight planes: 9.6 us a sweep;
// with a counter per group (fence, release, acquire, then the halo loads) in place
// of messages, and u loaded at its use, 10.4 for eleven of them.
#pragma once

#include "qslbm_kernels.cuh"
#include "qslbm_resident.cuh"

namespace qslbm {

constexpr int kGroupThreads = 1024;
// Nodes a CTA holds, at most: the shared-memory stride of one field component, a
// compile-time constant, so that the components of a node are one base address
// apart by immediate offsets.  The small stride leaves 44 KB to the IB tables
// (rings of up to some 200 markers), the large one, 20 KB, holds more planes of the
// smallest pipes (eight instead of seven of 27x27 nodes).
constexpr int kGroupStrideS = 5120;
constexpr int kGroupStrideL = 5888;

// One CTA's group: planes z0 .. z0 + G - 1 of instance inst; prev / next: the
// groups holding planes z0 - 1 and z0 + G (periodic; possibly itself); xoff:
// its messages, [2 parities][first, last plane][P], counted in uint4.
struct GroupDesc {
    int inst, z0, G, prev, next;
    long long xoff;
};

// What a CTA's threads look up per sweep (in shared memory: the sweep loop has no
// registers for it).
struct GroupJob {
    const float *u, *bin, *bxy;  // velocity, b before the first sweep, in-plane B^ext
    uint4* out;                  // messages, [parity][first, last plane][P]: own,
    const uint4 *prev, *next;    // the previous group's last plane, the next group's first
    float w0, w1, w1k, sq;
    unsigned base;               // sweeps done before the launch
    int P, GN;                   // nodes of a plane, of the group
    unsigned mP, mR, mS;         // magic_of P, R, S
    int abort;
};

// Messages of a group of planes of P nodes (uint4).
inline long long group_msgs(int P) { return 4LL * P; }

// Shared memory of one group (bytes): two buffers of b and one of e (stride nodes
// each), B^ext of its G planes and their two neighbours, the deltas of its G
// rings, the IB tables of one ring (R markers, S shell nodes, E list entries) and
// a bit per node of a plane.  A launch gives every CTA the largest group's size.
inline size_t group_smem_bytes(int stride, int R, int S, int E, int G, int P) {
    return 36 * (size_t)stride + 16 * (size_t)(G + 2) + 16 * (size_t)G * R + 8 * ((size_t)9 * R + E + S) +
           4 * ((size_t)R + (P + 31) / 32) + 16;
}

// XY: some instance has an in-plane applied field (QSLBM_B0_FIELD).
template <typename Desc, bool XY, int GS>
__global__ void __launch_bounds__(kGroupThreads, 1)
    k_batch_resident(const Desc* __restrict__ d, const GroupDesc* __restrict__ groups, uint4* xbuf, unsigned* counts,
                     int* err) {
    constexpr int NPT = (GS + kGroupThreads - 1) / kGroupThreads;  // nodes per thread, at most
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ GroupJob J;
    const GroupDesc gd = groups[blockIdx.x];
    const Desc& D = d[gd.inst];
    const int nmag = D.n_mag;
    if (nmag == 0) return;  // uniform: b keeps its parity
    const int nx = D.g.nx, ny = D.g.ny, nz = D.g.nz;
    const int P = nx * ny, n = (int)D.g.n;
    const int G = gd.G, z0 = gd.z0, GN = G * P;
    const unsigned mX = magic_of(nx);
    const bool whole = G == nz;  // the group holds every plane: no exchange
    const int tid = threadIdx.x;
    // the ring and shell of plane 0, which every plane carries (z-invariant tables)
    const int m0 = D.ibm.ring_off[0], R = D.ibm.ring_off[1] - m0;
    const int s0 = D.ibm.shell_off[0], S = D.ibm.shell_off[1] - s0;
    const int e0 = S > 0 ? D.ibm.csr_off[s0] : 0;
    const int E = S > 0 ? D.ibm.csr_off[s0 + S] - e0 : 0;
    const int zm = z0 == 0 ? nz - 1 : z0 - 1;  // plane below the group
    const int zp = z0 + G == nz ? 0 : z0 + G;  // plane above it
    // shared memory: b [2][3][GS] (sweep s reads b[s % 2], writes b[(s + 1) % 2]),
    // e [3][GS], B^ext, deltas, tables
    float* sb0 = reinterpret_cast<float*>(smem_raw);
    float* se = sb0 + 6 * GS;
    float4* sbz = reinterpret_cast<float4*>(se + 3 * GS);  // B^ext of planes zm, z0 .. z0 + G - 1, zp
    float4* sdelta = sbz + G + 2;                          // [G][R]
    int2* tqw = reinterpret_cast<int2*>(sdelta + G * R);   // [R][9] support (in-plane index), weight
    int2* tl = tqw + 9 * R;                                // [E] shell lists: marker (ring-relative), weight
    int2* tsh = tl + E;                                    // [S] shell nodes: in-plane index, list offset | length << 16
    float* tsc = reinterpret_cast<float*>(tsh + S);        // [R] s^m_j
    unsigned* shell = reinterpret_cast<unsigned*>(tsc + R);  // a bit per in-plane node: on the shell
    {
        const SweepCoef<float>& c = D.sc;
        if (tid == 0) {
            J.u = D.u[D.fpar];
            J.bin = D.b[D.bpar];
            J.bxy = XY ? c.bext_xy : nullptr;
            J.out = xbuf + gd.xoff;
            J.prev = xbuf + groups[gd.prev].xoff + P;
            J.next = xbuf + groups[gd.next].xoff;
            J.w0 = c.w0;
            J.w1 = c.w1;
            J.w1k = c.w1 * c.kappa;
            J.sq = c.sq;
            J.base = counts[blockIdx.x];
            J.abort = 0;
            J.P = P;
            J.GN = GN;
            J.mP = magic_of(P);
            J.mR = magic_of(R);
            J.mS = magic_of(S);
        }
        for (int t = tid; t < G + 2; t += kGroupThreads) {
            const int zz = t == 0 ? zm : (t == G + 1 ? zp : z0 + t - 1);
            float be[3];
            bext_at(c.bext_z, c.be, zz, be);
            sbz[t] = make_float4(be[0], be[1], be[2], 0.f);
        }
    }
    for (int i = tid; i < (P + 31) / 32; i += kGroupThreads) shell[i] = 0u;
    __syncthreads();
    for (int i = tid; i < 9 * R; i += kGroupThreads)
        tqw[i] = make_int2(D.ibm.mk_q[9 * m0 + i], __float_as_int(D.ibm.mk_w[9 * m0 + i]));
    for (int i = tid; i < R; i += kGroupThreads) tsc[i] = D.ibm.mk_s[m0 + i];
    for (int i = tid; i < S; i += kGroupThreads) {
        const int q = D.ibm.shell_xy[s0 + i], o = D.ibm.csr_off[s0 + i];
        tsh[i] = make_int2(q, (o - e0) | (D.ibm.csr_off[s0 + i + 1] - o) << 16);
        atomicOr(&shell[q >> 5], 1u << (q & 31));
    }
    for (int i = tid; i < E; i += kGroupThreads)
        tl[i] = make_int2(D.ibm.csr_m[e0 + i], __float_as_int(D.ibm.csr_w[e0 + i]));
    for (int i = tid; i < GN; i += kGroupThreads)
#pragma unroll
        for (int a = 0; a < 3; ++a) sb0[a * GS + i] = J.bin[a * n + z0 * P + i];
    float ur[NPT][3];  // u of nodes tid + k kGroupThreads, loaded ahead of their use
    auto load_u = [&] {
        const float* __restrict__ u = J.u + z0 * J.P + tid;
        const int GN = J.GN;
#pragma unroll
        for (int k = 0; k < NPT; ++k) {
            const int q = k * kGroupThreads;
            if (tid + q < GN) {
                ur[k][0] = __ldg(u + q);
                ur[k][1] = __ldg(u + n + q);
                ur[k][2] = __ldg(u + 2 * n + q);
            }
        }
    };
    load_u();
    __syncthreads();

    int s = 0;  // sweeps done
    for (; s < nmag; ++s) {
        const float* sb = sb0 + (s & 1) * 3 * GS;  // b after sweep s - 1
        float* sn = sb0 + ((s + 1) & 1) * 3 * GS;  // b after sweep s
        const bool send = !whole && s + 1 < nmag;
        // (a) every node's e from its b (shared memory) and u
        {
            const float sq = J.sq;
            const int P = J.P, GN = J.GN;
            const unsigned mP = J.mP;
#pragma unroll
            for (int k = 0; k < NPT; ++k) {
                const int i = tid + k * kGroupThreads;
                if (i < GN) {
                    const int g = magic_div(i, P, mP);
                    const float4 bz = sbz[g + 1];
                    float be[3] = {bz.x, bz.y, bz.z};
                    if constexpr (XY) bext_add_xy(J.bxy, P, i - g * P, be);
                    float r[6] = {sb[i], sb[GS + i], sb[2 * GS + i], ur[k][0], ur[k][1], ur[k][2]};
                    node_emf(r, be, sq);
                    se[i] = r[3];
                    se[GS + i] = r[4];
                    se[2 * GS + i] = r[5];
                }
            }
        }
        __syncthreads();
        // (b) the new b of this thread's nodes into the other buffer
        // (march_tile's expressions in its order)
        {
            const float w0 = J.w0, w1 = J.w1, w1k = J.w1k;
            // each thread walks whole z columns of the group: the column's b, e2 and
            // e3 (e1 enters in-plane differences only) at planes g - 1, g, g + 1
            // stay in registers
#pragma unroll 1
            for (int p = tid; p < P; p += kGroupThreads) {
                const int y = magic_div(p, nx, mX), x = p - y * nx;
                const int dl = x == 0 ? nx - 1 : -1, dr = x == nx - 1 ? 1 - nx : 1;
                const int du = y == 0 ? P - nx : -nx, dd = y == ny - 1 ? nx - P : nx;
                const bool now = send && !((shell[p >> 5] >> (p & 31)) & 1u);  // the IB leaves it as it is
                float prv[5], cur[5], nxt[5], top[5];  // top: the plane above the group
                if (whole) {
                    const int j = (G - 1) * P + p;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        prv[a] = sb[a * GS + j];
                        top[a] = sb[a * GS + p];
                    }
                    prv[3] = se[GS + j];
                    prv[4] = se[2 * GS + j];
                    top[3] = se[GS + p];
                    top[4] = se[2 * GS + p];
                } else {
                    // both neighbour planes' b: the fields' own before the first
                    // sweep, then the neighbour groups' messages of sweep s - 1
                    float r0[6], r1[6];
                    const float* __restrict__ u = J.u;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        r0[3 + a] = __ldg(u + a * n + zm * P + p);
                        r1[3 + a] = __ldg(u + a * n + zp * P + p);
                    }
                    if (s == 0) {
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            r0[a] = J.bin[a * n + zm * P + p];
                            r1[a] = J.bin[a * n + zp * P + p];
                        }
                    } else {
                        const uint4* xp = J.prev + ((s + 1) & 1) * 2 * P + p;
                        const uint4* xq = J.next + ((s + 1) & 1) * 2 * P + p;
                        const unsigned want = msg_seq2(J.base + (unsigned)s);
                        Msg mp, mq;
                        unsigned polls = 0;
                        unsigned long long t0 = 0;
                        for (;;) {
                            mp = msg_load(xp);
                            mq = msg_load(xq);
                            if (!(msg_stale(mp, want) || msg_stale(mq, want)) ||
                                msg_give_up(polls, t0, &J.abort, err))
                                break;
                        }
                        msg_values(mp, r0[0], r0[1], r0[2]);
                        msg_values(mq, r1[0], r1[1], r1[2]);
                    }
                    const float4 b0 = sbz[0], b1 = sbz[G + 1];
                    float be0[3] = {b0.x, b0.y, b0.z}, be1[3] = {b1.x, b1.y, b1.z};
                    if constexpr (XY) {
                        bext_add_xy(J.bxy, P, p, be0);
                        bext_add_xy(J.bxy, P, p, be1);
                    }
                    node_emf(r0, be0, J.sq);
                    node_emf(r1, be1, J.sq);
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        prv[a] = r0[a];
                        top[a] = r1[a];
                    }
                    prv[3] = r0[4];
                    prv[4] = r0[5];
                    top[3] = r1[4];
                    top[4] = r1[5];
                }
#pragma unroll
                for (int a = 0; a < 3; ++a) cur[a] = sb[a * GS + p];
                cur[3] = se[GS + p];
                cur[4] = se[2 * GS + p];
                int i = p;
#pragma unroll 1
                for (int g = 0; g < G; ++g, i += P) {
                    if (g < G - 1) {
#pragma unroll
                        for (int a = 0; a < 3; ++a) nxt[a] = sb[a * GS + i + P];
                        nxt[3] = se[GS + i + P];
                        nxt[4] = se[2 * GS + i + P];
                    } else {
#pragma unroll
                        for (int v = 0; v < 5; ++v) nxt[v] = top[v];
                    }
                    const int il = i + dl, ir = i + dr, iu = i + du, id = i + dd;
                    float nb[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const float* Ba = sb + a * GS;
                        const float sa = (Ba[il] + Ba[ir]) + (Ba[iu] + Ba[id]) + (prv[a] + nxt[a]);
                        float da;
                        if (a == 0)
                            da = (se[id] - se[iu]) + (nxt[3] - prv[3]);
                        else if (a == 1)
                            da = (se[il] - se[ir]) + (nxt[4] - prv[4]);
                        else
                            da = (se[GS + il] - se[GS + ir]) + (se[2 * GS + iu] - se[2 * GS + id]);
                        nb[a] = emf_update(w0, w1, w1k, cur[a], sa, da);
                        sn[a * GS + i] = nb[a];
                    }
                    if (now && (g == 0 || g == G - 1)) {
                        uint4* const xo = J.out + (s & 1) * 2 * P + p;
                        const unsigned seq2 = msg_seq2(J.base + (unsigned)s + 1u);
                        msg_store(g == 0, xo, nb[0], nb[1], nb[2], seq2);
                        msg_store(g == G - 1, xo + P, nb[0], nb[1], nb[2], seq2);
                    }
#pragma unroll
                    for (int v = 0; v < 5; ++v) {
                        prv[v] = cur[v];
                        cur[v] = nxt[v];
                    }
                }
            }
        }
        load_u();         // for the next sweep
        __syncthreads();  // the new b is complete
        if (J.abort) break;  // uniform: read by every thread after the barrier
        // (c) IB on each plane of the group: delta_j = -s^m_j D b* at every
        // marker, then b = b* + D^T delta on the shell (ib_plane's sums in its
        // order; the planes are independent)
        if (R > 0) {
            const unsigned mR = J.mR, mS = J.mS;
            const unsigned seq2 = msg_seq2(J.base + (unsigned)s + 1u);
            uint4* const xo = J.out + (s & 1) * 2 * P;
            for (int t = tid; t < G * R; t += kGroupThreads) {
                const int g = magic_div(t, R, mR), m = t - g * R;
                const float* f = sn + g * P;
                float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll
                for (int j = 0; j < 9; ++j) {
                    const int2 e = tqw[9 * m + j];
                    const float w = __int_as_float(e.y);
                    const int q = e.x;
                    a0 += w * f[q];
                    a1 += w * f[GS + q];
                    a2 += w * f[2 * GS + q];
                }
                const float sm = tsc[m];
                sdelta[t] = make_float4(-sm * a0, -sm * a1, -sm * a2, 0.f);
            }
            __syncthreads();
            // the first and last planes first: their nodes go to the neighbours
            for (int t = tid; t < G * S; t += kGroupThreads) {
                const int o = magic_div(t, S, mS), k = t - o * S;
                const int g = o == 0 ? 0 : (o == 1 ? G - 1 : o - 1);
                const int2 node = tsh[k];
                const float4* dl = sdelta + g * R;
                float c0 = 0.f, c1 = 0.f, c2 = 0.f;
                const int2* e = tl + (node.y & 0xffff);
                const int cnt = node.y >> 16;
                const int q = g * P + node.x;
                const float b0 = sn[q], b1 = sn[GS + q], b2 = sn[2 * GS + q];
#pragma unroll 3
                for (int j = 0; j < cnt; ++j) {
                    const int2 le = e[j];
                    const float w = __int_as_float(le.y);
                    const float4 dj = dl[le.x];
                    c0 += w * dj.x;
                    c1 += w * dj.y;
                    c2 += w * dj.z;
                }
                const float n0 = b0 + c0, n1 = b1 + c1, n2 = b2 + c2;
                sn[q] = n0;
                sn[GS + q] = n1;
                sn[2 * GS + q] = n2;
                msg_store(send && g == 0, xo + node.x, n0, n1, n2, seq2);
                msg_store(send && g == G - 1, xo + P + node.x, n0, n1, n2, seq2);
            }
            __syncthreads();
        }
    }
    // the b of the last sweep done (all of them unless a wait gave up)
    const float* sb = sb0 + (s & 1) * 3 * GS;
    float* __restrict__ bfin = D.b[(D.bpar + nmag) & 1];
    for (int i = tid; i < GN; i += kGroupThreads)
#pragma unroll
        for (int a = 0; a < 3; ++a) bfin[a * n + z0 * P + i] = sb[a * GS + i];
    if (tid == 0) counts[blockIdx.x] = J.base + (unsigned)nmag;
}

}  // namespace qslbm
