// Resident magnetic sub-iterations in FP64: one launch runs all N_mag sweeps
// (Sec. V.G) with the IB corrector on b after each (Sec. V.D, V.F).
//
// sm_103 issues about two FP64 operations per SM and clock (1/64 of the FP32
// rate), so an FP64 sweep is bound by its operation count: both kernels carry
// (b, e) per node, e = the three numbers of the antisymmetric flux, formed once
// per node and sweep with explicit fused multiply-adds.  That is 42 FP64
// operations per node (e 9, neighbour sums 15, flux differences 9, update 9)
// against about 135 when every neighbour's flux is formed from (b, u).
//   k_sweeps_resident64  3-D: one z plane per CTA, cooperative launch.
//   k_sweeps_cluster64   2-D: bands of rows over the CTAs of one thread-block
//                        cluster; a single CTA has one SM's FP64 rate only.
#pragma once

#include "qslbm_kernels.cuh"
#include "qslbm_resident.cuh"

namespace qslbm {

// ------------------------------------------------------------------- 3-D
// Each CTA keeps its plane's b and e in shared memory.  Per sweep: the
// in-plane part from its own plane; the bounded wait on the two neighbours'
// counters; the z terms from the neighbours' (b, e2, e3) of the previous
// sweep, a double-buffered exchange array in global memory (10 loads a node
// instead of forming e twice more, 8 operations); the plane-local IB; the new
// e of every node and its publication.  Operations at 2 per clock: 42 x 4096 nodes
// is 42 us a sweep for the 64x64x128 pipe, which takes 55.3 us (the marching sweep
// and its IB 65.6; 65x65x120 57.6 against 96.3, 48x48x128 32.7 against 55.8).  512
// threads keep the FP64 pipe as busy as 1024 do and have the registers for the new
// values of their nodes (1024, which spilled them: 57.7).
constexpr int kRes64Threads = 512;
// nodes per thread, at most: planes whose b and e fit shared memory have at most
// 4842; planes of up to 4096 take eight (ten cost a few spills)
constexpr int kRes64MaxNpt = 10;
constexpr int kRes64Fields = 5;  // exchanged per node: b, e2, e3

// Shared memory of a plane of P nodes with a ring of R markers, S shell nodes and E
// list entries.  The weights are kept once, with 16-bit indices (48 B a node leave 35
// KB of tables at 64x64, where separate weights and 32-bit indices took 44).
inline size_t resident64_smem_bytes(int P, int R, int S, int E) {
    return ((size_t)6 * P + 13 * R) * sizeof(double) + ((size_t)9 * R + 2 * S + 1 + E) * sizeof(unsigned short);
}

template <typename T, int kRes64Npt>
__global__ void __launch_bounds__(kRes64Threads, 1)
    k_sweeps_resident64(Geo g, const T* __restrict__ b_in, T* __restrict__ b_out, const T* __restrict__ u,
                        SweepCoef<T> c, IBView<T> ib, T* xbuf, ResidentSync* sync, int nsweeps, int max_ring,
                        int max_shell) {
    static_assert(sizeof(T) == 8, "the FP64 path");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned int s_epoch;
    __shared__ int s_abort;
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    const int P = nx * ny, n = (int)g.n;
    const int z = blockIdx.x;
    const int zm = wrap_dec(z, nz), zp = wrap_inc(z, nz);
    const int base = z * P;
    const int tid = threadIdx.x;
    double* sb = reinterpret_cast<double*>(smem_raw);  // [3][P] b
    double* se = sb + 3 * P;                           // [3][P] e
    double* sdelta = se + 3 * P;                       // [3 R]
    double* tw = sdelta + 3 * max_ring;                // [9 R]
    double* tsc = tw + 9 * max_ring;                   // [R]
    // 16 bits reach every index: a plane has at most 4842 nodes, and fewer list
    // entries than that fit
    unsigned short* tq = reinterpret_cast<unsigned short*>(tsc + max_ring);  // [9 R] support (in-plane index)
    unsigned short* tshell = tq + 9 * max_ring;                              // [S] shell nodes
    unsigned short* toff = tshell + max_shell;                               // [S + 1] list offsets
    unsigned short* tl = toff + max_shell + 1;                               // [E] the markers' entries (of tw, tq)
    if (tid == 0) {
        s_epoch = *(volatile unsigned int*)&sync->epoch;
        s_abort = 0;
    }
    const int tz = ib.zinv ? 0 : z;
    const int m0 = ib.ring_off[tz], R = ib.ring_off[tz + 1] - m0;
    const int s0 = ib.shell_off[tz], S = ib.shell_off[tz + 1] - s0;
    {
        const int e0 = S > 0 ? ib.csr_off[s0] : 0;
        for (int i = tid; i < 9 * R; i += kRes64Threads) {
            tq[i] = (unsigned short)ib.mk_q[9 * m0 + i];
            tw[i] = ib.mk_w[9 * m0 + i];
        }
        for (int i = tid; i < R; i += kRes64Threads) tsc[i] = ib.mk_s[m0 + i];
        __syncthreads();
        // a list entry is a marker's weight at the node: named by its place in tw
        for (int i = tid; i < S; i += kRes64Threads) {
            const int q = ib.shell_xy[s0 + i], o = ib.csr_off[s0 + i], o1 = ib.csr_off[s0 + i + 1];
            tshell[i] = (unsigned short)q;
            toff[i] = (unsigned short)(o - e0);
            if (i == S - 1) toff[S] = (unsigned short)(o1 - e0);
            for (int e = o; e < o1; ++e) {
                const int m = ib.csr_m[e];
                const double w = ib.csr_w[e];
                int at = 9 * m;
                for (int k = 9 * m; k < 9 * m + 9; ++k)
                    if (tq[k] == q && tw[k] == w) at = k;
                tl[e - e0] = (unsigned short)at;
            }
        }
    }
    double be[3];
    bext_at(c.bext_z, c.be, z, be);
    for (int p = tid; p < P; p += kRes64Threads)
#pragma unroll
        for (int a = 0; a < 3; ++a) sb[a * P + p] = b_in[a * n + base + p];
    __syncthreads();
    const unsigned int epoch = s_epoch;
    const long long xplane = (long long)kRes64Fields * P;
    const double w0 = c.w0, w1 = c.w1, w1k = c.w1 * c.kappa;
    // e of every own node from its b, and (b, e2, e3) to exchange buffer `par`
    auto form_e = [&](int par, bool publish) {
        double* xo = xbuf + ((long long)par * nz + z) * xplane;
        for (int p = tid; p < P; p += kRes64Threads) {
            double r[6] = {sb[p],          sb[P + p],          sb[2 * P + p], __ldg(u + base + p),
                           __ldg(u + n + base + p), __ldg(u + 2 * n + base + p)};
            node_emf(r, be, c.sq);
            se[p] = r[3];
            se[P + p] = r[4];
            se[2 * P + p] = r[5];
            if (publish) {
                __stcg(xo + p, r[0]);
                __stcg(xo + P + p, r[1]);
                __stcg(xo + 2 * P + p, r[2]);
                __stcg(xo + 3 * P + p, r[4]);
                __stcg(xo + 4 * P + p, r[5]);
            }
        }
        __syncthreads();
        if (publish && tid == 0) __threadfence();
    };
    form_e(1, true);
    if (tid == 0) st_release_u32(&sync->flags[z], epoch + 1u);
    for (int s = 0; s < nsweeps; ++s) {
        // (1) in-plane part, from this CTA's own plane
        double nv[kRes64Npt][3];
#pragma unroll
        for (int k = 0; k < kRes64Npt; ++k) {
            const int p = tid + k * kRes64Threads;
            if (p < P) {
                const int y = p / nx, x = p - y * nx;
                const int row = y * nx;
                const int il = row + wrap_dec(x, nx), ir = row + wrap_inc(x, nx);
                const int iu = wrap_dec(y, ny) * nx + x, id = wrap_inc(y, ny) * nx + x;
                const double *E1 = se, *E2 = se + P, *E3 = se + 2 * P;
                const double d[3] = {E1[id] - E1[iu], E1[il] - E1[ir], (E2[il] - E2[ir]) + (E3[iu] - E3[id])};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const double* B = sb + a * P;
                    nv[k][a] = emf_update(w0, w1, w1k, B[p], (B[il] + B[ir]) + (B[iu] + B[id]), d[a]);
                }
            }
        }
        // (2) the neighbour planes of the previous sweep
        if (tid == 0 &&
            !wait_counters(&sync->flags[zm], &sync->flags[zp], epoch + (unsigned int)s + 1u, kWaitTimeoutNs)) {
            atomicExch(&sync->err, 1);
            s_abort = 1;
        }
        __syncthreads();  // also: every in-plane read of the old plane is done
        if (s_abort) return;
        // (3) the z terms, and the plane's new values
        {
            const double* xin = xbuf + (long long)((s + 1) & 1) * nz * xplane;
            const double *xm = xin + zm * xplane, *xp = xin + zp * xplane;
#pragma unroll
            for (int k = 0; k < kRes64Npt; ++k) {
                const int p = tid + k * kRes64Threads;
                if (p < P) {
                    double vm[kRes64Fields], vp[kRes64Fields];
#pragma unroll
                    for (int f = 0; f < kRes64Fields; ++f) {
                        vm[f] = __ldcg(xm + f * P + p);
                        vp[f] = __ldcg(xp + f * P + p);
                    }
                    sb[p] = __fma_rn(w1k, vp[3] - vm[3], __fma_rn(w1, vm[0] + vp[0], nv[k][0]));
                    sb[P + p] = __fma_rn(w1k, vp[4] - vm[4], __fma_rn(w1, vm[1] + vp[1], nv[k][1]));
                    sb[2 * P + p] = __fma_rn(w1, vm[2] + vp[2], nv[k][2]);
                }
            }
        }
        __syncthreads();
        // (4) IB on the plane: every marker's delta, then the shell nodes; one
        // thread per (marker or node, component)
        if (R > 0) {
            for (int t = tid; t < 3 * R; t += kRes64Threads) {
                const int m = t / 3, a = t - 3 * m;
                const double* f = sb + a * P;
                double v = 0.0;
#pragma unroll
                for (int j = 0; j < 9; ++j) v = __fma_rn(tw[9 * m + j], f[tq[9 * m + j]], v);
                sdelta[t] = -tsc[m] * v;
            }
            __syncthreads();
            for (int t = tid; t < 3 * S; t += kRes64Threads) {
                const int i = t / 3, a = t - 3 * i;
                double v = 0.0;
                for (int e = toff[i]; e < toff[i + 1]; ++e) {
                    const int l = tl[e];
                    v = __fma_rn(tw[l], sdelta[3 * (l / 9) + a], v);
                }
                sb[a * P + tshell[i]] += v;
            }
            __syncthreads();
        }
        // (5) e of the corrected plane
        if (s + 1 < nsweeps) {
            form_e(s & 1, true);
            if (tid == 0) st_release_u32(&sync->flags[z], epoch + (unsigned int)s + 2u);
        }
    }
    for (int p = tid; p < P; p += kRes64Threads)
#pragma unroll
        for (int a = 0; a < 3; ++a) b_out[a * n + base + p] = sb[a * P + p];
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        const unsigned int prev = atomicAdd(&sync->done, 1u);
        if (prev == gridDim.x - 1) {
            sync->done = 0;
            sync->epoch = epoch + (unsigned int)nsweeps;
            __threadfence();
        }
    }
}

// ------------------------------------------------------------------- 2-D
// One thread-block cluster holds the plane, CTA r of it rows r RB .. r RB + RB
// - 1 (the last bands may be short or empty).  Per node in shared memory: b,
// e, b* (the swept field), u and S.  The flux of the (uniform) applied field is
// constant over the sweeps: its part S of the update is formed once, from
// differences of u, and e is that of b alone, so that no sum of large terms is
// rounded each sweep; 29 FP64 operations a node.  Neighbouring bands are read
// through distributed shared memory.  Per sweep:
//   b* of the own rows from (b, e) of the rows and their neighbours | cluster barrier
//   delta of every marker whose support touches the own rows, from b* (markers
//   across a band's edge are interpolated by both bands, bitwise alike) | barrier
//   the corrected b of the own rows and its e                       | cluster barrier
// b* and b are separate arrays, so those two cluster barriers order every
// read of a neighbour's rows against its writes.  Measured on the 64x32
// channel (465 sweeps a step): 2.9 us a sweep with 16 CTAs, against 56 us for
// the plane in one CTA; 128 nodes x 29 operations at two per clock are 0.9 us,
// the rest is the two cluster barriers and the chain of dependent operations.
constexpr int kC2Threads = 256;
constexpr int kC2MaxCluster = 16;

struct C2Geo {
    int nx, ny, RB;               // rows per band
    int mk_max, sh_max, nz_max;   // largest band's markers, shell nodes, list entries
};

// Bytes of shared memory of one band.
inline size_t cluster2d_smem_bytes(int nx, int RB, int R, int mk_max, int sh_max, int nz_max) {
    const size_t d = (size_t)15 * RB * nx + (size_t)13 * mk_max + nz_max;
    const size_t i = (size_t)9 * mk_max + 2 * mk_max + (size_t)sh_max + sh_max + 1 + nz_max + R + (size_t)RB * nx;
    return d * sizeof(double) + i * sizeof(int);
}

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned map_rank(unsigned addr, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ double ld_cluster(unsigned addr) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// (b, u) -> (b, u x b's three numbers) in place, 6 operations
__device__ __forceinline__ void emf_b(double r[6]) {
    const double u0 = r[3], u1 = r[4], u2 = r[5];
    r[3] = __fma_rn(u0, r[1], -__dmul_rn(u1, r[0]));
    r[4] = __fma_rn(u0, r[2], -__dmul_rn(u2, r[0]));
    r[5] = __fma_rn(u1, r[2], -__dmul_rn(u2, r[1]));
}

template <typename T>
__global__ void __launch_bounds__(kC2Threads, 1)
    k_sweeps_cluster64(C2Geo g, const T* __restrict__ b_in, T* __restrict__ b_out, const T* __restrict__ u,
                       SweepCoef<T> c, IBView<T> ib, int nsweeps) {
    static_assert(sizeof(T) == 8, "the FP64 path");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_cnt;
    const int nx = g.nx, ny = g.ny, RB = g.RB;
    const int n = nx * ny, NB = RB * nx;  // nodes of a full band
    const int rank = (int)cluster_rank();
    const int y0 = min(rank * RB, ny), y1 = min(y0 + RB, ny);
    const int N = (y1 - y0) * nx;
    const int tid = threadIdx.x;
    double* sb = reinterpret_cast<double*>(smem_raw);  // [3][NB] b
    double* se = sb + 3 * NB;                          // [3][NB] e
    double* ss = se + 3 * NB;                          // [3][NB] b*
    double* su = ss + 3 * NB;                          // [3][NB] u
    double* sS = su + 3 * NB;                          // [3][NB] S
    double* tw = sS + 3 * NB;                          // [9 mk_max] weights of the band's markers
    double* tsc = tw + 9 * g.mk_max;                   // [mk_max] scalings
    double* sdelta = tsc + g.mk_max;                   // [3 mk_max]
    double* tcw = sdelta + 3 * g.mk_max;               // [nz_max] list weights
    unsigned* tq = reinterpret_cast<unsigned*>(tcw + g.nz_max);  // [9 mk_max] cluster addresses of b* there
    int* tm = reinterpret_cast<int*>(tq + 9 * g.mk_max);         // [mk_max] the band's markers
    int* tcnt = tm + g.mk_max;                                   // [mk_max] nodes of nonzero weight of each
    int* tshell = tcnt + g.mk_max;                               // [sh_max] shell nodes (index in the band)
    int* toff = tshell + g.sh_max;                               // [sh_max + 1] list offsets
    int* tcm = toff + g.sh_max + 1;                              // [nz_max] markers (index in the band's list)
    int* isshell = tcm + g.nz_max;                               // [NB] 1: a shell node
    int* pos = isshell + NB;                                     // [R] marker -> index in the band's list
    const unsigned a_sb = (unsigned)__cvta_generic_to_shared(sb);
    const unsigned a_se = (unsigned)__cvta_generic_to_shared(se);
    const unsigned a_ss = (unsigned)__cvta_generic_to_shared(ss);
    const unsigned a_su = (unsigned)__cvta_generic_to_shared(su);
    double be[3];
    bext_at(c.bext_z, c.be, 0, be);
    for (int i = tid; i < N; i += kC2Threads) {
        double r[6];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            r[a] = b_in[a * n + y0 * nx + i];
            r[3 + a] = u[a * n + y0 * nx + i];
            sb[a * NB + i] = r[a];
            su[a * NB + i] = r[3 + a];
        }
        emf_b(r);
#pragma unroll
        for (int a = 0; a < 3; ++a) se[a * NB + i] = r[3 + a];
        isshell[i] = 0;
    }
    // the band's IB tables: its markers (any support row in the band) and its
    // shell nodes (a contiguous run: the shell list is sorted by in-plane index)
    const int R = ib.ring_off[1], S = ib.shell_off[1];
    if (tid == 0) s_cnt = 0;
    __syncthreads();
    for (int m = tid; m < R; m += kC2Threads) {
        bool own = false;
        for (int j = 0; j < 9; ++j) {
            const int y = ib.mk_q[9 * m + j] / nx;
            own = own || (y >= y0 && y < y1);
        }
        pos[m] = own ? atomicAdd(&s_cnt, 1) : -1;
        if (own) tm[pos[m]] = m;
    }
    int sA = 0, sB = 0;
    {
        int lo = 0, hi = S;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (ib.shell_xy[mid] < y0 * nx)
                lo = mid + 1;
            else
                hi = mid;
        }
        sA = lo;
        hi = S;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (ib.shell_xy[mid] < y1 * nx)
                lo = mid + 1;
            else
                hi = mid;
        }
        sB = lo;
    }
    __syncthreads();
    const int M = s_cnt, SB = sB - sA;
    const int e0 = SB > 0 ? ib.csr_off[sA] : 0;
    // support nodes of nonzero weight only: a wall on the nodes has one of nine
    for (int t = tid; t < M; t += kC2Threads) {
        const int m = tm[t];
        int k = 0;
        for (int j = 0; j < 9; ++j) {
            const double w = ib.mk_w[9 * m + j];
            if (w == 0.0) continue;
            const int q = ib.mk_q[9 * m + j], r = q / (nx * RB);
            tq[9 * t + k] = map_rank(a_ss, (unsigned)r) + 8u * (unsigned)(q - r * NB);
            tw[9 * t + k] = w;
            ++k;
        }
        tcnt[t] = k;
        tsc[t] = ib.mk_s[m];
    }
    for (int t = tid; t < SB; t += kC2Threads) {
        tshell[t] = ib.shell_xy[sA + t] - y0 * nx;
        isshell[tshell[t]] = 1;
        toff[t] = ib.csr_off[sA + t] - e0;
        for (int e = ib.csr_off[sA + t]; e < ib.csr_off[sA + t + 1]; ++e) {
            tcm[e - e0] = pos[ib.csr_m[e]];
            tcw[e - e0] = ib.csr_w[e];
        }
        if (t == SB - 1) toff[SB] = ib.csr_off[sB] - e0;
    }
    // the bands above and below (periodic), and the addresses of the rows next
    // to this band there
    const int last = (ny - 1) / RB;  // the last band with rows
    const int rp = rank == 0 ? last : rank - 1, rn = rank >= last ? 0 : rank + 1;
    const int prow = min(RB, ny - rp * RB) - 1;
    const unsigned ub_b = map_rank(a_sb, (unsigned)rp) + 8u * (unsigned)(prow * nx);
    const unsigned ub_e = map_rank(a_se, (unsigned)rp) + 8u * (unsigned)(prow * nx);
    const unsigned db_b = map_rank(a_sb, (unsigned)rn), db_e = map_rank(a_se, (unsigned)rn);
    const unsigned cs = 8u * (unsigned)NB;  // bytes between components
    const double w0 = c.w0, w1 = c.w1;
    const double w1k = c.sq == 0.0 ? 0.0 : c.w1 * c.kappa;  // strict QS: the flux has no b part
    __syncthreads();
    cluster_arrive();
    cluster_wait();  // every band's b, e and u are in place
    // S: the applied field's part of w1 kappa D, from differences of u (B^ext is uniform)
    {
        const double k = c.w1 * c.kappa;
        const unsigned uu = map_rank(a_su, (unsigned)rp) + 8u * (unsigned)(prow * nx), ud = map_rank(a_su, (unsigned)rn);
        for (int i = tid; i < N; i += kC2Threads) {
            const int y = i / nx, x = i - y * nx;
            const int il = y * nx + wrap_dec(x, nx), ir = y * nx + wrap_inc(x, nx);
            double dx[3], dy[3];  // u(-x) - u(+x), u(+y) - u(-y)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                dx[a] = su[a * NB + il] - su[a * NB + ir];
                dy[a] = (y == y1 - y0 - 1 ? ld_cluster(ud + a * cs + 8u * (unsigned)x) : su[a * NB + i + nx]) -
                        (y == 0 ? ld_cluster(uu + a * cs + 8u * (unsigned)x) : su[a * NB + i - nx]);
            }
            sS[i] = k * __fma_rn(dy[0], be[1], -dy[1] * be[0]);
            sS[NB + i] = k * __fma_rn(dx[0], be[1], -dx[1] * be[0]);
            sS[2 * NB + i] = k * (__fma_rn(dx[0], be[2], -dx[2] * be[0]) - __fma_rn(dy[1], be[2], -dy[2] * be[1]));
        }
    }
    // new b* of node i into r[0..2] and ss
    auto sweep = [&](int i, double r[6]) {
        const int y = i / nx, x = i - y * nx;
        const int il = y * nx + wrap_dec(x, nx), ir = y * nx + wrap_inc(x, nx);
        const bool first = y == 0, end = y == y1 - y0 - 1;
        double vu[5], vd[5];  // b, e1, e3 of the rows above and below
        if (first) {
            const unsigned bu = ub_b + 8u * (unsigned)x, eu = ub_e + 8u * (unsigned)x;
#pragma unroll
            for (int a = 0; a < 3; ++a) vu[a] = ld_cluster(bu + a * cs);
            vu[3] = ld_cluster(eu);
            vu[4] = ld_cluster(eu + 2 * cs);
        } else {
#pragma unroll
            for (int a = 0; a < 3; ++a) vu[a] = sb[a * NB + i - nx];
            vu[3] = se[i - nx];
            vu[4] = se[2 * NB + i - nx];
        }
        if (end) {
            const unsigned bd = db_b + 8u * (unsigned)x, ed = db_e + 8u * (unsigned)x;
#pragma unroll
            for (int a = 0; a < 3; ++a) vd[a] = ld_cluster(bd + a * cs);
            vd[3] = ld_cluster(ed);
            vd[4] = ld_cluster(ed + 2 * cs);
        } else {
#pragma unroll
            for (int a = 0; a < 3; ++a) vd[a] = sb[a * NB + i + nx];
            vd[3] = se[i + nx];
            vd[4] = se[2 * NB + i + nx];
        }
        const double d[3] = {vd[3] - vu[3], se[il] - se[ir], (se[NB + il] - se[NB + ir]) + (vu[4] - vd[4])};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double sum = (sb[a * NB + il] + sb[a * NB + ir]) + (vu[a] + vd[a]);
            r[a] = __fma_rn(w0, sb[a * NB + i], __fma_rn(w1k, d[a], __fma_rn(w1, sum, sS[a * NB + i])));
            ss[a * NB + i] = r[a];
        }
    };
    auto emf = [&](int i, double r[6]) {
#pragma unroll
        for (int a = 0; a < 3; ++a) r[3 + a] = su[a * NB + i];
        emf_b(r);
    };
    auto put = [&](int i, const double r[6]) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            sb[a * NB + i] = r[a];
            se[a * NB + i] = r[3 + a];
        }
    };
    __syncthreads();
    const bool one = N <= kC2Threads;  // a node per thread: its values stay in registers
    const bool mine = one && tid < N && !isshell[tid < N ? tid : 0];
    for (int s = 0; s < nsweeps; ++s) {
        double r[6];
        for (int i = tid; i < N; i += kC2Threads) sweep(i, r);
        cluster_arrive();
        if (mine) emf(tid, r);  // nodes off the shell keep b*
        cluster_wait();         // b* is complete everywhere; b and e may change
        for (int t = tid; t < 3 * M; t += kC2Threads) {
            const int m = t / 3, a = t - 3 * m;
            double v = 0.0;
            for (int j = 0; j < tcnt[m]; ++j) v = __fma_rn(tw[9 * m + j], ld_cluster(tq[9 * m + j] + a * cs), v);
            sdelta[t] = -tsc[m] * v;
        }
        if (mine) {
            put(tid, r);
        } else if (!one) {
            for (int i = tid; i < N; i += kC2Threads)
                if (!isshell[i]) {
                    double q[6] = {ss[i], ss[NB + i], ss[2 * NB + i], 0.0, 0.0, 0.0};
                    emf(i, q);
                    put(i, q);
                }
        }
        __syncthreads();  // the deltas
        for (int t = kC2Threads - 1 - tid; t < SB; t += kC2Threads) {
            const int i = tshell[t];
            double v[3] = {0.0, 0.0, 0.0};
            for (int e = toff[t]; e < toff[t + 1]; ++e)
#pragma unroll
                for (int a = 0; a < 3; ++a) v[a] = __fma_rn(tcw[e], sdelta[3 * tcm[e] + a], v[a]);
            double q[6] = {ss[i] + v[0], ss[NB + i] + v[1], ss[2 * NB + i] + v[2], 0.0, 0.0, 0.0};
            emf(i, q);
            put(i, q);
        }
        cluster_arrive();
        cluster_wait();  // the corrected b and its e; every read of b* is done
    }
    for (int i = tid; i < N; i += kC2Threads)
#pragma unroll
        for (int a = 0; a < 3; ++a) b_out[a * n + y0 * nx + i] = sb[a * NB + i];
}

}  // namespace qslbm
