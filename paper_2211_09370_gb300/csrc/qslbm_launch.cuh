// Kernel launchers for one storage precision T; included by qslbm_f32.cu and
// qslbm_f64.cu, which instantiate it for float and double.
#pragma once

#include <algorithm>

#include "qslbm_fused.cuh"
#include "qslbm_internal.h"
#include "qslbm_flow.cuh"
#include "qslbm_kernels.cuh"
#include "qslbm_resident.cuh"
#include "qslbm_resident64.cuh"
#include "qslbm_slab.cuh"

namespace qslbm {

template <typename T>
struct Launch {
    static Geo geo(const State& s) { return Geo{s.nx, s.ny, s.nz, s.n}; }

    static IBView<T> view(const State& s, bool magnetic) {
        IBView<T> v;
        v.ring_off = s.ib.ring_off;
        v.mk_q = s.ib.mk_q;
        v.mk_w = static_cast<const T*>(s.ib.mk_w);
        v.mk_s = static_cast<const T*>(magnetic ? s.ib.mk_sm : s.ib.mk_s);
        v.shell_off = s.ib.shell_off;
        v.shell_xy = s.ib.shell_xy;
        v.csr_off = s.ib.csr_off;
        v.csr_m = s.ib.csr_m;
        v.csr_w = static_cast<const T*>(s.ib.csr_w);
        v.mk_base = s.ib.mk_base;
        v.shell_node = s.ib.shell_node;
        v.csr_mg = s.ib.csr_mg;
        v.delta = static_cast<T*>(s.ib.delta);
        v.nm = s.ib.nm;
        v.ns = s.ib.ns;
        v.zinv = s.ib.zinv;
        v.mk_slot = s.ib.mk_slot;
        v.pad_m = s.ib.pad_m;
        v.pad_w = static_cast<const T*>(s.ib.pad_w);
        v.pad_k = s.ib.pad_k;
        return v;
    }

    // A launch that may begin while the previous kernel in the stream finishes
    // (programmatic dependent launch; the kernel calls pdl_wait before it
    // touches that kernel's results), or, without `early`, an ordinary one.
    template <typename... KArgs, typename... Args>
    static void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool early,
                           Args... args) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = block;
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = early ? 1 : 0;
        cudaLaunchKernelEx(&cfg, kernel, args...);  // errors surface at the next synchronising call
    }

    static size_t ib_smem(const State& s) { return (size_t)3 * (s.ib.max_ring > 0 ? s.ib.max_ring : 1) * sizeof(T); }

    static int grid_for(long long n, int threads) {
        long long b = (n + threads - 1) / threads;
        if (b > 152LL * 16) b = 152LL * 16;
        if (b < 1) b = 1;
        return (int)b;
    }

    static void init(State& s, cudaStream_t st) {
        int ncomp = s.dim == 3 ? 3 : 2;
        k_init<T><<<grid_for(s.n, 256), 256, 0, st>>>(geo(s), (T*)s.drho[0], (T*)s.u[0], (T*)s.b[0], s.p.seed,
                                                       s.p.perturb * s.units.U0, ncomp, s.p.geometry, s.cx,
                                                       s.cy, s.R, s.p.init_kind == QSLBM_INIT_POISEUILLE,
                                                       s.units.U0, s.axis);
    }

    // The staged IB corrector on every plane of f; early: scheduled as the CTAs of the
    // kernel before it exit.
    static void launch_ib_staged(const State& s, T* f, const IBView<T>& v, bool early, cudaStream_t st) {
        const int R = s.ib.max_ring, S = s.ib.max_shell;
        const size_t sm = s.ib_staged_smem;
        const dim3 ig((unsigned)s.nz), ib(kNodeThreads);
        switch (s.ib_staged_u) {
            case 1: launch_pdl(k_ib_staged<T, 1>, ig, ib, sm, st, early, geo(s), f, v, R, S); break;
            case 2: launch_pdl(k_ib_staged<T, 2>, ig, ib, sm, st, early, geo(s), f, v, R, S); break;
            case 4: launch_pdl(k_ib_staged<T, 4>, ig, ib, sm, st, early, geo(s), f, v, R, S); break;
            default: launch_pdl(k_ib_staged<T, 5>, ig, ib, sm, st, early, geo(s), f, v, R, S); break;
        }
    }

    // Planes per CTA of the marching force and flow kernels: two extra planes are read per
    // chunk, which a chunk as long as fills the device's resident CTAs in few waves hides.
    static cudaError_t plan_flow(State& s) {
        if (s.dim != 3) return cudaSuccess;
        int dev = 0, sms = 0, per_sm = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const void* kern = s.units.flow_q == 27 ? (const void*)k_flow_march<T, 27> : (const void*)k_flow_march<T, 19>;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kFlowThreads<T>, 0);
        if (e != cudaSuccess) return e;
        const long long tiles = (long long)((s.nx + kFlowTX - 1) / kFlowTX) * ((s.ny + kFlowTY<T> - 1) / kFlowTY<T>);
        const long long slots = (long long)std::max(1, sms) * std::max(1, per_sm);
        long long cost = 1LL << 62;
        for (int chunk = 1; chunk <= 32 && chunk <= s.nz; ++chunk) {
            const long long waves = (tiles * ((s.nz + chunk - 1) / chunk) + slots - 1) / slots;
            const long long c = waves * (chunk + 2);
            if (c < cost) {
                cost = c;
                s.flow_chunk = chunk;
            }
        }
        return cudaSuccess;
    }

    static void sweeps(State& s, int nsweeps, cudaStream_t st) {
        SweepCoef<T> c;
        sweep_weights(s, c.w0, c.w1, c.kappa);
        for (int a = 0; a < 3; ++a) c.be[a] = (T)s.be[a];
        c.bext_z = static_cast<const T*>(s.bext_z);
        c.bext_xy = static_cast<const T*>(s.bext_xy);
        c.strict_qs = s.p.strict_qs;
        c.sq = s.p.strict_qs ? T(0) : T(1);
        const IBView<T> v = view(s, true);
        const size_t smem = ib_smem(s);
        if (s.resident && nsweeps > 0) {
            launch_resident(s, nsweeps, c, v, st);
            s.bcur ^= 1;
            return;
        }
        if (s.fused) {
            for (int i = 0; i < nsweeps; ++i) {
                launch_fused(s, c, st);
                s.bcur ^= 1;
            }
            return;
        }
        if (s.p.sweep_kernel == QSLBM_SWEEP_SPLIT) {
            const int P = s.nx * s.ny;
            const dim3 grid((unsigned)((P + kNodeThreads - 1) / kNodeThreads), (unsigned)s.nz);
            const int chunk = s.march_chunk;
            const dim3 mgrid((unsigned)((s.nx + kMarchTX - 1) / kMarchTX), (unsigned)((s.ny + kMarchTY - 1) / kMarchTY),
                             (unsigned)((s.nz + chunk - 1) / chunk));
            for (int i = 0; i < nsweeps; ++i) {
                const T* bin = (const T*)s.b[s.bcur];
                T* bout = (T*)s.b[1 - s.bcur];
                const T* u = (const T*)s.u[s.fcur];
                if (pair_march(s)) {
                    if constexpr (sizeof(T) == 4) {
                        const int ty = 8 * s.march_rows;
                        const dim3 pgrid((unsigned)((s.nx + 2 * kPairTXP - 1) / (2 * kPairTXP)),
                                         (unsigned)((s.ny + ty - 1) / ty), (unsigned)((s.nz + chunk - 1) / chunk));
                        launch_pdl(pair_kernel(s.bext_xy != nullptr, s.march_rows), pgrid, dim3(kPairThreads), 0, st,
                                   true, geo(s), bin, bout, u, c, chunk);
                    }
                } else if (s.dim == 3) {
                    if (s.bext_xy)
                        k_sweep_march<T, true><<<mgrid, kMarchTX * kMarchTY, 0, st>>>(geo(s), bin, bout, u, c, chunk);
                    else if constexpr (sizeof(T) == 8)
                        k_sweep_march<T, false><<<mgrid, kMarchTX * kMarchTY, 0, st>>>(geo(s), bin, bout, u, c, chunk);
                } else {
                    k_sweep_nodes<T, 2><<<grid, kNodeThreads, 0, st>>>(geo(s), bin, bout, u, c);
                }
                if (s.ib.nm > 0 && s.ib_staged_smem > 0) {
                    launch_ib_staged(s, bout, v, s.ib_early, st);
                } else if (s.ib.nm > 0) {
                    k_ib_markers<T><<<(s.ib.nm + kNodeThreads - 1) / kNodeThreads, kNodeThreads, 0, st>>>(geo(s), bout, v);
                    k_ib_shell<T><<<(s.ib.ns + kNodeThreads - 1) / kNodeThreads, kNodeThreads, 0, st>>>(geo(s), bout, v);
                }
                s.bcur ^= 1;
            }
            return;
        }
        for (int i = 0; i < nsweeps; ++i) {
            const T* bin = (const T*)s.b[s.bcur];
            T* bout = (T*)s.b[1 - s.bcur];
            const T* u = (const T*)s.u[s.fcur];
            if (s.dim == 3)
                k_sweep_ib<T, 3><<<s.nz, kPlaneThreads, smem, st>>>(geo(s), bin, bout, u, c, v);
            else
                k_sweep_ib<T, 2><<<s.nz, kPlaneThreads, smem, st>>>(geo(s), bin, bout, u, c, v);
            s.bcur ^= 1;
        }
    }

    template <int DIM, bool UHALO, bool SMALL>
    static void resident_launch_one(State& s, int nsweeps, const SweepCoef<T>& c, const IBView<T>& v,
                                    cudaStream_t st) {
        constexpr int RT = ResidentShape<T, SMALL>::threads, NPT = ResidentShape<T, SMALL>::npt;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)s.nz);
        cfg.blockDim = dim3(RT);
        cfg.dynamicSmemBytes = s.resident_smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const T* bin = (const T*)s.b[s.bcur];
        T* bout = (T*)s.b[1 - s.bcur];
        const T* u = (const T*)s.u[s.fcur];
        cudaError_t e;
        if (s.nx % 2 == 0)
            e = cudaLaunchKernelEx(&cfg, k_sweeps_resident<T, DIM, UHALO, RT, NPT, true>, geo(s), bin, bout, u, c, v,
                                   (T*)s.xbuf, (ResidentSync*)s.rsync, nsweeps, s.ib.max_ring, s.ib.max_shell,
                                   s.ib.max_nnz);
        else
            e = cudaLaunchKernelEx(&cfg, k_sweeps_resident<T, DIM, UHALO, RT, NPT, false>, geo(s), bin, bout, u, c,
                                   v, (T*)s.xbuf, (ResidentSync*)s.rsync, nsweeps, s.ib.max_ring, s.ib.max_shell,
                                   s.ib.max_nnz);
        // a failed launch is recorded for the caller
        if (e != cudaSuccess) s.launch_error = true;
    }

    static FusedIB fused_ib(const State& s) {
        FusedIB t;
        t.mk_cnt = s.fu_mk_cnt;
        t.mk_off = s.fu_mk_off;
        t.mk_w = s.fu_mk_w;
        t.mk_s = s.fu_mk_s;
        t.sh_cnt = s.fu_sh_cnt;
        t.sh_off = s.fu_sh_off;
        t.sh_m = s.fu_sh_m;
        t.sh_w = s.fu_sh_w;
        t.sh_cnt_e = s.fu_sh_ce;
        t.Mmax = s.fu_Mmax;
        t.Smax = s.fu_Smax;
        t.K = s.fu_K;
        return t;
    }

    // the instantiation for this handle's shape: compile-time (nx, rows per
    // band, slots) for common plane widths, the general one otherwise
    static decltype(&k_sweep_fused<false>) fused_kernel(const State& s) {
        if (s.bext_xy) return k_sweep_fused<true>;
        if (s.nx == 96 && s.fu_TY == 12 && s.fu_slots == 4) return k_sweep_fused<false, 96, 12, 4>;
        if (s.nx == 64 && s.fu_TY == 20 && s.fu_slots == 4) return k_sweep_fused<false, 64, 20, 4>;
        if (s.nx == 128 && s.fu_TY == 8 && s.fu_slots == 4) return k_sweep_fused<false, 128, 8, 4>;
        return k_sweep_fused<false>;
    }

    // one sweep + IB on b, bin = b[bcur] -> b[1 - bcur], u = u[fcur]
    static void launch_fused(State& s, const SweepCoef<T>& c, cudaStream_t st) {
        if constexpr (sizeof(T) == 4) {
            const dim3 grid((unsigned)s.fu_bands, (unsigned)s.fu_chunks);
            const FusedGeo g{s.nx, s.ny, s.nz, s.fu_TY, s.fu_chunk, (int)s.n, s.fu_slots};
            const int bc = s.bcur, fc = s.fcur;
            launch_pdl(fused_kernel(s), grid, dim3(s.fu_threads), s.fu_smem, st, true, s.fu_map_b3[bc], s.fu_map_bt[bc],
                       s.fu_map_u3[fc], s.fu_map_ut[fc], (float*)s.b[1 - bc], c, fused_ib(s), g, s.fu_err);
        } else {
            s.launch_error = true;  // never planned: the fused sweep is the FP32 path
        }
    }

    // threads, and z planes per CTA so that the grid is one CTA per SM
    static cudaError_t plan_fused(State& s) {
        if constexpr (sizeof(T) != 4) {
            s.fused = false;
            return cudaSuccess;
        } else {
            // one node pair per thread and pass over the band's swept rows
            const int pairs = (s.fu_TY + 4) * s.nx / 2;
            s.fu_threads = std::min(kFusedMaxThreads, (pairs + 31) / 32 * 32);
            auto kern = fused_kernel(s);
            cudaError_t e = allow_smem((const void*)kern, s.fu_smem);
            if (e != cudaSuccess) {
                cudaGetLastError();
                s.fused = false;
                return cudaSuccess;
            }
            int dev = 0, sms = 0, per_sm = 0;
            if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
            if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
            if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, s.fu_threads, s.fu_smem)) !=
                cudaSuccess)
                return e;
            if (per_sm < 1) {
                s.fused = false;
                return cudaSuccess;
            }
            const int slots_total = per_sm * sms;
            const int chunks = std::max(1, slots_total / s.fu_bands);
            s.fu_chunk = (s.nz + chunks - 1) / chunks;
            s.fu_chunks = (s.nz + s.fu_chunk - 1) / s.fu_chunk;
            return cudaSuccess;
        }
    }

    // Times the fused kernel and the split path on this handle's own fields and takes
    // the fused one only when it is at least 2 % faster: the split path is the simpler
    // one and wins ties, so that the choice does not flip on timing noise.  Both are
    // timed from a graph, as steps run them: on a stream the split path's second launch
    // per sweep costs more than in a graph, and 24x24x96 in an in-plane field went to the
    // fused kernel (7.4 us a sweep) for a split path of 5.5.  Two interleaved rounds of
    // 8 sweeps each after a warm-up, the faster round kept.  Every timed sweep reads
    // b[bcur] and writes the other buffer, so the state is left as it was.
    static cudaError_t tune_fused(State& s, double* us_fused, double* us_split) {
        constexpr int kSweeps = 8;
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        cudaGraphExec_t run[2] = {nullptr, nullptr};
        cudaError_t e = cudaEventCreate(&e0);
        if (e == cudaSuccess) e = cudaEventCreate(&e1);
        double us[2] = {1e300, 1e300};
        for (int k = 0; k < 2 && e == cudaSuccess; ++k) {
            s.fused = k == 0;
            s.p.sweep_kernel = k == 0 ? QSLBM_SWEEP_FUSED : QSLBM_SWEEP_SPLIT;
            cudaGraph_t g = nullptr;
            e = cudaStreamBeginCapture(s.stream, cudaStreamCaptureModeThreadLocal);
            if (e != cudaSuccess) break;
            for (int r = 0; r < kSweeps; ++r) {
                sweeps(s, 1, s.stream);
                s.bcur ^= 1;  // undo the sweep's swap: the next reads the same b
            }
            e = cudaStreamEndCapture(s.stream, &g);
            if (e == cudaSuccess) e = cudaGraphInstantiate(&run[k], g, 0);
            if (g) cudaGraphDestroy(g);
        }
        for (int round = 0; round < 2; ++round)
            for (int k = 0; k < 2 && e == cudaSuccess; ++k) {
                e = cudaGraphLaunch(run[k], s.stream);
                if (e == cudaSuccess) e = cudaEventRecord(e0, s.stream);
                if (e == cudaSuccess) e = cudaGraphLaunch(run[k], s.stream);
                if (e == cudaSuccess) e = cudaEventRecord(e1, s.stream);
                if (e == cudaSuccess) e = cudaEventSynchronize(e1);
                float ms = 0.f;
                if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
                us[k] = std::min(us[k], 1e3 * ms / kSweeps);
            }
        for (cudaGraphExec_t x : run)
            if (x) cudaGraphExecDestroy(x);
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
        if (e == cudaSuccess) e = cudaGetLastError();
        *us_fused = us[0];
        *us_split = us[1];
        s.fused = e == cudaSuccess && us[0] < 0.98 * us[1];
        s.p.sweep_kernel = s.fused ? QSLBM_SWEEP_FUSED : QSLBM_SWEEP_SPLIT;
        return e;
    }

    static bool small_plane(const State& s) { return (long long)s.nx * s.ny <= (long long)kResidentSmallPlane; }

    // FP32: a slab of planes per CTA
    static auto slab_kernel(int K) {
        return K == 1   ? k_sweeps_slab<1>
               : K == 2 ? k_sweeps_slab<2>
               : K == 3 ? k_sweeps_slab<3>
               : K == 4 ? k_sweeps_slab<4>
                        : k_sweeps_slab<5>;
    }
    static void launch_slab(State& s, int nsweeps, const SweepCoef<float>& c, const IBView<float>& v,
                            cudaStream_t st) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)s.slab_ctas);
        cfg.blockDim = dim3((unsigned)s.slab_threads);
        cfg.dynamicSmemBytes = s.resident_smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t e =
            cudaLaunchKernelEx(&cfg, slab_kernel(s.slab_rows), geo(s), (const float*)s.b[s.bcur],
                               (float*)s.b[1 - s.bcur], (const float*)s.u[s.fcur], c, v, s.slab_S, (float*)s.xbuf,
                               (ResidentSync*)s.rsync, nsweeps, s.slab_more);
        if (e != cudaSuccess) s.launch_error = true;
    }

    // Estimated us per sweep, where k_sweeps_resident does not apply: of the slab kernel
    // with K rows a thread and `columns` threads at work on slabs of G planes, its start
    // (tables, S) included, and of the split sweep and its IB pass.  A slab's time is that
    // of one CTA, however many there are; the split sweep's grows with the planes of its
    // chunk (pair_shape), so that a device half full of slabs can lose to it.  Fitted to
    // 740 domains with and without walls, ramps and in-plane fields.  Measured, slab /
    // split: 57x57 (five rows) x153 16.4 / 11.6, x245 16.6 / 15.1, x304 16.6 / 17.0; 54x54
    // (four) x153 13.5 / 9.8, x245 13.5 / 13.1, x304 13.6 / 15.1; without walls 53x53 (four)
    // x200 11.6 / 8.8, 37x37 (two) x153 6.3 / 5.4; 20x300x40 in an in-plane field 13.2 /
    // 8.4.  A step of few sweeps does not earn the start back: 40x40x192 (three) at 5
    // sweeps 89 us a step against 67, at 40 358 against 368.
    static double slab_us(const State& s, int K, int columns, int G) {
        const int XP = slab_pairs(s.nx);
        double t;
        if (K == 1)
            t = 1.0 + 0.0022 * columns;
        else if (K == 2)  // (rows of an odd number of pairs, unpadded, conflict in their banks)
            t = XP % 2 && slab_row_stride(s.nx, s.ny, G, K) == XP ? 2.6 + 0.0052 * columns : 0.0066 * columns;
        else if (K == 3)
            t = G > 1 ? 1.65 + 0.0068 * columns : 3.5 + 0.0033 * columns;
        else if (K == 4)  // (wide planes, and slabs of several low ones, have fewer conflicts)
            t = (XP >= 32 ? 0.0125 : G > 2 ? 0.0132 : 0.0155) * columns;
        else
            t = 6.3 + 0.01 * columns;
        const double ib[] = {0.8, 1.5, G > 1 ? 2.0 : 1.0, 1.9, 3.0};
        if (s.ib.nm > 0) t += ib[K - 1];
        const double start = 9.0 + 0.0037 * G * s.nx * s.ny + (s.bext_xy ? 3.5 : 0.0);
        return t + start / std::max(1, s.units.n_mag);
    }
    static cudaError_t split_us(const State& s, double* us) {
        int rows = 2, chunk = 1;
        const cudaError_t e = pair_shape(s, 1, &rows, &chunk);
        double t = rows == 1 ? 1.7 + 1.03 * chunk : 1.55 + 1.42 * chunk;
        if (s.nx % 2) t += rows == 1 ? 1.0 : 1.0 + 0.1 * chunk;
        if (s.bext_xy) t *= s.nx % 2 ? 1.2 : 1.3;
        if (s.ib.nm > 0) t += 2.2 + 0.004 * s.ib.max_shell;
        *us = t;
        return e;
    }

    // The slab kernel for this domain: the fewest planes per CTA at which every
    // CTA is co-resident.
    static cudaError_t plan_slab(State& s, int optin, int sms) {
        s.slab_ctas = 0;
        if (s.dim != 3 || (long long)s.nx * s.ny > kResidentMaxPlane || !s.ib.zinv) return cudaSuccess;
        const int ctas = (s.nz + (s.nz + sms - 1) / sms - 1) / ((s.nz + sms - 1) / sms);
        const int G = (s.nz + ctas - 1) / ctas;  // the largest slab of the balanced split
        const int K = slab_rows(s.nx, s.ny, G);
        if (K == 0 || (long long)G * slab_plane_stride(s.nx, s.ny, G, K) > slab_half(K)) return cudaSuccess;
        // Where it is not the faster one (measured, us per sweep, slab against the
        // other): even-width planes of one per CTA beyond one row per thread stay
        // with k_sweeps_resident (48x48: 5.3 against 5.0, 64x64: 7.1 against 7.05;
        // at one row 24x24: 2.0 against 3.6, 36x36: 3.3 against 4.0), whose pairs an
        // odd width does without (47x46: 5.3 against 6.8); even-width slabs of
        // several planes at five rows stay with the marching sweep (60x60x304: 17.6
        // against 16.4).
        if (s.nx % 2 == 0 && ((G == 1 && K > 1 && s.resident) || (G > 1 && K == kSlabMaxK))) return cudaSuccess;
        // its start (tables, S) takes about 5 us longer than k_sweeps_resident's: a
        // step of few sweeps does not earn that back
        if (s.resident && s.units.n_mag < 24) return cudaSuccess;
        if (!s.resident) {
            double split = 0.0;
            const cudaError_t e = split_us(s, &split);
            if (e != cudaSuccess) return e;
            // (the estimates are within some 5 %)
            if (slab_us(s, K, G * slab_pairs(s.nx) * ((s.ny + K - 1) / K), G) > 1.05 * split) return cudaSuccess;
        }
        const int R = s.ib.max_ring, S = s.ib.max_shell;
        int more = 0;
        for (int i = 0; i < S; ++i) more += std::max(0, s.hib.csr_off[i + 1] - s.hib.csr_off[i] - 4);
        const size_t smem = slab_direct_smem_bytes(s.nx, s.ny, G, R, S, more);
        if (smem + 1024 > (size_t)optin) return cudaSuccess;
        const auto kern = slab_kernel(K);
        cudaError_t e = allow_smem((const void*)kern, smem);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return cudaSuccess;
        }
        int per_sm = 0;
        // a thread per column of rows, and enough for a marker component or a
        // shell node each
        const int columns = G * slab_pairs(s.nx) * ((s.ny + K - 1) / K);
        const int threads = std::min(kSlabThreads, (std::max(columns, std::max(3 * G * R, G * S)) + 31) / 32 * 32);
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        if (e != cudaSuccess) return e;
        if ((long long)per_sm * sms < ctas) return cudaSuccess;
        s.slab_ctas = ctas;
        s.slab_rows = K;
        s.slab_threads = threads;
        s.slab_more = more;
        s.slab_xbytes = (size_t)ctas * 4 * slab_msg_floats(s.nx, s.ny, G, K);
        s.resident_smem = smem;
        return cudaSuccess;
    }

    static auto resident64_kernel(const State& s) {
        return s.nx * s.ny <= 8 * kRes64Threads ? k_sweeps_resident64<T, 8> : k_sweeps_resident64<T, kRes64MaxNpt>;
    }

    // FP64: one plane per CTA in 3-D, one thread-block cluster in 2-D.
    static void launch_resident64(State& s, int nsweeps, const SweepCoef<T>& c, const IBView<T>& v,
                                  cudaStream_t st) {
        cudaLaunchConfig_t cfg = {};
        cfg.stream = st;
        cfg.dynamicSmemBytes = s.resident_smem;
        cudaLaunchAttribute attr[1];
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const T* bin = (const T*)s.b[s.bcur];
        T* bout = (T*)s.b[1 - s.bcur];
        const T* u = (const T*)s.u[s.fcur];
        cudaError_t e;
        if (s.dim == 3) {
            cfg.gridDim = dim3((unsigned)s.nz);
            cfg.blockDim = dim3(kRes64Threads);
            attr[0].id = cudaLaunchAttributeCooperative;
            attr[0].val.cooperative = 1;
            e = cudaLaunchKernelEx(&cfg, resident64_kernel(s), geo(s), bin, bout, u, c, v, (T*)s.xbuf,
                                   (ResidentSync*)s.rsync, nsweeps, s.ib.max_ring, s.ib.max_shell);
        } else {
            cfg.gridDim = dim3((unsigned)s.c2_ctas);
            cfg.blockDim = dim3(kC2Threads);
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)s.c2_ctas;
            attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            const C2Geo g{s.nx, s.ny, s.c2_rows, s.c2_mk, s.c2_sh, s.c2_nnz};
            e = cudaLaunchKernelEx(&cfg, k_sweeps_cluster64<T>, g, bin, bout, u, c, v, nsweeps);
        }
        if (e != cudaSuccess) s.launch_error = true;
    }

    static void launch_resident(State& s, int nsweeps, const SweepCoef<T>& c, const IBView<T>& v,
                                cudaStream_t st) {
        if constexpr (sizeof(T) == 8) {
            if (s.dim == 3 || s.c2_ctas > 0) {
                launch_resident64(s, nsweeps, c, v, st);
                return;
            }
        }
        if constexpr (sizeof(T) == 4) {
            if (s.slab_ctas > 0) {
                launch_slab(s, nsweeps, c, v, st);
                return;
            }
        }
        const bool small = small_plane(s);
        if constexpr (sizeof(T) == 4) if (s.dim == 3) {
            if (s.resident_uhalo) {
                if (small)
                    resident_launch_one<3, true, true>(s, nsweeps, c, v, st);
                else
                    resident_launch_one<3, true, false>(s, nsweeps, c, v, st);
            } else {
                if (small)
                    resident_launch_one<3, false, true>(s, nsweeps, c, v, st);
                else
                    resident_launch_one<3, false, false>(s, nsweeps, c, v, st);
            }
            return;
        }
        if (small)
            resident_launch_one<2, false, true>(s, nsweeps, c, v, st);
        else
            resident_launch_one<2, false, false>(s, nsweeps, c, v, st);
    }

    template <int DIM, bool UHALO, bool SMALL>
    static cudaError_t try_resident_shape(State& s, size_t smem, bool& ok) {
        constexpr int RT = ResidentShape<T, SMALL>::threads, NPT = ResidentShape<T, SMALL>::npt;
        ok = false;
        auto kern = k_sweeps_resident<T, DIM, UHALO, RT, NPT, false>;
        auto kern2 = k_sweeps_resident<T, DIM, UHALO, RT, NPT, true>;
        cudaError_t e = allow_smem((const void*)kern, smem);
        if (e == cudaSuccess) e = allow_smem((const void*)kern2, smem);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return cudaSuccess;  // too much shared memory: not resident
        }
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, RT, smem);
        if (e != cudaSuccess) return e;
        int dev = 0, sms = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        ok = per_sm >= 1 && (long long)per_sm * sms >= s.nz;
        return cudaSuccess;
    }

    template <int DIM, bool UHALO>
    static cudaError_t try_resident(State& s, size_t smem, bool& ok) {
        if (small_plane(s)) return try_resident_shape<DIM, UHALO, true>(s, smem, ok);
        return try_resident_shape<DIM, UHALO, false>(s, smem, ok);
    }

    // The pair kernel serves FP32 3-D domains, but not odd widths in an in-plane field:
    // two scalar accesses per pair for the field too (87x86x255 32.4 us a sweep with one
    // node per thread, 34.5 in pairs; 96x96x298, even, 47.4 and 38.5).
    static bool pair_march(const State& s) { return sizeof(T) == 4 && s.dim == 3 && (s.nx % 2 == 0 || !s.bext_xy); }
    static void sweep_plan(const State& s, qslbm_sweep_plan_t* out) {
        if (s.resident && s.slab_ctas > 0)
            *out = {QSLBM_KERNEL_SLAB, s.slab_ctas, s.slab_threads, s.slab_rows,
                    (s.nz + s.slab_ctas - 1) / s.slab_ctas};
        else if (s.resident && s.c2_ctas > 0)
            *out = {QSLBM_KERNEL_CLUSTER64, s.c2_ctas, kC2Threads, s.c2_rows, 1};
        else if (s.resident && sizeof(T) == 8 && s.dim == 3)
            *out = {QSLBM_KERNEL_RESIDENT64, s.nz, kRes64Threads, 0, 1};
        else if (s.resident)
            *out = {QSLBM_KERNEL_RESIDENT, s.nz,
                    small_plane(s) ? ResidentShape<T, true>::threads : ResidentShape<T, false>::threads, 0, 1};
        else if (s.fused)
            *out = {QSLBM_KERNEL_FUSED, s.fu_bands * s.fu_chunks, s.fu_threads, s.fu_TY, s.fu_chunk};
        else if (s.p.sweep_kernel != QSLBM_SWEEP_SPLIT)
            *out = {QSLBM_KERNEL_PLANES, s.nz, kPlaneThreads, 0, 1};
        else if (s.dim == 2)
            *out = {QSLBM_KERNEL_NODES, (s.nx * s.ny + kNodeThreads - 1) / kNodeThreads, kNodeThreads, 0, 1};
        else {
            const bool pair = s.march_rows > 0;
            const int tx = pair ? 2 * kPairTXP : kMarchTX, ty = pair ? 8 * s.march_rows : kMarchTY;
            *out = {pair ? QSLBM_KERNEL_MARCH_PAIR : QSLBM_KERNEL_MARCH,
                    ((s.nx + tx - 1) / tx) * ((s.ny + ty - 1) / ty) * ((s.nz + s.march_chunk - 1) / s.march_chunk),
                    pair ? kPairThreads : kMarchTX * kMarchTY, s.march_rows, s.march_chunk, s.ib_early};
        }
    }
    static auto pair_kernel(bool xy, int rows) {
        return rows == 1 ? (xy ? k_sweep_march_pair<T, true, 1> : k_sweep_march_pair<T, false, 1>)
                         : (xy ? k_sweep_march_pair<T, true, 2> : k_sweep_march_pair<T, false, 2>);
    }
    // z planes per CTA such that a grid of tiles of tx x ty columns fills one wave of
    // the kernel's resident CTAs (`share`: of which so many such grids run at a time),
    // at least `least`.
    static cudaError_t wave_chunk(const State& s, const void* kern, int threads, int tx, int ty, int least, int share,
                                  int& chunk) {
        int dev = 0, sms = 0, per_sm = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0);
        const long long tiles = (long long)((s.nx + tx - 1) / tx) * ((s.ny + ty - 1) / ty);
        const long long slots = (long long)std::max(1, per_sm) * std::max(1, sms) / share;
        const long long per_column = std::max<long long>(1, slots / tiles);
        chunk = (int)std::min<long long>(std::max<long long>((s.nz + per_column - 1) / per_column, least), s.nz);
        return e;
    }

    // The pair sweep's rows per thread and planes per CTA, on a domain that shares the
    // device with share - 1 others: one wave either way.  Two rows (chunk c2) where a
    // CTA's chunk is of four planes or more; below, the time is that of one CTA's chain
    // of planes, and a plane costs one row a thread (chunk c1) about 0.7 of what it costs
    // two.  Sweep alone, us: 64x64x128 c2 = 3 6.2, c1 = 4 6.0; 48x48x128 c2 = 2 5.0, c1 =
    // 3 5.1; 128x128x16 c2 = 2 4.9, c1 = 2 4.0; 40x40x300 c2 = 4 7.5, c1 = 5 8.1 (chunks of
    // at least four planes: 7.4, 7.6, 7.7, 7.5).  A grid that would need more than four
    // planes only because of the others keeps four.
    static cudaError_t pair_shape(const State& s, int share, int* rows, int* chunk) {
        if constexpr (sizeof(T) == 4) {
            const bool xy = s.bext_xy != nullptr;
            const void *k1 = (const void*)pair_kernel(xy, 1), *k2 = (const void*)pair_kernel(xy, 2);
            int c1 = 1, c2 = 1, alone = 1;
            cudaError_t e = wave_chunk(s, k2, kPairThreads, 2 * kPairTXP, kPairTY<2>, 1, 1, alone);
            if (e == cudaSuccess) e = wave_chunk(s, k2, kPairThreads, 2 * kPairTXP, kPairTY<2>, 1, share, c2);
            if (e == cudaSuccess) e = wave_chunk(s, k1, kPairThreads, 2 * kPairTXP, kPairTY<1>, 1, share, c1);
            c2 = std::min(c2, std::max(alone, 4));
            // (a grid has at most 65535 tiles of rows)
            *rows = c2 < 4 && 10 * c1 <= 14 * c2 && s.ny <= 65535LL * kPairTY<1> ? 1 : 2;
            *chunk = *rows == 1 ? c1 : c2;
            return e;
        }
        return cudaErrorNotSupported;  // FP64 has no pair sweep
    }

    // The marching sweep's planes per CTA and, for pairs, rows per thread.
    static cudaError_t plan_march(State& s) {
        cudaError_t e;
        if (pair_march(s)) {
            e = pair_shape(s, 1, &s.march_rows, &s.march_chunk);
        } else {
            const void* kern = (const void*)k_sweep_march<T, true>;
            if constexpr (sizeof(T) == 8)
                if (!s.bext_xy) kern = (const void*)k_sweep_march<T, false>;
            // (at least four planes, to keep the z halo's share small)
            e = wave_chunk(s, kern, kMarchTX * kMarchTY, kMarchTX, kMarchTY, 4, 1, s.march_chunk);
            s.march_rows = 0;
        }
        if (e == cudaSuccess) e = plan_flow(s);
        if (e != cudaSuccess) return e;
        // the staged IB corrector, when the plane's shell fits shared memory
        // and the shell nodes' marker lists are padded
        s.ib_staged_smem = 0;
        if (s.ib.nm > 0 && s.ib.pad_k > 0) {
            const size_t smem = ib_staged_smem_bytes<T>(s.ib.max_ring, s.ib.max_shell);
            int dev = 0, sms = 0, max_optin = 0;
            e = cudaGetDevice(&dev);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
            if (e != cudaSuccess) return e;
            if (smem <= (size_t)max_optin) {
                s.ib_staged_u = ib_staged_unroll(s.ib.max_shell, s.nz, sms);
                const int U = s.ib_staged_u;
                const auto kern = U == 1   ? k_ib_staged<T, 1>
                                  : U == 2 ? k_ib_staged<T, 2>
                                  : U == 4 ? k_ib_staged<T, 4>
                                           : k_ib_staged<T, 5>;
                e = allow_smem((const void*)kern, smem);
                if (e != cudaSuccess) return e;
                s.ib_staged_smem = smem;
                // Early CTAs gather on the SMs whose sweep CTAs end first, two and more to
                // an SM: where the planes have an SM each, spreading them is worth more
                // than the earlier start (us a sweep, early / not: 99x99x64 16.6 / 14.3,
                // 96x96x40 12.1 / 9.3, 128x128x60 23.6 / 17.3, 64x64x128 10.6 / 9.6; with
                // more planes than SMs 40x40x192 8.6 / 9.3, 96x96x512 48.8 / 51.7).
                s.ib_early = s.nz > sms;
            }
        }
        return cudaSuccess;
    }

    // FP64, 3-D: shared memory for b, e and the IB tables, every plane's CTA
    // co-resident.
    static cudaError_t try_resident64(State& s, size_t smem, int sms, bool& ok) {
        ok = false;
        if ((long long)s.nx * s.ny > (long long)kRes64Threads * kRes64MaxNpt) return cudaSuccess;
        const auto kern = resident64_kernel(s);
        if (allow_smem((const void*)kern, smem) != cudaSuccess) {
            cudaGetLastError();
            return cudaSuccess;
        }
        int per_sm = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kRes64Threads, smem);
        if (e != cudaSuccess) return e;
        ok = per_sm >= 1 && (long long)per_sm * sms >= s.nz;
        return cudaSuccess;
    }

    // FP64, 2-D: the plane's rows over the CTAs of one cluster, the largest
    // cluster (at most 16) that the device can hold with a row or more per
    // CTA: one SM does about two FP64 operations per clock, so the sweep time
    // falls nearly with the CTA count.
    static cudaError_t plan_cluster2d(State& s, int optin) {
        s.c2_ctas = 0;
        const HostIB& h = s.hib;
        const int R = s.ib.max_ring, S = s.ib.max_shell;
        for (int C = kC2MaxCluster; C >= 1; C /= 2) {
            if (C > s.ny) continue;
            const int RB = (s.ny + C - 1) / C;
            int mk = 1, sh = 1, nnz = 1;
            for (int r = 0; r * RB < s.ny; ++r) {
                const int y0 = r * RB, y1 = std::min(y0 + RB, s.ny);
                int m = 0, k = 0, e = 0;
                for (int j = 0; j < R; ++j) {
                    bool own = false;
                    for (int b = 0; b < 3; ++b) own = own || (h.iy[3 * j + b] >= y0 && h.iy[3 * j + b] < y1);
                    m += own;
                }
                for (int i = 0; i < S; ++i) {
                    const int y = h.shell_xy[i] / s.nx;
                    if (y >= y0 && y < y1) {
                        ++k;
                        e += h.csr_off[i + 1] - h.csr_off[i];
                    }
                }
                mk = std::max(mk, m);
                sh = std::max(sh, k);
                nnz = std::max(nnz, e);
            }
            const size_t smem = cluster2d_smem_bytes(s.nx, RB, R, mk, sh, nnz);
            if (smem + 1024 > (size_t)optin) continue;
            cudaError_t e = cudaSuccess;
            if (C > 8) e = cudaFuncSetAttribute(k_sweeps_cluster64<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e == cudaSuccess)
                e = allow_smem((const void*)k_sweeps_cluster64<T>, smem);
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)C);
            cfg.blockDim = dim3(kC2Threads);
            cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)C;
            attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int clusters = 0;
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, k_sweeps_cluster64<T>, &cfg);
            if (e != cudaSuccess) {
                cudaGetLastError();
                continue;
            }
            if (clusters < 1) continue;
            s.c2_ctas = C;
            s.c2_rows = RB;
            s.c2_mk = mk;
            s.c2_sh = sh;
            s.c2_nnz = nnz;
            s.resident_smem = smem;
            return cudaSuccess;
        }
        return cudaSuccess;
    }

    // FP32, 3-D: the slab kernel wherever it fits.  A handle that asks for the
    // resident kernel by name gets it where one plane per CTA fits the device
    // (and no in-plane field is applied), as before the slab kernel.
    static cudaError_t plan_resident(State& s) {
        const cudaError_t e = plan_planes(s);
        if constexpr (sizeof(T) == 4) {
            if (e != cudaSuccess || (!s.resident && s.p.sweep_kernel == QSLBM_SWEEP_RESIDENT)) return e;
            int dev = 0, optin = 0, sms = 0;
            cudaError_t f = cudaGetDevice(&dev);
            if (f == cudaSuccess) f = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
            if (f == cudaSuccess) f = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (f == cudaSuccess) f = plan_slab(s, optin, sms);
            if (s.slab_ctas > 0) s.resident = true;
            return f;
        }
        return e;
    }

    // One plane per CTA (k_sweeps_resident, k_sweeps_resident64) or, in FP64
    // and 2-D, one cluster.
    static cudaError_t plan_planes(State& s) {
        s.resident = false;
        const long long P = (long long)s.nx * s.ny;
        if (P > (long long)kResidentMaxPlane) return cudaSuccess;
        if (s.bext_xy) return cudaSuccess;  // an in-plane applied field takes the split path
        int dev = 0, optin = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess)
            return e;
        const size_t base = resident_smem_bytes<T>((int)P, false, s.ib.max_ring, s.ib.max_shell, s.ib.max_nnz);
        const size_t halo = (size_t)6 * P * sizeof(T);
        const size_t reserve = 1024;  // static shared variables and the runtime's own share
        bool ok = false;
        if constexpr (sizeof(T) == 8) {
            if (s.dim == 2) {
                if ((e = plan_cluster2d(s, optin)) != cudaSuccess) return e;
                s.resident = s.c2_ctas > 0;
                if (s.resident) return cudaSuccess;
            } else {
                int sms = 0;
                if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
                const size_t smem = resident64_smem_bytes((int)P, s.ib.max_ring, s.ib.max_shell, s.ib.max_nnz);
                if (smem + reserve > (size_t)optin) return cudaSuccess;
                if ((e = try_resident64(s, smem, sms, ok)) != cudaSuccess) return e;
                s.resident = ok;
                s.resident_smem = smem;
                return cudaSuccess;
            }
        }
        if (sizeof(T) == 4 && s.dim == 3 && base + halo + reserve <= (size_t)optin) {
            if constexpr (sizeof(T) == 4)
                if ((e = try_resident<3, true>(s, base + halo, ok)) != cudaSuccess) return e;
            if (ok) {
                s.resident = true;
                s.resident_uhalo = true;
                s.resident_smem = base + halo;
                return cudaSuccess;
            }
        }
        if (base + reserve > (size_t)optin) return cudaSuccess;
        if (s.dim == 2)
            e = try_resident<2, false>(s, base, ok);
        else if constexpr (sizeof(T) == 4)
            e = try_resident<3, false>(s, base, ok);
        if (e != cudaSuccess) return e;
        if (ok) {
            s.resident = true;
            s.resident_uhalo = false;
            s.resident_smem = base;
        }
        return cudaSuccess;
    }

    static void force_flow(State& s, cudaStream_t st) {
        ForceCoef<T> fc;
        fc.F0 = s.units.F0;
        fc.amp = s.p.force_amp;
        fc.omega = s.omega;
        fc.axis = s.axis;
        for (int a = 0; a < 3; ++a) fc.be[a] = (T)s.be[a];
        fc.bext_z = static_cast<const T*>(s.bext_z);
        fc.bext_xy = static_cast<const T*>(s.bext_xy);
        FlowCoef<T> c;
        c.tau = (T)s.units.tau;
        c.kforce = (T)(1.0 - 1.0 / (2.0 * s.units.tau));
        c.mac = s.p.flow_scheme == QSLBM_FLOW_MACROSCOPIC;
        c.ig = (T)s.ig;
        c.ig2 = (T)(s.ig * s.ig);
        const IBView<T> v = view(s, false);
        const T* b = (const T*)s.b[s.bcur];
        const T* dr = (const T*)s.drho[s.fcur];
        const T* u = (const T*)s.u[s.fcur];
        T* dro = (T*)s.drho[1 - s.fcur];
        T* uo = (T*)s.u[1 - s.fcur];
        T* F = (T*)s.F;
        if (s.dim == 2) {
            const int blocks = (s.nx * s.ny + kFlowNodeThreads - 1) / kFlowNodeThreads;
            k_force_nodes<T, 9><<<blocks, kFlowNodeThreads, 0, st>>>(geo(s), b, F, fc, s.tdev);
            k_flow_nodes<T, 9><<<blocks, kFlowNodeThreads, 0, st>>>(geo(s), dr, u, F, dro, uo, c, s.tdev);
        } else {
            const int chunk = s.flow_chunk;
            const unsigned grid = (unsigned)((s.nx + kFlowTX - 1) / kFlowTX) *
                                  (unsigned)((s.ny + kFlowTY<T> - 1) / kFlowTY<T>) *
                                  (unsigned)((s.nz + chunk - 1) / chunk);
            constexpr int threads = kFlowThreads<T>;
            // Short CTAs start as those of the kernel before them end; longer ones crowd the
            // SMs that are done first (us a step of one sweep, early / not: 16^3 16.9 / 18.9,
            // 40x40x64 26.3 / 27.8, 40x40x192 in chunks of four 39.0 / 38.3, 96x96x512 204.7
            // / 198.6), and FP64's are long anyway.
            const bool early = sizeof(T) == 4 && chunk <= 2;
            if (s.units.flow_q == 27) {
                launch_pdl(k_force_march<T, 27>, dim3(grid), dim3(threads), 0, st, early, geo(s), b, F, fc,
                           (const long long*)s.tdev, chunk, early);
                launch_pdl(k_flow_march<T, 27>, dim3(grid), dim3(threads), 0, st, early, geo(s), dr, u, (const T*)F, dro,
                           uo, c, s.tdev, chunk, early);
            } else {
                launch_pdl(k_force_march<T, 19>, dim3(grid), dim3(threads), 0, st, early, geo(s), b, F, fc,
                           (const long long*)s.tdev, chunk, early);
                launch_pdl(k_flow_march<T, 19>, dim3(grid), dim3(threads), 0, st, early, geo(s), dr, u, (const T*)F, dro,
                           uo, c, s.tdev, chunk, early);
            }
        }
        if (s.ib.nm > 0 && s.ib_staged_smem > 0)
            launch_ib_staged(s, uo, v, true, st);
        else if (s.ib.nm > 0)
            k_ib_planes<T><<<s.nz, kNodeThreads, ib_smem(s), st>>>(geo(s), uo, v);
        s.fcur ^= 1;
    }

    static ObsCoef<T> obs_coef(const State& s, double fb) {
        ObsCoef<T> c;
        c.eta = s.units.eta;
        c.fb = fb;
        c.axis = s.axis;
        c.geometry = s.p.geometry;
        c.strict_qs = s.p.strict_qs;
        c.dim = s.dim;
        c.cx = s.cx;
        c.cy = s.cy;
        c.rin = s.R - 2.0;
        for (int a = 0; a < 3; ++a) c.be[a] = (T)s.be[a];
        c.bext_z = static_cast<const T*>(s.bext_z);
        c.bext_xy = static_cast<const T*>(s.bext_xy);
        return c;
    }

    static void observe_fields(const State& s, const void* drho, const void* u, const void* b, const void* usnap,
                               double fb, int blocks, double* partial, double* sums, cudaStream_t st) {
        const ObsCoef<T> c = obs_coef(s, fb);
        const T* dr = (const T*)drho;
        const T* uu = (const T*)u;
        const T* bb = (const T*)b;
        const T* us = (const T*)usnap;
        if (s.dim == 3 && s.units.flow_q == 27)
            k_observe<T, 3, 27><<<blocks, kReduceThreads, 0, st>>>(geo(s), dr, uu, bb, us, c, partial);
        else if (s.dim == 3)
            k_observe<T, 3><<<blocks, kReduceThreads, 0, st>>>(geo(s), dr, uu, bb, us, c, partial);
        else
            k_observe<T, 2><<<blocks, kReduceThreads, 0, st>>>(geo(s), dr, uu, bb, us, c, partial);
        k_fold<T><<<1, 32 * kObs, 0, st>>>(partial, blocks, sums);
    }

    static void observe(State& s, double fb, cudaStream_t st) {
        observe_fields(s, s.drho[s.fcur], s.u[s.fcur], s.b[s.bcur], s.usnap, fb, s.nblocks_obs, s.partial,
                       s.obs_dev, st);
    }

    static void to_f64(State& s, cudaStream_t st) {
        k_to_f64<T><<<grid_for(s.n, 256), 256, 0, st>>>(s.n, (const T*)s.drho[s.fcur], (const T*)s.u[s.fcur],
                                                        (const T*)s.b[s.bcur], s.staging);
    }

    static void from_f64(State& s, int mask, cudaStream_t st) {
        k_from_f64<T><<<grid_for(s.n, 256), 256, 0, st>>>(s.n, s.staging, (T*)s.drho[s.fcur], (T*)s.u[s.fcur],
                                                          (T*)s.b[s.bcur], mask);
    }

    static const Ops& table() {
        static const Ops o = {&init,     &sweeps,        &force_flow, &observe,     &observe_fields,
                              &to_f64,   &from_f64,      &plan_resident, &plan_march, &pair_shape, &sweep_plan,
                              &plan_fused, &tune_fused};
        return o;
    }
};

}  // namespace qslbm
