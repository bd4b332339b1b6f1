// usp_kernels.cu -- sm_103a kernels of the plain (one kernel per stage)
// USP-ESBGK step.  Each kernel walks a device-resident tile table, so the
// same launches serve one simulation or a batch of them and stay valid when
// captured in a CUDA graph.
//
// Stage order of one step n (Table 2 of the paper, unit particle weights):
//   k_stream   advection + boundaries, new cell, cell histogram,    (Table 2 step 3)
//              net count through the counting plane                 (Eq. 41)
//   k_scan     exclusive scan of the histogram                      (counting sort)
//   k_scatter  particles to their sorted slots                      (counting sort)
//   k_inject   refill of reservoir buffer cells
//   k_moments  per-cell sums of shifted velocities                  (Eq. 1)
//   k_params   per-cell P_ne, sigma*, q*, Cholesky, fields, Eq. 34  (Eqs. 16-18, 33, 35-36, 6c)
//   k_relax    Bernoulli or fixed-count selection, ES Gaussian or   (Eqs. 8b, 9, 27, 29-32,
//              Gallis-Torczynski sampling, conservation              10-11)
//   k_finish   advance the step counter and swap buffers
#include <algorithm>

#include "usp_device.cuh"

#include <cstdio>

namespace usp {

// ---------------------------------------------------------------------------
// K1: advection, new cell, histogram
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(kPUnit) k_stream(const SimDev* __restrict__ sims, const int2* __restrict__ tiles,
                                                const int* __restrict__ ntiles) {
    __shared__ SimDev sim_sh;
    const int nu = *ntiles * (kPTile / kPUnit);
    int loaded = -1;
    for (int t = blockIdx.x; t < nu; t += gridDim.x) {
        const int2 tile = unit_of(tiles, t);
        if (tile.x != loaded) {
            __syncthreads();
            load_sim(sim_sh, sims[tile.x]);
            __syncthreads();
            loaded = tile.x;
        }
        const SimDev& s = sim_sh;
        const uint32_t n = s.dyn->n;
        const uint32_t step = s.dyn->step;
        const int cur = s.dyn->cur;
        PView<T> P = view<T>(s, cur);
        const int64_t i = (int64_t)tile.y + threadIdx.x;
        if (i < (int64_t)n) {
            T x = s.dim == 2 ? P.x[i] : (T)0;
            T y = P.y[i];
            T c[3] = {P.c0[i], P.c1[i], P.c2[i]};
            const uint32_t pid = P.pid[i];
            const T x0 = x, y0 = y;
            bool alive = true;
            if (!advect_clear<T>(s, x, y, c)) alive = advect<T>(s, step, pid, x, y, c);
            if (s.flux_axis) count_flux<T>(s, x0, y0, x, y);
            int cell = s.K;
            if (alive) {
                cell = cell_index<T>(s, x, y);
                if (in_buffer(s, cell)) {
                    cell = s.K;
                    atomicAdd(&s.dyn->counters[kCntRemoved], 1ull);
                }
            }
            if (s.dim == 2) P.x[i] = x;
            P.y[i] = y;
            P.c0[i] = c[0];
            P.c1[i] = c[1];
            P.c2[i] = c[2];
            s.cell[i] = (uint32_t)cell;
            if (cell < s.K) aggregated_add(s.count, (uint32_t)cell);
        }
    }
}

// cell of every particle without moving it (ordering an arbitrary loaded state)
template <class T>
__global__ void __launch_bounds__(kPUnit) k_assign(const SimDev* __restrict__ sims, const int2* __restrict__ tiles,
                                                const int* __restrict__ ntiles) {
    __shared__ SimDev sim_sh;
    const int nu = *ntiles * (kPTile / kPUnit);
    int loaded = -1;
    for (int t = blockIdx.x; t < nu; t += gridDim.x) {
        const int2 tile = unit_of(tiles, t);
        if (tile.x != loaded) {
            __syncthreads();
            load_sim(sim_sh, sims[tile.x]);
            __syncthreads();
            loaded = tile.x;
        }
        const SimDev& s = sim_sh;
        const uint32_t n = s.dyn->n;
        PView<T> P = view<T>(s, s.dyn->cur);
        const int64_t i = (int64_t)tile.y + threadIdx.x;
        if (i < (int64_t)n) {
            // local cell of a slab (row0 = 0 without a decomposition),
            // clamped into the slab's cell range
            const int cell = min(max(cell_index<T>(s, s.dim == 2 ? P.x[i] : (T)0, P.y[i]) - s.row0 * s.nx, 0),
                                 s.K - 1);
            s.cell[i] = (uint32_t)cell;
            aggregated_add(s.count, (uint32_t)cell);
        }
    }
}

// ---------------------------------------------------------------------------
// K2: per-simulation exclusive scan of counts (+ injected) -> start
// ---------------------------------------------------------------------------
// with_inj: leave room for the reservoir refill of the step (the plain step);
// 0 when a loaded state is only being sorted (fused set-up)
__global__ void __launch_bounds__(1024) k_scan(const SimDev* __restrict__ sims, int nsims, int with_inj) {
    __shared__ uint32_t warp_sums[32];
    __shared__ uint32_t carry;
    for (int si = blockIdx.x; si < nsims; si += gridDim.x) {
        const SimDev& s = sims[si];
        const int K = s.K;
        if (threadIdx.x == 0) carry = 0;
        __syncthreads();
        for (int base = 0; base <= K; base += blockDim.x) {
            const int c = base + threadIdx.x;
            uint32_t v = 0;
            if (c < K) {
                v = s.count[c] + (with_inj && s.has_reservoir ? s.inj_count[c] : 0u);
                s.count[c] = 0;
            } else if (c == K) {
                s.count[c] = 0;   // removed particles are not kept
            }
            // inclusive warp scan
            uint32_t x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if ((threadIdx.x & 31) >= o) x += y;
            }
            if ((threadIdx.x & 31) == 31) warp_sums[threadIdx.x >> 5] = x;
            __syncthreads();
            if (threadIdx.x < 32) {
                uint32_t ws = threadIdx.x < (blockDim.x >> 5) ? warp_sums[threadIdx.x] : 0u;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    uint32_t y = __shfl_up_sync(0xffffffffu, ws, o);
                    if (threadIdx.x >= o) ws += y;
                }
                warp_sums[threadIdx.x] = ws;
            }
            __syncthreads();
            const uint32_t before = (threadIdx.x >= 32 ? warp_sums[(threadIdx.x >> 5) - 1] : 0u) + carry;
            if (c <= K) s.start[c] = before + x - v;
            __syncthreads();
            if (threadIdx.x == blockDim.x - 1) carry = before + x;
            __syncthreads();
        }
        if (threadIdx.x == 0) s.start[K + 1] = carry;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// K3: scatter to sorted slots
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(kPUnit) k_scatter(const SimDev* __restrict__ sims, const int2* __restrict__ tiles,
                                                 const int* __restrict__ ntiles) {
    __shared__ SimDev sim_sh;
    const int nu = *ntiles * (kPTile / kPUnit);
    int loaded = -1;
    for (int t = blockIdx.x; t < nu; t += gridDim.x) {
        const int2 tile = unit_of(tiles, t);
        if (tile.x != loaded) {
            __syncthreads();
            load_sim(sim_sh, sims[tile.x]);
            __syncthreads();
            loaded = tile.x;
        }
        const SimDev& s = sim_sh;
        const uint32_t n = s.dyn->n;
        const int cur = s.dyn->cur;
        PView<T> A = view<T>(s, cur), B = view<T>(s, cur ^ 1);
        const int64_t i = (int64_t)tile.y + threadIdx.x;
        if (i < (int64_t)n) {
            const uint32_t cell = s.cell[i];
            if (cell >= (uint32_t)s.K) continue;   // (the block's other threads take theirs)
            const uint32_t slot = s.start[cell] + aggregated_add(s.fill, cell);
            if ((int64_t)slot >= s.cap) {
                atomicAdd(&s.dyn->counters[kCntOverflow], 1ull);
                continue;
            }
            if (s.dim == 2) B.x[slot] = A.x[i];
            B.y[slot] = A.y[i];
            B.c0[slot] = A.c0[i];
            B.c1[slot] = A.c1[i];
            B.c2[slot] = A.c2[i];
            B.pid[slot] = A.pid[i];
        }
    }
}

// ---------------------------------------------------------------------------
// K4: reservoir buffer cells: fresh particles from the reservoir Maxwellian
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(256) k_inject(const SimDev* __restrict__ sims, const int2* __restrict__ tiles,
                                                const int* __restrict__ ntiles) {
    __shared__ SimDev sim_sh;
    const int nt = *ntiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int t = blockIdx.x; t < nt; t += gridDim.x) {
        const int2 tile = tiles[t];
        __syncthreads();
        load_sim(sim_sh, sims[tile.x]);
        __syncthreads();
        const SimDev& s = sim_sh;
        if (!s.has_reservoir) continue;
        const uint32_t step = s.dyn->step, next_pid = s.dyn->next_pid;
        PView<T> B = view<T>(s, s.dyn->cur ^ 1);
        for (int cc = warp; cc < kCTile; cc += nwarps) {
            const int cell = tile.y + cc;
            if (cell >= s.K) break;
            const uint32_t cnt = s.inj_count[cell];
            if (cnt == 0) continue;
            const int f = buffer_face(s, cell);
            const FaceDev& F = s.face[f];
            const uint32_t base = s.start[cell] + s.fill[cell];
            for (uint32_t k = lane; k < cnt; k += 32) {
                const uint32_t slot = base + k;
                if ((int64_t)slot >= s.cap) {
                    atomicAdd(&s.dyn->counters[kCntOverflow], 1ull);
                    continue;
                }
                const uint32_t pid = next_pid + s.inj_pidoff[cell] + k;
                T x, y, c[3];
                make_particle<T>(s, cell, pid, step, kInject, F.theta, F.u, x, y, c);
                if (s.dim == 2) B.x[slot] = x;
                B.y[slot] = y;
                B.c0[slot] = c[0];
                B.c1[slot] = c[1];
                B.c2[slot] = c[2];
                B.pid[slot] = pid;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// K5: per-cell sums of velocities shifted by the previous cell mean (Eq. 1)
// ---------------------------------------------------------------------------
// src_cur: the sums of the current buffer (the weighted step's moments of
// f^n) instead of the sorted one; with weighted particles every sum is
// W-weighted and the cell's weight sum goes to wneff
// One warp per block, the blocks striding over single cells: the FP64 sums
// are latency-bound, so even a domain of a hundred cells should spread
// over a hundred SMs.
template <class T>
__global__ void __launch_bounds__(32) k_moments(const SimDev* __restrict__ sims, const int2* __restrict__ tiles,
                                                const int* __restrict__ ntiles, int src_cur) {
    __shared__ SimDev sim_sh;
    const int nt = *ntiles;
    const int lane = threadIdx.x & 31;
    int loaded = -1;
    for (int g = blockIdx.x; g < nt * kCTile; g += gridDim.x) {
        const int2 tile = tiles[g / kCTile];
        if (tile.x != loaded) {
            __syncwarp();
            load_sim(sim_sh, sims[tile.x]);
            __syncwarp();
            loaded = tile.x;
        }
        const SimDev& s = sim_sh;
        const int K = s.K;
        const int buf = src_cur ? s.dyn->cur : s.dyn->cur ^ 1;
        PView<T> B = view<T>(s, buf);
        const double* Wt = s.weighted ? s.wgt[buf] : nullptr;
        const int cell = tile.y + g % kCTile;
        if (cell == 0 && lane == 0) s.fill[K] = 0;
        if (cell >= K) continue;
        {
            const uint32_t cap = (uint32_t)s.cap;
            const uint32_t b = min(s.start[cell], cap), e = min(s.start[cell + 1], cap);
            const double sh0 = s.ushift[cell], sh1 = s.ushift[K + cell], sh2 = s.ushift[2 * K + cell];
            double a[12], we = 0.0;
#pragma unroll
            for (int m = 0; m < 12; ++m) a[m] = 0.0;
            for (uint32_t i = b + lane; i < e; i += 32) {
                const double C0 = (double)B.c0[i] - sh0, C1 = (double)B.c1[i] - sh1, C2 = (double)B.c2[i] - sh2;
                const double c2 = C0 * C0 + C1 * C1 + C2 * C2;
                if (Wt) {
                    const double w = Wt[i];
                    we += w;
                    a[0] += w * C0; a[1] += w * C1; a[2] += w * C2;
                    a[3] += w * C0 * C0; a[4] += w * C1 * C1; a[5] += w * C2 * C2;
                    a[6] += w * C0 * C1; a[7] += w * C0 * C2; a[8] += w * C1 * C2;
                    a[9] += w * c2 * C0; a[10] += w * c2 * C1; a[11] += w * c2 * C2;
                    continue;
                }
                a[0] += C0; a[1] += C1; a[2] += C2;
                a[3] += C0 * C0; a[4] += C1 * C1; a[5] += C2 * C2;
                a[6] += C0 * C1; a[7] += C0 * C2; a[8] += C1 * C2;
                a[9] += c2 * C0; a[10] += c2 * C1; a[11] += c2 * C2;
            }
            // the twelve sums (and the weights') as a warp reduce-scatter: lane
            // 2 v ends with value v (16 FP64 additions instead of 60)
            double v[16];
#pragma unroll
            for (int m = 0; m < 12; ++m) v[m] = a[m];
            v[12] = we;
            v[13] = v[14] = v[15] = 0.0;
#pragma unroll
            for (int half = 8; half >= 1; half >>= 1) {
                const bool up = (lane & (2 * half)) != 0;
#pragma unroll
                for (int i = 0; i < half; ++i) {
                    const double send = up ? v[i] : v[i + half];
                    const double recv = __shfl_xor_sync(0xffffffffu, send, 2 * half);
                    v[i] = (up ? v[i + half] : v[i]) + recv;
                }
            }
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
            if ((lane & 1) == 0 && lane < 24) s.mom[(size_t)(lane / 2 + 1) * K + cell] = v[0];
            if (Wt && lane == 24) s.wneff[cell] = v[0];
            if (s.gloc) {
                // n, T and |u| for the neighbours' Kn_GLL
                double S[6];
#pragma unroll
                for (int m = 0; m < 6; ++m) S[m] = __shfl_sync(0xffffffffu, v[0], 2 * m);
                const double w = Wt ? __shfl_sync(0xffffffffu, v[0], 24) : (double)(e - b);
                double T = 0.0, um = 0.0;
                bool ok = false;
                if (e > b && w > 0.0) {
                    const double inv = 1.0 / w;
                    const double d0 = S[0] * inv, d1 = S[1] * inv, d2 = S[2] * inv;
                    const double th = ((S[3] * inv - d0 * d0) + (S[4] * inv - d1 * d1) + (S[5] * inv - d2 * d2)) *
                                      (1.0 / 3.0);
                    ok = e - b >= 2 && (!Wt || w > 1.0) && th > 0.0;
                    if (ok) {
                        const double u0 = sh0 + d0, u1 = sh1 + d1, u2 = sh2 + d2;
                        T = th * s.inv_R;
                        um = sqrt(u0 * u0 + u1 * u1 + u2 * u2);
                    }
                }
                if (lane == 0) store_grad_state(s, cell, ok, w * s.w, T, um);
            }
            if (lane == 0) {
                s.mom[cell] = (double)(e - b);
                s.fill[cell] = 0;
                if (gll_averaged(s)) snap_avg(s, cell);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// K6: per-cell USP parameters, fields and the Eq. 34 average
//
// A lane per cell, a warp per block: as long as one cell's chain of FP64
// instructions, about 20 us, on domains of a few thousand cells (100 cells: 30 us
// with plain divisions and the stencil's states formed again, 22 with loads
// where they were needed, 20 with all of them first; 4e4 cells 67 -> 56).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(32) k_params(const SimDev* __restrict__ sims, const int2* __restrict__ tiles,
                                               const int* __restrict__ ntiles) {
    __shared__ SimDev sim_sh;
    const int nt = *ntiles;
    for (int t = blockIdx.x; t < nt; t += gridDim.x) {
        const int2 tile = tiles[t];
        __syncthreads();
        load_sim(sim_sh, sims[tile.x]);
        __syncthreads();
        const SimDev& s = sim_sh;
        const int K = s.K;
        for (int cc = threadIdx.x; cc < kCTile; cc += blockDim.x) {
            const int cell = tile.y + cc;
            if (cell >= K) break;
            // every load of the cell first, as one round of latency (stores
            // to the fields would hold the averages' loads back one by one):
            // the running averages, the neighbours' stencil states, the sums
            const bool first = s.dyn->nsamples == 0;
            double av[kNFields];
#pragma unroll
            for (int k = 0; k < kNFields; ++k) av[k] = first ? 0.0 : s.avg[(size_t)k * K + cell];
            const bool avg = gll_averaged(s);
            GradState Nb[2][2];   // by axis and side
            bool has[2][2] = {{false, false}, {false, false}};
            if (s.mode == kModeUSP) {
#pragma unroll
                for (int axis = 0; axis < 2; ++axis) {
                    if (axis == 0 && s.dim == 1) continue;
#pragma unroll
                    for (int side = 0; side < 2; ++side) {
                        const int c = neighbor(s, cell, axis, side ? +1 : -1);
                        if (c < 0) continue;
                        if (avg) grad_from_avg(s, c, Nb[axis][side], false);
                        else load_grad_state(s, c, Nb[axis][side]);
                        has[axis][side] = Nb[axis][side].valid != 0;
                    }
                }
            }
            Local L;
            double P[6], Q[3];
            local_state(s, cell, L, P, Q);
            double f[kNFields];
            for (int k = 0; k < kNFields; ++k) f[k] = 0.0;
            f[0] = L.n;
            f[15] = L.N;
            if (L.N >= 1) {
                f[1] = L.u[0];
                f[2] = L.u[1];
                f[3] = L.u[2];
            }
            double* prm = s.prm;
            double pr[kNPrm];
            for (int k = 0; k < kNPrm; ++k) pr[k] = 0.0;
            pr[0] = L.u[0];
            pr[1] = L.u[1];
            pr[2] = L.u[2];
            pr[3] = L.theta;
            if (L.valid) {
                local_transport(s, L);
                double pne;
                if (s.mode == kModeSP || s.mode == kModeSPESBGK) pne = 0.0;
                else if (s.mode == kModeFixed) pne = s.fixed_pne;
                else {
                    // gradient-length local Knudsen number (Eqs. 17-18): central
                    // differences, one-sided next to a missing or invalid neighbour
                    GradState G;
                    if (avg) grad_from_avg(s, cell, G, true);
                    else grad_from_local(L, G);
                    double kn = 0.0;   // no stencil state of its own: no gradient
                    if (G.valid) {
                        const double Qc[3] = {G.n, G.T, G.umag};
                        double g2[3] = {0.0, 0.0, 0.0};
#pragma unroll
                        for (int axis = 0; axis < 2; ++axis) {
                            if (axis == 0 && s.dim == 1) continue;
                            const double ih = s.inv_d[axis];
                            const GradState &Gm = Nb[axis][0], &Gp = Nb[axis][1];
                            const int m = has[axis][0] ? 1 : -1, p = has[axis][1] ? 1 : -1;
                            double Qm[3], Qp[3];
                            if (m >= 0) { Qm[0] = Gm.n; Qm[1] = Gm.T; Qm[2] = Gm.umag; }
                            if (p >= 0) { Qp[0] = Gp.n; Qp[1] = Gp.T; Qp[2] = Gp.umag; }
                            for (int q = 0; q < 3; ++q) {
                                double d = 0.0;
                                if (m >= 0 && p >= 0) d = (Qp[q] - Qm[q]) * (0.5 * ih);
                                else if (p >= 0) d = (Qp[q] - Qc[q]) * ih;
                                else if (m >= 0) d = (Qc[q] - Qm[q]) * ih;
                                g2[q] += d * d;
                            }
                        }
                        // Eq. 17: lambda max over Q of |grad Q| / Q, in squares
                        const double r0 = 1.0 / G.n, r1 = 1.0 / G.T, r2 = 1.0 / fmax(G.umag, G.a_sound);
                        kn = G.lambda * sqrt(fmax(g2[0] * r0 * r0, fmax(g2[1] * r1 * r1, g2[2] * r2 * r2)));
                    }
                    pne = exp(kn * (-1.0 / kKnC));                           // Eq. 16
                }
                const double ifs = 1.0 / (1.0 + 0.5 * s.dt * L.nu * pne);   // Eq. 33
                const double ifq = 1.0 / (1.0 + 0.5 * s.dt * L.nu * s.Pr * pne);
                const double sig[6] = {(P[0] - L.theta) * ifs, (P[1] - L.theta) * ifs, (P[2] - L.theta) * ifs,
                                       P[3] * ifs, P[4] * ifs, P[5] * ifs};
                const double b = s.es_b;                                    // Eq. 6c: 1 - 1/Pr
                const double A00 = L.theta + b * sig[0], A11 = L.theta + b * sig[1], A22 = L.theta + b * sig[2];
                const double A10 = b * sig[3], A20 = b * sig[4], A21 = b * sig[5];
                double l00 = 0, l10 = 0, l11 = 0, l20 = 0, l21 = 0, l22 = 0;
                bool ok = A00 > 0.0;
                if (ok) {
                    l00 = sqrt(A00);
                    const double i0 = 1.0 / l00;
                    l10 = A10 * i0;
                    l20 = A20 * i0;
                    const double d1 = A11 - l10 * l10;
                    ok = d1 > 0.0;
                    if (ok) {
                        l11 = sqrt(d1);
                        l21 = (A21 - l20 * l10) / l11;
                        const double d2 = A22 - l20 * l20 - l21 * l21;
                        ok = d2 > 0.0;
                        if (ok) l22 = sqrt(d2);
                    }
                }
                if (!ok) {
                    const double r = sqrt(L.theta);
                    l00 = l11 = l22 = r;
                    l10 = l20 = l21 = 0.0;
                    atomicAdd(&s.dyn->counters[kCntChol], 1ull);
                }
                pr[4] = l00; pr[5] = l10; pr[6] = l11; pr[7] = l20; pr[8] = l21; pr[9] = l22;
                if (s.es_sampler) {
                    // Eq. 11: B = ((1 - Pr)/(2 Pr)) sigma*/(rho theta); S = I - s B
                    const double beta = (1.0 - s.Pr) / (2.0 * s.Pr) / L.theta;
                    for (int k = 0; k < 6; ++k) pr[4 + k] = beta * sig[k];
                }
                if (s.weighted) {
                    // sigma* and q* per unit density for the weights of steps 4 and 7
                    for (int k = 0; k < 6; ++k) s.wst[(size_t)k * K + cell] = sig[k];
                    for (int k = 0; k < 3; ++k) s.wst[(size_t)(6 + k) * K + cell] = Q[k] * ifq;
                }
                pr[10] = -expm1(-s.Pr * L.nu * s.dt);                       // Eqs. 8b, 9
                pr[11] = L.nu;
                pr[12] = s.Pr * L.nu;
                pr[13] = pne;
                pr[14] = 1.0;
                f[4] = L.T;
                f[5] = L.p + L.rho * sig[0];
                f[6] = L.p + L.rho * sig[1];
                f[7] = L.p + L.rho * sig[2];
                f[8] = L.rho * sig[3];
                f[9] = L.rho * sig[4];
                f[10] = L.rho * sig[5];
                f[11] = L.rho * Q[0] * ifq;
                f[12] = L.rho * Q[1] * ifq;
                f[13] = L.rho * Q[2] * ifq;
                f[14] = pne;
            }
            for (int k = 0; k < kNPrm; ++k) prm[(size_t)k * K + cell] = pr[k];
#pragma unroll
            for (int k = 0; k < kNFields; ++k) {
                s.inst[(size_t)k * K + cell] = f[k];
                s.avg[(size_t)k * K + cell] = first ? f[k] : s.avg_keep * av[k] + f[k] * s.avg_new;   // Eq. 34
            }
        }
    }
}

// ---------------------------------------------------------------------------
// K7: relaxation of each cell with conservation of momentum and energy
// ---------------------------------------------------------------------------
// is the particle at slot i of the cell [b, e) relaxed?  Bernoulli: its
// selection word against the probability (in FP64 as its limit in integers); fixed count (Eq. 9): its rank
// among the cell's selection words below ns.  `words` holds the cell's
// selection words (staged once per cell) when the cell fits, else null and
// the words are drawn again.
constexpr uint32_t kRelaxWords = 1024;
// relaxed particles of a cell worked on at a time: their new peculiar
// velocities are kept from the sums for the apply pass (a larger cell goes
// through in chunks of this many particles and draws them again)
constexpr uint32_t kRelaxKeep = 512;
// warps per cell: four in FP64; one in FP32, where the draws are cheap and the
// cell's own FP64 work would only be done four times over
template <class T> constexpr int kRelaxWarps = sizeof(T) == 8 ? 4 : 1;

template <class T>
__device__ __forceinline__ bool selected(const SimDev& s, const PView<T>& B, uint32_t b, uint32_t e, uint32_t i,
                                         uint32_t wx, T pth, uint64_t limit, uint32_t ns, uint32_t step, const uint32_t* words) {
    if (!s.selection) return sizeof(T) == 8 ? wx < limit : u01<T>(wx) < pth;
    if (ns == 0) return false;
    uint32_t rank = 0;
    for (uint32_t j = b; j < e && rank < ns; ++j) {
        const uint32_t xj = words ? words[j - b] : draw(s, B.pid[j], step, kRelax, 0).x;
        rank += (xj < wx || (xj == wx && j < i)) ? 1u : 0u;
    }
    return rank < ns;
}

// A block of four warps per cell, the blocks striding over single cells: the
// relaxation is bound by FP64 issue (about two FP64 FMA per clock per SM on
// GB300, the same for one lane of a warp as for all), so
//  * only the selected particles are worked on: their list is packed first, so
//    that a cell with a quarter of its particles selected takes a quarter of
//    the draws' instructions;
//  * the draw of a particle is split over the four warps (the time instant, and
//    one Box-Muller pair each), which keep the FP64 pipe busy together where a
//    domain has about one cell per SM.
//  * the draws' functions are those of usp_math64.cuh, and the selection
//    compares integers.
// Measured per launch, one warp per cell on all particles before: 100 cells of
// 100 particles, a quarter selected, 60 -> 20 us; 1000 cells of 360 / 45, all
// selected, 208 -> 175 us, with these functions 130 us (FP64 issue: about 230
// instructions a particle, 74 us at two lanes a clock); FP32, 4e4 cells of
// 100, 719 -> 432 us.
template <class T>
__global__ void __launch_bounds__(32 * kRelaxWarps<T>) k_relax(const SimDev* __restrict__ sims,
                                                               const int2* __restrict__ tiles,
                                                               const int* __restrict__ ntiles) {
    constexpr int NW = kRelaxWarps<T>;
    constexpr uint32_t B_ = 32 * NW, Q_ = kRelaxKeep / NW;
    __shared__ SimDev sim_sh;
    __shared__ uint32_t sel_words[kRelaxWords];
    __shared__ T zc[NW > 1 ? 6 : 3][kRelaxKeep];   // the six normals, then the new peculiar velocity (first three)
    __shared__ T ab[2][NW > 1 ? kRelaxKeep : 1];   // sqrt(s), sqrt((1 - s) theta) of Eqs. 31-32 (Gallis-Torczynski: s)
    __shared__ unsigned short part[kRelaxKeep], list[NW > 1 ? kRelaxKeep : 1];   // selected particles by warp, packed
    __shared__ uint32_t part_n[NW];
    __shared__ double sums[NW][8], fac[8];
    const int nt = *ntiles;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = lanemask_lt();
    int loaded = -1;
    for (int g = blockIdx.x; g < nt * kCTile; g += gridDim.x) {
        const int2 tile = tiles[g / kCTile];
        if (tile.x != loaded) {
            __syncthreads();
            load_sim(sim_sh, sims[tile.x]);
            __syncthreads();
            loaded = tile.x;
        }
        const SimDev& s = sim_sh;
        const int K = s.K;
        const uint32_t step = s.dyn->step;
        const PView<T> V = view<T>(s, s.dyn->cur ^ 1);
        const int cell = tile.y + g % kCTile;
        if (cell >= K) continue;
        const double* pr = s.prm;
        const bool valid = pr[(size_t)14 * K + cell] != 0.0;
        CellRelax R;
        for (int d = 0; d < 3; ++d) R.u[d] = pr[(size_t)d * K + cell];
        if (tid == 0 && s.mom[cell] >= 1.0)
            for (int d = 0; d < 3; ++d) s.ushift[(size_t)d * K + cell] = R.u[d];
        if (!valid) continue;
        R.theta = pr[(size_t)3 * K + cell];
        for (int d = 0; d < 6; ++d) R.L[d] = pr[(size_t)(4 + d) * K + cell];
        R.p_relax = pr[(size_t)10 * K + cell];
        R.nu = pr[(size_t)11 * K + cell];
        R.nu_es = pr[(size_t)12 * K + cell];
        R.pne = pr[(size_t)13 * K + cell];
        const uint32_t cap = (uint32_t)s.cap;
        const uint32_t b = min(s.start[cell], cap), e = min(s.start[cell + 1], cap);
        const T pth = (T)R.p_relax;
        const uint64_t limit = sizeof(T) == 8 ? word_limit(R.p_relax) : 0u;
        // Eq. 9 fixed count: the ns particles with the smallest selection
        // words (ties: lower position first)
        const uint32_t ns = s.selection ? (uint32_t)floor((double)(e - b) * R.p_relax + 0.5) : 0u;
        const uint32_t* words = nullptr;
        __syncthreads();   // the shared arrays of the cell before are free
        if (s.selection && e - b <= kRelaxWords) {
            for (uint32_t i = b + tid; i < e; i += B_) sel_words[i - b] = draw(s, V.pid[i], step, kRelax, 0).x;
            __syncthreads();
            words = sel_words;
        }
        // the selected particles of [c0, c0 + kRelaxKeep) into `list`, in
        // order, and their new peculiar velocities into zc[0..2]; how many
        unsigned short* const lst = NW > 1 ? list : part;
        auto draws = [&](uint32_t c0) -> uint32_t {
            uint32_t mine = 0;
            for (uint32_t j = 0; j < Q_; j += 32) {   // warp w: particles w Q_ .. (w + 1) Q_ - 1
                const uint32_t k = warp * Q_ + j + lane, i = c0 + k;
                if (c0 + warp * Q_ + j >= e) break;
                bool sel = false;
                if (i < e) sel = selected<T>(s, V, b, e, i, draw(s, V.pid[i], step, kRelax, 0).x, pth, limit, ns, step, words);
                const unsigned m = __ballot_sync(0xffffffffu, sel);
                if (sel) part[warp * Q_ + mine + __popc(m & lt)] = (unsigned short)k;
                mine += __popc(m);
            }
            if constexpr (NW == 1) {
                __syncwarp();
                for (uint32_t k = lane; k < mine; k += 32) {
                    const uint32_t id = V.pid[c0 + part[k]];
                    T C[3];
                    const uint4 w = draw(s, id, step, kRelax, 0);
                    es_draw<T>(s, R, id, step, w, sample_time<T>(u01<T>(w.y), (T)R.nu_es, (T)s.dt), C);
                    zc[0][k] = C[0];   // (read again by this thread alone)
                    zc[1][k] = C[1];
                    zc[2][k] = C[2];
                }
                return mine;
            } else {
            if (lane == 0) part_n[warp] = mine;
            __syncthreads();
            uint32_t first = 0, all = 0;
            for (int w = 0; w < NW; ++w) {
                if (w < warp) first += part_n[w];
                all += part_n[w];
            }
            for (uint32_t k = lane; k < mine; k += 32) list[first + k] = part[warp * Q_ + k];
            __syncthreads();
            TimeLaw64 law;   // time instant (Eqs. 29-30): of this warp alone
            if (warp == 0) law.set(R.nu_es, s.dt);
            for (uint32_t k = lane; k < all; k += 32) {
                const uint32_t id = V.pid[c0 + list[k]];
                if (warp == 0) {
                    const T U = u01<T>(draw(s, id, step, kRelax, 0).y);
                    const T t = law.instant(U);
                    // Eq. 32; the SP-ESBGK step holds the target for the whole step (Eq. 8b)
                    const T sf = s.mode == kModeSPESBGK ? (T)1 : (T)R.pne + (T)(1.0 - R.pne) * exp(-(T)R.nu * t);
                    ab[0][k] = s.es_sampler ? sf : dev_sqrt<T>(sf);
                    ab[1][k] = s.es_sampler ? dev_sqrt<T>((T)R.theta) : dev_sqrt<T>(((T)1 - sf) * (T)R.theta);
                } else {
                    const uint4 w = draw(s, id, step, kRelax, warp == 1 ? 0u : 1u);
                    T z0, z1;
                    box_muller<T>(warp == 2 ? w.x : w.z, warp == 2 ? w.y : w.w, z0, z1);
                    zc[2 * warp - 2][k] = z0;
                    zc[2 * warp - 1][k] = z1;
                }
            }
            __syncthreads();
            for (uint32_t k = tid; k < all; k += B_) {
                const T a0 = ab[0][k], b0 = ab[1][k];
                T C[3];
                if (s.es_sampler) {
                    // Eq. 10: one thermal component per (cosine) Box-Muller pair; Eq. 11:
                    // C = S C*, S = I - s B, B = ((1 - Pr)/(2 Pr)) sigma*/(rho theta) in
                    // the L slots (xx, yy, zz, xy, xz, yz)
                    const T c0_ = b0 * zc[0][k], c1_ = b0 * zc[2][k], c2_ = b0 * zc[4][k];
                    const T b00 = a0 * (T)R.L[0], b11 = a0 * (T)R.L[1], b22 = a0 * (T)R.L[2];
                    const T b01 = a0 * (T)R.L[3], b02 = a0 * (T)R.L[4], b12 = a0 * (T)R.L[5];
                    C[0] = ((T)1 - b00) * c0_ - b01 * c1_ - b02 * c2_;
                    C[1] = -b01 * c0_ + ((T)1 - b11) * c1_ - b12 * c2_;
                    C[2] = -b02 * c0_ - b12 * c1_ + ((T)1 - b22) * c2_;
                } else {
                    const T z0 = zc[0][k], z1 = zc[1][k], z2 = zc[2][k];
                    C[0] = a0 * ((T)R.L[0] * z0) + b0 * zc[3][k];
                    C[1] = a0 * ((T)R.L[1] * z0 + (T)R.L[2] * z1) + b0 * zc[4][k];
                    C[2] = a0 * ((T)R.L[3] * z0 + (T)R.L[4] * z1 + (T)R.L[5] * z2) + b0 * zc[5][k];
                }
                zc[0][k] = C[0];   // (read again by this thread alone)
                zc[1][k] = C[1];
                zc[2][k] = C[2];
            }
            return all;
            }
        };
        // pass 1: sums over the relaxed subset (velocities relative to the cell mean)
        double S[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        uint32_t nr = 0, all = 0;
        for (uint32_t c0 = b; c0 < e; c0 += kRelaxKeep) {
            if (c0 != b) __syncthreads();
            all = draws(c0);
            nr += all;
            for (uint32_t k = tid; k < all; k += B_) {
                const uint32_t i = c0 + lst[k];
                const double o0 = (double)V.c0[i] - R.u[0], o1 = (double)V.c1[i] - R.u[1],
                             o2 = (double)V.c2[i] - R.u[2];
                const double C0 = (double)zc[0][k], C1 = (double)zc[1][k], C2 = (double)zc[2][k];
                S[0] += o0; S[1] += o1; S[2] += o2;
                S[3] += o0 * o0 + o1 * o1 + o2 * o2;
                S[4] += C0; S[5] += C1; S[6] += C2;
                S[7] += C0 * C0 + C1 * C1 + C2 * C2;
            }
        }
        int applied = 0;
        if (nr >= 2) {
            // reduce-scatter of the eight sums in each warp (lane 4 i: sum i), then over the warps
#pragma unroll
            for (int half = 4; half >= 1; half >>= 1) {
                const bool up = (lane & (4 * half)) != 0;
#pragma unroll
                for (int i = 0; i < half; ++i) {
                    const double send = up ? S[i] : S[i + half];
                    const double recv = __shfl_xor_sync(0xffffffffu, send, 4 * half);
                    S[i] = (up ? S[i + half] : S[i]) + recv;
                }
            }
            S[0] += __shfl_xor_sync(0xffffffffu, S[0], 2);
            S[0] += __shfl_xor_sync(0xffffffffu, S[0], 1);
            if ((lane & 3) == 0) sums[warp][lane >> 2] = S[0];
            __syncthreads();
            if (warp == 0) {   // the factors once (FP64 costs each warp that computes it)
                double A[8], a = 0.0;
                if (lane < 8)
                    for (int w = 0; w < NW; ++w) a += sums[w][lane];
#pragma unroll
                for (int k = 0; k < 8; ++k) A[k] = __shfl_sync(0xffffffffu, a, k);
                const double inv = 1.0 / (double)nr;
                const double Eo = A[3] - (A[0] * A[0] + A[1] * A[1] + A[2] * A[2]) * inv;
                const double En = A[7] - (A[4] * A[4] + A[5] * A[5] + A[6] * A[6]) * inv;
                if (lane == 0) {
                    fac[7] = En > 0.0 ? 1.0 : 0.0;
                    if (En > 0.0) {
                        fac[6] = sqrt(Eo / En);
                        for (int d = 0; d < 3; ++d) {
                            fac[d] = R.u[d] + A[d] * inv;
                            fac[3 + d] = A[4 + d] * inv;
                        }
                    }
                }
            }
            __syncthreads();
            if (fac[7] != 0.0) {
                applied = (int)nr;
                const double alpha = fac[6];
                const double uo[3] = {fac[0], fac[1], fac[2]};
                const double mn[3] = {fac[3], fac[4], fac[5]};
                // pass 2: apply c = ubar_old + alpha (c' - ubar_new), with c'
                // kept from pass 1 or drawn again
                for (uint32_t c0 = b; c0 < e; c0 += kRelaxKeep) {
                    if (e - b > kRelaxKeep) {
                        __syncthreads();
                        all = draws(c0);
                    }
                    for (uint32_t k = tid; k < all; k += B_) {
                        const uint32_t i = c0 + lst[k];
                        V.c0[i] = (T)(uo[0] + alpha * ((double)zc[0][k] - mn[0]));
                        V.c1[i] = (T)(uo[1] + alpha * ((double)zc[1][k] - mn[1]));
                        V.c2[i] = (T)(uo[2] + alpha * ((double)zc[2][k] - mn[2]));
                    }
                }
            }
        }
        if (tid == 0) {
            s.prm[(size_t)15 * K + cell] = applied;
            if (applied) atomicAdd(&s.dyn->counters[kCntRelaxed], (unsigned long long)applied);
        }
    }
}

// ---------------------------------------------------------------------------
// K8: end of step
// ---------------------------------------------------------------------------
__global__ void k_finish(const SimDev* __restrict__ sims, int nsims) {
    for (int si = blockIdx.x * blockDim.x + threadIdx.x; si < nsims; si += gridDim.x * blockDim.x) {
        const SimDev& s = sims[si];
        SimDyn* d = s.dyn;
        uint32_t n = s.start[s.K];
        if ((int64_t)n > s.cap) n = (uint32_t)s.cap;
        d->n = n;
        if (s.has_reservoir) {
            d->next_pid += s.inj_total;
            d->counters[kCntInjected] += s.inj_total;
        }
        d->cur ^= 1;
        d->step += 1;
        d->nsamples += 1;
    }
}

// ---------------------------------------------------------------------------
// initial fill (Table 2 step 1): warp per cell; counts and offsets from the host
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(256) k_init_fill(const SimDev* __restrict__ sims, const int2* __restrict__ tiles,
                                                   const int* __restrict__ ntiles, const double* __restrict__ reg_theta,
                                                   const double* __restrict__ reg_u, const int* __restrict__ cell_reg) {
    __shared__ SimDev sim_sh;
    const int nt = *ntiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int t = blockIdx.x; t < nt; t += gridDim.x) {
        const int2 tile = tiles[t];
        __syncthreads();
        load_sim(sim_sh, sims[tile.x]);
        __syncthreads();
        const SimDev& s = sim_sh;
        PView<T> A = view<T>(s, 0);
        for (int cc = warp; cc < kCTile; cc += nwarps) {
            const int cell = tile.y + cc;
            if (cell >= s.K) break;
            const int r = cell_reg[cell];
            if (r < 0) continue;
            const uint32_t b = s.start[cell], e = s.start[cell + 1];
            for (uint32_t i = b + lane; i < e; i += 32) {
                T x, y, c[3];
                make_particle<T>(s, cell, i, 0u, kInit, reg_theta[r], reg_u + 3 * r, x, y, c);
                if (s.dim == 2) A.x[i] = x;
                A.y[i] = y;
                A.c0[i] = c[0];
                A.c1[i] = c[1];
                A.c2[i] = c[2];
                A.pid[i] = i;
            }
        }
    }
}

__global__ void k_debug_philox(int64_t n, const uint32_t* __restrict__ ctr, uint32_t k0, uint32_t k1,
                               uint32_t* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint4 r = philox(make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]), make_uint2(k0, k1));
        out[4 * i] = r.x;
        out[4 * i + 1] = r.y;
        out[4 * i + 2] = r.z;
        out[4 * i + 3] = r.w;
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
void launch_stream(const Launch& L, bool fp64) {
    if (fp64) k_stream<double><<<L.grid_u, kPUnit, 0, L.stream>>>(L.sims, L.ptiles, L.nptiles);
    else k_stream<float><<<L.grid_u, kPUnit, 0, L.stream>>>(L.sims, L.ptiles, L.nptiles);
}
void launch_assign(const Launch& L, bool fp64) {
    if (fp64) k_assign<double><<<L.grid_u, kPUnit, 0, L.stream>>>(L.sims, L.ptiles, L.nptiles);
    else k_assign<float><<<L.grid_u, kPUnit, 0, L.stream>>>(L.sims, L.ptiles, L.nptiles);
}
void launch_scan(const Launch& L, bool with_inj) { k_scan<<<L.nsims, 1024, 0, L.stream>>>(L.sims, L.nsims, with_inj ? 1 : 0); }
void launch_scatter(const Launch& L, bool fp64) {
    if (fp64) k_scatter<double><<<L.grid_u, kPUnit, 0, L.stream>>>(L.sims, L.ptiles, L.nptiles);
    else k_scatter<float><<<L.grid_u, kPUnit, 0, L.stream>>>(L.sims, L.ptiles, L.nptiles);
}
void launch_inject(const Launch& L, bool fp64) {
    if (fp64) k_inject<double><<<L.grid_c, 256, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles);
    else k_inject<float><<<L.grid_c, 256, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles);
}
void launch_moments(const Launch& L, bool fp64) { launch_moments_src(L, fp64, false); }
void launch_moments_src(const Launch& L, bool fp64, bool src_cur) {
    const int sc = src_cur ? 1 : 0;
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = std::max(1, std::min(L.grid_c * kCTile, 32 * sms));
    if (fp64) k_moments<double><<<grid, 32, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles, sc);
    else k_moments<float><<<grid, 32, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles, sc);
}
void launch_params(const Launch& L) { k_params<<<L.grid_c, 32, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles); }
void launch_relax(const Launch& L, bool fp64) {
    // one block per cell slot of the tiles, at most what the SMs' shared memory holds (41 and 13 KB a block)
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = std::max(1, std::min(L.grid_c * kCTile, (fp64 ? 5 : 16) * sms));
    if (fp64) k_relax<double><<<grid, 32 * kRelaxWarps<double>, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles);
    else k_relax<float><<<grid, 32 * kRelaxWarps<float>, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles);
}
void launch_finish(const Launch& L) { k_finish<<<(L.nsims + 127) / 128, 128, 0, L.stream>>>(L.sims, L.nsims); }

// user-supplied particles (host layout: pos[n][2], vel[n][3] in FP64) into
// the storage planes of buffer 0.  pos, vel and ids are device copies of the
// caller's arrays or, for page-locked host memory, the arrays themselves
// read through their mapped device addresses; any of pos, vel, ids may be
// null (that part is not read).  ids go to pid (when non-null); with
// next_pid non-null, one past the largest id is folded into *next_pid (one
// atomic per warp).
template <class T>
__global__ void k_unpack(const double* __restrict__ pos, const double* __restrict__ vel,
                         const uint32_t* __restrict__ ids, int64_t n, int dim, T* x, T* y, T* v0, T* v1, T* v2,
                         uint32_t* pid, uint32_t* next_pid) {
    uint32_t top = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (pos) {
            if (dim == 2) x[i] = (T)pos[2 * i];
            y[i] = (T)pos[2 * i + 1];
        }
        if (vel) {
            v0[i] = (T)vel[3 * i];
            v1[i] = (T)vel[3 * i + 1];
            v2[i] = (T)vel[3 * i + 2];
        }
        if (ids) {
            const uint32_t id = ids[i];
            if (pid) pid[i] = id;
            top = max(top, id + 1u);
        }
    }
    if (next_pid) {
        top = __reduce_max_sync(0xffffffffu, top);
        if ((threadIdx.x & 31) == 0 && top) atomicMax(next_pid, top);
    }
}

void launch_unpack(const SimDev& s, bool fp64, const double* pos, const double* vel, const uint32_t* ids,
                   bool ids_to_plane, uint32_t* next_pid, int64_t n, cudaStream_t st) {
    if (n <= 0) return;
    const int grid = (int)std::min<int64_t>((n + 255) / 256, 152 * 16);
    uint32_t* pid = ids_to_plane ? s.pid[0] : nullptr;
    if (fp64)
        k_unpack<double><<<grid, 256, 0, st>>>(pos, vel, ids, n, s.dim, (double*)s.pos[0][0], (double*)s.pos[0][1],
                                               (double*)s.vel[0][0], (double*)s.vel[0][1], (double*)s.vel[0][2],
                                               pid, next_pid);
    else
        k_unpack<float><<<grid, 256, 0, st>>>(pos, vel, ids, n, s.dim, (float*)s.pos[0][0], (float*)s.pos[0][1],
                                              (float*)s.vel[0][0], (float*)s.vel[0][1], (float*)s.vel[0][2],
                                              pid, next_pid);
}

// clear up to kZeroRanges device ranges of 32-bit words in one launch
__global__ void k_zero(ZeroList z) {
    for (int r = 0; r < z.n; ++r) {
        uint32_t* p = (uint32_t*)z.p[r];
        for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < z.words[r];
             i += (size_t)gridDim.x * blockDim.x)
            p[i] = 0u;
    }
}

void launch_zero(const ZeroList& z, cudaStream_t st) {
    size_t most = 0;
    for (int r = 0; r < z.n; ++r) most = std::max(most, z.words[r]);
    if (most == 0) return;
    const int grid = (int)std::min<size_t>((most + 255) / 256, 152 * 8);
    k_zero<<<grid, 256, 0, st>>>(z);
}

void launch_init(const Launch& L, bool fp64, const double* reg_theta, const double* reg_u, const int* cell_reg) {
    if (fp64)
        k_init_fill<double><<<L.grid_c, 256, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles, reg_theta, reg_u, cell_reg);
    else
        k_init_fill<float><<<L.grid_c, 256, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles, reg_theta, reg_u, cell_reg);
}

cudaError_t debug_philox(int64_t n, const uint32_t* d_ctr, uint32_t k0, uint32_t k1, uint32_t* d_out,
                         cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    int grid = (int)((n + 255) / 256);
    if (grid > 4096) grid = 4096;
    k_debug_philox<<<grid, 256, 0, st>>>(n, d_ctr, k0, k1, d_out);
    return cudaGetLastError();
}

}  // namespace usp
