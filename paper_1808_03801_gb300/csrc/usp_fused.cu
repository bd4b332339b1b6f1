// usp_fused.cu -- the fused FP32 pipeline of the USP-ESBGK step (sm_103a).
//
// One step n reads buffer p = cur and writes buffer q = cur ^ 1:
//   k_g2      per cell (one warp; k_g2b: a block, where there are few or
//             very dense cells): the relaxation of step n-1 still pending on
//             the cell's particles (Eqs. 8b, 9, 27, 29-32 with the per-cell
//             momentum / energy conservation), then advection of step n with
//             the boundaries, the new cell, and the write into that cell's
//             bucket of buffer q (the scatter of the counting sort; the
//             bucket sizes come from the previous histogram plus slack).
//   k_inject  reservoir buffer cells refilled into buffer q.
//   k_g1      per cell (one warp): moments of Eq. 1 in one pass, as sums
//             about the cell's mean velocity of the previous step, and the
//             cell's n, T, |u| for its neighbours' Kn_GLL.
//   k_params_f  per cell: Kn_GLL and P_ne (Eqs. 16-18), sigma* and q* (Eq. 33),
//             the Cholesky factor of the ES covariance (Eq. 6c), the fields
//             and the average of Eq. 34.
//   k_lay_small, or k_lay_sum, k_lay_scan and k_lay_put in larger domains:
//             histogram -> bucket sizes -> exclusive scan, the layout that
//             the next step writes with (beside k_g1 and k_params_f).
//   k_step_end  per simulation: swap buffers, advance the step.
// All arithmetic of a step is FP32 except the number density and the Eq. 34
// running averages (FP64, in k_params_f).  FP64 issue rate is scarce on
// GB300 (about two FP64 FMA per clock per SM).  The moments are sums about
// the previous step's cell mean and the conservation factors use sums about
// the cell mean, so no subtraction cancels: the per-cell state, Eq. 33 and
// the Cholesky factor lose nothing in FP32 that the FP32 sums still carry.
// Each particle is read once and written once by k_g2 and its velocity is
// read once more by k_g1.
#include <algorithm>
#include <cstddef>

#include "usp_device.cuh"

namespace usp {

namespace {

constexpr uint32_t kNoCell = 0xFFFFFFFFu;

// f(rank, i) for each entry i of buffer b's spill list that belongs to `cell`,
// rank counting them (a warp; its lanes take entries side by side); returns
// how many there are
template <class F>
__device__ __forceinline__ uint32_t each_spilled(const SimDev& s, int b, int cell, int lane, const F& f) {
    const uint32_t n = min(s.dyn->sp_n[b], (uint32_t)kSpillCap);
    uint32_t found = 0;
    for (uint32_t base = 0; base < n; base += 32) {
        const uint32_t i = base + lane;
        const bool hit = i < n && s.sp_cell[b][i] == (uint32_t)cell;
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (hit) f(found + __popc(m & lanemask_lt()), i);
        found += __popc(m);
    }
    return found;
}

template <int DIM>
__device__ __forceinline__ void load_particle(const SimDev& s, int b, uint32_t base, uint32_t nb, const uint16_t* spl,
                                              uint32_t j, float& x, float& y, float& v0, float& v1, float& v2,
                                              uint32_t& id) {
    if (j < nb) {
        const uint32_t i = base + j;
        if (DIM == 2) x = ((const float*)s.pos[b][0])[i];
        y = ((const float*)s.pos[b][1])[i];
        v0 = ((const float*)s.vel[b][0])[i];
        v1 = ((const float*)s.vel[b][1])[i];
        v2 = ((const float*)s.vel[b][2])[i];
        id = s.pid[b][i];
    } else {
        const uint32_t i = spl[j - nb];
        if (DIM == 2) x = s.sp_pos[b][0][i];
        y = s.sp_pos[b][1][i];
        v0 = s.sp_vel[b][0][i];
        v1 = s.sp_vel[b][1][i];
        v2 = s.sp_vel[b][2][i];
        id = s.sp_pid[b][i];
    }
}

__device__ __forceinline__ void store_velocity(const SimDev& s, int b, uint32_t base, uint32_t nb, const uint16_t* spl,
                                               uint32_t j, float v0, float v1, float v2) {
    if (j < nb) {
        const uint32_t i = base + j;
        ((float*)s.vel[b][0])[i] = v0;
        ((float*)s.vel[b][1])[i] = v1;
        ((float*)s.vel[b][2])[i] = v2;
    } else {
        const uint32_t i = spl[j - nb];
        s.sp_vel[b][0][i] = v0;
        s.sp_vel[b][1][i] = v1;
        s.sp_vel[b][2][i] = v2;
    }
}

// a particle whose bucket is full: into the spill list of buffer b
template <int DIM>
__device__ __forceinline__ void spill(const SimDev& s, int b, int cell, float x, float y, float v0, float v1, float v2,
                                      uint32_t id) {
    const uint32_t k = atomicAdd(&s.dyn->sp_n[b], 1u);
    atomicAdd(&s.dyn->counters[kCntSpilled], 1ull);
    if (k < (uint32_t)kSpillCap) {
        if (DIM == 2) s.sp_pos[b][0][k] = x;
        s.sp_pos[b][1][k] = y;
        s.sp_vel[b][0][k] = v0;
        s.sp_vel[b][1][k] = v1;
        s.sp_vel[b][2][k] = v2;
        s.sp_pid[b][k] = id;
        s.sp_cell[b][k] = (uint32_t)cell;
    } else {
        atomicAdd(&s.dyn->counters[kCntOverflow], 1ull);
    }
}

// ---------------------------------------------------------------------------
// k_g2b: pending relaxation + advection + bucket scatter, one block of G warps
// per cell.
//
// A block takes units of consecutive cells from one counter and works on one
// cell at a time; thread t holds the particles t, t + 32 G, ... (at most kG2P)
// in registers from the load to the write:
//   relax    relaxation draws of the pending step (one Philox call per
//            particle), conservation sums over the block;
//   move     conservation, advection, destination cell and its slot in the
//            cell's 64-cell destination window; each particle's rank among
//            the arrivals of its slot from one shared-memory atomic;
//   reserve  one global atomic per occupied slot in the destination buckets
//            (one round trip for the whole cell);
//   write    each particle at its slot's reserved start plus its rank, so
//            the lanes of one slot write consecutive words of one bucket.
// It is for domains of few cells, where a step takes as long as its slowest
// cell: spread over several warps a cell's latency is that of a few particles
// per thread (measured per launch, one warp per cell -> block per cell: 100
// cells of 200 particles 21 -> 13 us, one shock tube of 1000 cells 30 -> 18 us;
// with 4e4 cells of 100 particles the barriers and the per-warp share of the
// cell's work cost more than they give, 117 -> 230 us).
// Cells above 32 G kG2P particles go through in chunks: a first sweep for the
// conservation sums, a second one (in reverse, so that the last chunk is
// still in registers) that draws the same counter-based random numbers again.
// ---------------------------------------------------------------------------
// the general advection (wall and plate hits), out of line; the particle
// goes in and out by value so that the common path keeps it in registers
// (reference arguments to a call would pass through local memory)
struct AdvOut {
    float x, y, c0, c1, c2;
    int alive;
};

__device__ __noinline__ AdvOut advect_slow(const SimDev& s, uint32_t step, uint32_t pid, float x, float y, float c0,
                                           float c1, float c2) {
    float c[3] = {c0, c1, c2};
    AdvOut o;
    o.alive = advect<float>(s, step, pid, x, y, c) ? 1 : 0;
    o.x = x;
    o.y = y;
    o.c0 = c[0];
    o.c1 = c[1];
    o.c2 = c[2];
    return o;
}

// row and column of an FP32 position: floor of the scaled offset, clamped to
// the grid (1-D: ix = 0)
template <int DIM>
__device__ __forceinline__ void cell_xy(const SimDev& s, float x, float y, int& ix, int& iy) {
    iy = min(max(__float2int_rd((y - s.f_lo[1]) * s.f_inv_dy), 0), s.ny - 1);
    ix = DIM == 1 ? 0 : min(max(__float2int_rd((x - s.f_lo[0]) * s.f_inv_dx), 0), s.nx - 1);
}

template <int DIM>
__device__ __forceinline__ bool advect_fast(const SimDev& s, uint32_t step, uint32_t pid, float& x, float& y,
                                            float* c) {
    const float yn = y + c[1] * s.f_dt;
    bool inside = yn > s.f_lo[1] && yn < s.f_hi[1];
    float xn = x;
    if (DIM == 2) {
        xn = x + c[0] * s.f_dt;
        inside = inside && xn > s.f_lo[0] && xn < s.f_hi[0];
        for (int g = 0; g < s.nseg; ++g) {
            const float ps = s.f_seg_pos[g];
            if ((x - ps) * (xn - ps) <= 0.0f) inside = false;
        }
    }
    if (inside) {
        y = yn;
        if (DIM == 2) x = xn;
        c[0] += s.f_bdt[0];
        c[1] += s.f_bdt[1];
        c[2] += s.f_bdt[2];
        return true;
    }
    const AdvOut o = advect_slow(s, step, pid, x, y, c[0], c[1], c[2]);
    x = o.x;
    y = o.y;
    c[0] = o.c0;
    c[1] = o.c1;
    c[2] = o.c2;
    return o.alive != 0;
}

// reservoir buffer cell (column ix, global row iy)?
__device__ __forceinline__ bool in_buffer_xy(const SimDev& s, int ix, int iy) {
    return ix < s.buf_lo[0] || ix >= s.buf_hi[0] || iy < s.buf_lo[1] || iy >= s.buf_hi[1];
}

// Destination window of a cell: the 64 cells that its particles can reach in
// one step without leaving it (1-D: offsets -32..31; 2-D: an 8 x 8 block
// around the cell).  The block counts its arrivals per window slot in shared
// memory, reserves each slot's range in the destination bucket with one
// global atomic, then writes; particles that land outside the window reserve
// their place one at a time.
constexpr int kWin = 64;
constexpr uint32_t kSlotNone = 0xFF;   // removed, nothing to write
constexpr uint32_t kSlotFar = 0xFE;    // outside the window
constexpr uint32_t kSlotOther = 0xFD;  // in another slab of a decomposed domain

template <int DIM>
__device__ __forceinline__ int win_slot_xy(int ix, int iy, int cell, int cx, int cy) {
    if (DIM == 1) {
        const int o = iy - cell + 32;
        return (unsigned)o < (unsigned)kWin ? o : -1;
    }
    const int oy = iy - cy + 4, ox = ix - cx + 4;
    return ((unsigned)oy < 8u && (unsigned)ox < 8u) ? oy * 8 + ox : -1;
}

template <int DIM>
__device__ __forceinline__ int win_cell(int k, int cell, int cx, int cy, int nx) {
    if (DIM == 1) return cell + k - 32;
    return (cy + (k >> 3) - 4) * nx + (cx + (k & 7) - 4);
}

// a particle that crossed into another slab of a decomposed domain: its
// place is reserved in that slab's bucket (or spill list) of buffer q, all
// slabs of a domain stepping together
template <int DIM>
__device__ __noinline__ void emit_other(const SimDev* __restrict__ sims, const SimDev& s, int q, float x, float y,
                                        float v0, float v1, float v2, uint32_t id) {
    int ix, row;
    cell_xy<DIM>(s, x, y, ix, row);
    const int gc = DIM == 2 ? row * s.nx + ix : row;
    const SimDev& o = sims[s.slab_first + row / s.rows];
    const int dc = gc - o.row0 * o.nx;
    const uint32_t i = o.lay[q][dc] + atomicAdd(&o.cnt[q][dc], 1u);
    const uint32_t hi = min(o.lay[q][dc + 1], (uint32_t)o.cap);
    if (i < hi) {
        if (DIM == 2) ((float*)o.pos[q][0])[i] = x;
        ((float*)o.pos[q][1])[i] = y;
        ((float*)o.vel[q][0])[i] = v0;
        ((float*)o.vel[q][1])[i] = v1;
        ((float*)o.vel[q][2])[i] = v2;
        o.pid[q][i] = id;
        return;
    }
    spill<DIM>(o, q, dc, x, y, v0, v1, v2, id);
}

// kFullSlab: kFull for batches holding slabs of a decomposed domain (routes
// particles that leave the slab; the plain kFull code carries no such check).
// kFullFlux: kFull for batches where some simulation counts particles
// through a plane (kFullSlab counts too).  kRelaxOnly applies the pending
// relaxation in place (before the particles are read back).
enum { kFull = 0, kRelaxOnly = 1, kFullSlab = 2, kFullFlux = 3 };

constexpr int kG2P = 4;         // particles per thread and chunk
constexpr int kG2Warps = 16;    // resident warps per SM

// shared state of one block of k_g2b
template <int G>
struct G2Shared {
    SimDev sim;                 // the simulation the block works on
    uint32_t wcnt[kWin];        // arrivals per window slot (zero between cells)
    uint32_t wstart[kWin];      // first reserved index of each slot in its bucket
    uint32_t wend[kWin];        // end of that bucket
    float part[G][8];           // per-warp conservation sums
    uint32_t part_n[G];         // per-warp relaxed particles
    uint32_t key[20];           // the ten round keys of the relaxation's Philox calls
    uint32_t hist[256];         // fixed-count selection: digits
    uint16_t spl[kSpillCap];    // the cell's spill-list entries (all of them, if need be)
    uint32_t nsp;
    uint32_t next;              // next unit
    uint32_t sel[4];            // fixed-count selection: broadcast words
};

// approximate functions with subnormal inputs and results flushed: the
// arguments here are never subnormal, and the plain forms scale for that
__device__ __forceinline__ float lg2_ftz(float x) { float y; asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float ex2_ftz(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float sqrt_ftz(float x) { float y; asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float rsqrt_ftz(float x) { float y; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float sin_ftz(float x) { float y; asm("sin.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float cos_ftz(float x) { float y; asm("cos.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

// per-cell constants of the relaxation: the record k_params_f writes.  X:
// e^a - 1 where a = nu_ES dt < 1, else -e^-a.
struct G2Prm {
    float u[3], th, M[6], pr, nu, inv_nues, pne, X, inv_pr;
};

__device__ __forceinline__ G2Prm g2_prm(const float* fprm, int cell) {
    const float4* r = reinterpret_cast<const float4*>(fprm) + (size_t)cell * (kNFPrm / 4);
    const float4 a = r[0], b = r[1], c = r[2], d = r[3];
    G2Prm f;
    f.u[0] = a.x; f.u[1] = a.y; f.u[2] = a.z; f.th = a.w;
    f.M[0] = b.x; f.M[1] = b.y; f.M[2] = b.z; f.M[3] = b.w;
    f.M[4] = c.x; f.M[5] = c.y; f.pr = c.z; f.nu = c.w;
    f.inv_nues = d.x; f.pne = d.y; f.X = d.z; f.inv_pr = d.w;
    return f;
}

// Philox4x32-10 for the relaxation of one particle, counter (pid, step,
// relax, 0): the round keys come from shared memory (five 16-byte broadcast
// loads instead of eighteen additions)
__device__ __forceinline__ uint4 philox_keys(uint32_t pid, uint32_t step, const uint32_t* key) {
    uint4 c = make_uint4(pid, step, kRelax, 0u);
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c.x;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c.z;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ key[2 * r], (uint32_t)p1,
                       (uint32_t)(p0 >> 32) ^ c.w ^ key[2 * r + 1], (uint32_t)p0);
    }
    return c;
}

// three independent normals from the four words of one Philox call: a
// Box-Muller pair (w.y, w.z) and a third one whose radius comes from w.w and
// whose angle comes from the 23 low bits that the uniforms of w.x, w.y and
// w.z leave unused (each takes the top 23 bits; lo + 1/2 over 2^23 is built
// from the bits, exactly).
__device__ __forceinline__ void g2_normals(const uint4& w, float* z) {
    const float r = sqrt_ftz(-1.3862943611198906f * lg2_ftz(u01<float>(w.y)));
    const float a = 6.283185307179586f * u01<float>(w.z) - 3.14159265358979f;
    z[0] = r * cos_ftz(a);
    z[1] = r * sin_ftz(a);
    const uint32_t lo = (w.x & 511u) | ((w.y & 511u) << 9) | ((w.z & 31u) << 18);
    const float r2 = sqrt_ftz(-1.3862943611198906f * lg2_ftz(u01<float>(w.w)));
    const float v = __uint_as_float(0x3F800000u | lo) - 0.99999994039535522f;
    z[2] = r2 * cos_ftz(6.283185307179586f * v - 3.14159265358979f);
}

// s of Eq. 32 at the time instant of Eq. 30.  u = u01(w.x) selects the
// particle (u < P_relax); given the selection u / P_relax is uniform on (0, 1]
// and gives the instant, in the overflow-free form of its range of a.
__device__ __forceinline__ float g2_instant(const SimDev& s, const G2Prm& f, float u) {
    const float U1 = fminf(u * f.inv_pr, 1.0f);
    const bool small = f.X > 0.0f;
    const float arg = (small ? U1 : 1.0f - U1) * fabsf(f.X) + (small ? 1.0f : U1);
    const float t = 0.6931471805599453f * lg2_ftz(arg) * f.inv_nues + (small ? 0.0f : s.f_dt);
    return f.pne + (1.0f - f.pne) * ex2_ftz(1.4426950408889634f * (-f.nu * t));
}

// new peculiar velocity: the sum sqrt(s) L xi1 + sqrt((1 - s) theta) xi2 of
// Eqs. 31-32 is one Gaussian of covariance s L L^T + (1 - s) theta I =
// theta I + s M, sampled through its own Cholesky factor
__device__ __forceinline__ void es_draw1(const SimDev& s, const G2Prm& f, float u, const uint4& w, float* C) {
    const float sf = g2_instant(s, f, u);
    float z[3];
    g2_normals(w, z);
    const float S00 = f.th + sf * f.M[0], S10 = sf * f.M[1], S11 = f.th + sf * f.M[2];
    const float S20 = sf * f.M[3], S21 = sf * f.M[4], S22 = f.th + sf * f.M[5];
    const float r0 = rsqrt_ftz(S00);
    const float l00 = S00 * r0, l10 = S10 * r0, l20 = S20 * r0;
    const float d1 = fmaxf(S11 - l10 * l10, 1e-12f * f.th);
    const float r1 = rsqrt_ftz(d1);
    const float l11 = d1 * r1, l21 = (S21 - l20 * l10) * r1;
    const float l22 = sqrt_ftz(fmaxf(S22 - l20 * l20 - l21 * l21, 0.0f));
    C[0] = l00 * z[0];
    C[1] = l10 * z[0] + l11 * z[1];
    C[2] = l20 * z[0] + l21 * z[1] + l22 * z[2];
}

// The Gallis-Torczynski draw (Eqs. 10-11) of the SP-ESBGK ablations: a
// thermal velocity sqrt(theta) z transformed by S = I - s B, B = ((1 - Pr) /
// (2 Pr)) sigma* / (rho theta) (symmetric; M holds its lower triangle) and s
// of Eq. 32 at the time instant.
__device__ __forceinline__ void es_draw_gt(const SimDev& s, const G2Prm& f, float u, const uint4& w, float* C) {
    const float sf = g2_instant(s, f, u);
    float z[3];
    g2_normals(w, z);
    const float st = sqrt_ftz(f.th);
    const float c0 = st * z[0], c1 = st * z[1], c2 = st * z[2];
    const float b00 = f.M[0], b10 = f.M[1], b11 = f.M[2], b20 = f.M[3], b21 = f.M[4], b22 = f.M[5];
    C[0] = c0 - sf * (b00 * c0 + b10 * c1 + b20 * c2);
    C[1] = c1 - sf * (b10 * c0 + b11 * c1 + b21 * c2);
    C[2] = c2 - sf * (b20 * c0 + b21 * c1 + b22 * c2);
}

// counters of one simulation, added when the block leaves it
struct G2Acc {
    uint32_t relaxed, removed;   // relaxed: thread 0's
};

__device__ __forceinline__ void g2_flush(G2Acc& a, SimDyn* dyn, int tid) {
    if (tid == 0 && a.relaxed) atomicAdd(&dyn->counters[kCntRelaxed], (unsigned long long)a.relaxed);
    const uint32_t r = __reduce_add_sync(0xffffffffu, a.removed);
    if ((tid & 31) == 0 && r) atomicAdd(&dyn->counters[kCntRemoved], (unsigned long long)r);
    a.relaxed = a.removed = 0;
}

// the id of particle j of a cell (bucket, then its spill-list entries)
__device__ __forceinline__ uint32_t g2_id(const SimDev& s, int p, uint32_t base, uint32_t nb, const uint16_t* spl,
                                          uint32_t j) {
    return j < nb ? s.pid[p][base + j] : s.sp_pid[p][spl[j - nb]];
}

// Eq. 9 fixed count for one cell: the ns = nearest-int(n P_relax) particles
// with the smallest selection words w.x (ties: lower position in the
// bucket).  T is the ns-th smallest word and `quota` the number of particles
// with word T that are taken; the (ns+1)-th smallest word T2 scales the time
// instants (given T2, the ns smallest words are independent and uniform
// below it).
struct G2Fixed {
    uint32_t T, quota, eq, ns;
    float inv_thr;
};

// the digit of the rem-th smallest word among the counted ones (one warp; lane l
// looks at digits [8 l, 8 l + 8)); below: how many words have a smaller digit
__device__ __forceinline__ uint32_t radix_digit(const uint32_t* hist, uint32_t rem, int lane, uint32_t& below) {
    uint32_t h[8], tot = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        h[i] = hist[8 * lane + i];
        tot += h[i];
    }
    uint32_t inc = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    const uint32_t exc = inc - tot;
    const unsigned own = __ballot_sync(0xffffffffu, exc < rem && rem <= inc);
    const int L = __ffs(own) - 1;
    uint32_t d = 0;
    below = exc;
    if (lane == L) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (below + h[i] >= rem) {
                d = 8u * lane + i;
                break;
            }
            below += h[i];
        }
    }
    d = __shfl_sync(0xffffffffu, d, L);
    below = __shfl_sync(0xffffffffu, below, L);
    return d;
}

// radix select of the ns-th smallest word: four passes of 8-bit digits
// counted in shared memory, then the ties and T2; every pass draws the words
// again
template <int G>
__device__ __noinline__ G2Fixed g2_fixed(G2Shared<G>& sh, int p, uint32_t step, uint32_t base, uint32_t nb, uint32_t n,
                                         float pr, int tid) {
    const SimDev& s = sh.sim;
    const int lane = tid & 31;
    G2Fixed F;
    F.ns = min((uint32_t)floorf((float)n * pr + 0.5f), n);
    F.T = 0xFFFFFFFFu;
    F.quota = F.eq = 0;
    F.inv_thr = 1.0f;
    if (F.ns == 0) return F;
    auto word = [&](uint32_t j) { return philox_keys(g2_id(s, p, base, nb, sh.spl, j), step, sh.key).x; };
    uint32_t prefix = 0, mask = 0, rem = F.ns;
    for (int shift = 24; shift >= 0; shift -= 8) {
        __syncthreads();
        for (int b = tid; b < 256; b += 32 * G) sh.hist[b] = 0u;
        __syncthreads();
        for (uint32_t j = tid; j < n; j += 32 * G) {
            const uint32_t k = word(j);
            if ((k & mask) == prefix) atomicAdd(&sh.hist[(k >> shift) & 255u], 1u);
        }
        __syncthreads();
        uint32_t below;
        const uint32_t d = radix_digit(sh.hist, rem, lane, below);   // (every warp for itself)
        rem -= below;
        prefix |= d << shift;
        mask |= 0xFFu << shift;
    }
    F.T = prefix;
    F.quota = rem;
    // words equal to T, and the smallest word above it
    __syncthreads();
    if (tid == 0) {
        sh.sel[0] = 0u;            // words equal to T
        sh.sel[1] = 0xFFFFFFFFu;   // smallest word above T
        sh.sel[2] = 0u;            // whether there is one
    }
    __syncthreads();
    uint32_t eq = 0, above = 0xFFFFFFFFu;
    bool any_above = false;
    for (uint32_t j = tid; j < n; j += 32 * G) {
        const uint32_t k = word(j);
        eq += k == F.T;
        if (k > F.T) {
            any_above = true;
            above = min(above, k);
        }
    }
    if (eq) atomicAdd(&sh.sel[0], eq);
    if (any_above) {
        atomicMin(&sh.sel[1], above);
        sh.sel[2] = 1u;
    }
    __syncthreads();
    F.eq = sh.sel[0];
    if (F.eq > F.quota) F.inv_thr = 1.0f / u01<float>(F.T);
    else if (sh.sel[2]) F.inv_thr = 1.0f / u01<float>(sh.sel[1]);
    return F;
}

// is particle j with word x among the fixed count?  Ties beyond the quota go
// to the lower positions (counted by drawing the words before j again).
template <int G>
__device__ __forceinline__ bool g2_fixed_takes(G2Shared<G>& sh, const G2Fixed& X, int p, uint32_t step, uint32_t base,
                                               uint32_t nb, uint32_t j, uint32_t x) {
    if (X.ns == 0 || x > X.T) return false;
    if (x < X.T || X.eq <= X.quota) return true;
    uint32_t rank = 0;
    for (uint32_t i = 0; i < j; ++i)
        rank += philox_keys(g2_id(sh.sim, p, base, nb, sh.spl, i), step, sh.key).x == X.T;
    return rank < X.quota;
}

// the cell's spill-list entries into sh.spl (whole block); returns their count
template <int G>
__device__ __noinline__ uint32_t g2_collect(G2Shared<G>& sh, int p, int cell, int tid) {
    const SimDev& s = sh.sim;
    __syncthreads();
    if (tid == 0) sh.nsp = 0;
    __syncthreads();
    const uint32_t n = min(s.dyn->sp_n[p], (uint32_t)kSpillCap);
    for (uint32_t i = tid; i < n; i += 32 * G)
        if (s.sp_cell[p][i] == (uint32_t)cell) sh.spl[atomicAdd(&sh.nsp, 1u)] = (uint16_t)i;
    __syncthreads();
    return sh.nsp;
}

// one cell: bucket [base, base + nb) of buffer p, `arrived` arrivals
template <int DIM, int MODE, bool ABL, int G>
__device__ __forceinline__ void g2_cell(const SimDev* __restrict__ sims, G2Shared<G>& sh, int cell, uint32_t base,
                                        uint32_t nb, uint32_t arrived, int p, uint32_t step, bool pending, int tid,
                                        G2Acc& acc) {
    constexpr uint32_t T = 32 * G, CAP = T * kG2P;
    const SimDev& s = sh.sim;
    const int lane = tid & 31, warp = tid >> 5, q = p ^ 1;
    uint32_t nsp = 0;
    if (arrived > nb) nsp = g2_collect<G>(sh, p, cell, tid);
    const uint32_t n = nb + nsp;
    if (n == 0) return;
    G2Prm f = g2_prm(s.fprm, cell);
    const bool relax = pending && f.pr > 0.0f;
    if (MODE == kRelaxOnly && !relax) return;
    // the window: thread k < 64 looks after slot k, its bucket bounds read ahead
    const int cy = DIM == 2 ? cell / s.nx : 0;
    const int cx = DIM == 2 ? cell - cy * s.nx : 0;
    const int gcell = cell + (MODE == kFullSlab && DIM == 1 ? s.row0 : 0);   // 1-D: global cell of the slab's cell
    const int row0 = MODE == kFullSlab && DIM == 2 ? s.row0 : 0;
    const int cell0 = MODE == kFullSlab ? s.row0 * s.nx : 0;
    int dest = -1;
    uint32_t dlo = 0, dhi = 0;
    if (MODE != kRelaxOnly && tid < kWin) {
        dest = win_cell<DIM>(tid, cell, cx, cy, s.nx);
        if ((unsigned)dest < (unsigned)s.K) {
            dlo = s.lay[q][dest];
            dhi = min(s.lay[q][dest + 1], (uint32_t)s.cap);
        }
    }
    G2Fixed X = {0u, 0u, 0u, 0u, 1.0f};
    if (ABL && relax && s.selection) {
        X = g2_fixed<G>(sh, p, step, base, nb, n, f.pr, tid);
        f.inv_pr = X.inv_thr;   // the instants scale with the threshold word instead of P_relax
    }
    const uint32_t nch = (n + CAP - 1) / CAP;
    float R[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) R[k] = 0.0f;
    uint32_t nr = 0;
    float uo0 = 0, uo1 = 0, uo2 = 0, mn0 = 0, mn1 = 0, mn2 = 0, alpha = 1.0f;
    bool apply = false;
    // sweep 1: chunks 0 .. nch - 1 (sums); sweep 2: nch - 1 .. 0 (moves)
#pragma unroll 1
    for (uint32_t it = relax ? 0 : nch - 1; it < 2 * nch - 1; ++it) {
        const uint32_t off = (it < nch ? it : 2 * nch - 2 - it) * CAP;
        const uint32_t cnt = min(CAP, n - off);      // particles of the chunk
        float x[kG2P], y[kG2P], v[kG2P][3];
        uint32_t id[kG2P], selm = 0;
#pragma unroll
        for (int k = 0; k < kG2P; ++k) {
            const uint32_t j = tid + k * T;
            x[k] = y[k] = v[k][0] = v[k][1] = v[k][2] = 0.0f;
            id[k] = 0;
            if (j < cnt)
                load_particle<DIM>(s, p, base, nb, sh.spl, off + j, x[k], y[k], v[k][0], v[k][1], v[k][2], id[k]);
        }
        if (relax) {
#pragma unroll
            for (int k = 0; k < kG2P; ++k) {
                if (32u * warp + k * T >= cnt) break;
                const uint32_t j = tid + k * T;
                const uint4 w = philox_keys(id[k], step, sh.key);
                const float u = u01<float>(w.x);
                bool sel;
                if (ABL && s.selection) {
                    sel = j < cnt && g2_fixed_takes<G>(sh, X, p, step, base, nb, off + j, w.x);
                } else {
                    sel = j < cnt && u < f.pr;
                }
                if (sel) {
                    float C[3];
                    if (ABL && s.es_sampler) es_draw_gt(s, f, u, w, C);
                    else es_draw1(s, f, u, w, C);
                    const float o0 = v[k][0] - f.u[0], o1 = v[k][1] - f.u[1], o2 = v[k][2] - f.u[2];
                    R[0] += o0; R[1] += o1; R[2] += o2;
                    R[3] += o0 * o0 + o1 * o1 + o2 * o2;
                    R[4] += C[0]; R[5] += C[1]; R[6] += C[2];
                    R[7] += C[0] * C[0] + C[1] * C[1] + C[2] * C[2];
                    v[k][0] = C[0]; v[k][1] = C[1]; v[k][2] = C[2];
                    selm |= 1u << k;
                }
                if (it < nch) nr += (uint32_t)__popc(__ballot_sync(0xffffffffu, sel));
            }
        }
        if (it + 1 < nch) continue;
        if (it + 1 == nch && relax) {
            // conservation factors from the block's sums.  Warp: reduce-scatter
            // of the eight sums (lane 4 i holds sum i); block: through shared
            // memory, every warp adding the G partial sums.
#pragma unroll
            for (int half = 4; half >= 1; half >>= 1) {
                const bool up = (lane & (4 * half)) != 0;
#pragma unroll
                for (int i = 0; i < half; ++i) {
                    const float send = up ? R[i] : R[i + half];
                    const float recv = __shfl_xor_sync(0xffffffffu, send, 4 * half);
                    R[i] = (up ? R[i + half] : R[i]) + recv;
                }
            }
            R[0] += __shfl_xor_sync(0xffffffffu, R[0], 2);
            R[0] += __shfl_xor_sync(0xffffffffu, R[0], 1);
            if ((lane & 3) == 0) sh.part[warp][lane >> 2] = R[0];
            if (lane == 0) sh.part_n[warp] = nr;
            __syncthreads();
            float t = sh.part[lane >> 3][lane & 7];
#pragma unroll
            for (int g = 4; g < G; g += 4) t += sh.part[g + (lane >> 3)][lane & 7];
            t += __shfl_xor_sync(0xffffffffu, t, 8);
            t += __shfl_xor_sync(0xffffffffu, t, 16);
            uint32_t nall = 0;
#pragma unroll
            for (int g = 0; g < G; ++g) nall += sh.part_n[g];
            float Q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) Q[k] = __shfl_sync(0xffffffffu, t, k);
            if (nall >= 2) {
                // FP32: the sums are taken about the cell mean, so the
                // differences below do not cancel; every thread computes the
                // same factors from the same values
                const float inv = 1.0f / (float)nall;
                const float Eo = Q[3] - (Q[0] * Q[0] + Q[1] * Q[1] + Q[2] * Q[2]) * inv;
                const float En = Q[7] - (Q[4] * Q[4] + Q[5] * Q[5] + Q[6] * Q[6]) * inv;
                if (En > 0.0f && Eo >= 0.0f) {
                    apply = true;
                    alpha = sqrtf(Eo / En);
                    uo0 = f.u[0] + Q[0] * inv;
                    uo1 = f.u[1] + Q[1] * inv;
                    uo2 = f.u[2] + Q[2] * inv;
                    mn0 = Q[4] * inv;
                    mn1 = Q[5] * inv;
                    mn2 = Q[6] * inv;
                    if (tid == 0) acc.relaxed += nall;
                }
            }
        }
        if (MODE == kRelaxOnly) {
            if (apply) {
#pragma unroll
                for (int k = 0; k < kG2P; ++k)
                    if (selm & (1u << k))
                        store_velocity(s, p, base, nb, sh.spl, off + tid + k * T, uo0 + alpha * (v[k][0] - mn0),
                                       uo1 + alpha * (v[k][1] - mn1), uo2 + alpha * (v[k][2] - mn2));
            }
            continue;
        }
        uint32_t sr[kG2P];   // slot, rank << 8
#pragma unroll
        for (int k = 0; k < kG2P; ++k) {
            sr[k] = kSlotNone;
            if (32 * warp + k * T >= cnt) break;
            const uint32_t j = tid + k * T;
            if (j >= cnt) continue;
            if (selm & (1u << k)) {
                if (apply) {
                    v[k][0] = uo0 + alpha * (v[k][0] - mn0);
                    v[k][1] = uo1 + alpha * (v[k][1] - mn1);
                    v[k][2] = uo2 + alpha * (v[k][2] - mn2);
                } else {   // a single relaxed particle: reverted
                    float ox, oy;
                    uint32_t oid;
                    load_particle<DIM>(s, p, base, nb, sh.spl, off + j, ox, oy, v[k][0], v[k][1], v[k][2], oid);
                }
            }
            const float x0 = x[k], y0 = y[k];
            const bool alive = advect_fast<DIM>(s, step, id[k], x[k], y[k], v[k]);
            if ((MODE == kFullFlux || MODE == kFullSlab) && s.flux_axis) count_flux<float>(s, x0, y0, x[k], y[k]);
            if (!alive) continue;
            int ix, iy;
            cell_xy<DIM>(s, x[k], y[k], ix, iy);
            const int dc = (DIM == 2 ? iy * s.nx + ix : iy) - cell0;   // local
            if (MODE == kFullSlab && (unsigned)dc >= (unsigned)s.K) {
                sr[k] = kSlotOther;
            } else if (s.has_reservoir && in_buffer_xy(s, ix, iy)) {
                ++acc.removed;
            } else {
                const int slot = win_slot_xy<DIM>(ix, iy - row0, gcell, cx, cy);
                sr[k] = kSlotFar;
                // the particle's rank among the arrivals of its slot: one shared
                // atomic (lanes of one slot are served one after another)
                if (slot >= 0) sr[k] = (uint32_t)slot | (atomicAdd(&sh.wcnt[slot], 1u) << 8);
            }
        }
        __syncthreads();
        // one reservation per occupied slot, all in flight together
        if (tid < kWin) {
            const uint32_t c = sh.wcnt[tid];
            if (c) {
                sh.wstart[tid] = dlo + atomicAdd(&s.cnt[q][dest], c);
                sh.wend[tid] = dhi;
                sh.wcnt[tid] = 0;
            }
        }
        __syncthreads();
        // consecutive lanes write particles of the same few destination
        // buckets (a window slot's particles go to consecutive slots of its
        // bucket, in rank order); particles leaving the window or the slab
        // take their own reservation
#pragma unroll
        for (int k = 0; k < kG2P; ++k) {
            if (32 * warp + k * T >= cnt) break;
            const uint32_t slot = sr[k] & 255u;
            if (slot == kSlotNone) continue;
            uint32_t i, hi;
            if (slot < (uint32_t)kWin) {
                i = sh.wstart[slot] + (sr[k] >> 8);
                hi = sh.wend[slot];
            } else if (MODE == kFullSlab && slot == kSlotOther) {   // into the buckets of another slab
                emit_other<DIM>(sims, s, q, x[k], y[k], v[k][0], v[k][1], v[k][2], id[k]);
                continue;
            } else {   // outside the window: a reservation of its own
                int ix, iy;
                cell_xy<DIM>(s, x[k], y[k], ix, iy);
                const int dc = (DIM == 2 ? iy * s.nx + ix : iy) - cell0;
                i = s.lay[q][dc] + atomicAdd(&s.cnt[q][dc], 1u);
                hi = min(s.lay[q][dc + 1], (uint32_t)s.cap);
            }
            if (i < hi) {
                if (DIM == 2) ((float*)s.pos[q][0])[i] = x[k];
                ((float*)s.pos[q][1])[i] = y[k];
                ((float*)s.vel[q][0])[i] = v[k][0];
                ((float*)s.vel[q][1])[i] = v[k][1];
                ((float*)s.vel[q][2])[i] = v[k][2];
                s.pid[q][i] = id[k];
            } else {   // the bucket is full
                int ix, iy;
                cell_xy<DIM>(s, x[k], y[k], ix, iy);
                spill<DIM>(s, q, (DIM == 2 ? iy * s.nx + ix : iy) - cell0, x[k], y[k], v[k][0], v[k][1], v[k][2],
                           id[k]);
            }
        }
    }
    // kRelaxOnly has no barrier after the sums are read: the next cell's
    // partial sums wait for it
    if (MODE == kRelaxOnly) __syncthreads();
}

// DIMS: bit 0 / 1: the batch holds 1-D / 2-D simulations
template <int DIMS, int MODE, bool ABL, int G>
__global__ void __launch_bounds__(32 * G, kG2Warps / G) k_g2b(const SimDev* __restrict__ sims, const int2* __restrict__ tiles,
                                                       const int* __restrict__ ntiles, uint32_t* __restrict__ wq) {
    __shared__ __align__(16) G2Shared<G> sh;
    const int tid = threadIdx.x;
    const uint32_t slots = (uint32_t)*ntiles * kCTile;
    // units of 1 to 8 cells, at least 32 units per block where there are enough cells
    uint32_t U = 1;
    while (U < 8 && slots >= U * 64 * gridDim.x) U *= 2;
    const uint32_t nunits = slots / U;
    if (tid < kWin) sh.wcnt[tid] = 0;
    G2Acc acc = {0u, 0u};
    int loaded = -1, p = 0;
    uint32_t step = 0;
    bool pending = false;
    for (uint32_t unit = blockIdx.x; unit < nunits;) {
        uint32_t nxt = 0;
        if (tid == 0) nxt = gridDim.x + atomicAdd(&wq[0], 1u);
        const uint32_t slot0 = unit * U;
        const int2 tile = tiles[slot0 / kCTile];
        if (tile.x != loaded) {
            if (loaded >= 0) g2_flush(acc, sh.sim.dyn, tid);
            __syncthreads();
            load_sim(sh.sim, sims[tile.x]);
            __syncthreads();
            loaded = tile.x;
            p = sh.sim.dyn->cur;
            step = sh.sim.dyn->step;
            pending = sh.sim.dyn->relax_pending != 0;
            if (tid < 10) {   // round keys: the key plus r times the Weyl constants
                sh.key[2 * tid] = sh.sim.key0 + (uint32_t)tid * 0x9E3779B9u;
                sh.key[2 * tid + 1] = sh.sim.key1 + (uint32_t)tid * 0xBB67AE85u;
            }
            __syncthreads();
        }
        const SimDev& s = sh.sim;
        const int c0 = tile.y + (int)(slot0 % kCTile), c1 = min(c0 + (int)U, s.K);
        if (c0 < c1 && !(MODE == kRelaxOnly && !pending)) {
            const uint32_t cap = (uint32_t)s.cap;
            uint32_t lo = s.lay[p][c0], hi = s.lay[p][c0 + 1], ar = s.cnt[p][c0];
            for (int cell = c0; cell < c1; ++cell) {
                const uint32_t base = lo, top = min(hi, cap), arrived = ar;
                if (cell + 1 < c1) {   // the next cell's bounds
                    lo = hi;
                    hi = s.lay[p][cell + 2];
                    ar = s.cnt[p][cell + 1];
                }
                const uint32_t nb = min(arrived, top > base ? top - base : 0u);
                if (DIMS == 1 || (DIMS == 3 && s.dim == 1))
                    g2_cell<1, MODE, ABL, G>(sims, sh, cell, base, nb, arrived, p, step, pending, tid, acc);
                else
                    g2_cell<2, MODE, ABL, G>(sims, sh, cell, base, nb, arrived, p, step, pending, tid, acc);
            }
        }
        __syncthreads();
        if (tid == 0) sh.next = nxt;
        __syncthreads();
        unit = sh.next;
    }
    if (loaded >= 0) g2_flush(acc, sh.sim.dyn, tid);
    if (tid == 0) {
        __threadfence();
        const uint32_t done = atomicAdd(&wq[1], 1u);
        if (done == gridDim.x - 1) wq[0] = wq[1] = 0;   // the last block resets the counters for the next launch
    }
}

// copy one simulation descriptor into shared memory (one warp)
__device__ __forceinline__ void load_sim_warp(SimDev& dst, const SimDev& src, int lane) {
    const int4* a = reinterpret_cast<const int4*>(&src);
    int4* b = reinterpret_cast<int4*>(&dst);
    for (int i = lane; i < (int)(sizeof(SimDev) / 16); i += 32) b[i] = a[i];
}

// ---------------------------------------------------------------------------
// k_g2: the same work for domains of many cells, one warp per cell.
//
// With many cells per SM the work is bound by instruction issue, not by a
// cell's latency: a warp of its own per cell needs no block barriers, wastes
// no lanes on the per-cell part and leaves at most 31 lanes of a cell idle.
// The warps of a block are independent; each keeps its own copy of the
// simulation descriptor and its own staging area in shared memory.  A cell:
//   copy     its planes and parameter record come in by bulk asynchronous
//            copies (one per plane), started while the cell before it is worked on wherever both fit
//            the staging area (its bounds are read another cell ahead, the
//            unit number yet another), so that a cell finds its data there;
//   sweep 1  relaxation draw, conservation sums, the new velocity staged;
//   sweep 2  conservation, flight, destination slot and rank, staged;
//   reserve  one global atomic per occupied slot;
//   sweep 3  the writes, consecutive lanes to consecutive slots.
// The two particles per lane and iteration are independent chains.  16 warps
// per SM with 128 registers and no spills measured best (12 and 14 warps with
// more staging, 18 and 20 with less and some spills: 3-50 % slower), and so did
// bulk copies (per-lane 16-byte copies took three times as long to issue).
// Two codings of the same cell can differ by 1 % in 2-D, where the kernel is at
// the edge of the instruction cache (the window as one array: 157.5 -> 158.3 us a
// step of the cavity).
// What bounds it: the warps' dependent instructions (370 per 32 particles in
// 1-D, 48 % issue) and, for dense cells, the copy that cannot start before the
// cell ahead is written.  Against the form before it (a producer warp feeding
// seven consumer warps): 64 shock tubes 301 -> 255 us, cavity 200 x 200 168 ->
// 119 us, slit 522 -> 388 us per launch.
// Cells above the staging area, and cells with spill-list entries, take the
// general form of the same code: loaded by the lanes (asynchronously, a chunk
// at once: 20 000 cells of 600 particles 692 -> 324 us a step), in chunks, the
// draws of all but one chunk made twice.  Domains whose cells are mostly above
// the area of four blocks per SM run three with more staging (choose_form).
//
// The wait for a copy is bounded (kG2WaitNs of global time); one that runs out
// adds kG2TimeoutMark to the overflow counter of simulation 0 and ends the
// warp's work, so that a fault shows up as lost particles, not as a hang.
// ---------------------------------------------------------------------------
constexpr int kG2wWarps = 4;    // warps per block

template <int DIMS, bool ABL, int BLOCKS>   // BLOCKS per SM
struct alignas(16) G2Warp {
    // staged particles (an ablation's larger window takes some of three blocks' space)
    static constexpr uint32_t CAP = kG2Stage[BLOCKS - 3][DIMS - 1] - (ABL && BLOCKS == 3 ? 32u : 0u);
    float stage[(DIMS == 1 ? 5 : 6) * CAP + CAP / 2];                 // (x,) y, v0, v1, v2, id and 16-bit slots
    float prm[2][kNFPrm];  // parameter records of the cell and of the next one
    SimDev sim;
    uint32_t key[20];
    uint32_t wst[kWin];    // arrivals per window slot, then its first reserved index
    uint32_t wlo[kWin];    // start and end of the slot's bucket
    uint32_t wend[ABL ? 2 * kWin : kWin];
    // the digit counts of a fixed-count selection, before the window is used
    __device__ __forceinline__ uint32_t* hist() {
        return reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(this) + offsetof(G2Warp, wst));
    }
    int2 ptile[4];         // the cells on their way: tile,
    uint32_t pbound[4][4]; // bucket start, end and arrivals,
    uint32_t punit[4];     // unit number
    uint64_t full[2];      // the copies of a cell have landed (cells alternate)
};

// slot and rank of a staged particle in 16 bits (at most 1023 arrivals of one
// cell share a slot)
constexpr uint32_t kPackNone = 0xFFFFu;   // removed, nothing to write
constexpr uint32_t kPackFar = 0xFFFEu;    // outside the window
constexpr uint32_t kPackOther = 0xFFFDu;  // in another slab of a decomposed domain

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// per-lane asynchronous global -> shared copies (completion waited with
// cp.async.wait_group by the issuing lane, then made visible to the warp
// with __syncwarp)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }


constexpr unsigned long long kG2WaitNs = 2000000000ull;   // bound of one mbarrier wait
constexpr unsigned long long kG2TimeoutMark = 1ull << 40;

// ---- mbarrier and bulk-copy primitives (PTX, sm_90+) ----------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_tx(uint64_t* bar, uint32_t tx) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(smem_u32(bar)),
                 "r"(tx)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// wait for the phase of `bar` with the given parity to complete, at most
// kG2WaitNs; false when the bound ran out
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (;;) {
        for (int k = 0; k < 64; ++k)
            if (mbar_try_wait(bar, parity)) return true;
        if (global_ns() - t0 > kG2WaitNs) return false;
    }
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// the same range into L2 only
__device__ __forceinline__ void bulk_prefetch(const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// order this thread's generic-proxy accesses to shared memory before later
// bulk copies (async proxy) into the same bytes
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// registers of one warp's current simulation
struct G2Sim {
    uint32_t step;
    int p;
    bool pending, aligned;   // aligned: every plane starts on a 16-byte boundary
};

__device__ __forceinline__ uint32_t atom_add_global(uint32_t* p, uint32_t v) {
    uint32_t r;
    asm volatile("atom.global.add.u32 %0, [%1], %2;" : "=r"(r) : "l"(__cvta_generic_to_global(p)), "r"(v) : "memory");
    return r;
}

// a cell on its way through a warp: its bounds, and where it is staged
struct G2Job {
    int cell;              // -1: none
    uint32_t base, nb, arrived;
    uint32_t ro;           // first staged particle
};

// start the bulk copies of a cell's bucket and parameter record (lane 0):
// whole 16-byte groups, bucket starts and the capacity being multiples of
// four slots
template <int DIM, class Sh>
__device__ __forceinline__ void g2w_copy(Sh& sh, const G2Job& J, int p, uint32_t parity) {
    constexpr uint32_t CAP = Sh::CAP;
    const SimDev& s = sh.sim;
    float* const d = sh.stage + J.ro;
    const uint32_t bytes = 4u * ((J.nb + 3u) & ~3u);
    uint64_t* const bar = &sh.full[parity];
    mbar_arrive_tx(bar, (DIM == 2 ? 6u : 5u) * bytes + 4u * kNFPrm);
    bulk_g2s(sh.prm[parity], s.fprm + (size_t)J.cell * kNFPrm, 4u * kNFPrm, bar);
    bulk_g2s(d + 4 * CAP, s.pid[p] + J.base, bytes, bar);
    bulk_g2s(d + 1 * CAP, (const float*)s.vel[p][0] + J.base, bytes, bar);
    bulk_g2s(d + 2 * CAP, (const float*)s.vel[p][1] + J.base, bytes, bar);
    bulk_g2s(d + 3 * CAP, (const float*)s.vel[p][2] + J.base, bytes, bar);
    bulk_g2s(d, (const float*)s.pos[p][1] + J.base, bytes, bar);
    if (DIM == 2) bulk_g2s(d + 5 * CAP, (const float*)s.pos[p][0] + J.base, bytes, bar);
}

// the same by the lanes, for buckets that are not 16-byte aligned (the
// compact layout right after a set-up sort)
template <int DIM, class Sh>
__device__ __noinline__ void g2w_load(Sh& sh, G2Job J, int p, uint32_t parity, int lane) {
    constexpr uint32_t CAP = Sh::CAP;
    const SimDev& s = sh.sim;
    float* const d = sh.stage + J.ro;
    if (lane < kNFPrm) sh.prm[parity][lane] = s.fprm[(size_t)J.cell * kNFPrm + lane];
    for (uint32_t k = lane; k < J.nb; k += 32u) {
        const uint32_t i = J.base + k;
        d[k] = ((const float*)s.pos[p][1])[i];
        d[k + 1 * CAP] = ((const float*)s.vel[p][0])[i];
        d[k + 2 * CAP] = ((const float*)s.vel[p][1])[i];
        d[k + 3 * CAP] = ((const float*)s.vel[p][2])[i];
        reinterpret_cast<uint32_t*>(d)[k + 4 * CAP] = s.pid[p][i];
        if (DIM == 2) d[k + 5 * CAP] = ((const float*)s.pos[p][0])[i];
    }
    __syncwarp();
}

template <int V>
struct Num {
    static constexpr int value = V;
};

// the fixed count of one cell by one warp, its ids staged at J.ro or (GEN) read
// from the bucket and the spill list.  f(j, word) for every particle j
template <bool GEN, class Sh, class F>
__device__ __forceinline__ void g2w_words(const Sh& sh, const G2Sim& S, const G2Job& J, uint32_t nsp, int lane,
                                          const F& f) {
    const SimDev& s = sh.sim;
    const uint32_t* const st_id = reinterpret_cast<const uint32_t*>(sh.stage + 4 * Sh::CAP) + J.ro;
    for (uint32_t j = lane; j < J.nb; j += 32)
        f(j, philox_keys(GEN ? s.pid[S.p][J.base + j] : st_id[j], S.step, sh.key).x);
    if (GEN && nsp)
        each_spilled(s, S.p, J.cell, lane, [&](uint32_t rank, uint32_t i) {
            f(J.nb + rank, philox_keys(s.sp_pid[S.p][i], S.step, sh.key).x);
        });
}

template <bool GEN, class Sh>
__device__ __noinline__ G2Fixed g2w_fixed(Sh& sh, G2Sim S, G2Job J, uint32_t nsp, float pr, int lane) {
    const uint32_t n = J.nb + nsp;
    G2Fixed F;
    F.ns = min((uint32_t)floorf((float)n * pr + 0.5f), n);
    F.T = 0xFFFFFFFFu;
    F.quota = F.eq = 0;
    F.inv_thr = 1.0f;
    if (F.ns == 0) return F;
    uint32_t* const hist = sh.hist();
    uint32_t prefix = 0, mask = 0, rem = F.ns;
    for (int shift = 24; shift >= 0; shift -= 8) {
        __syncwarp();
        for (int b = lane; b < 256; b += 32) hist[b] = 0u;
        __syncwarp();
        g2w_words<GEN>(sh, S, J, nsp, lane, [&](uint32_t, uint32_t k) {
            if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1u);
        });
        __syncwarp();
        uint32_t below;
        const uint32_t d = radix_digit(hist, rem, lane, below);
        rem -= below;
        prefix |= d << shift;
        mask |= 0xFFu << shift;
    }
    F.T = prefix;
    F.quota = rem;
    // words equal to T, and the smallest word above it
    uint32_t eq = 0, above = 0xFFFFFFFFu;
    bool any_above = false;
    g2w_words<GEN>(sh, S, J, nsp, lane, [&](uint32_t, uint32_t k) {
        eq += k == F.T;
        if (k > F.T) {
            any_above = true;
            above = min(above, k);
        }
    });
    __syncwarp();
    F.eq = __reduce_add_sync(0xffffffffu, eq);
    above = __reduce_min_sync(0xffffffffu, above);
    if (F.eq > F.quota) F.inv_thr = 1.0f / u01<float>(F.T);
    else if (__any_sync(0xffffffffu, any_above)) F.inv_thr = 1.0f / u01<float>(above);
    return F;
}

// is particle j with word x among the fixed count?  (one lane; as g2_fixed_takes)
template <bool GEN, class Sh>
__device__ __noinline__ bool g2w_fixed_takes(const Sh& sh, G2Sim S, G2Job J, G2Fixed X, uint32_t j, uint32_t x) {
    if (X.ns == 0 || x > X.T) return false;
    if (x < X.T || X.eq <= X.quota) return true;
    const SimDev& s = sh.sim;
    const uint32_t* const st_id = reinterpret_cast<const uint32_t*>(sh.stage + 4 * Sh::CAP) + J.ro;
    uint32_t rank = 0;
    for (uint32_t i = 0; i < min(j, J.nb); ++i)
        rank += philox_keys(GEN ? s.pid[S.p][J.base + i] : st_id[i], S.step, sh.key).x == X.T;
    if (GEN && j > J.nb) {
        const uint32_t m = min(s.dyn->sp_n[S.p], (uint32_t)kSpillCap);
        for (uint32_t i = 0, k = J.nb; i < m && k < j; ++i)
            if (s.sp_cell[S.p][i] == (uint32_t)J.cell) {
                rank += philox_keys(s.sp_pid[S.p][i], S.step, sh.key).x == X.T;
                ++k;
            }
    }
    return rank < X.quota;
}

// one cell.  GEN: loaded here, in chunks, with spill-list entries; else it is
// staged at J.ro
template <int DIM, int MODE, bool ABL, bool GEN, class Sh>
__device__ __forceinline__ void g2w_cell_impl(const SimDev* __restrict__ sims, Sh& sh, const G2Sim& S, const G2Job& J,
                                              uint32_t parity, uint32_t nsp, int lane, G2Acc& acc) {
    constexpr uint32_t CAP = Sh::CAP;
    const SimDev& s = sh.sim;
    const int p = S.p, q = p ^ 1, cell = J.cell;
    const uint32_t base = J.base, nb = J.nb, n = nb + nsp, ro = GEN ? 0u : J.ro;
    float* const st_y = sh.stage;
    float* const st_0 = st_y + CAP;
    float* const st_1 = st_0 + CAP;
    float* const st_2 = st_1 + CAP;
    uint32_t* const st_id = reinterpret_cast<uint32_t*>(st_2 + CAP);
    float* const st_x = st_2 + 2 * CAP;   // 2-D only
    uint16_t* const st_r = reinterpret_cast<uint16_t*>(st_2 + (DIM == 2 ? 3 : 2) * CAP);
    G2Prm f = GEN ? g2_prm(s.fprm, cell) : g2_prm(sh.prm[parity], 0);
    const bool relax = S.pending && f.pr > 0.0f;
    if (MODE == kRelaxOnly && !relax) return;
    G2Fixed X = {0u, 0u, 0u, 0u, 1.0f};
    if (ABL && relax && s.selection) {
        X = g2w_fixed<GEN>(sh, S, J, nsp, f.pr, lane);
        f.inv_pr = X.inv_thr;   // the instants scale with the threshold word instead of P_relax
        __syncwarp();
    }
    // the window: lane k looks after slots k and k + 32, their bucket bounds read ahead
    const int cy = DIM == 2 ? cell / s.nx : 0;
    const int cx = DIM == 2 ? cell - cy * s.nx : 0;
    const int gcell = cell + (MODE == kFullSlab && DIM == 1 ? s.row0 : 0);   // 1-D: global cell of the slab's cell
    const int row0 = MODE == kFullSlab && DIM == 2 ? s.row0 : 0;
    const int cell0 = MODE == kFullSlab ? s.row0 * s.nx : 0;
#pragma unroll
    for (int h = 0; MODE != kRelaxOnly && h < 2; ++h) {
        const int k = lane + 32 * h, dest = win_cell<DIM>(k, cell, cx, cy, s.nx);
        if ((unsigned)dest < (unsigned)s.K) {
            cp_async4(&sh.wlo[k], &s.lay[q][dest]);
            cp_async4(&sh.wend[k], &s.lay[q][dest + 1]);
        }
        sh.wst[k] = 0;
    }
    const uint32_t nch = GEN ? (n + CAP - 1) / CAP : 1u;
    float R[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) R[k] = 0.0f;
    uint32_t nr = 0;
    // GEN: particles [off, off + cnt) of the cell, the bucket's and then the spill list's
    auto load_chunk = [&](uint32_t off, uint32_t cnt) {
        // (all of the chunk in flight at once)
#pragma unroll 1
        for (uint32_t j = lane; j < cnt && off + j < nb; j += 32) {
            const uint32_t i = base + off + j;
            if (DIM == 2) cp_async4(st_x + j, (const float*)s.pos[p][0] + i);
            cp_async4(st_y + j, (const float*)s.pos[p][1] + i);
            cp_async4(st_0 + j, (const float*)s.vel[p][0] + i);
            cp_async4(st_1 + j, (const float*)s.vel[p][1] + i);
            cp_async4(st_2 + j, (const float*)s.vel[p][2] + i);
            cp_async4(st_id + j, s.pid[p] + i);
        }
        if (off + cnt > nb) each_spilled(s, p, cell, lane, [&](uint32_t rank, uint32_t i) {
            const uint32_t j = nb + rank - off;   // (far above cnt where it lies before off)
            if (j >= cnt) return;
            if (DIM == 2) st_x[j] = s.sp_pos[p][0][i];
            st_y[j] = s.sp_pos[p][1][i];
            st_0[j] = s.sp_vel[p][0][i];
            st_1[j] = s.sp_vel[p][1][i];
            st_2[j] = s.sp_vel[p][2][i];
            st_id[j] = s.sp_pid[p][i];
        });
        cp_async_wait_all();
        __syncwarp();
    };
    float al = 1.0f, uo0 = 0, uo1 = 0, uo2 = 0, mn0 = 0, mn1 = 0, mn2 = 0;
    bool apply = false;
#pragma unroll 1
    for (uint32_t it = relax || !GEN ? 0 : nch - 1; it < 2 * nch - 1; ++it) {
        const uint32_t off = GEN ? (it < nch ? it : 2 * nch - 2 - it) * CAP : 0u;
        const uint32_t cnt = GEN ? min(CAP, n - off) : n;
        if (GEN) {
            __syncwarp();
            load_chunk(off, cnt);
        }
        uint32_t selm = 0;   // bit i: the lane's particle of iteration i is relaxed
        // ---- sweep 1: each lane on its own particles, two at a time (lanes
        // past the end work on what is there, unselected) ----
        if (relax) {
            auto draw = [&](auto nt, uint32_t b) {
                constexpr int N = decltype(nt)::value;
                uint4 w[N];
                float u[N], C[N][3];
                bool sel[N], any = false;
#pragma unroll
                for (int t = 0; t < N; ++t) w[t] = philox_keys(st_id[ro + b + 32 * t + lane], S.step, sh.key);
#pragma unroll
                for (int t = 0; t < N; ++t) {
                    u[t] = u01<float>(w[t].x);
                    sel[t] = b + 32 * t + lane < cnt;
                    if (ABL && s.selection)
                        sel[t] = sel[t] && g2w_fixed_takes<GEN>(sh, S, J, X, off + b + 32 * t + lane, w[t].x);
                    else
                        sel[t] = sel[t] && u[t] < f.pr;
                    any = any || sel[t];
                }
                if (!__any_sync(0xffffffffu, any)) return;
#pragma unroll
                for (int t = 0; t < N; ++t) {
                    if (ABL && s.es_sampler) es_draw_gt(s, f, u[t], w[t], C[t]);
                    else es_draw1(s, f, u[t], w[t], C[t]);
                }
#pragma unroll
                for (int t = 0; t < N; ++t) {
                    const uint32_t j = ro + b + 32 * t + lane;
                    const float o0 = st_0[j] - f.u[0], o1 = st_1[j] - f.u[1], o2 = st_2[j] - f.u[2];
                    if (sel[t]) {
                        R[0] += o0; R[1] += o1; R[2] += o2;
                        R[3] += o0 * o0 + o1 * o1 + o2 * o2;
                        R[4] += C[t][0]; R[5] += C[t][1]; R[6] += C[t][2];
                        R[7] += C[t][0] * C[t][0] + C[t][1] * C[t][1] + C[t][2] * C[t][2];
                        st_0[j] = C[t][0];
                        st_1[j] = C[t][1];
                        st_2[j] = C[t][2];
                        selm |= 1u << ((b >> 5) + t);
                    }
                }
            };
            uint32_t b = 0;
#pragma unroll 1
            for (; b + 32 < cnt; b += 64) draw(Num<2>{}, b);
            if (b < cnt) draw(Num<1>{}, b);
            if (!GEN || it < nch) nr += (uint32_t)__popc(selm);
        }
        if (GEN && it + 1 < nch) continue;
        if ((!GEN || it + 1 == nch) && relax) {
            // conservation factors: reduce-scatter of the eight sums (lane
            // 4 i holds sum i), every lane then reads all eight
            __syncwarp();
#pragma unroll
            for (int half = 4; half >= 1; half >>= 1) {
                const bool up = (lane & (4 * half)) != 0;
#pragma unroll
                for (int i = 0; i < half; ++i) {
                    const float send = up ? R[i] : R[i + half];
                    const float recv = __shfl_xor_sync(0xffffffffu, send, 4 * half);
                    R[i] = (up ? R[i + half] : R[i]) + recv;
                }
            }
            R[0] += __shfl_xor_sync(0xffffffffu, R[0], 2);
            R[0] += __shfl_xor_sync(0xffffffffu, R[0], 1);
            const uint32_t nall = __reduce_add_sync(0xffffffffu, nr);
            float Q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) Q[k] = __shfl_sync(0xffffffffu, R[0], 4 * k);
            if (nall >= 2) {
                // FP32: the sums are taken about the cell mean, so the
                // differences below do not cancel
                const float inv = 1.0f / (float)nall;
                const float Eo = Q[3] - (Q[0] * Q[0] + Q[1] * Q[1] + Q[2] * Q[2]) * inv;
                const float En = Q[7] - (Q[4] * Q[4] + Q[5] * Q[5] + Q[6] * Q[6]) * inv;
                if (En > 0.0f && Eo >= 0.0f) {
                    // c = ubar_old + alpha (c' - ubar_new) with c' about the cell mean
                    apply = true;
                    al = sqrtf(Eo / En);
                    uo0 = f.u[0] + Q[0] * inv;
                    uo1 = f.u[1] + Q[1] * inv;
                    uo2 = f.u[2] + Q[2] * inv;
                    mn0 = Q[4] * inv;
                    mn1 = Q[5] * inv;
                    mn2 = Q[6] * inv;
                    if (lane == 0) acc.relaxed += nall;
                }
            }
        }
        if (MODE == kRelaxOnly) {   // the new velocities back in place
            if (!apply) return;
#pragma unroll 1
            for (uint32_t b = lane; b < cnt; b += 32, selm >>= 1) {
                if (!(selm & 1u)) continue;
                const uint32_t j = ro + b;
                st_0[j] = uo0 + al * (st_0[j] - mn0);
                st_1[j] = uo1 + al * (st_1[j] - mn1);
                st_2[j] = uo2 + al * (st_2[j] - mn2);
                if (off + b >= nb) continue;
                ((float*)s.vel[p][0])[base + off + b] = st_0[j];
                ((float*)s.vel[p][1])[base + off + b] = st_1[j];
                ((float*)s.vel[p][2])[base + off + b] = st_2[j];
            }
            __syncwarp();
            if (GEN && off + cnt > nb)   // (entries not relaxed get back what they hold)
                each_spilled(s, p, cell, lane, [&](uint32_t rank, uint32_t i) {
                    const uint32_t j = nb + rank - off;
                    if (j >= cnt) return;
                    s.sp_vel[p][0][i] = st_0[j];
                    s.sp_vel[p][1][i] = st_1[j];
                    s.sp_vel[p][2][i] = st_2[j];
                });
            continue;
        }
        if (GEN) {   // fewer than two relaxed particles in the cell: reverted
            if (!apply && __any_sync(0xffffffffu, selm)) {
                __syncwarp();
                load_chunk(off, cnt);
                selm = 0;
            }
        } else if (!apply && selm) {
#pragma unroll 1
            for (uint32_t b = lane; b < cnt; b += 32, selm >>= 1)
                if (selm & 1u) {
                    st_0[ro + b] = ((const float*)s.vel[p][0])[base + b];
                    st_1[ro + b] = ((const float*)s.vel[p][1])[base + b];
                    st_2[ro + b] = ((const float*)s.vel[p][2])[base + b];
                }
            selm = 0;
        }
        // ---- sweep 2 ----
        const float tau = s.f_dt, lo1 = s.f_lo[1], hi1 = s.f_hi[1], idy = s.f_inv_dy;
        const float lo0 = s.f_lo[0], hi0 = s.f_hi[0], idx = s.f_inv_dx;
        const int nym1 = s.ny - 1, nxm1 = s.nx - 1, nseg = DIM == 2 ? s.nseg : 0;
        const bool res = s.has_reservoir != 0;
        const float b0 = s.f_bdt[0], b1 = s.f_bdt[1], b2 = s.f_bdt[2];
        uint32_t slow = 0;   // bit i: the lane's particle of iteration i meets a wall or plate
        // destination slot of a moved particle, its rank among the arrivals
        // of the slot from one shared atomic (lanes of one slot are served
        // one after another)
        auto place = [&](bool alive, float x, float y) -> uint32_t {
            const int iy = min(max(__float2int_rd((y - lo1) * idy), 0), nym1);
            const int ix = DIM == 1 ? 0 : min(max(__float2int_rd((x - lo0) * idx), 0), nxm1);
            if (res && alive && in_buffer_xy(s, ix, iy)) {
                ++acc.removed;
                alive = false;
            }
            if (MODE == kFullSlab && alive) {
                const int dc = (DIM == 2 ? iy * s.nx + ix : iy) - cell0;
                if ((unsigned)dc >= (unsigned)s.K) return kPackOther;
            }
            const int slot = win_slot_xy<DIM>(ix, iy - row0, gcell, cx, cy);
            uint32_t sr = alive ? kPackFar : kPackNone;
            if (alive && slot >= 0) sr = (uint32_t)slot | (atomicAdd(&sh.wst[slot], 1u) << 6);
            return sr;
        };
        auto fly = [&](auto nt, uint32_t b) {
            constexpr int N = decltype(nt)::value;
            float x[N], y[N], c[N][3], xn[N], yn[N];
            bool has[N], inside[N];
#pragma unroll
            for (int t = 0; t < N; ++t) {
                const uint32_t j = ro + b + 32 * t + lane;
                x[t] = DIM == 2 ? st_x[j] : 0.0f;
                y[t] = st_y[j];
                c[t][0] = st_0[j];
                c[t][1] = st_1[j];
                c[t][2] = st_2[j];
            }
#pragma unroll
            for (int t = 0; t < N; ++t) {
                has[t] = b + 32 * t + lane < cnt;
                if (selm >> ((b >> 5) + t) & 1u) {
                    c[t][0] = uo0 + al * (c[t][0] - mn0);
                    c[t][1] = uo1 + al * (c[t][1] - mn1);
                    c[t][2] = uo2 + al * (c[t][2] - mn2);
                }
                yn[t] = y[t] + c[t][1] * tau;
                xn[t] = x[t];
                inside[t] = yn[t] > lo1 && yn[t] < hi1;
                if (DIM == 2) {
                    xn[t] = x[t] + c[t][0] * tau;
                    inside[t] = inside[t] && xn[t] > lo0 && xn[t] < hi0;
                }
            }
            if (DIM == 2)
                for (int g = 0; g < nseg; ++g) {
                    const float ps = s.f_seg_pos[g];
#pragma unroll
                    for (int t = 0; t < N; ++t)
                        if ((x[t] - ps) * (xn[t] - ps) <= 0.0f) inside[t] = false;
                }
            if ((MODE == kFullFlux || MODE == kFullSlab) && s.flux_axis) {
#pragma unroll
                for (int t = 0; t < N; ++t)
                    if (has[t] && inside[t]) count_flux<float>(s, x[t], y[t], xn[t], yn[t]);
            }
#pragma unroll
            for (int t = 0; t < N; ++t) {
                const uint32_t j = ro + b + 32 * t + lane;
                const uint32_t sr = place(has[t] && inside[t], xn[t], yn[t]);
                if (has[t] && !inside[t]) slow |= 1u << ((b >> 5) + t);   // left as it is for the loop below
                if (DIM == 2) st_x[j] = inside[t] ? xn[t] : x[t];
                st_y[j] = inside[t] ? yn[t] : y[t];
                st_0[j] = inside[t] ? c[t][0] + b0 : c[t][0];
                st_1[j] = inside[t] ? c[t][1] + b1 : c[t][1];
                st_2[j] = inside[t] ? c[t][2] + b2 : c[t][2];
                st_r[j] = (uint16_t)sr;
            }
        };
        __syncwarp();   // the window is clear
        {
            uint32_t b = 0;
#pragma unroll 1
            for (; b + 32 < cnt; b += 64) fly(Num<2>{}, b);
            if (b < cnt) fly(Num<1>{}, b);
        }
        // walls and plates
        for (; __any_sync(0xffffffffu, slow); slow &= slow - 1u) {
            if (!slow) continue;
            const uint32_t j = ro + 32u * (uint32_t)(__ffs(slow) - 1) + lane;
            const float x = DIM == 2 ? st_x[j] : 0.0f, y = st_y[j];
            const AdvOut o = advect_slow(s, S.step, st_id[j], x, y, st_0[j], st_1[j], st_2[j]);
            if ((MODE == kFullFlux || MODE == kFullSlab) && s.flux_axis) count_flux<float>(s, x, y, o.x, o.y);
            st_r[j] = (uint16_t)place(o.alive != 0, o.x, o.y);
            if (DIM == 2) st_x[j] = o.x;
            st_y[j] = o.y;
            st_0[j] = o.c0;
            st_1[j] = o.c1;
            st_2[j] = o.c2;
        }
        __syncwarp();
        // ---- reserve: all slots in flight together (each lane with the bounds it asked for) ----
        cp_async_wait_all();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = lane + 32 * h;
            const uint32_t c = sh.wst[k];
            if (c) sh.wst[k] = sh.wlo[k] + atom_add_global(&s.cnt[q][win_cell<DIM>(k, cell, cx, cy, s.nx)], c);
            sh.wend[k] = min(sh.wend[k], (uint32_t)s.cap);
        }
        // ---- sweep 3 ----
        float* const dx = (float*)s.pos[q][0];
        float* const dy = (float*)s.pos[q][1];
        float* const d0 = (float*)s.vel[q][0];
        float* const d1 = (float*)s.vel[q][1];
        float* const d2 = (float*)s.vel[q][2];
        uint32_t* const did = s.pid[q];
        auto put = [&](auto nt, uint32_t b) {
            constexpr int N = decltype(nt)::value;
            uint32_t sr[N], id[N], i[N];
            float x[N], y[N], v[N][3];
            bool in[N], odd = false;
#pragma unroll
            for (int t = 0; t < N; ++t) {
                const uint32_t j = ro + b + 32 * t + lane;
                sr[t] = b + 32 * t + lane < cnt ? st_r[j] : kPackNone;
                id[t] = st_id[j];
                x[t] = DIM == 2 ? st_x[j] : 0.0f;
                y[t] = st_y[j];
                v[t][0] = st_0[j];
                v[t][1] = st_1[j];
                v[t][2] = st_2[j];
            }
#pragma unroll
            for (int t = 0; t < N; ++t) {
                i[t] = sh.wst[sr[t] & 63u] + (sr[t] >> 6);
                in[t] = sr[t] < kPackOther && i[t] < sh.wend[sr[t] & 63u];
                odd = odd || (!in[t] && sr[t] != kPackNone);
            }
            if (__any_sync(0xffffffffu, odd)) {   // not in the window, or the bucket is full
                int dc[N];
                uint32_t r[N], lo[N], hi[N];
#pragma unroll
                for (int t = 0; t < N; ++t) {   // reservations of their own, all in flight together
                    int ix, iy;
                    cell_xy<DIM>(s, x[t], y[t], ix, iy);
                    dc[t] = (DIM == 2 ? iy * s.nx + ix : iy) - cell0;
                    r[t] = lo[t] = hi[t] = 0;
                    if (sr[t] == kPackFar) {
                        r[t] = atom_add_global(&s.cnt[q][dc[t]], 1u);
                        lo[t] = __ldg(&s.lay[q][dc[t]]);
                        hi[t] = __ldg(&s.lay[q][dc[t] + 1]);
                    }
                }
#pragma unroll
                for (int t = 0; t < N; ++t) {
                    if (sr[t] == kPackFar) {
                        i[t] = lo[t] + r[t];
                        in[t] = i[t] < min(hi[t], (uint32_t)s.cap);
                    }
                    if (MODE == kFullSlab && sr[t] == kPackOther)   // into the buckets of another slab
                        emit_other<DIM>(sims, s, q, x[t], y[t], v[t][0], v[t][1], v[t][2], id[t]);
                    else if (!in[t] && sr[t] != kPackNone)
                        spill<DIM>(s, q, dc[t], x[t], y[t], v[t][0], v[t][1], v[t][2], id[t]);
                }
            }
#pragma unroll
            for (int t = 0; t < N; ++t)
                if (in[t]) {
                    if (DIM == 2) __stcg(dx + i[t], x[t]);
                    __stcg(dy + i[t], y[t]);
                    __stcg(d0 + i[t], v[t][0]);
                    __stcg(d1 + i[t], v[t][1]);
                    __stcg(d2 + i[t], v[t][2]);
                    __stcg(did + i[t], id[t]);
                }
        };
        __syncwarp();
        {
            uint32_t b = 0;
#pragma unroll 1
            for (; b + 32 < cnt; b += 64) put(Num<2>{}, b);
            if (b < cnt) put(Num<1>{}, b);
        }
        if (GEN && it + 1 < 2 * nch - 1) {   // the window of the next chunk
            __syncwarp();
            sh.wst[lane] = 0;
            sh.wst[lane + 32] = 0;
        }
    }
    __syncwarp();
}

// a cell out of line: the general form, and the ablations' (inline their state
// spills: the 200 x 200 cavity with the fixed count 338 us a step, 330 like this)
template <int DIM, int MODE, bool ABL, bool GEN, class Sh>
__device__ __noinline__ G2Acc g2w_cell_call(const SimDev* __restrict__ sims, Sh& sh, G2Sim S, G2Job J, uint32_t parity,
                                            int lane) {
    G2Acc acc = {0u, 0u};
    uint32_t nsp = 0;
    if (GEN) {
        if (J.arrived > J.nb) nsp = each_spilled(sh.sim, S.p, J.cell, lane, [](uint32_t, uint32_t) {});
        if (J.nb + nsp == 0) return acc;   // no bucket, and the spill list was full when its particles arrived
    }
    g2w_cell_impl<DIM, MODE, ABL, GEN>(sims, sh, S, J, parity, nsp, lane, acc);
    return acc;
}

// DIMS 1 or 2: the dimension of every cell of the tiles *first .. *first +
// *ntiles (first null: 0)
template <int DIMS, int MODE, bool ABL, int BLOCKS>
__global__ void __launch_bounds__(32 * kG2wWarps, BLOCKS) k_g2(const SimDev* __restrict__ sims,
                                                                   const int2* __restrict__ tiles,
                                                                   const int* __restrict__ ntiles,
                                                                   const int* __restrict__ first_tile,
                                                                   uint32_t* __restrict__ wq) {
    extern __shared__ __align__(16) unsigned char g2_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    using Sh = G2Warp<DIMS, ABL, BLOCKS>;
    Sh& sh = reinterpret_cast<Sh*>(g2_smem)[warp];
    const SimDev& s = sh.sim;
    const uint32_t nunits = (uint32_t)*ntiles * kCTile;   // a unit is one cell slot of a tile
    if (first_tile) tiles += *first_tile;
    const uint32_t nwarps = gridDim.x * kG2wWarps;
    G2Acc acc = {0u, 0u};
    G2Sim S = {0u, 0, false};
    int loaded = -1;
    // Four cells are on their way through the warp.  While cell i is worked
    // on, the copies of i + 1, the bounds of i + 2 and the tile of i + 3 come
    // in asynchronously, each from what had arrived by the start of cell i;
    // the unit number of i + 4 (lane 0's `ahead`) comes from the counter.  The
    // first four units of a warp are dealt out by its number.
    const uint32_t first = blockIdx.x * kG2wWarps + warp;
    uint32_t ahead = 0;
    if (lane == 0) {
        ahead = atom_add_global(&wq[0], 1u);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t u = first + k * nwarps;
            sh.punit[k] = u;
            if (k < 3 && u < nunits) cp_async8(&sh.ptile[k], &tiles[u / kCTile]);
        }
    }
    if (lane == 0) {
        mbar_init(&sh.full[0], 1);
        mbar_init(&sh.full[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    uint32_t phase = 0;    // bit b: parity of the next phase of full[b]
    bool ok = true;
    uint32_t known = 0;    // bit k: pbound[k] holds the bounds of the cell in slot k
    bool staged = false;   // the copies of the next cell have been started, to `ro`
    uint32_t ro = 0;
    for (uint32_t i = 0;; ++i) {
        const uint32_t k0 = i & 3u, k1 = (i + 1) & 3u, k2 = (i + 2) & 3u, k3 = (i + 3) & 3u;
        cp_async_wait_all();
        __syncwarp();
        const uint32_t unit = sh.punit[k0];
        if (unit >= nunits) break;   // unit numbers of a warp only grow
        const int2 tile = sh.ptile[k0];
        if (tile.x != loaded) {
            if (loaded >= 0) g2_flush(acc, s.dyn, lane);
            __syncwarp();
            load_sim_warp(sh.sim, sims[tile.x], lane);
            __syncwarp();
            loaded = tile.x;
            S.p = s.dyn->cur;
            S.step = s.dyn->step;
            S.pending = s.dyn->relax_pending != 0;
            uintptr_t al = (uintptr_t)s.pos[S.p][1] | (uintptr_t)s.vel[S.p][0] | (uintptr_t)s.vel[S.p][1] |
                           (uintptr_t)s.vel[S.p][2] | (uintptr_t)s.pid[S.p];
            if (DIMS == 2) al |= (uintptr_t)s.pos[S.p][0];
            S.aligned = (al & 15u) == 0;
            if (lane < 10) {   // round keys: the key plus r times the Weyl constants
                sh.key[2 * lane] = s.key0 + (uint32_t)lane * 0x9E3779B9u;
                sh.key[2 * lane + 1] = s.key1 + (uint32_t)lane * 0xBB67AE85u;
            }
            __syncwarp();
            known = 0;
            staged = false;
        }
        const uint32_t room = sh.CAP, cap = (uint32_t)s.cap;
        G2Job J;
        J.cell = tile.y + (int)(unit % kCTile);
        J.base = J.nb = J.arrived = 0;
        J.ro = staged ? ro : 0u;
        if (J.cell < s.K) {
            uint32_t lo, hi;
            if (known >> k0 & 1u) {
                lo = sh.pbound[k0][0];
                hi = sh.pbound[k0][1];
                J.arrived = sh.pbound[k0][2];
            } else {
                lo = __ldg(&s.lay[S.p][J.cell]);
                hi = __ldg(&s.lay[S.p][J.cell + 1]);
                J.arrived = __ldg(&s.cnt[S.p][J.cell]);
            }
            hi = min(hi, cap);
            J.base = lo;
            J.nb = min(J.arrived, hi > lo ? hi - lo : 0u);
        }
        const bool general = J.arrived > J.nb || J.nb > room;
        const uint32_t par = i & 1u;
        if (J.arrived && !general) {
            bool bulk = staged;
            if (!staged) {
                bulk = S.aligned && (J.base & 3u) == 0u;
                if (bulk) {
                    if (lane == 0) g2w_copy<DIMS>(sh, J, S.p, par);
                } else {
                    g2w_load<DIMS>(sh, J, S.p, par, lane);
                }
            }
            if (bulk) {
                // one outcome for the warp: near the limit some lanes may see the copy land and others not
                ok = __all_sync(0xffffffffu, mbar_wait(&sh.full[par], phase >> par & 1u));
                if (!ok) break;
                phase ^= 1u << par;
            }
        }
        // the next cell's copies, where it fits the staging area beside this one
        staged = false;
        if (known >> k1 & 1u) {
            G2Job N;
            const uint32_t lo = sh.pbound[k1][0], hi = min(sh.pbound[k1][1], cap);
            N.cell = sh.ptile[k1].y + (int)(sh.punit[k1] % kCTile);
            N.base = lo;
            N.arrived = sh.pbound[k1][2];
            N.nb = min(N.arrived, hi > lo ? hi - lo : 0u);
            const uint32_t m = (J.nb + 31u) & ~31u, mn = (N.nb + 31u) & ~31u;
            staged = !general && S.aligned && (lo & 3u) == 0u && N.arrived == N.nb && N.nb > 0 &&
                     (J.ro + m + mn <= room || mn <= J.ro);
            if (staged) {
                ro = J.ro + m + mn <= room ? J.ro + m : 0u;
                N.ro = ro;
                if (lane == 0) g2w_copy<DIMS>(sh, N, S.p, par ^ 1u);
            } else if (S.aligned && (lo & 3u) == 0u && N.nb > 0 && lane == 0) {   // at least into L2
                const uint32_t bytes = 4u * ((N.nb + 3u) & ~3u);
                bulk_prefetch(s.pid[S.p] + lo, bytes);
                for (int d = 0; d < 3; ++d) bulk_prefetch((const float*)s.vel[S.p][d] + lo, bytes);
                bulk_prefetch((const float*)s.pos[S.p][1] + lo, bytes);
                if (DIMS == 2) bulk_prefetch((const float*)s.pos[S.p][0] + lo, bytes);
            }
        }
        __syncwarp();   // every lane has read the slots of cell i
        {   // bounds of i + 2, tile of i + 3, unit of i + 4
            const uint32_t u2 = sh.punit[k2], u3 = sh.punit[k3];
            known &= ~(1u << k2);
            if (u2 < nunits && sh.ptile[k2].x == loaded) {
                const int c = sh.ptile[k2].y + (int)(u2 % kCTile);
                if (c < s.K) {
                    if (lane < 3) cp_async4(&sh.pbound[k2][lane], lane < 2 ? &s.lay[S.p][c + lane] : &s.cnt[S.p][c]);
                    known |= 1u << k2;
                }
            }
            if (lane == 0) {
                if (u3 < nunits) cp_async8(&sh.ptile[k3], &tiles[u3 / kCTile]);
                sh.punit[k0] = 4 * nwarps + ahead;
                ahead = atom_add_global(&wq[0], 1u);   // not looked at before the next cell
            }
        }
        if (J.arrived) {
            if (ABL || general) {
                const G2Acc a = !ABL || general ? g2w_cell_call<DIMS, MODE, ABL, true>(sims, sh, S, J, 0u, lane)
                                                : g2w_cell_call<DIMS, MODE, ABL, false>(sims, sh, S, J, par, lane);
                acc.relaxed += a.relaxed;
                acc.removed += a.removed;
            } else {
                g2w_cell_impl<DIMS, MODE, ABL, false>(sims, sh, S, J, par, 0u, lane, acc);
            }
            fence_proxy_async_smem();   // later copies come after these accesses
            __syncwarp();
        }
    }
    if (loaded >= 0) g2_flush(acc, s.dyn, lane);
    if (!ok) {   // copies in flight land before the block may exit
        if (lane == 0) atomicAdd(&sims[0].dyn->counters[kCntOverflow], kG2TimeoutMark);
        mbar_wait(&sh.full[0], phase & 1u);
        mbar_wait(&sh.full[1], phase >> 1 & 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const uint32_t done = atomicAdd(&wq[1], 1u);
        if (done == gridDim.x - 1) wq[0] = wq[1] = 0;   // the last block resets the counters for the next launch
    }
}

// ---------------------------------------------------------------------------
// k_g1: per-cell moments (Eq. 1) in one pass, as sums of C = c - u_s about a
// shift u_s: the cell's mean velocity of the previous step (the parameters
// of that step, still in fprm).  The mean moves little in one step, so the
// FP32 sums of the centred velocities do not cancel; k_params_f forms the
// state from them in FP32 with the shift taken into account.
// ---------------------------------------------------------------------------
constexpr int kG1Warps = 4;     // warps per block; a block takes one 32-cell tile at a time
constexpr int kG1Stage = 384;   // slots of one pipeline stage (a multiple of 4)

__global__ void __launch_bounds__(32 * kG1Warps) k_g1(const SimDev* __restrict__ sims, const int2* __restrict__ tiles,
                                                     const int* __restrict__ ntiles) {
    // the unit's per-cell headers, fetched in one round for all its cells:
    // bucket start, particles in the bucket, arrivals, and the shift u_s
    __shared__ uint32_t h_base[kCTile], h_nb[kCTile], h_arr[kCTile];
    __shared__ float4 h_us[kCTile];
    // each warp's two pipeline stages of the three velocity planes
    __shared__ __align__(16) float stage[kG1Warps][2][3][kG1Stage];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ SimDev sim_sh;
    // A unit is a whole tile or, until every block has one, a
    // half, quarter or eighth of one (down to one cell per warp), so that few
    // cells spread over all SMs: one shock tube of 1000 cells 16.6 -> 8.9 us.
    // More units than blocks cost what the next cell's copy ahead gains
    // (cavity 200 x 200: 34 us with one per block, 37 / 42 / 54 us with 2 / 4 / 8).
    const int nt = *ntiles;
    int parts = 1;
    while (parts < kCTile / kG1Warps && nt * parts < (int)gridDim.x) parts *= 2;
    const int ncell = kCTile / parts;   // cells of a unit
    int loaded = -1;
    for (int t = blockIdx.x; t < nt * parts; t += gridDim.x) {
        int2 tile = tiles[t / parts];
        tile.y += (t % parts) * ncell;
        __syncthreads();
        if (tile.x != loaded) {
            load_sim(sim_sh, sims[tile.x]);
            __syncthreads();
            loaded = tile.x;
        }
        const SimDev& s = sim_sh;
        const int K = s.K;
        const int q = s.dyn->cur ^ 1;
        if ((int)threadIdx.x < ncell && tile.y + (int)threadIdx.x < K) {
            const int cell = tile.y + (int)threadIdx.x;
            const uint32_t base = s.lay[q][cell];
            const uint32_t top = min(s.lay[q][cell + 1], (uint32_t)s.cap);
            const uint32_t capc = top > base ? top - base : 0u;
            const uint32_t arrived = s.cnt[q][cell];
            h_base[threadIdx.x] = base;
            h_nb[threadIdx.x] = min(arrived, capc);
            h_arr[threadIdx.x] = arrived;
            h_us[threadIdx.x] = reinterpret_cast<const float4*>(s.fprm)[(size_t)cell * (kNFPrm / 4)];
        }
        __syncthreads();
        const float* V0 = (const float*)s.vel[q][0];
        const float* V1 = (const float*)s.vel[q][1];
        const float* V2 = (const float*)s.vel[q][2];
        // The warp's cells (cc = warp, warp + kG1Warps, ...) are read as a
        // sequence of chunks of at most kG1Stage slots, each copied into one
        // of two stages while the chunk before it is summed: a cell's whole
        // bucket is in flight at once, and its round trip overlaps the
        // previous chunk's work.  (c, o) is the next chunk to copy.
        auto live = [&](int c) { return c < ncell && tile.y + c < K; };
        auto copy_chunk = [&](int c, uint32_t o, int b) {
            const uint32_t g = h_base[c] + o;
            const uint32_t len = min(h_nb[c] - o, (uint32_t)kG1Stage);
            float* d0 = stage[warp][b][0];
            float* d1 = stage[warp][b][1];
            float* d2 = stage[warp][b][2];
            if ((g & 3u) == 0u) {
                // 16-byte groups up to the next multiple of four slots: the
                // bucket start and the capacity are multiples of four, so the
                // copy stays inside the plane
                const uint32_t n4 = (len + 3u) >> 2;
                for (uint32_t k = lane; k < n4; k += 32) {
                    cp_async16(d0 + 4 * k, V0 + g + 4 * k);
                    cp_async16(d1 + 4 * k, V1 + g + 4 * k);
                    cp_async16(d2 + 4 * k, V2 + g + 4 * k);
                }
            } else {   // the compact layout right after a set-up sort
                for (uint32_t k = lane; k < len; k += 32) {
                    cp_async4(d0 + k, V0 + g + k);
                    cp_async4(d1 + k, V1 + g + k);
                    cp_async4(d2 + k, V2 + g + k);
                }
            }
            cp_async_commit();
        };
        // the chunk after (c, o), skipping cells with an empty bucket
        auto advance = [&](int& c, uint32_t& o) {
            o += kG1Stage;
            if (o < h_nb[c]) return;
            o = 0;
            c += kG1Warps;
            while (live(c) && h_nb[c] == 0) c += kG1Warps;
        };
        int ic = warp;
        uint32_t io = 0;
        while (live(ic) && h_nb[ic] == 0) ic += kG1Warps;
        if (live(ic)) copy_chunk(ic, io, 0);
        int done = 0;   // chunks summed so far (stage done & 1 holds the next)
        for (int cc = warp; live(cc); cc += kG1Warps) {
            const int cell = tile.y + cc;
            const uint32_t nb = h_nb[cc];
            const uint32_t arrived = h_arr[cc];
            const float4 us = h_us[cc];
            const float u0 = us.x, u1 = us.y, u2 = us.z;
            uint32_t n = nb;
            float S[12];
#pragma unroll
            for (int k = 0; k < 12; ++k) S[k] = 0.0f;
            auto add = [&](float a, float b, float c) {
                const float C0 = a - u0, C1 = b - u1, C2 = c - u2;
                const float c2 = C0 * C0 + C1 * C1 + C2 * C2;
                S[0] += C0; S[1] += C1; S[2] += C2;
                S[3] += C0 * C0; S[4] += C1 * C1; S[5] += C2 * C2;
                S[6] += C0 * C1; S[7] += C0 * C2; S[8] += C1 * C2;
                S[9] += c2 * C0; S[10] += c2 * C1; S[11] += c2 * C2;
            };
            for (uint32_t o = 0; o < nb; o += kG1Stage) {
                // (ic, io) is this chunk: copy the next one, then wait for this one
                advance(ic, io);
                if (live(ic)) {
                    copy_chunk(ic, io, (done + 1) & 1);
                    cp_async_wait<1>();
                } else {
                    cp_async_wait<0>();
                }
                __syncwarp();
                const float* b0 = stage[warp][done & 1][0];
                const float* b1 = stage[warp][done & 1][1];
                const float* b2 = stage[warp][done & 1][2];
                const uint32_t len = min(nb - o, (uint32_t)kG1Stage);
#pragma unroll 4
                for (uint32_t j = lane; j < len; j += 32) add(b0[j], b1[j], b2[j]);
                __syncwarp();   // the stage is refilled by the copy issued two chunks on
                ++done;
            }
            if (arrived > nb)
                n += each_spilled(s, q, cell, lane, [&](uint32_t, uint32_t i) {
                    add(s.sp_vel[q][0][i], s.sp_vel[q][1][i], s.sp_vel[q][2][i]);
                });
            // The cell's 64-byte record [N, 12 sums, shift u_s] as a warp
            // reduce-scatter: at each of four halving stages a lane keeps half
            // of its values and adds the partner's copy of that half (16
            // shuffles instead of 60 for twelve butterfly sums); lane 2v then
            // holds entry v of the record and writes it.  N and u_s come from
            // lane 0 alone.
            float v[16];
            v[0] = lane == 0 ? (float)n : 0.0f;
#pragma unroll
            for (int k = 0; k < 12; ++k) v[1 + k] = S[k];
            v[13] = lane == 0 ? u0 : 0.0f;
            v[14] = lane == 0 ? u1 : 0.0f;
            v[15] = lane == 0 ? u2 : 0.0f;
#pragma unroll
            for (int half = 8; half >= 1; half >>= 1) {
                const bool up = (lane & (2 * half)) != 0;
#pragma unroll
                for (int i = 0; i < half; ++i) {
                    const float send = up ? v[i] : v[i + half];
                    const float recv = __shfl_xor_sync(0xffffffffu, send, 2 * half);
                    v[i] = (up ? v[i + half] : v[i]) + recv;
                }
            }
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
            if ((lane & 1) == 0) s.momf[(size_t)cell * 16 + (lane >> 1)] = v[0];   // one 64-byte record per cell
            // the totals of the first six sums (entries 1..6, on lanes 2..12) for the local state
#pragma unroll
            for (int k = 0; k < 6; ++k) S[k] = __shfl_sync(0xffffffffu, v[0], 2 * (k + 1));
            if (lane == 31) {
                // local state of the cell for its neighbours' Kn_GLL (FP32):
                // the instantaneous one, or the Eq. 34 average as it stood at
                // the start of the step (k_params_f updates it later)
                float nn = (float)n * s.f_w, T = 0.0f, um = 0.0f, valid = 0.0f;
                if (s.gll_average && s.dyn->nsamples > 0) {
                    const int K = s.K;
                    const double a1 = s.avg[(size_t)1 * K + cell], a2 = s.avg[(size_t)2 * K + cell],
                                 a3 = s.avg[(size_t)3 * K + cell];
                    nn = (float)s.avg[cell];
                    T = (float)s.avg[(size_t)4 * K + cell];
                    um = (float)sqrt(a1 * a1 + a2 * a2 + a3 * a3);
                    valid = nn > 0.0f && T > 0.0f ? 1.0f : 0.0f;
                } else if (n >= 2) {
                    const float inv2 = 1.0f / (float)n;
                    const float d0 = S[0] * inv2, d1 = S[1] * inv2, d2 = S[2] * inv2;
                    const float th = ((S[3] + S[4] + S[5]) * inv2 - (d0 * d0 + d1 * d1 + d2 * d2)) * (1.0f / 3.0f);
                    if (th > 0.0f) {
                        valid = 1.0f;
                        T = th * s.f_inv_R;
                        const float w0 = u0 + d0, w1 = u1 + d1, w2 = u2 + d2;
                        um = sqrtf(w0 * w0 + w1 * w1 + w2 * w2);
                    }
                }
                reinterpret_cast<float4*>(s.floc)[cell] = make_float4(nn, T, um, valid);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// k_params_f: per-cell parameters in FP32; the number density and the Eq. 34
// averages in FP64
// ---------------------------------------------------------------------------
// A warp per tile of 32 cells, which takes as long as one cell's chain of
// loads and arithmetic (10 us): all tiles in one wave where they fit.  16 blocks
// of one warp per SM are what 128 registers a thread allow (18 and 24 with fewer
// registers: small domains 1 us slower).  Against 8 per SM: 4e4 cells 19.5 ->
// 14.2 us, 8e4 28.5 -> 26 us, 64 x 1000 cells 20.4 -> 17.7 us; a second warp for
// the fields and averages gave no more.
constexpr int kParamsBlocks = 16;

struct LocalF {
    int valid, N;
    float n, T, umag;
};

// the cell's state from its FP32 shifted sums: mean velocity, pressure
// tensor per unit density (P / rho) and theta = R T; inv = 1 / N.  The sums
// are about the previous mean, so the subtractions below do not cancel and
// FP32 keeps the accuracy the FP32 sums carry.
__device__ __forceinline__ void local_f(const SimDev& s, const float* M, LocalF& L, float* u, float* P, float* theta,
                                        float& inv) {
    const int N = (int)M[0];
    L.N = N;
    L.valid = 0;
    L.n = (float)N * s.f_w;
    L.T = 0;
    L.umag = 0;
    inv = 0.0f;
    if (N < 1) return;
    inv = 1.0f / (float)N;
    const float d0 = M[1] * inv, d1 = M[2] * inv, d2 = M[3] * inv;
    u[0] = M[13] + d0; u[1] = M[14] + d1; u[2] = M[15] + d2;
    P[0] = M[4] * inv - d0 * d0;
    P[1] = M[5] * inv - d1 * d1;
    P[2] = M[6] * inv - d2 * d2;
    P[3] = M[7] * inv - d0 * d1;
    P[4] = M[8] * inv - d0 * d2;
    P[5] = M[9] * inv - d1 * d2;
    const float th = (P[0] + P[1] + P[2]) * (1.0f / 3.0f);
    *theta = th;
    L.valid = N >= 2 && th > 0.0f;
    if (!L.valid) return;
    L.T = th * s.f_inv_R;
    L.umag = sqrtf(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
}

// neighbour state for the Kn_GLL stencil, written in FP32 by k_g1
__device__ __forceinline__ void local_nb(const SimDev& s, int cell, LocalF& L) {
    const float4 f = reinterpret_cast<const float4*>(s.floc)[cell];
    L.n = f.x;
    L.T = f.y;
    L.umag = f.z;
    L.valid = f.w != 0.0f;
    L.N = 0;
}

// state of the neighbour of cell (ix, iy) along `axis` (dir = -1 / +1) for the
// Kn_GLL stencil; across a slab boundary it is the adjacent slab's row.
// Returns whether the neighbour exists and is valid.
__device__ __forceinline__ bool nb_state(const SimDev* __restrict__ sims, const SimDev& s, int ix, int iy, int axis,
                                         int dir, LocalF& L) {
    const SimDev* t = &s;
    int c;
    if (axis == 0) {
        int j = ix + dir;
        if (j < 0 || j >= s.nx) {
            if (!s.periodic_x) return false;
            j = j < 0 ? j + s.nx : j - s.nx;
        }
        c = iy * s.nx + j;
    } else {
        int gj = s.row0 + iy + dir;   // global row
        if (gj < 0 || gj >= s.ny) {
            if (!s.periodic_y) return false;
            gj = gj < 0 ? gj + s.ny : gj - s.ny;
        }
        const int r = gj - s.row0;
        if (r >= 0 && r < s.rows) {
            c = r * s.nx + ix;
        } else {
            t = &sims[s.slab_first + gj / s.rows];
            c = (gj - t->row0) * s.nx + ix;
        }
    }
    local_nb(*t, c, L);
    return L.valid != 0;
}

__global__ void __launch_bounds__(32, kParamsBlocks) k_params_f(const SimDev* __restrict__ sims,
                                                                const int2* __restrict__ tiles,
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
            // every load of the cell first (one round of latency): the
            // running averages, the neighbours' states for the stencil, then
            // the cell's own sums
            const bool first = s.dyn->nsamples == 0;
            double av[kNFields];
#pragma unroll
            for (int k = 0; k < kNFields; ++k) av[k] = first ? 0.0 : s.avg[(size_t)k * K + cell];
            LocalF Nm[2] = {}, Np[2] = {};
            bool hm[2] = {false, false}, hp[2] = {false, false};
            if (s.mode == kModeUSP) {
                const int iy = s.dim == 1 ? cell : cell / s.nx, ix = s.dim == 1 ? 0 : cell - iy * s.nx;
#pragma unroll
                for (int axis = 0; axis < 2; ++axis) {
                    if (axis == 0 && s.dim == 1) continue;
                    hm[axis] = nb_state(sims, s, ix, iy, axis, -1, Nm[axis]);
                    hp[axis] = nb_state(sims, s, ix, iy, axis, +1, Np[axis]);
                }
            }
            LocalF L;
            const float* M = s.momf + (size_t)cell * 16;   // N, 12 sums, shift[3]
            float u[3] = {0, 0, 0}, P[6], th = 0, inv;
            local_f(s, M, L, u, P, &th, inv);
            float f[kNFields];
            for (int k = 0; k < kNFields; ++k) f[k] = 0.0f;
            f[0] = L.n;
            f[15] = (float)L.N;
            if (L.N >= 1) {
                f[1] = u[0]; f[2] = u[1]; f[3] = u[2];
            }
            float pr[kNFPrm];
            for (int k = 0; k < kNFPrm; ++k) pr[k] = 0.0f;
            pr[0] = u[0]; pr[1] = u[1]; pr[2] = u[2];
            pr[3] = th;
            if (L.valid) {
                const float thf = th;
                const float rho = L.n * s.f_mass;
                const float pf = rho * thf;
                const float mu = s.f_mu_ref * __powf(L.T / s.f_T_ref, s.f_omega);   // Eq. 35
                const float nu = pf / mu;
                const float lam = 1.2766152f * mu / sqrtf(rho * pf);     // Eq. 36: 16 / (5 sqrt(2 pi))
                float pne;
                if (s.mode == kModeSP || s.mode == kModeSPESBGK) pne = 0.0f;
                else if (s.mode == kModeFixed) pne = s.f_fixed_pne;
                else {
                    // the cell's own stencil state: instantaneous, or the
                    // Eq. 34 average (loaded above, before this step's update)
                    float gn = L.n, gT = L.T, gu = L.umag, glam = lam, ga = sqrtf((float)kGammaMono * thf);
                    bool gvalid = true;
                    if (s.gll_average && !first) {
                        gn = (float)av[0];
                        gT = (float)av[4];
                        gu = (float)sqrt(av[1] * av[1] + av[2] * av[2] + av[3] * av[3]);
                        gvalid = gn > 0.0f && gT > 0.0f;
                        if (gvalid) {
                            const float gth = gT * s.f_R;
                            const float grho = gn * s.f_mass;
                            const float gmu = s.f_mu_ref * __powf(gT / s.f_T_ref, s.f_omega);
                            glam = 1.2766152f * gmu / sqrtf(grho * grho * gth);   // Eq. 36 at the averaged state
                            ga = sqrtf((float)kGammaMono * gth);
                        }
                    }
                    // the gradients are taken relative to the cell's own value
                    // (|grad Q| / Q): absolute density gradients (~1e25 m^-3 over
                    // sub-micron cells) would overflow FP32 when squared
                    const float a_s = ga;
                    const float Qc[3] = {gn, gT, gu};
                    const float rq[3] = {1.0f / gn, 1.0f / gT, 1.0f / fmaxf(gu, a_s)};
                    float g2[3] = {0, 0, 0};
#pragma unroll
                    for (int axis = 0; axis < 2; ++axis) {
                        if (axis == 0 && s.dim == 1) continue;
                        const float h = s.f_h[axis];
                        const LocalF& Lm = Nm[axis];
                        const LocalF& Lp = Np[axis];
                        const int m = hm[axis] ? 1 : -1;
                        const int p = hp[axis] ? 1 : -1;
                        const float Qm[3] = {Lm.n, Lm.T, Lm.umag}, Qp[3] = {Lp.n, Lp.T, Lp.umag};
                        for (int k = 0; k < 3; ++k) {
                            float d = 0.0f;
                            if (m >= 0 && p >= 0) d = (Qp[k] - Qm[k]) * rq[k] / (2.0f * h);
                            else if (p >= 0) d = (Qp[k] - Qc[k]) * rq[k] / h;
                            else if (m >= 0) d = (Qc[k] - Qm[k]) * rq[k] / h;
                            g2[k] += d * d;
                        }
                    }
                    const float kn = gvalid ? glam * sqrtf(fmaxf(g2[0], fmaxf(g2[1], g2[2]))) : 0.0f;
                    pne = __expf(-kn / (float)kKnC);                                              // Eqs. 16-18
                }
                // Eq. 33
                const float ifs = 1.0f / (1.0f + 0.5f * s.f_dt * nu * pne);
                const float ifq = 1.0f / (1.0f + 0.5f * s.f_dt * nu * s.f_Pr * pne);
                const float sig[6] = {(P[0] - th) * ifs, (P[1] - th) * ifs, (P[2] - th) * ifs, P[3] * ifs, P[4] * ifs,
                                      P[5] * ifs};
                const float b = s.f_es_b;                                                  // Eq. 6c
                const float A00 = th + b * sig[0], A11 = th + b * sig[1], A22 = th + b * sig[2];
                const float A10 = b * sig[3], A20 = b * sig[4], A21 = b * sig[5];
                float l00 = 0, l10 = 0, l11 = 0, l20 = 0, l21 = 0, l22 = 0;
                bool ok = A00 > 0.0f;
                if (ok) {
                    const float r0 = rsqrtf(A00);
                    l00 = A00 * r0;
                    l10 = A10 * r0;
                    l20 = A20 * r0;
                    const float d1 = A11 - l10 * l10;
                    ok = d1 > 0.0f;
                    if (ok) {
                        const float r1 = rsqrtf(d1);
                        l11 = d1 * r1;
                        l21 = (A21 - l20 * l10) * r1;
                        const float d2 = A22 - l20 * l20 - l21 * l21;
                        ok = d2 > 0.0f;
                        if (ok) l22 = d2 * rsqrtf(d2);
                    }
                }
                if (s.es_sampler) {
                    // Gallis-Torczynski (Eq. 11): B = ((1 - Pr)/(2 Pr)) sigma* / (rho theta)
                    // in M's slots, lower triangle row-major
                    const float beta = (1.0f - s.f_Pr) / (2.0f * s.f_Pr * th);
                    pr[4] = beta * sig[0]; pr[5] = beta * sig[3]; pr[6] = beta * sig[1];
                    pr[7] = beta * sig[4]; pr[8] = beta * sig[5]; pr[9] = beta * sig[2];
                } else {
                    if (!ok) {   // no Cholesky factor: an isotropic Gaussian
                        l00 = l11 = l22 = sqrtf(th);
                        l10 = l20 = l21 = 0.0f;
                        atomicAdd(&s.dyn->counters[kCntChol], 1ull);
                    }
                    // M = L L^T - theta I (lower triangle, row-major)
                    pr[4] = l00 * l00 - th;
                    pr[5] = l10 * l00;
                    pr[6] = l10 * l10 + l11 * l11 - th;
                    pr[7] = l20 * l00;
                    pr[8] = l20 * l10 + l21 * l11;
                    pr[9] = l20 * l20 + l21 * l21 + l22 * l22 - th;
                }
                const float nues = s.f_Pr * nu;
                const float at = nues * s.f_dt;
                pr[10] = -expm1f(-nues * s.f_dt);                                             // Eqs. 8b, 9
                // the decay rate of Eq. 32; the SP-ESBGK step holds its target
                // for the whole step (Eq. 8b): with P_ne = 0 a rate of 0 gives s = 1
                pr[11] = s.mode == kModeSPESBGK ? 0.0f : nu;
                pr[12] = 1.0f / nues;
                pr[13] = pne;
                pr[14] = at < 1.0f ? expm1f(at) : -__expf(-at);
                pr[15] = pr[10] > 0.0f ? 1.0f / pr[10] : 0.0f;
                // heat flux from the third central moment of the shifted sums
                const float d0 = M[1] * inv, d1 = M[2] * inv, d2 = M[3] * inv;
                const float m00 = M[4] * inv, m11 = M[5] * inv, m22 = M[6] * inv;
                const float m01 = M[7] * inv, m02 = M[8] * inv, m12 = M[9] * inv;
                const float t0 = M[10] * inv, t1 = M[11] * inv, t2 = M[12] * inv;
                const float tr = m00 + m11 + m22, dd = d0 * d0 + d1 * d1 + d2 * d2;
                const float Q0 = 0.5f * (t0 - d0 * tr - 2.0f * (m00 * d0 + m01 * d1 + m02 * d2) + 2.0f * d0 * dd);
                const float Q1 = 0.5f * (t1 - d1 * tr - 2.0f * (m01 * d0 + m11 * d1 + m12 * d2) + 2.0f * d1 * dd);
                const float Q2 = 0.5f * (t2 - d2 * tr - 2.0f * (m02 * d0 + m12 * d1 + m22 * d2) + 2.0f * d2 * dd);
                const float rhod = rho, pd = pf;
                f[4] = L.T;
                f[5] = pd + rhod * sig[0];
                f[6] = pd + rhod * sig[1];
                f[7] = pd + rhod * sig[2];
                f[8] = rhod * sig[3];
                f[9] = rhod * sig[4];
                f[10] = rhod * sig[5];
                f[11] = rhod * Q0 * ifq;
                f[12] = rhod * Q1 * ifq;
                f[13] = rhod * Q2 * ifq;
                f[14] = pne;
            }
            {   // one 64-byte parameter record per cell
                float4* dst = reinterpret_cast<float4*>(s.fprm) + (size_t)cell * (kNFPrm / 4);
#pragma unroll
                for (int k = 0; k < kNFPrm / 4; ++k) dst[k] = make_float4(pr[4 * k], pr[4 * k + 1], pr[4 * k + 2], pr[4 * k + 3]);
            }
            // the number density in FP64 (N w exactly as the FP64 paths form
            // it: a closed box keeps its domain total to the last bit)
            const double n_d = (double)L.N * s.w;
#pragma unroll
            for (int k = 0; k < kNFields; ++k) {
                const double fk = k == 0 ? n_d : (double)f[k];
                s.inst[(size_t)k * K + cell] = fk;
                s.avg[(size_t)k * K + cell] = first ? fk : s.avg_keep * av[k] + fk * s.avg_new;   // Eq. 34, FP64
            }
        }
    }
}

// append one particle to the bucket of its cell (all 32 lanes call this
// together; key == kNoCell for lanes with nothing to write)
template <int DIM>
__device__ __forceinline__ void emit_c(const SimDev& s, int b, uint32_t key, float x, float y, float v0, float v1,
                                       float v2, uint32_t id, int lane) {
    const unsigned grp = __match_any_sync(0xffffffffu, key);
    if (key == kNoCell) return;
    const int leader = __ffs(grp) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(&s.cnt[b][key], (uint32_t)__popc(grp));
    base = __shfl_sync(grp, base, leader);
    const uint32_t i = s.lay[b][key] + base + (uint32_t)__popc(grp & lanemask_lt());
    if (i < min(s.lay[b][key + 1], (uint32_t)s.cap)) {
        if (DIM == 2) ((float*)s.pos[b][0])[i] = x;
        ((float*)s.pos[b][1])[i] = y;
        ((float*)s.vel[b][0])[i] = v0;
        ((float*)s.vel[b][1])[i] = v1;
        ((float*)s.vel[b][2])[i] = v2;
        s.pid[b][i] = id;
    } else {
        spill<DIM>(s, b, (int)key, x, y, v0, v1, v2, id);
    }
}

// ---------------------------------------------------------------------------
// k_inject_f: reservoir buffer cells, written into buffer q
// ---------------------------------------------------------------------------
template <int DIM>
__global__ void __launch_bounds__(256) k_inject_f(const SimDev* __restrict__ sims, const int2* __restrict__ tiles,
                                                  const int* __restrict__ ntiles) {
    __shared__ SimDev sim_sh;
    const int nt = *ntiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int t = blockIdx.x; t < nt; t += gridDim.x) {
        const int2 tile = tiles[t];
        __syncthreads();
        load_sim(sim_sh, sims[tile.x]);
        __syncthreads();
        const SimDev& s = sim_sh;
        if (!s.has_reservoir || s.dim != DIM) continue;
        const uint32_t step = s.dyn->step, next_pid = s.dyn->next_pid;
        const int q = s.dyn->cur ^ 1;
        for (int cc = warp; cc < kCTile; cc += 8) {
            const int cell = tile.y + cc;
            if (cell >= s.K) break;
            const uint32_t cnt = s.inj_count[cell];
            if (cnt == 0) continue;
            const FaceDev& F = s.face[buffer_face(s, cell)];
            for (uint32_t k0 = 0; k0 < cnt; k0 += 32) {
                const uint32_t k = k0 + lane;
                uint32_t key = kNoCell;
                float x = 0, y = 0, c[3] = {0, 0, 0};
                uint32_t pid = 0;
                if (k < cnt) {
                    pid = next_pid + s.inj_pidoff[cell] + k;
                    make_particle<float>(s, cell, pid, step, kInject, F.theta, F.u, x, y, c);
                    key = (uint32_t)cell;
                }
                emit_c<DIM>(s, q, key, x, y, c[0], c[1], c[2], pid, lane);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// k_layout: histogram -> bucket sizes (slack for arrivals) -> exclusive scan, the
// write layout of buffer cur ^ 1 right after the initial fill (counts of buffer
// cur from the exact start offsets)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t bucket_size(const SimDev& s, const uint32_t* cnt, int c) {
    const int ix = c % s.nx, iy = c / s.nx;
    uint32_t m = 0;
    for (int dy = -1; dy <= 1; ++dy) {
        const int jy = iy + dy;
        if (jy < 0 || jy >= s.rows) continue;   // (the counts of a slab are those of its own rows)
        for (int dx = (s.dim == 2 ? -1 : 0); dx <= (s.dim == 2 ? 1 : 0); ++dx) {
            const int jx = ix + dx;
            if (jx < 0 || jx >= s.nx) continue;
            m = max(m, cnt[jy * s.nx + jx]);
        }
    }
    // a multiple of four slots, so that every bucket starts on a 16-byte
    // boundary (the bulk copies of k_g2 need it)
    return (m + (m >> 2) + 16u + (s.has_reservoir ? s.inj_count[c] : 0u) + 3u) & ~3u;
}

__global__ void __launch_bounds__(1024) k_layout(const SimDev* __restrict__ sims, int nsims) {
    __shared__ uint32_t warp_sums[32];
    __shared__ unsigned long long tot_full, tot_exact;
    __shared__ uint32_t carry;
    for (int si = blockIdx.x; si < nsims; si += gridDim.x) {
        const SimDev& s = sims[si];
        SimDyn* dyn = s.dyn;
        const int K = s.K;
        const int cur = dyn->cur;
        const int dst = cur ^ 1;   // layout for the next write
        for (int c = threadIdx.x; c <= K; c += blockDim.x) {
            s.lay[cur][c] = s.start[c];
            if (c < K) s.cnt[cur][c] = s.start[c + 1] - s.start[c];
        }
        __syncthreads();
        const uint32_t* C = s.cnt[cur];
        if (threadIdx.x == 0) {
            tot_full = 0;
            tot_exact = 0;
            carry = 0;
        }
        __syncthreads();
        unsigned long long lf = 0, le = 0;
        for (int c = threadIdx.x; c < K; c += blockDim.x) {
            lf += bucket_size(s, C, c);
            le += C[c];
        }
        // warp sums first: one shared atomic per warp instead of per thread
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lf += __shfl_xor_sync(0xffffffffu, lf, o);
            le += __shfl_xor_sync(0xffffffffu, le, o);
        }
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&tot_full, lf);
            atomicAdd(&tot_exact, le);
        }
        __syncthreads();
        // bucket sizes with slack when they fit, else the exact demand plus an even share of what is left
        const unsigned long long demand = tot_exact + (s.has_reservoir ? s.inj_total : 0u);
        const bool full = tot_full <= (unsigned long long)s.cap;
        // (each bucket rounded up to a multiple of four: up to 3 K more slots)
        const unsigned long long room = demand + 3ull * (unsigned long long)K;
        const uint32_t extra = (!full && room < (unsigned long long)s.cap)
                                   ? (uint32_t)(((unsigned long long)s.cap - room) / (unsigned long long)K)
                                   : 0u;
        if (!full && demand > (unsigned long long)s.cap && threadIdx.x == 0)
            atomicAdd(&dyn->counters[kCntOverflow], 1ull);
        for (int base = 0; base < K; base += blockDim.x) {
            const int c = base + threadIdx.x;
            uint32_t v = 0;
            if (c < K) v = full ? bucket_size(s, C, c) : (C[c] + (s.has_reservoir ? s.inj_count[c] : 0u) + extra + 3u) & ~3u;
            uint32_t x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if ((threadIdx.x & 31) >= o) x += y;
            }
            if ((threadIdx.x & 31) == 31) warp_sums[threadIdx.x >> 5] = x;
            __syncthreads();
            if (threadIdx.x < 32) {
                uint32_t ws = threadIdx.x < (blockDim.x >> 5) ? warp_sums[threadIdx.x] : 0u;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, ws, o);
                    if (threadIdx.x >= o) ws += y;
                }
                warp_sums[threadIdx.x] = ws;
            }
            __syncthreads();
            const uint32_t before = (threadIdx.x >= 32 ? warp_sums[(threadIdx.x >> 5) - 1] : 0u) + carry;
            if (c < K) s.lay[dst][c] = before + x - v;
            __syncthreads();
            if (threadIdx.x == blockDim.x - 1) carry = before + x;
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            s.lay[dst][K] = carry;
            dyn->sp_n[dst] = 0;
            dyn->sp_n[cur] = 0;
            dyn->relax_pending = 0;
        }
        for (int c = threadIdx.x; c < K; c += blockDim.x) s.cnt[dst][c] = 0;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Per-step layout of the next write, over tiles of kLayTile cells so that a
// large domain is laid out by many blocks at once:
//   k_lay_sum   per tile: sums of the bucket sizes with slack (bucket_size),
//               of the counts rounded up to four slots (tight) and of the
//               exact counts;
//   k_lay_scan  per simulation: the choice between slack and tight buckets
//               (tight ones get an even share of the spare slots, a multiple
//               of four), the exclusive scan of the tile sums into tile
//               offsets, the totals, and the end of the step;
//   k_lay_put   per tile: the bucket offsets of its cells and cleared counts.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t tight_size(const SimDev& s, const uint32_t* C, int c) {
    return (C[c] + (s.has_reservoir ? s.inj_count[c] : 0u) + 3u) & ~3u;
}

// sum over a block of 1024 threads (every thread gets the total)
__device__ __forceinline__ unsigned long long block_sum_1024(unsigned long long v, unsigned long long* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    v = threadIdx.x < 32 ? sh[threadIdx.x] : 0ull;
    if (threadIdx.x < 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) sh[32] = v;
    }
    __syncthreads();
    return sh[32];
}

// exclusive scan over a block of 1024 threads; *total receives the sum
__device__ __forceinline__ unsigned long long block_scan_1024(unsigned long long v, unsigned long long* sh,
                                                              unsigned long long* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        unsigned long long t = sh[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        sh[lane] = t;   // inclusive warp totals
    }
    __syncthreads();
    *total = sh[31];
    return (w ? sh[w - 1] : 0ull) + x - v;
}

__global__ void __launch_bounds__(kLayTile) k_lay_sum(const SimDev* __restrict__ sims) {
    __shared__ unsigned long long sh[33];
    const SimDev& s = sims[blockIdx.y];
    const int K = s.K;
    const int T = (K + kLayTile - 1) / kLayTile;
    const int src = s.dyn->cur ^ 1;   // counts of the buffer this step wrote
    const uint32_t* C = s.cnt[src];
    for (int t = blockIdx.x; t < T; t += gridDim.x) {
        const int c = t * kLayTile + threadIdx.x;
        unsigned long long f = 0, g = 0, e = 0;
        if (c < K) {
            f = bucket_size(s, C, c);
            g = tight_size(s, C, c);
            e = C[c];
        }
        f = block_sum_1024(f, sh);
        g = block_sum_1024(g, sh);
        e = block_sum_1024(e, sh);
        if (threadIdx.x == 0) {
            s.lay_part[3 * t] = f;
            s.lay_part[3 * t + 1] = g;
            s.lay_part[3 * t + 2] = e;
        }
    }
}

__global__ void __launch_bounds__(kLayTile) k_lay_scan(const SimDev* __restrict__ sims, int nsims) {
    __shared__ unsigned long long sh[33];
    __shared__ unsigned long long carry;
    for (int si = blockIdx.x; si < nsims; si += gridDim.x) {
        const SimDev& s = sims[si];
        SimDyn* dyn = s.dyn;
        const int K = s.K;
        const int T = (K + kLayTile - 1) / kLayTile;
        const int cur = dyn->cur;
        unsigned long long P = 0, G = 0, E = 0;
        for (int t = threadIdx.x; t < T; t += blockDim.x) {
            P += s.lay_part[3 * t];
            G += s.lay_part[3 * t + 1];
            E += s.lay_part[3 * t + 2];
        }
        const unsigned long long tot_full = block_sum_1024(P, sh);
        const unsigned long long tot_tight = block_sum_1024(G, sh);
        const unsigned long long tot_exact = block_sum_1024(E, sh);
        const unsigned long long cap = (unsigned long long)s.cap;
        const bool full = tot_full <= cap;
        const unsigned long long extra =
            (!full && tot_tight < cap) ? ((cap - tot_tight) / (unsigned long long)K) & ~3ull : 0ull;
        const unsigned long long demand = tot_exact + (s.has_reservoir ? s.inj_total : 0u);
        if (threadIdx.x == 0) {
            carry = 0;
            if (!full && demand > cap) atomicAdd(&dyn->counters[kCntOverflow], 1ull);
        }
        __syncthreads();
        for (int base = 0; base < T; base += blockDim.x) {
            const int t = base + threadIdx.x;
            unsigned long long v = 0;
            if (t < T) {
                const int cells = min(kLayTile, K - t * kLayTile);
                v = full ? s.lay_part[3 * t] : s.lay_part[3 * t + 1] + extra * (unsigned long long)cells;
            }
            unsigned long long tot;
            const unsigned long long x = block_scan_1024(v, sh, &tot);
            if (t < T) s.lay_part[3 * t] = carry + x;   // tile offset
            __syncthreads();
            if (threadIdx.x == 0) carry += tot;
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            s.lay_part[3 * T] = full ? 1ull : 0ull;
            s.lay_part[3 * T + 1] = extra;
            s.lay[cur][K] = (uint32_t)min(carry, 0xFFFFFFFFull);
            dyn->n = (uint32_t)min(tot_exact, 0xFFFFFFFFull);
            dyn->sp_n[cur] = 0;
            dyn->lay_dst = (uint32_t)cur;
        }
        __syncthreads();
    }
}

// the three in one, a block per simulation, where every simulation has at
// most kLaySmall cells (each thread a run of consecutive cells): the layout
// then takes one latency instead of three (measured on one simulation of 1000
// cells: 20 -> 8 us), so that it stays behind k_g1 and k_params_f
constexpr int kLaySmall = 8 * 1024;

__global__ void __launch_bounds__(1024) k_lay_small(const SimDev* __restrict__ sims) {
    __shared__ unsigned long long sh[33];
    const SimDev& s = sims[blockIdx.x];
    SimDyn* dyn = s.dyn;
    const int K = s.K, cur = dyn->cur;
    const uint32_t* C = s.cnt[cur ^ 1];
    uint32_t* const lay = s.lay[cur];
    uint32_t* const cnt = s.cnt[cur];
    const int per = (K + 1023) / 1024;   // at most 8
    const int c0 = min((int)threadIdx.x * per, K), c1 = min(c0 + per, K);
    uint32_t slack[8], tight[8];
    unsigned long long f = 0, g = 0, e = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        slack[k] = tight[k] = 0;
        if (c0 + k < c1) {
            slack[k] = bucket_size(s, C, c0 + k);
            tight[k] = tight_size(s, C, c0 + k);
            f += slack[k];
            g += tight[k];
            e += C[c0 + k];
        }
    }
    unsigned long long tot_full, tot_tight;
    const unsigned long long xf = block_scan_1024(f, sh, &tot_full);
    const unsigned long long xg = block_scan_1024(g, sh, &tot_tight);
    const unsigned long long tot_exact = block_sum_1024(e, sh);
    const unsigned long long cap = (unsigned long long)s.cap;
    const bool full = tot_full <= cap;
    const unsigned long long extra =
        (!full && tot_tight < cap) ? ((cap - tot_tight) / (unsigned long long)K) & ~3ull : 0ull;
    unsigned long long x = full ? xf : xg + extra * (unsigned long long)c0;
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (c0 + k < c1) {
            lay[c0 + k] = (uint32_t)min(x, 0xFFFFFFFFull);
            cnt[c0 + k] = 0;
            x += full ? slack[k] : tight[k] + extra;
        }
    if (threadIdx.x == 0) {
        const unsigned long long demand = tot_exact + (s.has_reservoir ? s.inj_total : 0u);
        if (!full && demand > cap) atomicAdd(&dyn->counters[kCntOverflow], 1ull);
        lay[K] = (uint32_t)min(full ? tot_full : tot_tight + extra * (unsigned long long)K, 0xFFFFFFFFull);
        dyn->n = (uint32_t)min(tot_exact, 0xFFFFFFFFull);
        dyn->sp_n[cur] = 0;
        dyn->lay_dst = (uint32_t)cur;
    }
}

// end of the step (after the layout and the parameters): buffers swap, the
// step counter and the sample count advance, the relaxation becomes pending
__global__ void k_step_end(const SimDev* __restrict__ sims, int nsims) {
    for (int si = blockIdx.x * blockDim.x + threadIdx.x; si < nsims; si += gridDim.x * blockDim.x) {
        const SimDev& s = sims[si];
        SimDyn* dyn = s.dyn;
        if (s.has_reservoir) {
            dyn->next_pid += s.inj_total;
            dyn->counters[kCntInjected] += s.inj_total;
        }
        dyn->cur ^= 1;
        dyn->step += 1;
        dyn->nsamples += 1;
        dyn->relax_pending = 1;
    }
}

__global__ void __launch_bounds__(kLayTile) k_lay_put(const SimDev* __restrict__ sims) {
    __shared__ unsigned long long sh[33];
    const SimDev& s = sims[blockIdx.y];
    const int K = s.K;
    const int T = (K + kLayTile - 1) / kLayTile;
    const int dst = (int)s.dyn->lay_dst;
    const uint32_t* C = s.cnt[dst ^ 1];
    const bool full = s.lay_part[3 * T] != 0;
    const uint32_t extra = (uint32_t)s.lay_part[3 * T + 1];
    for (int t = blockIdx.x; t < T; t += gridDim.x) {
        const int c = t * kLayTile + threadIdx.x;
        unsigned long long v = 0;
        if (c < K) v = full ? bucket_size(s, C, c) : tight_size(s, C, c) + extra;
        unsigned long long tot;
        const unsigned long long x = block_scan_1024(v, sh, &tot);
        if (c < K) {
            s.lay[dst][c] = (uint32_t)min(s.lay_part[3 * t] + x, 0xFFFFFFFFull);
            s.cnt[dst][c] = 0;
        }
        __syncthreads();
    }
}

// clears the pending relaxation once it has been applied in place before a
// read-back
__global__ void k_clear_pending(const SimDev* __restrict__ sims, int nsims) {
    for (int si = blockIdx.x * blockDim.x + threadIdx.x; si < nsims; si += gridDim.x * blockDim.x)
        sims[si].dyn->relax_pending = 0;
}

// ---------------------------------------------------------------------------
// k_g2 launch configuration: one wave of resident blocks
// ---------------------------------------------------------------------------
static int sm_count() {
    static const int sms = [] {
        int dev = 0, n = 152;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return n;
    }();
    return sms;
}

// blocks of a kernel resident on the device (the same on every GB300), with its
// shared memory allowed; each launcher asks once (the initialisation of its
// static is the one that threads wait for)
template <class K>
int wave_of(K* kernel, int threads, int smem) {
    int per = 0;
    if (smem) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem);
    return sm_count() * std::max(per, 1);
}

template <int DIMS, int MODE, bool ABL, int G>
void launch_g2b_one(const Launch& L) {
    static const int wave = wave_of(k_g2b<DIMS, MODE, ABL, G>, 32 * G, 0);
    const int grid = std::max(1, std::min(wave, L.cells));
    k_g2b<DIMS, MODE, ABL, G><<<grid, 32 * G, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles, L.wq);
}

template <int DIMS, int MODE, bool ABL, int BLOCKS>
void launch_g2_blocks(const Launch& L, int group, cudaStream_t st) {
    constexpr int smem = (int)(kG2wWarps * sizeof(G2Warp<DIMS, ABL, BLOCKS>));
    static const int wave = wave_of(k_g2<DIMS, MODE, ABL, BLOCKS>, 32 * kG2wWarps, smem);
    const int grid = std::max(1, std::min(wave, (L.cells + kG2wWarps - 1) / kG2wWarps));
    k_g2<DIMS, MODE, ABL, BLOCKS><<<grid, 32 * kG2wWarps, smem, st>>>(
        L.sims, L.ctiles, L.gtiles ? L.gtiles + group : L.nctiles, L.gtiles ? L.gtiles + kG2Groups + group : nullptr,
        L.wq + 2 * group);
}

template <int DIMS, int MODE, bool ABL>
void launch_g2_one(const Launch& L, int group, cudaStream_t st) {
    if constexpr (MODE != kRelaxOnly) {
        if (L.g2_blocks == 3) return launch_g2_blocks<DIMS, MODE, ABL, 3>(L, group, st);
    }
    launch_g2_blocks<DIMS, MODE, ABL, 4>(L, group, st);
}

// the cells of one group (g2_group).  The ablations' kernel counts the flux too,
// and the one that relaxes in place holds the ablations' code.
template <int MODE>
void launch_g2_group(const Launch& L, int group, cudaStream_t st) {
    constexpr int M = MODE == kFull ? kFullFlux : MODE;
    const bool abl = MODE == kRelaxOnly || (group & 1);
    if (group < 2) {
        if (abl) return launch_g2_one<1, M, true>(L, group, st);
        if constexpr (MODE != kRelaxOnly) launch_g2_one<1, MODE, false>(L, group, st);
    } else {
        if (abl) return launch_g2_one<2, M, true>(L, group, st);
        if constexpr (MODE != kRelaxOnly) launch_g2_one<2, MODE, false>(L, group, st);
    }
}

// A mixed batch runs the kernels of its groups side by side: one kernel with the
// bodies of both dimensions overflows the instruction cache where a block's warps
// are in different ones, and one that holds the ablations' code too costs the
// other cells a sixth (64 shock tubes 325 -> 380 us a step).  One group of
// ordinary cells takes the step's stream; the others follow on the second one,
// an ablation's cells (few, and slow) before the rest, and their blocks run
// where those of the first are done.
template <int MODE>
void launch_g2(const Launch& L) {
    constexpr int order[kG2Groups] = {1, 3, 0, 2};   // the ablations' first
    int main = -1;
    for (int g : {0, 2, 1, 3})
        if (main < 0 && (L.groups >> g & 1)) main = g;
    const bool fork = L.side && (L.groups & (L.groups - 1));
    if (fork) {
        cudaEventRecord(L.ev_fork, L.stream);
        cudaStreamWaitEvent(L.side, L.ev_fork, 0);
    }
    for (int g : order)
        if (L.groups >> g & 1) launch_g2_group<MODE>(L, g, fork && g != main ? L.side : L.stream);
    if (fork) {
        cudaEventRecord(L.ev_join, L.side);
        cudaStreamWaitEvent(L.stream, L.ev_join, 0);
    }
}

template <int MODE, bool ABL, int G>
void launch_g2b(const Launch& L) {
    if constexpr (ABL || MODE == kRelaxOnly || MODE == kFullSlab) {   // seldom run: one form for both dimensions
        launch_g2b_one<3, MODE, ABL, G>(L);
    } else {
        if (L.dims == 3) launch_g2b_one<3, MODE, ABL, G>(L);
        else if (L.dims == 1) launch_g2b_one<1, MODE, ABL, G>(L);
        else launch_g2b_one<2, MODE, ABL, G>(L);
    }
}

// R (tuning): 4 one warp per cell, 8 and 12 a block of 4 or 8 warps
template <int MODE>
void launch_g2_R(const Launch& L, int R) {
    if (R <= 4) {
        launch_g2<MODE>(L);
    } else if (L.ablation) {
        launch_g2b<MODE, true, 4>(L);
    } else if constexpr (MODE == kRelaxOnly || MODE == kFullSlab) {
        launch_g2b<MODE, false, 4>(L);
    } else if (R <= 8) {
        launch_g2b<MODE, false, 4>(L);
    } else {
        launch_g2b<MODE, false, 8>(L);
    }
}

}  // namespace

void launch_fused_setup(const Launch& L) { k_layout<<<L.nsims, 1024, 0, L.stream>>>(L.sims, L.nsims); }

void launch_fused_relax_stream(const Launch& L, int R, bool flush_only) {
    if (flush_only) {
        launch_g2_R<kRelaxOnly>(L, R);
        k_clear_pending<<<(L.nsims + 127) / 128, 128, 0, L.stream>>>(L.sims, L.nsims);
        return;
    }
    if (L.slabs) launch_g2_R<kFullSlab>(L, R);
    else if (L.flux) launch_g2_R<kFullFlux>(L, R);
    else launch_g2_R<kFull>(L, R);
}

void launch_fused_inject(const Launch& L) {
    if (L.dims & 1) k_inject_f<1><<<L.grid_c, 256, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles);
    if (L.dims & 2) k_inject_f<2><<<L.grid_c, 256, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles);
}

void launch_fused_moments(const Launch& L) {
    k_g1<<<L.grid_f, 32 * kG1Warps, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles);
}

void launch_fused_params(const Launch& L) {
    const int grid = std::max(1, std::min((L.cells - 1) / kCTile + 1, kParamsBlocks * sm_count()));
    k_params_f<<<grid, 32, 0, L.stream>>>(L.sims, L.ctiles, L.nctiles);
}

// the bucket layout of the next step's destination buffer (reads only the
// arrivals of this step, so it may run beside k_g1 and k_params_f)
void launch_fused_layout_parts(const Launch& L) {
    if (L.lay_tiles * kLayTile <= kLaySmall) {
        k_lay_small<<<L.nsims, 1024, 0, L.stream>>>(L.sims);
        return;
    }
    const dim3 grid((unsigned)std::min(L.lay_tiles, 1024), (unsigned)L.nsims);
    k_lay_sum<<<grid, kLayTile, 0, L.stream>>>(L.sims);
    k_lay_scan<<<L.nsims, kLayTile, 0, L.stream>>>(L.sims, L.nsims);
    k_lay_put<<<grid, kLayTile, 0, L.stream>>>(L.sims);
}

void launch_fused_step_end(const Launch& L) { k_step_end<<<(L.nsims + 127) / 128, 128, 0, L.stream>>>(L.sims, L.nsims); }

void launch_fused_layout(const Launch& L) {
    launch_fused_layout_parts(L);
    launch_fused_step_end(L);
}


}  // namespace usp
