// WMCD kernels for sm_103a: cell list, slot generation and bucketing, the concurrent wavelet
// kernels, the serial wavelet kernels and the plane-wave kernels.
//
// Nothing here is a dense contraction, so there are no tensor-core paths: the work is
// gathers of 32-byte bead records through per-cell linked lists, pair energies and
// warp / block reductions. See the host file for the order of launches in a sweep.
#include <algorithm>
#include <cfloat>
#include <type_traits>
#include "wmcd_internal.h"
#include "wmcd_limits.h"

namespace wmcd {

__device__ __forceinline__ void set_err(const SimView& v, int bit) { atomicOr(v.err, bit); }

// Acceptance threshold of a move on its draw w (accept iff dU <= threshold): Metropolis
// (Eq. 20), -kT ln(1 - u) with u in [0, 1); Glauber (Secs. V.C, VIII), accept with probability
// 1 / (1 + exp(dU / kT)), i.e. kT (ln(1 - u) - ln u) with u in (0, 1).
// Centre uniform in the box (Sec. V.D, the homogeneous scheme, P_b = 1/L^3): each coordinate L
// times a 32-bit uniform of the slot's own draw.
__device__ __forceinline__ void uniform_centre(const SimView& v, int l, uint64_t sweep, uint32_t j, double b[3]) {
    const u4 w = draw(v.k0, v.k1, K_BUNI, l, sweep, j, 0);
    b[0] = mul(v.L, (double)w.x * (1.0 / 4294967296.0));
    b[1] = mul(v.L, (double)w.y * (1.0 / 4294967296.0));
    b[2] = mul(v.L, (double)w.z * (1.0 / 4294967296.0));
}
// Amplitude with a uniform centre: A0 lam / sqrt(nbar), nbar = N (4 pi / 3) lam^3 / L^3 the mean
// support at the global density (Eq. 29 with the mean count)
__device__ __forceinline__ double uniform_aw(const SimView& v, double lam) {
    const double nbar = dvd(mul((double)v.N, mul(4.0 * kPi / 3.0, mul(mul(lam, lam), lam))), mul(mul(v.L, v.L), v.L));
    return dvd(mul(v.A0, lam), sqr_t(nbar));
}
// Largest displacement of a concurrent move as its region rule counts it: A0 lam / 4, which bounds
// A_w / 4 of every support (Eq. 29, n >= 1); with a uniform centre A_w / 4 itself where the mean
// support is below one bead and A_w therefore above A0 lam
// (aw: uniform_aw, read only then)
__device__ __forceinline__ double rule_disp(const SimView& v, double lam, double aw) {
    const double d = mul(mul(0.25, v.A0), lam);
    return v.centring == 1 ? fmax(d, mul(0.25, aw)) : d;
}
__device__ __forceinline__ double rule_disp(const SimView& v, double lam) {
    return rule_disp(v, lam, v.centring == 1 ? uniform_aw(v, lam) : 0.0);
}
__device__ __forceinline__ double accept_threshold(const SimView& v, const u4& w) {
    if (v.acceptance == 1) {
        const double u = u_open(w.x, w.y);
        return v.kT * (log(1.0 - u) - log(u));
    }
    return -v.kT * log(1.0 - u53(w.x, w.y));
}

// One audited mixed-precision decision: d32 and band as the decision used them, thr_cmp the
// threshold d32 was compared with, d64 the binary64 energy change and thr64 its threshold.
__device__ void audit_record(const SimView& v, double d32, double band, double thr_cmp, double d64, double thr64) {
    AuditDev* A = v.audit;
    const unsigned long long k = atomicAdd(&A->n, 1ull);
    const bool outside = isfinite(d32) && isfinite(band) && fabs(d32 - thr_cmp) > band;
    double ratio = 0.0;
    if (isfinite(d32) && isfinite(d64) && isfinite(band) && band > 0.0) ratio = fabs(d32 - d64) / band;
    if (outside) atomicAdd(&A->outside, 1ull);
    if (ratio >= 1.0) atomicAdd(&A->viol, 1ull);
    if (outside && ((d32 <= thr_cmp) != (d64 <= thr64))) atomicAdd(&A->flip, 1ull);
    atomicMax(&A->max_ratio, __float_as_uint((float)ratio));
    if ((long long)k < A->cap) {
        A->rec[4 * k] = d32; A->rec[4 * k + 1] = d64; A->rec[4 * k + 2] = band; A->rec[4 * k + 3] = thr64;
    }
}

// wrap and minimum image with the rare correction behind a branch that the lanes of `mask` take
// together: written plainly, the correction's binary64 add is predicated and, on this part,
// occupies the binary64 pipe even when no lane needs it
__device__ __forceinline__ double wrap_u(double x, double L, unsigned mask, int* im) {
    if (__any_sync(mask, ge_pos(x, L) || lt_zero(x))) x = wrap(x, L, im);
    return x;
}
__device__ __forceinline__ double mi_u(double d, double L, double h, unsigned mask) {
    if (__any_sync(mask, gt_pos(d, h) || lt_neg(d, h))) d = mi(d, L, h);
    return d;
}
// the same for the three components of a vector, with one vote for all three
__device__ __forceinline__ void wrap3_u(double x[3], double L, unsigned mask, int* im) {
    const bool need = ge_pos(x[0], L) || lt_zero(x[0]) || ge_pos(x[1], L) || lt_zero(x[1]) || ge_pos(x[2], L) ||
                      lt_zero(x[2]);
    if (__any_sync(mask, need))
        for (int a = 0; a < 3; a++) x[a] = wrap(x[a], L, im ? &im[a] : nullptr);
}
__device__ __forceinline__ void mi3_u(double d[3], double L, double h, unsigned mask) {
    const bool need = gt_pos(d[0], h) || lt_neg(d[0], h) || gt_pos(d[1], h) || lt_neg(d[1], h) || gt_pos(d[2], h) ||
                      lt_neg(d[2], h);
    if (__any_sync(mask, need))
        for (int a = 0; a < 3; a++) d[a] = mi(d[a], L, h);
}

// Every kernel serves a group of simulations: blockIdx.y selects one, whose view is copied
// into shared memory once per block. SIM_EXIT_IF tests a condition on the view in global
// memory first, so blocks of a simulation with no work in this launch leave without the copy.
#define SIM_EXIT_IF(cond)                                                                     \
    {                                                                                         \
        const SimView& gv = vs[blockIdx.y];                                                   \
        if (cond) return;                                                                     \
    }
#define SIM_PROLOGUE                                                                          \
    __shared__ SimView sv_;                                                                   \
    {                                                                                         \
        const int* src_ = (const int*)(vs + blockIdx.y);                                      \
        int* dst_ = (int*)&sv_;                                                               \
        for (int w_ = threadIdx.x; w_ < (int)(sizeof(SimView) / 4); w_ += blockDim.x)        \
            dst_[w_] = src_[w_];                                                              \
    }                                                                                         \
    __syncthreads();                                                                          \
    const SimView& v = sv_;

__device__ __forceinline__ int cell_lin(const SimView& v, double x, double y, double z) {
    return fine_cell(x, v.invf, v.Gf) + v.Gf * (fine_cell(y, v.invf, v.Gf) + v.Gf * fine_cell(z, v.invf, v.Gf));
}
// Fine cell of a coordinate from its shadow: the binary32 quotient is within 4 units of Gf 2^-24 of
// the exact one, so away from a cell face its floor is the cell of the definition; the others (a few
// in a thousand) take it. The definition's binary64 product and floor hold their pipe for every warp.
__device__ __forceinline__ int fine_cell32(const SimView& v, float h, double x) {
    const float f = h * (float)v.invf, c = floorf(f), eps = 2.4e-7f * (float)v.Gf + 1e-6f;
    if (f - c > eps && f - c < 1.0f - eps && c >= 0.0f && c < (float)v.Gf) return (int)c;
    return fine_cell(x, v.invf, v.Gf);
}
__device__ __forceinline__ int fine_cell32(const SimView& v, float h, const double* x) {
    const float f = h * (float)v.invf, c = floorf(f), eps = 2.4e-7f * (float)v.Gf + 1e-6f;
    if (f - c > eps && f - c < 1.0f - eps && c >= 0.0f && c < (float)v.Gf) return (int)c;
    return fine_cell(*x, v.invf, v.Gf);
}

__device__ __forceinline__ int wrapi(int c, int G) { c %= G; return c < 0 ? c + G : c; }

// occupancy bit of fine cell c (atomic: cells of neighbouring regions share a word)
__device__ __forceinline__ void occ_bit(const SimView& v, int c, bool on) {
    if (!v.occ) return;
    const int x = c % v.Gf, yz = c / v.Gf;
    uint32_t* w = &v.occ[(size_t)yz * v.occ_w + (x >> 5)];
    if (on) atomicOr(w, 1u << (x & 31));
    else atomicAnd(w, ~(1u << (x & 31)));
}
// the bits of occupancy word wi of a row that lie in the cell range [a, b) of the row
__device__ __forceinline__ uint32_t occ_masked(uint32_t word, int a, int b, int wi) {
    const int lo = max(a - (wi << 5), 0), hi = min(b - (wi << 5), 32);
    if (hi <= lo) return 0u;
    return word & (hi >= 32 ? 0xffffffffu : ((1u << hi) - 1u)) & ~((1u << lo) - 1u);
}
// Move bead m from the list of fine cell oc to the head of the list of ncl (lists doubly linked
// through Bead::next and prev[]), keeping both cells' occupancy bits.
__device__ __forceinline__ void relink(const SimView& v, int m, int oc, int ncl) {
    const int pr = v.prev[m], nx = v.bead[m].next;
    if (pr >= 0) v.bead[pr].next = nx; else v.head[oc] = nx;
    if (nx >= 0) v.prev[nx] = pr;
    if (pr < 0 && nx < 0) occ_bit(v, oc, false);
    const int hd = v.head[ncl];
    v.bead[m].next = hd;
    v.prev[m] = -1;
    if (hd >= 0) v.prev[hd] = m;
    v.head[ncl] = m;
    occ_bit(v, ncl, true);
}

// The cell changes of one accepted move, (bead, old cell, new cell) in cm/co/cn, applied by the
// nt threads of a block together: one thread per old cell unlinks that cell's leaving beads,
// then one thread per new cell pushes its arriving beads in entry order, so the lists end as
// the one-at-a-time relinks leave them. Every thread of the block calls it (two barriers).
__device__ void grouped_relink(const SimView& v, const int* cm, const int* co, const int* cn, int nch, int tid, int nt) {
    for (int c = tid; c < nch; c += nt) {
        const int oc = co[c];
        bool first = true;
        for (int e = 0; e < c && first; e++) first = co[e] != oc;
        if (!first) continue;
        for (int e = c; e < nch; e++) {
            if (co[e] != oc) continue;
            const int m = cm[e], pr = v.prev[m], nx = v.bead[m].next;
            if (pr >= 0) v.bead[pr].next = nx; else v.head[oc] = nx;
            if (nx >= 0) v.prev[nx] = pr;
            if (pr < 0 && nx < 0) occ_bit(v, oc, false);
        }
    }
    __syncthreads();
    for (int c = tid; c < nch; c += nt) {
        const int ncl = cn[c];
        bool first = true;
        for (int e = 0; e < c && first; e++) first = cn[e] != ncl;
        if (!first) continue;
        for (int e = c; e < nch; e++) {
            if (cn[e] != ncl) continue;
            const int m = cm[e], hd = v.head[ncl];
            v.bead[m].next = hd;
            v.prev[m] = -1;
            if (hd >= 0) v.prev[hd] = m;
            v.head[ncl] = m;
        }
        occ_bit(v, ncl, true);
    }
    __syncthreads();
}

// ======================================================================================
// Cell list: per fine cell a singly linked list through Bead::next plus prev[] for O(1)
// removal. Built in canonical order (ascending bead id within a cell) so runs repeat.
// use_flag 0: always rebuilt; 1: after an accepted plane wave moved the beads; 2: before an
// active plane-wave move if the shared-memory serial phase left the lists stale; 3 + l: before
// the global-memory serial phase of layer l if they are stale.
// ======================================================================================
__device__ __forceinline__ bool cl_skip(const SimView& v, int use_flag) {
    if (use_flag == 1) return !*v.pw_rebuild;
    if (use_flag == 2) return !(v.pw->active && !v.pw->null_move && *v.cl_stale);
    if (use_flag >= 3) return !(*v.cl_stale && !((v.smem_layers >> (use_flag - 3)) & 1));
    return false;
}
__global__ void k_cl_clear(const SimView* __restrict__ vs, int use_flag) {
    SIM_EXIT_IF(cl_skip(gv, use_flag))
    SIM_PROLOGUE
    if (v.occ && use_flag != 0) {
        // lists and bits agree since the last full rebuild: empty only the occupied cells
        const int64_t nw = (int64_t)v.Gf * v.Gf * v.occ_w;
        for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < nw; w += (int64_t)gridDim.x * blockDim.x) {
            const uint32_t bits0 = v.occ[w];
            if (!bits0) continue;
            const int64_t base = (w % v.occ_w) * 32 + (int64_t)v.Gf * (w / v.occ_w);
            for (uint32_t bits = bits0; bits; bits &= bits - 1u) v.head[base + __ffs(bits) - 1] = -1;
            v.occ[w] = 0u;
        }
        return;
    }
    // full rebuild (creation, new positions or state): every cell and every bit
    int64_t nc = (int64_t)v.Gf * v.Gf * v.Gf;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nc; c += (int64_t)gridDim.x * blockDim.x)
        v.head[c] = -1;
    if (v.occ) {
        const int64_t nw = (int64_t)v.Gf * v.Gf * v.occ_w;
        for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < nw; w += (int64_t)gridDim.x * blockDim.x)
            v.occ[w] = 0u;
    }
}
__global__ void k_cl_insert(const SimView* __restrict__ vs, int use_flag) {
    SIM_EXIT_IF(cl_skip(gv, use_flag))
    SIM_PROLOGUE
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < v.N; i += (int64_t)gridDim.x * blockDim.x) {
        Bead b = v.bead[i];
        if (!(b.x >= 0.0 && b.x < v.L && b.y >= 0.0 && b.y < v.L && b.z >= 0.0 && b.z < v.L)) set_err(v, E_NONFINITE);
        int c = cell_lin(v, b.x, b.y, b.z);
        int old = atomicExch(&v.head[c], (int)i);
        v.bead[i].next = old;
        if (old < 0) occ_bit(v, c, true);
    }
}
// put the list of fine cell c in ascending bead-id order and set prev[]
__device__ void canon_cell(const SimView& v, int64_t c) {
    int ids[32];
    int n = 0, p = v.head[c];
    bool small = true;
    while (p >= 0) {
        if (n < 32) ids[n] = p;
        n++;
        if (n > 32) small = false;
        if (n > kMaxWalk) { set_err(v, E_WALK); break; }
        p = v.bead[p].next;
    }
    if (n == 0) return;
    if (small) {
        for (int a = 1; a < n; a++) {      // insertion sort by bead id
            int x = ids[a], b = a - 1;
            while (b >= 0 && ids[b] > x) { ids[b + 1] = ids[b]; b--; }
            ids[b + 1] = x;
        }
        v.head[c] = ids[0];
        for (int a = 0; a < n; a++) {
            v.bead[ids[a]].next = (a + 1 < n) ? ids[a + 1] : -1;
            v.prev[ids[a]] = (a > 0) ? ids[a - 1] : -1;
        }
    } else {
        int pr = -1;
        for (int q = v.head[c]; q >= 0; q = v.bead[q].next) { v.prev[q] = pr; pr = q; }
    }
}
__global__ void k_cl_canon(const SimView* __restrict__ vs, int use_flag) {
    SIM_EXIT_IF(cl_skip(gv, use_flag))
    SIM_PROLOGUE
    if (v.occ) {
        // only the occupied cells (the bits were set by the insert pass just before)
        const int64_t nw = (int64_t)v.Gf * v.Gf * v.occ_w;
        for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < nw; w += (int64_t)gridDim.x * blockDim.x) {
            const int64_t yz = w / v.occ_w;
            const int xb = (int)(w % v.occ_w) << 5;
            for (uint32_t bits = v.occ[w]; bits; bits &= bits - 1u)
                canon_cell(v, (int64_t)(xb + __ffs(bits) - 1) + (int64_t)v.Gf * yz);
        }
        return;
    }
    int64_t nc = (int64_t)v.Gf * v.Gf * v.Gf;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nc; c += (int64_t)gridDim.x * blockDim.x)
        canon_cell(v, c);
}
// blocks per simulation for a grid-stride kernel: what the largest simulation needs, but no
// more than keeps about 8k blocks over the whole group
static unsigned gx(int64_t needed_blocks, int S) {
    const int64_t cap = std::max<int64_t>(1, 8192 / std::max(S, 1));
    return (unsigned)std::max<int64_t>(1, std::min(needed_blocks, cap));
}
void launch_cl_rebuild(const SimView* d, const GroupDims& g, cudaStream_t s, int use_flag) {
    const dim3 bc(gx((g.maxCells + 255) / 256, g.S), g.S);
    const dim3 bb(gx((g.maxN + 255) / 256, g.S), g.S);
    k_cl_clear<<<bc, 256, 0, s>>>(d, use_flag);
    k_cl_insert<<<bb, 256, 0, s>>>(d, use_flag);
    k_cl_canon<<<bc, 256, 0, s>>>(d, use_flag);
}

// Slot counts of the sweep about to run, from the counter stream: floor(x) plus one more
// with probability frac(x), per layer and for the plane waves.
__global__ void k_counts(const SimView* __restrict__ vs) {
    SIM_PROLOGUE
    if (threadIdx.x != 0) return;
    const uint64_t sw = v.step[0];
    for (int l = 0; l < v.nL; l++) {
        const u4 w = draw(v.k0, v.k1, K_COUNT, l, sw, 0u, 0u);
        const double x = v.layer[l].expect, f = floor(x);
        v.counts[l] = (int)f + ((u53(w.x, w.y) < x - f) ? 1 : 0);
    }
    int mf = 0;
    if (v.pw_on) {
        const u4 w = draw(v.k0, v.k1, K_PWCOUNT, 0, sw, 0u, 0u);
        const double x = v.expect_F, f = floor(x);
        mf = (int)f + ((u53(w.x, w.y) < x - f) ? 1 : 0);
    }
    v.counts[kMaxLayers] = mf;
}
__global__ void k_advance(const SimView* __restrict__ vs, int which) {
    SIM_PROLOGUE
    if (threadIdx.x == 0) v.step[which] += 1;
}
void launch_counts(const SimView* d, const GroupDims& g, cudaStream_t s) {
    k_counts<<<dim3(1, g.S), 32, 0, s>>>(d);
}
void launch_advance(const SimView* d, const GroupDims& g, int which, cudaStream_t s) {
    k_advance<<<dim3(1, g.S), 32, 0, s>>>(d, which);
}

// ======================================================================================
// Slots of a layer: scale in the band (Eq. 32 restricted to [lo, hi), inverse transform of
// Appendix D) and the picked bead; then bucketing by coarse cell in colour-major order.
// ======================================================================================
__global__ void k_slots(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(l >= gv.nL || (int)(blockIdx.x * blockDim.x) >= gv.counts[l])
    SIM_PROLOGUE
    if (l >= v.nL) return;
    const int M = v.counts[l];
    const uint64_t sweep = v.step[0];
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    const LayerDev& Ly = v.layer[l];
    u4 w = draw(v.k0, v.k1, K_SLOT, l, sweep, (uint32_t)j, 0);
    double u = u53(w.x, w.y);
    double wv = sub(Ly.ilo3, mul(u, sub(Ly.ilo3, Ly.ihi3)));
    v.slot_lam[j] = inv_cbrt_band(wv, Ly.lo);
    v.slot_bead[j] = (int)pick(w.z, w.w, v.N);
    v.tr_out[Ly.tr_off + j] = 0;
    v.tr_n[Ly.tr_off + j] = 0;
    v.tr_du[Ly.tr_off + j] = 0.0;
    // the rest of the slot's draws, whichever phase runs it: centre offset V in the unit ball
    // (or the centre itself, uniform in the box), unit polarisation p by rejection (Appendix D),
    // and the acceptance threshold (Eq. 20); one slot per thread, so full warps share the
    // binary64 work
    double V[3] = {0.0, 0.0, 0.0}, p[3] = {0.0, 0.0, 1.0};
    // the first attempt in the ball; a binary32 test decides away from the sphere and the centre (its
    // error is below 1e-6), the binary64 one of the definition near them: fourteen binary64
    // instructions an attempt held the pipe of this kernel longer than everything else in it
    auto ball = [&](uint32_t kind, bool nonzero, double* out) {
        for (uint32_t a = 0; a < 64; a++) {
            const u4 w = draw(v.k0, v.k1, kind, l, sweep, (uint32_t)j, a);
            const float fx = (float)(int)(w.x ^ 0x80000000u), fy = (float)(int)(w.y ^ 0x80000000u), fz = (float)(int)(w.z ^ 0x80000000u);
            const float f = (fx * fx + fy * fy + fz * fz) * (1.0f / 4611686018427387904.0f);
            bool in = f < 1.0f;
            if (fabsf(f - 1.0f) < 1e-5f || f < 1e-5f) {
                const double q = norm2(sym(w.x), sym(w.y), sym(w.z));
                in = q <= 1.0 && (!nonzero || q > 0.0);
            }
            if (in) { out[0] = sym(w.x); out[1] = sym(w.y); out[2] = sym(w.z); break; }
        }
    };
    ball(K_VB, false, V);
    ball(K_VP, true, p);
    const double r = sqr_t(norm2(p[0], p[1], p[2]));
    if (v.centring == 1) uniform_centre(v, l, sweep, (uint32_t)j, V);   // slot_V holds the centre itself
    // p / r as div_by, through one reciprocal (not for a significand of ones)
    const double ir = dvd(1.0, r);
    const bool ones = (__double_as_longlong(r) & 0xfffffffffffffLL) == 0xfffffffffffffLL;
    for (int a = 0; a < 3; a++) {
        v.slot_V[3 * j + a] = V[a];
        v.slot_p[3 * j + a] = ones ? dvd(p[a], r) : div_by(p[a], r, ir);
    }
    const u4 wa = draw(v.k0, v.k1, K_ACC, l, sweep, (uint32_t)j, 0);
    v.slot_thr[j] = accept_threshold(v, wa);
}
void launch_slots(const SimView* d, const GroupDims& g, int l, cudaStream_t s) {
    k_slots<<<dim3((g.Mmax[l] + 255) / 256, g.S), 256, 0, s>>>(d, l);
}

// The layer record of schedule index l: layer l itself, or (l >= kLevel2) the second colouring
// of layer l - kLevel2, with its grid and carries in place of the layer's own.
__device__ __forceinline__ LayerDev sched_layer(const SimView& v, int l) {
    if (l < kLevel2) return v.layer[l];
    LayerDev y = v.layer[l - kLevel2];
    y.G = y.G2;
    y.invG = y.invG2;
    y.carry_off = y.carry_off2;
    return y;
}
__device__ __forceinline__ bool sched_on(const SimView& v, int l) {
    return layer_real(l) < v.nL && (l < kLevel2 ? v.layer[l].G : v.layer[l - kLevel2].G2) > 0;
}
// slots a schedule index buckets: the layer's slots, or the ones its first colouring deferred
__device__ __forceinline__ int sched_count(const SimView& v, int l) { return l < kLevel2 ? v.counts[l] : *v.serial_count; }
// largest support a concurrent move of the index takes
__device__ __forceinline__ int sched_ncap(const SimView& v, int l) { return l < kLevel2 ? v.n_cap : kNCapMax; }

// The slots of schedule index l by coarse cell (of the picked bead now, or of the centre):
// entry t is slot t of the layer, or for a second colouring the t-th slot its first deferred.
__global__ void k_bucket_count(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(!sched_on(gv, l) || (int)(blockIdx.x * blockDim.x) >= sched_count(gv, l))
    SIM_PROLOGUE
    if (!sched_on(v, l)) return;
    const int M = sched_count(v, l);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= M) return;
    const int j = l < kLevel2 ? t : v.serial_list[t];
    const LayerDev Ly = sched_layer(v, l);
    const int G = Ly.G, K = v.K, Q = G / K;
    double xs[3];
    if (v.centring == 1) uniform_centre(v, layer_real(l), v.step[0], (uint32_t)j, xs);      // bucket by the centre
    else {
        const Bead b = v.bead[v.slot_bead[j]];
        xs[0] = b.x; xs[1] = b.y; xs[2] = b.z;
    }
    int c[3];
    for (int a = 0; a < 3; a++) {
        double f = floor(mul(xs[a], Ly.invG));
        int ci = (int)f;
        if (f < 0.0) ci = 0;
        if (ci >= G) ci = G - 1;
        c[a] = ci;
    }
    int colour = (c[0] % K) + K * ((c[1] % K) + K * (c[2] % K));
    int q = (c[0] / K) + Q * ((c[1] / K) + Q * (c[2] / K));
    int key = colour * Q * Q * Q + q;
    v.slot_key[t] = key;
    atomicAdd(&v.q_count[key], 1);
}
// Exclusive prefix of one value per thread over a block of NW warps: a shuffle scan per warp, the warp
// totals scanned by warp 0; two block barriers. *total receives the sum.
template <int NW = 32>
__device__ __forceinline__ int block_excl_scan(int x, int* s_w, int* total) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = x;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_w[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const int c = lane < NW ? s_w[lane] : 0;
        int ci = c;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, ci, o);
            if (lane >= o) ci += y;
        }
        if (lane < NW) s_w[lane] = ci - c;
        if (lane == 31) s_w[32] = ci;
    }
    __syncthreads();
    *total = s_w[32];
    return s_w[wid] + incl - x;
}
constexpr int kScanPer = 8;   // consecutive entries per thread in the single-block scans

// exclusive scan of n ints by one block of 1,024 threads per simulation: mode 0 = bucket counts
// of layer l (G^3 keys), mode 1 = region counts of layer l (Q^3 queues); each thread takes
// kScanPer consecutive entries of a chunk. With heavy_lo >= 0 (mode 1) it also lists the queues
// of the colour phase that have slots and more than heavy_lo beads in their region or more than heavy_slots
// slots, in no particular order: those with at most heavy_mid beads from the front of hq_list, the others
// from its back, and resets the two lists' work counters.
// parts > 1: `parts` blocks per simulation, each with its share of the chunks, after k_scan_sums left
// every share's sum in scan_part (1.6 million buckets by one block: 1.1 ms).
__global__ void k_scan_sums(const SimView* __restrict__ vs, int mode, int l) {
    SIM_EXIT_IF(!sched_on(gv, l))
    SIM_PROLOGUE
    if (!sched_on(v, l)) return;
    const int G = sched_layer(v, l).G, Q = G / v.K;
    const int n = mode == 0 ? G * G * G : Q * Q * Q;
    const int* in = mode == 0 ? v.q_count : v.rcount;
    const int chunks = (n + kScanPer * 1024 - 1) / (kScanPer * 1024), per = (chunks + gridDim.x - 1) / gridDim.x;
    const int i0 = blockIdx.x * per * kScanPer * 1024, i1 = min(n, i0 + per * kScanPer * 1024);
    int sum = 0;
    for (int i = i0 + threadIdx.x; i < i1; i += 1024) sum += in[i];
    __shared__ int s_w[33];
    int total;
    block_excl_scan(sum, s_w, &total);
    if (threadIdx.x == 0) v.scan_part[blockIdx.x] = total;
    if (mode == 1 && blockIdx.x == 0 && threadIdx.x < 4) v.hq_ctl[threadIdx.x] = 0;
}
__global__ void k_scan(const SimView* __restrict__ vs, int mode, int l, int colour, int heavy_lo, int heavy_slots, int heavy_mid) {
    SIM_EXIT_IF(!sched_on(gv, l))
    SIM_PROLOGUE
    if (!sched_on(v, l)) return;
    const int G = sched_layer(v, l).G, Q = G / v.K;
    const int n = mode == 0 ? G * G * G : Q * Q * Q;
    const int* in = mode == 0 ? v.q_count : v.rcount;
    int* out = mode == 0 ? v.q_start : v.rstart;
    __shared__ int s_w[33];
    const bool parts = gridDim.x > 1;
    const int chunks = (n + kScanPer * 1024 - 1) / (kScanPer * 1024), per = (chunks + gridDim.x - 1) / gridDim.x;
    const int b0 = blockIdx.x * per * kScanPer * 1024, b1 = min(n, b0 + per * kScanPer * 1024);
    int carry = 0;
    if (parts) {
        int x = 0;
        for (int i = threadIdx.x; i < (int)blockIdx.x; i += 1024) x += v.scan_part[i];
        block_excl_scan(x, s_w, &carry);
        __syncthreads();
    }
    for (int base = b0; base < b1; base += kScanPer * 1024) {
        const int i0 = base + kScanPer * (int)threadIdx.x;
        int x[kScanPer], sum = 0;
#pragma unroll
        for (int u = 0; u < kScanPer; u++) { x[u] = i0 + u < n ? in[i0 + u] : 0; sum += x[u]; }
        int total;
        int pre = carry + block_excl_scan(sum, s_w, &total);
#pragma unroll
        for (int u = 0; u < kScanPer; u++) {
            if (i0 + u < n) out[i0 + u] = pre;
            pre += x[u];
        }
        carry += total;
        __syncthreads();                          // s_w is rewritten by the next chunk
    }
    if (mode == 1 && heavy_lo >= 0 && parts) {
        for (int q = b0 + threadIdx.x; q < b1; q += blockDim.x)
            if (const int slots = v.q_count[colour * n + q]; slots > 0 && (in[q] > heavy_lo || slots > heavy_slots)) {
                if (in[q] <= heavy_mid) v.hq_list[atomicAdd(&v.hq_ctl[0], 1)] = q;
                else v.hq_list[n - 1 - atomicAdd(&v.hq_ctl[2], 1)] = q;
            }
    } else if (mode == 1 && heavy_lo >= 0) {
        __shared__ int hc[2];
        if (threadIdx.x < 2) hc[threadIdx.x] = 0;
        __syncthreads();
        for (int q = threadIdx.x; q < n; q += blockDim.x)
            if (const int slots = v.q_count[colour * n + q]; slots > 0 && (in[q] > heavy_lo || slots > heavy_slots)) {
                if (in[q] <= heavy_mid) v.hq_list[atomicAdd(&hc[0], 1)] = q;
                else v.hq_list[n - 1 - atomicAdd(&hc[1], 1)] = q;
            }
        __syncthreads();
        if (threadIdx.x == 0) { v.hq_ctl[0] = hc[0]; v.hq_ctl[1] = 0; v.hq_ctl[2] = hc[1]; v.hq_ctl[3] = 0; }
    }
}
// blocks per simulation of a scan of n entries: one up to four chunks, else one per chunk (at most
// kScanParts); below that the second launch costs more than it saves
constexpr int kScanParts = 256;
static int launch_scan(const SimView* d, const GroupDims& g, int64_t n, int mode, int l, int colour, int heavy_lo, int heavy_slots,
                       int heavy_mid, cudaStream_t s) {
    const int64_t chunks = (n + kScanPer * 1024 - 1) / (kScanPer * 1024);
    const unsigned parts = chunks > 4 ? (unsigned)std::min<int64_t>(chunks, kScanParts) : 1u;
    if (parts > 1) k_scan_sums<<<dim3(parts, g.S), 1024, 0, s>>>(d, mode, l);
    k_scan<<<dim3(parts, g.S), 1024, 0, s>>>(d, mode, l, colour, heavy_lo, heavy_slots, heavy_mid);
    return parts > 1 ? 2 : 1;
}
// zero the per-phase counters: mode 0 = bucket counts, fills and deferral flags of layer l,
// mode 1 = region counts
__global__ void k_zero(const SimView* __restrict__ vs, int mode, int l) {
    SIM_EXIT_IF(!sched_on(gv, l))
    SIM_PROLOGUE
    if (!sched_on(v, l)) return;
    const int G = sched_layer(v, l).G, Q = G / v.K;
    const int n = mode == 0 ? G * G * G : Q * Q * Q;
    int* a = mode == 0 ? v.q_count : v.rcount;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        a[i] = 0;
        if (mode == 0) v.q_fill[i] = 0;
    }
    if (mode == 0) {
        const int M = v.layer[layer_real(l)].Mmax;
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += gridDim.x * blockDim.x) v.defer[i] = 0;
    }
}
__global__ void k_bucket_scatter(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(!sched_on(gv, l) || (int)(blockIdx.x * blockDim.x) >= sched_count(gv, l))
    SIM_PROLOGUE
    if (!sched_on(v, l)) return;
    const int M = sched_count(v, l);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= M) return;
    int key = v.slot_key[t];
    int pos = v.q_start[key] + atomicAdd(&v.q_fill[key], 1);
    v.q_slots[pos] = t;
}
// slots of one queue in ascending slot id (the order of the sequential schedule); a second
// colouring sorts its entries in first-schedule order and then names their slots. A short queue is
// sorted by its thread; a longer one by the warp, every entry placed at its rank (the count of smaller
// entries) by way of slot_key, free once the entries are scattered: one thread's insertion sort of the
// ~270 slots of a queue took 2 ms (65k semi-dilute beads, 34.0 -> 31.1 ms a sweep; a chain of 1,001 beads 3.3 -> 2.6).
constexpr int kSortThread = 16;
__global__ void k_bucket_sort(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(!sched_on(gv, l))
    SIM_PROLOGUE
    if (!sched_on(v, l)) return;
    const int G = sched_layer(v, l).G, nkeys = G * G * G;
    const int key = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    const int s = key < nkeys ? v.q_start[key] : 0, n = key < nkeys ? v.q_count[key] : 0;
    int* a = v.q_slots + s;
    if (n <= kSortThread) {
        for (int i = 1; i < n; i++) {
            int x = a[i], b = i - 1;
            while (b >= 0 && a[b] > x) { a[b + 1] = a[b]; b--; }
            a[b + 1] = x;
        }
    }
    for (unsigned bits = __ballot_sync(FULL, n > kSortThread); bits; bits &= bits - 1u) {
        const int src = __ffs(bits) - 1, s1 = __shfl_sync(FULL, s, src), n1 = __shfl_sync(FULL, n, src);
        int* const q = v.q_slots + s1;
        int* const t = v.slot_key + s1;
        for (int i = lane; i < n1; i += 32) {
            const int x = q[i];
            int r = 0;
#pragma unroll 4
            for (int j = 0; j < n1; j++) r += q[j] < x;
            t[r] = x;
        }
        __syncwarp();
        for (int i = lane; i < n1; i += 32) q[i] = t[i];
        __syncwarp();
    }
    if (l >= kLevel2)
        for (int i = 0; i < n; i++) a[i] = v.serial_list[a[i]];
}
int launch_bucket(const SimView* d, const GroupDims& g, int l, cudaStream_t s) {
    const int keys = g.keys[l], M = g.Mmax[l];
    k_zero<<<dim3(gx((std::max(keys, M) + 255) / 256, g.S), g.S), 256, 0, s>>>(d, 0, l);
    k_bucket_count<<<dim3((M + 255) / 256, g.S), 256, 0, s>>>(d, l);
    const int scans = launch_scan(d, g, keys, 0, l, 0, -1, 0, 0, s);
    k_bucket_scatter<<<dim3((M + 255) / 256, g.S), 256, 0, s>>>(d, l);
    k_bucket_sort<<<dim3((keys + 127) / 128, g.S), 128, 0, s>>>(d, l);
    return 4 + scans;
}

// deferred slots in schedule order -> serial list
__global__ void k_defer_compact(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(!sched_on(gv, l))
    SIM_PROLOGUE
    if (!sched_on(v, l)) return;
    // (a second colouring's entries are the first one's deferred slots: read before the barriers
    // below, ahead of the new count written at the end)
    const int M = sched_count(v, l);
    // the deferred slots in schedule order: each thread takes kScanPer consecutive entries of a
    // chunk, a block prefix of the per-thread counts places them; chunks without a deferred slot
    // (nearly all) cost one block vote
    __shared__ int s_w[33];
    int carry = 0;
    for (int base = 0; base < M; base += kScanPer * 1024) {
        const int i0 = base + kScanPer * (int)threadIdx.x;
        unsigned f = 0u;
#pragma unroll
        for (int u = 0; u < kScanPer; u++)
            if (i0 + u < M && v.defer[i0 + u]) f |= 1u << u;
        if (!__syncthreads_or(f != 0u)) continue;
        int total;
        int pos = carry + block_excl_scan(__popc(f), s_w, &total);
        for (; f; f &= f - 1u) v.serial_list[pos++] = v.q_slots[i0 + __ffs(f) - 1];
        carry += total;
        __syncthreads();                          // s_w is rewritten by the next chunk
    }
    if (threadIdx.x == 0) *v.serial_count = carry;
}
void launch_defer_compact(const SimView* d, const GroupDims& g, int l, cudaStream_t s) {
    k_defer_compact<<<dim3(1, g.S), 1024, 0, s>>>(d, l);
}

}  // namespace wmcd

namespace wmcd {

// ======================================================================================
// Concurrent wavelet moves: one warp per queue (coarse cell) of one colour.
// ======================================================================================
struct WarpSmem {
    int ids[kNCapMax];          // support, in gather order
    double op[kNCapMax][3];     // old positions
    double np[kNCapMax][3];     // new (wrapped) positions
    double nu[kNCapMax][3];     // new unwrapped positions (old + delta)
    int dimg[kNCapMax];         // packed image change
    int sid[kNCapMax];          // support ids ascending
    int cpre[kNCapMax + 1];     // prefix of partner-search columns per member
    int cbox[kNCapMax][6];      // partner-search box per member: first cell c0[3], cells nc[3]
};

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}
__device__ __forceinline__ int warp_sum_i(int x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}
__device__ __forceinline__ bool sorted_has(const int* a, int n, int x) {
    int lo = 0, hi = n - 1;
    while (lo <= hi) {
        int m = (lo + hi) >> 1;
        if (a[m] == x) return true;
        if (a[m] < x) lo = m + 1; else hi = m - 1;
    }
    return false;
}

// Uniform point of the unit ball by rejection (Appendix D): attempt a uses counter attempt a;
// the warp tries 32 attempts at once and takes the first accepted one, which is what a
// sequential loop over the attempts would return.
__device__ void warp_ball_point(const SimView& v, uint32_t kind, int l, uint64_t sweep, uint32_t j, bool nonzero,
                                int lane, double V[3]) {
    for (int base = 0; base < 64; base += 32) {
        u4 w = draw(v.k0, v.k1, kind, l, sweep, j, (uint32_t)(base + lane));
        double x = sym(w.x), y = sym(w.y), z = sym(w.z);
        double q = norm2(x, y, z);
        unsigned ok = __ballot_sync(0xffffffffu, q <= 1.0 && (!nonzero || q > 0.0));
        if (ok) {
            int src = __ffs(ok) - 1;
            V[0] = __shfl_sync(0xffffffffu, x, src);
            V[1] = __shfl_sync(0xffffffffu, y, src);
            V[2] = __shfl_sync(0xffffffffu, z, src);
            return;
        }
    }
    V[0] = 0.0; V[1] = 0.0; V[2] = nonzero ? 1.0 : 0.0;
}

// cell box [floor((lo) invf), floor((hi) invf)] per axis, at most Gf cells
__device__ __forceinline__ void cell_box(const SimView& v, const double lo[3], const double hi[3], int c0[3], int nc[3]) {
    for (int a = 0; a < 3; a++) {
        int t0 = (int)floor(mul(lo[a], v.invf));
        int t1 = (int)floor(mul(hi[a], v.invf));
        c0[a] = t0;
        nc[a] = min(t1 - t0 + 1, v.Gf);
    }
}
__device__ __forceinline__ int box_cell(const SimView& v, const int c0[3], const int nc[3], int k) {
    int kx = k % nc[0], ky = (k / nc[0]) % nc[1], kz = k / (nc[0] * nc[1]);
    return wrapi(c0[0] + kx, v.Gf) + v.Gf * (wrapi(c0[1] + ky, v.Gf) + v.Gf * wrapi(c0[2] + kz, v.Gf));
}

// cell index modulo G: one add or subtract in the common case, a remainder otherwise
__device__ __forceinline__ int wrapc(int c, int G) {
    if (c < 0) c += G;
    else if (c >= G) c -= G;
    if ((unsigned)c >= (unsigned)G) { c %= G; if (c < 0) c += G; }
    return c;
}

// fn(cell) for the occupied fine cells of a box (first cell c0, cells per axis nc), in ascending z, y
// and x from c0: a row's x range is read as one or two occupancy words, which stay in L2 where the
// heads of the cells (mostly empty) do not
template <class F>
__device__ __forceinline__ void for_occupied(const SimView& v, const int c0[3], const int nc[3], F&& fn) {
    const int Gf = v.Gf, x0 = wrapc(c0[0], Gf);
    for (int kz = 0; kz < nc[2]; kz++) {
        const int z = wrapc(c0[2] + kz, Gf);
        for (int ky = 0; ky < nc[1]; ky++) {
            const int yz = wrapc(c0[1] + ky, Gf) + Gf * z;
            if (!v.occ) {                             // no bits kept: every cell
                for (int kx = 0; kx < nc[0]; kx++) fn(Gf * yz + wrapc(c0[0] + kx, Gf));
                continue;
            }
            const uint32_t* row = v.occ + (size_t)yz * v.occ_w;
            // the x range [x0, x0 + nc) as at most two pieces inside [0, Gf)
            for (int piece = 0; piece < 2; piece++) {
                const int xa = piece == 0 ? x0 : 0, xb = piece == 0 ? min(x0 + nc[0], Gf) : x0 + nc[0] - Gf;
                for (int wi = xa >> 5; xa < xb && wi <= (xb - 1) >> 5; wi++)
                    for (uint32_t bits = occ_masked(row[wi], xa, xb, wi); bits; bits &= bits - 1u)
                        fn(Gf * yz + (wi << 5) + __ffs(bits) - 1);
            }
        }
    }
}

// difference a - b of two wrapped coordinates in binary32, minimum image applied
__device__ __forceinline__ float dif32(double a, double b, double L, float hLf) {
    const double d = sub(a, b);
    float f = (float)d;
    if (fabsf(f) > hLf) f = (float)(d > 0.0 ? sub(d, L) : add(d, L));
    return f;
}
// minimum image of a binary32 difference
__device__ __forceinline__ float wrapn(float f, float L, float hL) { return fabsf(f) > hL ? f - copysignf(L, f) : f; }
__device__ __forceinline__ float norm2f(float x, float y, float z) { return x * x + y * y + z * z; }

// binary32 pair energies with a magnitude m such that |error| <= 64 u m  (u = 2^-24)
struct Pot32 {
    float sig2, eps, rc2, bk, br0, br02, R02, kappa, hL;
    int bond, kappa_on, eps_on;
};
__device__ __forceinline__ Pot32 pot32(const Pot& P) {
    Pot32 q;
    q.sig2 = (float)P.sig2; q.eps = (float)P.eps; q.rc2 = (float)P.rc2; q.bk = (float)P.bk; q.br0 = (float)P.br0;
    q.br02 = q.br0 * q.br0; q.R02 = (float)P.R02; q.kappa = (float)P.kappa; q.hL = (float)P.halfL; q.bond = P.bond;
    q.kappa_on = P.kappa != 0.0; q.eps_on = P.eps != 0.0;
    return q;
}
__device__ __forceinline__ void wca32(const Pot32& P, float r2, float& u, float& m) {
    if (P.eps == 0.0f || !(r2 < P.rc2)) { u = 0.0f; m = 0.0f; return; }
    const float s2 = __fdiv_rn(P.sig2, r2), s6 = s2 * s2 * s2, s12 = s6 * s6;
    u = 4.0f * P.eps * (s12 - s6) + P.eps;
    m = 4.0f * P.eps * (s12 + s6) + P.eps;
}
__device__ __forceinline__ void bond32(const Pot32& P, float r2, float& u, float& m) {
    if (P.bond == 1) {
        // |error| <= 5 ulp * k (|d| r + d^2): r2 carries ~7 ulp, sqrt halves it, one more for
        // the subtraction and two for the products (scaled by 80 ulp in the band: ample)
        const float r = __fsqrt_rn(r2), d = r - P.br0;
        u = 0.5f * P.bk * d * d;
        m = P.bk * (fabsf(d) * r + d * d + 1e-6f * P.br02);
    } else if (P.bond == 2) {
        const float x = __fdiv_rn(r2, P.R02);
        if (!(x < 0.98f)) { u = 0.0f; m = __int_as_float(0x7f800000); return; }   // near R0: decide in FP64
        const float lg = log1pf(-x);
        u = -0.5f * P.bk * P.R02 * lg;
        m = 0.5f * P.bk * P.R02 * (fabsf(lg) + 8.0f * x / (1.0f - x) + 1.0f);
    } else {
        u = 0.0f; m = 0.0f;
    }
}

// Partner-search boxes of the support: [min(old, new) - rc, max(old, new) + rc] per member;
// columns (x, y) are spread over lanes, z is looped. Returns the column count and max z extent.
__device__ void partner_boxes(const SimView& v, WarpSmem& sm, int n, int lane, int* ncols, int* nzmax) {
    int nz = 0;
    for (int k = lane; k < n; k += 32) {
        int c0[3], nc[3];
        for (int a = 0; a < 3; a++) {
            const double o = sm.op[k][a], u = sm.nu[k][a];
            c0[a] = (int)floor(mul(sub(fmin(o, u), v.rc + 1e-9), v.invf));
            const int t1 = (int)floor(mul(add(fmax(o, u), v.rc + 1e-9), v.invf));
            nc[a] = min(t1 - c0[a] + 1, v.Gf);
        }
        for (int a = 0; a < 3; a++) { sm.cbox[k][a] = c0[a]; sm.cbox[k][3 + a] = nc[a]; }
        sm.cpre[k + 1] = nc[0] * nc[1];
        nz = max(nz, nc[2]);
    }
    __syncwarp();
    if (lane == 0) { sm.cpre[0] = 0; for (int k = 0; k < n; k++) sm.cpre[k + 1] += sm.cpre[k]; }
    for (int o = 16; o > 0; o >>= 1) nz = max(nz, __shfl_xor_sync(0xffffffffu, nz, o));
    __syncwarp();
    *ncols = sm.cpre[n];
    *nzmax = nz;
}

// Energy change of the move (Eqs. 1, 2; external well): support-support pairs, bonds to beads
// outside the support, WCA to beads outside the support (cell lists). F32: binary32 terms,
// returns the sum, the magnitude sum and the term count; otherwise binary64.
template <bool F32>
__device__ void energy(const SimView& v, WarpSmem& sm, int n, int lane, int ncols, int nzmax, double* dU64,
                       float* dU32, float* mag32, int* terms, int* pe_out) {
    const double L = v.L, hL = v.halfL;
    const Pot& P = v.pot;
    const Pot32 P32 = pot32(P);
    const float hLf = (float)hL;
    double a64 = 0.0;
    float a32 = 0.0f, m32 = 0.0f;
    int T = 0, pe = 0;
    // external well and bonds to partners outside the support
    for (int k = lane; k < n; k += 32) {
        if (P.kappa != 0.0) {
            if (F32) {
                float x = dif32(sm.np[k][0], hL, L, hLf), y = dif32(sm.np[k][1], hL, L, hLf), z = dif32(sm.np[k][2], hL, L, hLf);
                float un = 0.5f * P32.kappa * norm2f(x, y, z);
                x = dif32(sm.op[k][0], hL, L, hLf); y = dif32(sm.op[k][1], hL, L, hLf); z = dif32(sm.op[k][2], hL, L, hLf);
                float uo = 0.5f * P32.kappa * norm2f(x, y, z);
                a32 += un - uo; m32 += un + uo; T += 2;
            } else {
                a64 += U_ext(P, sm.np[k][0], sm.np[k][1], sm.np[k][2]) - U_ext(P, sm.op[k][0], sm.op[k][1], sm.op[k][2]);
            }
        }
        const int m = sm.ids[k];
        for (int e = 0; e < 2; e++) {
            const int q = e ? m + 1 : m - 1;
            if (q < 0 || q >= v.N || !(e ? v.bnext[m] : v.bnext[q]) || sorted_has(sm.sid, n, q)) continue;
            const Bead bq = v.bead[q];
            if (F32) {
                float r2n = norm2f(dif32(sm.np[k][0], bq.x, L, hLf), dif32(sm.np[k][1], bq.y, L, hLf), dif32(sm.np[k][2], bq.z, L, hLf));
                float r2o = norm2f(dif32(sm.op[k][0], bq.x, L, hLf), dif32(sm.op[k][1], bq.y, L, hLf), dif32(sm.op[k][2], bq.z, L, hLf));
                float un, mn, uo, mo;
                bond32(P32, r2n, un, mn);
                bond32(P32, r2o, uo, mo);
                a32 += un - uo; m32 += mn + mo; T += 2;
            } else {
                double r2n = norm2(mi(sm.np[k][0] - bq.x, L, hL), mi(sm.np[k][1] - bq.y, L, hL), mi(sm.np[k][2] - bq.z, L, hL));
                double r2o = norm2(mi(sm.op[k][0] - bq.x, L, hL), mi(sm.op[k][1] - bq.y, L, hL), mi(sm.op[k][2] - bq.z, L, hL));
                a64 += U_bond(P, r2n) - U_bond(P, r2o);
            }
        }
    }
    // pairs inside the support
    const int npairs = n * (n - 1) / 2;
    for (int t = lane; t < npairs; t += 32) {
        int a = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
        while (a * (a + 1) / 2 > t) a--;
        while ((a + 1) * (a + 2) / 2 <= t) a++;
        const int k1 = t - a * (a + 1) / 2, k2 = a + 1;
        const int m1 = sm.ids[k1], m2 = sm.ids[k2];
        const int lo_ = min(m1, m2), hi_ = max(m1, m2);
        const bool bonded = hi_ == lo_ + 1 && v.bnext[lo_];
        if (F32) {
            float r2n = norm2f(dif32(sm.np[k1][0], sm.np[k2][0], L, hLf), dif32(sm.np[k1][1], sm.np[k2][1], L, hLf),
                               dif32(sm.np[k1][2], sm.np[k2][2], L, hLf));
            float r2o = norm2f(dif32(sm.op[k1][0], sm.op[k2][0], L, hLf), dif32(sm.op[k1][1], sm.op[k2][1], L, hLf),
                               dif32(sm.op[k1][2], sm.op[k2][2], L, hLf));
            float un, mn, uo, mo;
            wca32(P32, r2n, un, mn);
            wca32(P32, r2o, uo, mo);
            a32 += un - uo; m32 += mn + mo; T += 2;
            if (bonded) { bond32(P32, r2n, un, mn); bond32(P32, r2o, uo, mo); a32 += un - uo; m32 += mn + mo; T += 2; }
        } else {
            double r2n = norm2(mi(sm.np[k1][0] - sm.np[k2][0], L, hL), mi(sm.np[k1][1] - sm.np[k2][1], L, hL),
                               mi(sm.np[k1][2] - sm.np[k2][2], L, hL));
            double r2o = norm2(mi(sm.op[k1][0] - sm.op[k2][0], L, hL), mi(sm.op[k1][1] - sm.op[k2][1], L, hL),
                               mi(sm.op[k1][2] - sm.op[k2][2], L, hL));
            double u = U_wca(P, r2n) - U_wca(P, r2o);
            if (bonded) u += U_bond(P, r2n) - U_bond(P, r2o);
            a64 += u;
        }
    }
    // WCA with beads outside the support, through the cell lists
    if (P.eps != 0.0) {
        const int Gf = v.Gf;
        for (int base = 0; base < ncols; base += 32) {
            const int w = base + lane;
            int k = 0, cx = 0, cy = 0, c0z = 0, nz = 0;
            const bool valid = w < ncols;
            if (valid) {
                while (sm.cpre[k + 1] <= w) k++;
                const int col = w - sm.cpre[k], nx = sm.cbox[k][3];
                cx = wrapc(sm.cbox[k][0] + col % nx, Gf);
                cy = wrapc(sm.cbox[k][1] + col / nx, Gf);
                c0z = sm.cbox[k][2];
                nz = sm.cbox[k][5];
            }
            const int m = sm.ids[k];
            const int colbase = cx + Gf * cy;
            for (int kz = 0; kz < nzmax; kz++) {
                int q = (valid && kz < nz) ? v.head[colbase + Gf * Gf * wrapc(c0z + kz, Gf)] : -1;
                int guard = 0;
                while (q >= 0) {
                    const Bead bq = v.bead[q];
                    if (q != m && !sorted_has(sm.sid, n, q)) {
                        if (F32) {
                            float r2n = norm2f(dif32(sm.np[k][0], bq.x, L, hLf), dif32(sm.np[k][1], bq.y, L, hLf),
                                               dif32(sm.np[k][2], bq.z, L, hLf));
                            float r2o = norm2f(dif32(sm.op[k][0], bq.x, L, hLf), dif32(sm.op[k][1], bq.y, L, hLf),
                                               dif32(sm.op[k][2], bq.z, L, hLf));
                            if (r2n < P32.rc2 || r2o < P32.rc2) {
                                float un, mn, uo, mo;
                                wca32(P32, r2n, un, mn);
                                wca32(P32, r2o, uo, mo);
                                a32 += un - uo; m32 += mn + mo; T += 2; pe++;
                            }
                        } else {
                            double r2n = norm2(mi(sm.np[k][0] - bq.x, L, hL), mi(sm.np[k][1] - bq.y, L, hL),
                                               mi(sm.np[k][2] - bq.z, L, hL));
                            double r2o = norm2(mi(sm.op[k][0] - bq.x, L, hL), mi(sm.op[k][1] - bq.y, L, hL),
                                               mi(sm.op[k][2] - bq.z, L, hL));
                            if (r2n < P.rc2 || r2o < P.rc2) { a64 += U_wca(P, r2n) - U_wca(P, r2o); pe++; }
                        }
                    }
                    q = bq.next;
                    if (++guard > kMaxWalk) { set_err(v, E_WALK); break; }
                }
            }
        }
    }
    // lane 0's sums for every lane (a butterfly leaves lanes with differently rounded totals)
    const unsigned FULL = 0xffffffffu;
    if (F32) {
        float s = a32, mm = m32;
        int tt = T;
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(FULL, s, o);
            mm += __shfl_xor_sync(FULL, mm, o);
            tt = max(tt, __shfl_xor_sync(FULL, tt, o));
        }
        *dU32 = __shfl_sync(FULL, s, 0);
        *mag32 = __shfl_sync(FULL, mm, 0);
        *terms = __shfl_sync(FULL, tt, 0) + 5;   // summation depth: one lane's terms, then the butterfly
    } else {
        *dU64 = __shfl_sync(FULL, warp_sum(a64), 0);
    }
    *pe_out = warp_sum_i(pe);
}

template <int PREC>
__device__ int warp_attempt(const SimView& v, WarpSmem& sm, int ls, int j, int i, double lam, uint64_t sweep,
                            const int64_t rlo[3], const int64_t rhi[3], int lane, int* n_out, int* pe_out,
                            int* recheck_out, double* du_out) {
    const unsigned FULL = 0xffffffffu;
    const int l = layer_real(ls), ncap = sched_ncap(v, ls);   // draws are the layer's own
    const double L = v.L, hL = v.halfL;
    const float hLf = (float)hL;
    *du_out = 0.0;
    const int Gf = v.Gf;
    // centre b = r_i + lam V (Appendix D), wrapped into the box; or uniform in the box
    double V[3], b[3];
    if (v.centring == 1) uniform_centre(v, l, sweep, (uint32_t)j, b);
    else {
        const double ri[3] = {v.bead[i].x, v.bead[i].y, v.bead[i].z};
        warp_ball_point(v, K_VB, l, sweep, (uint32_t)j, false, lane, V);
        for (int a = 0; a < 3; a++) b[a] = wrap(add(ri[a], mul(lam, V[a])), L, nullptr);
    }
    // the influence ball must lie in fine cells wholly inside the queue's region
    const double R = add(add(lam, rule_disp(v, lam)), v.r_reach);
    for (int a = 0; a < 3; a++) {
        const int64_t t0 = (int64_t)floor(mul(sub(b[a], R), v.invf));
        const int64_t t1 = (int64_t)floor(mul(add(b[a], R), v.invf));
        if (!range_inside(t0, t1, rlo[a], rhi[a], Gf)) return DEFER;
    }
    // gather the support: beads strictly inside the ball (one image each, lambda <= L/2);
    // binary32 prefilter, exact binary64 test within 1e-6 of the sphere
    const double lam2 = mul(lam, lam);
    const float lam2f = (float)lam2, lin = lam2f * (1.0f - 1e-6f), lout = lam2f * (1.0f + 1e-6f);
    int c0[3], nc[3];
    for (int a = 0; a < 3; a++) {
        c0[a] = (int)floor(mul(sub(b[a], lam + 1e-9), v.invf));
        const int t1 = (int)floor(mul(add(b[a], lam + 1e-9), v.invf));
        nc[a] = min(t1 - c0[a] + 1, Gf);
    }
    int n = 0;
    // one bead per lane per step: test it, vote, append the members in vote order; a support
    // above n_cap means the move is deferred, so the walk stops there
    auto step = [&](int& ptr) {
        bool in = false;
        int nxt = -1;
        Bead bb;
        if (ptr >= 0) {
            bb = v.bead[ptr];
            nxt = bb.next;
            const float d2f = norm2f(dif32(bb.x, b[0], L, hLf), dif32(bb.y, b[1], L, hLf), dif32(bb.z, b[2], L, hLf));
            if (d2f < lin) in = true;
            else if (d2f <= lout) {
                const double e2 = norm2(mi(sub(bb.x, b[0]), L, hL), mi(sub(bb.y, b[1]), L, hL), mi(sub(bb.z, b[2]), L, hL));
                in = e2 < lam2;
            }
        }
        const unsigned msk = __ballot_sync(FULL, in);
        const int slot = n + __popc(msk & ((1u << lane) - 1u));
        if (in && slot < kNCapMax) {
            sm.ids[slot] = ptr;
            sm.op[slot][0] = bb.x; sm.op[slot][1] = bb.y; sm.op[slot][2] = bb.z;
        }
        n += __popc(msk);
        ptr = nxt;
    };
    if (v.occ) {
        // rows (y, z) of the ball's cell box over the lanes; each lane takes the occupied cells of
        // its row's x range from the occupancy words, one list at a time
        const int rows = nc[1] * nc[2], x0 = wrapi(c0[0], Gf);
        int guard = 0;
        for (int base = 0; base < rows; base += 32) {
            const int r = base + lane;
            bool live = r < rows;
            const uint32_t* row = nullptr;
            int rowcell = 0, piece = 0, a = x0, bnd = min(x0 + nc[0], Gf), wi = x0 >> 5;
            uint32_t bits = 0u;
            if (live) {
                const int y = wrapi(c0[1] + r % nc[1], Gf), z = wrapi(c0[2] + r / nc[1], Gf);
                row = v.occ + ((size_t)y + (size_t)Gf * z) * v.occ_w;
                rowcell = Gf * (y + Gf * z);
                bits = occ_masked(row[wi], a, bnd, wi);
            }
            int ptr = -1;
            while (true) {
                while (live && ptr < 0) {
                    if (bits) { ptr = v.head[rowcell + (wi << 5) + __ffs(bits) - 1]; bits &= bits - 1u; continue; }
                    if (wi < ((bnd - 1) >> 5)) { wi++; bits = occ_masked(row[wi], a, bnd, wi); continue; }
                    if (piece == 0 && x0 + nc[0] > Gf) {
                        piece = 1; a = 0; bnd = x0 + nc[0] - Gf; wi = 0;
                        bits = occ_masked(row[0], a, bnd, 0);
                        continue;
                    }
                    live = false;
                }
                if (!__any_sync(FULL, ptr >= 0)) break;
                step(ptr);
                if (n > ncap) { *n_out = n; return DEFER; }
                if (++guard > kMaxWalk) { if (lane == 0) set_err(v, E_WALK); return DEFER; }
            }
        }
    } else {
        const int nxy = nc[0] * nc[1];
        int guard = 0;
        for (int base = 0; base < nxy; base += 32) {
            const int w = base + lane;
            const bool col = w < nxy;
            const int colbase = col ? wrapc(c0[0] + w % nc[0], Gf) + Gf * wrapc(c0[1] + w / nc[0], Gf) : 0;
            for (int kz = 0; kz < nc[2]; kz++) {
                int ptr = col ? v.head[colbase + Gf * Gf * wrapc(c0[2] + kz, Gf)] : -1;
                while (__any_sync(FULL, ptr >= 0)) {
                    step(ptr);
                    if (n > ncap) { *n_out = n; return DEFER; }
                    if (++guard > kMaxWalk) { if (lane == 0) set_err(v, E_WALK); return DEFER; }
                }
            }
        }
    }
    *n_out = n;
    if (n > ncap) return DEFER;
    __syncwarp();
    if (n == 0) {                        // no bead moves: dU = 0 against the threshold
        const u4 w0 = draw(v.k0, v.k1, K_ACC, l, sweep, (uint32_t)j, 0);
        return 0.0 <= accept_threshold(v, w0) ? ACCEPT : REJECT;
    }
    // polarisation and amplitude A_w = A0 lam / sqrt(n) (Eq. 29)
    double p[3];
    warp_ball_point(v, K_VP, l, sweep, (uint32_t)j, true, lane, p);
    {
        const double r = sqr_t(norm2(p[0], p[1], p[2]));
        p[0] = dvd(p[0], r); p[1] = dvd(p[1], r); p[2] = dvd(p[2], r);
    }
    const double Aw = v.centring == 1 ? uniform_aw(v, lam) : dvd(mul(v.A0, lam), sqr_t((double)n));
    for (int k = lane; k < n; k += 32) {
        double d[3];
        for (int a = 0; a < 3; a++) d[a] = mi(sub(sm.op[k][a], b[a]), L, hL);
        const double d2 = norm2(d[0], d[1], d[2]);
        double dl[3];
        if (PREC == 0) wavelet_disp64(d, d2, lam, Aw, p, dl);
        else wavelet_disp32(d, lam, Aw, p, dl);
        int im[3] = {0, 0, 0};
        for (int a = 0; a < 3; a++) {
            const double u = add(sm.op[k][a], dl[a]);
            sm.nu[k][a] = u;
            sm.np[k][a] = wrap(u, L, &im[a]);
        }
        sm.dimg[k] = pack_img(im[0], im[1], im[2]);
        const int me = sm.ids[k];
        int r = 0;
        for (int t = 0; t < n; t++) r += sm.ids[t] < me;
        sm.sid[r] = me;
    }
    __syncwarp();
    // bonded partners outside the support must lie in the region
    bool bad = false;
    for (int k = lane; k < n; k += 32) {
        const int m = sm.ids[k];
        for (int e = 0; e < 2; e++) {
            const int q = e ? m + 1 : m - 1;
            if (q < 0 || q >= v.N || !(e ? v.bnext[m] : v.bnext[q]) || sorted_has(sm.sid, n, q)) continue;
            const Bead bq = v.bead[q];
            const int64_t cq[3] = {fine_cell(bq.x, v.invf, Gf), fine_cell(bq.y, v.invf, Gf), fine_cell(bq.z, v.invf, Gf)};
            for (int a = 0; a < 3; a++) if (!range_inside(cq[a], cq[a], rlo[a], rhi[a], Gf)) bad = true;
        }
    }
    if (__any_sync(FULL, bad)) return DEFER;
    int ncols = 0, nzmax = 0;
    partner_boxes(v, sm, n, lane, &ncols, &nzmax);
    // Metropolis threshold (Eq. 20): accept iff dU <= -kT ln(1 - u)
    const u4 w = draw(v.k0, v.k1, K_ACC, l, sweep, (uint32_t)j, 0);
    const double thr = accept_threshold(v, w);
    bool acc;
    int pe = 0;
    if (PREC == 1) {
        // binary32 energy change; decided in binary64 only within the rigorous error band
        float d32 = 0.0f, m32 = 0.0f;
        int T = 0;
        energy<true>(v, sm, n, lane, ncols, nzmax, nullptr, &d32, &m32, &T, &pe);
        const double band = 2.0 * (double)(80 + T + 6) * 5.9604644775390625e-08 * (double)m32 + 1e-9 * v.kT;
        if (isfinite(d32) && isfinite(m32) && fabs((double)d32 - thr) > band) {
            acc = (double)d32 <= thr;
            *du_out = (double)d32;
            if (v.audit) {
                double d64 = 0.0;
                int pe2 = 0;
                energy<false>(v, sm, n, lane, ncols, nzmax, &d64, nullptr, nullptr, nullptr, &pe2);
                if (lane == 0) audit_record(v, (double)d32, band, thr, d64, thr);
            }
        } else {
            double d64 = 0.0;
            int pe2 = 0;
            energy<false>(v, sm, n, lane, ncols, nzmax, &d64, nullptr, nullptr, nullptr, &pe2);
            acc = d64 <= thr;
            *du_out = d64;
            (*recheck_out)++;
            if (v.audit && lane == 0) audit_record(v, (double)d32, isfinite(m32) ? band : (double)INFINITY, thr, d64, thr);
        }
    } else {
        double d64 = 0.0;
        energy<false>(v, sm, n, lane, ncols, nzmax, &d64, nullptr, nullptr, nullptr, &pe);
        acc = d64 <= thr;
        *du_out = d64;
    }
    *pe_out += pe;
    if (!acc) return REJECT;
    // commit: positions, image counters, then cell-list moves (lane 0, in support order)
    for (int k = lane; k < n; k += 32) {
        const int m = sm.ids[k];
        put_bead(v.bead, v.bf, m, sm.np[k][0], sm.np[k][1], sm.np[k][2]);
        if (sm.dimg[k] != pack_img(0, 0, 0)) {
            int dd[3];
            unpack_img(sm.dimg[k], dd);
            v.img[3 * m] += dd[0]; v.img[3 * m + 1] += dd[1]; v.img[3 * m + 2] += dd[2];
        }
    }
    __syncwarp();
    if (lane == 0) {
        for (int k = 0; k < n; k++) {
            const int m = sm.ids[k];
            const int oc = cell_lin(v, sm.op[k][0], sm.op[k][1], sm.op[k][2]);
            const int ncl = cell_lin(v, sm.np[k][0], sm.np[k][1], sm.np[k][2]);
            if (oc == ncl) continue;
            relink(v, m, oc, ncl);
        }
    }
    __syncwarp();
    return ACCEPT;
}

}  // namespace wmcd

namespace wmcd {

// ======================================================================================
// Serial wavelet moves: a layer's deferred slots (schedule order), or every slot of a serial
// layer, taking effect one after another; a lone simulation's blocks evaluate them ahead of their
// turn. Supports of any size. The slot kernel drew every slot's parameters.
// ======================================================================================

// pairs a serial move keeps for its binary64 recheck (dynamic shared memory of the serial kernel
// in its mixed-precision 512-thread form, the one lone simulations use; other forms walk again)
constexpr int kSerialPairCap = 4096;
template <int PREC, int NT> __host__ __device__ constexpr int serial_pair_cap() { return (PREC == 1 && NT >= 512) ? kSerialPairCap : 0; }
// support members the gather keeps in shared memory (the 512-thread forms): written there by the
// few lanes that find a member, then to the global arrays in whole warps by the displacement
// pass; single-lane global stores from the gather held the block's memory pipe ~37k cycles a move
template <int NT> __host__ __device__ constexpr int serial_mem_cap() { return NT >= 512 ? kSerialMemCap : 0; }
// (member, occupied partner cell) entries of a move's pair search, walked one per thread
constexpr int kSerialEntCap = 4096;
template <int NT> __host__ __device__ constexpr int serial_ent_cap() { return NT >= 512 ? kSerialEntCap : 0; }
// ---- the window walk of speculative moves ------------------------------------------------------
// Hypothesis c = w(w+1)/2 + r of a window: its w-th move on the scale that the r rejections before
// it hand on. rec[c] holds the outcomes of the first nh hypotheses (at most 160); left = slots from
// the window's start. Follows the outcomes that hold in schedule order, up to the first move that is
// not known, has no hypothesis or may have read what an accepted move of the window wrote (balls
// about the centres, margin between them; pad is added between two balls that are both written). Run
// by one warp, alike in every warp that runs it: the path from a shuffle per step, then lane w holds
// the path's w-th move and all conflicts are tested side by side. Returns the moves that hold;
// *taken: hypothesis `mine` is one of them; *carry: the recycled scale before the window, and after.
template <class REC>
__device__ __forceinline__ int window_walk(const REC* rec, int nh, int left, float L, float hL, float margin, float pad,
                                           int mine, int lane, int* taken, double* carry) {
    const unsigned FULL = 0xffffffffu;
    int flags = 0;                               // 3 bits per hypothesis 32 j + lane: known (2 bits), accepted
    for (int j = 0; 32 * j < nh; j++)
        if (32 * j + lane < nh) flags |= (rec[32 * j + lane].known | (rec[32 * j + lane].acc ? 4 : 0)) << (3 * j);
    int w = 0, r = 0, myc = 0;
    bool has = *carry > 0.0;
    while (w < left) {
        const int c = w * (w + 1) / 2 + r;
        if (c >= nh) break;
        const int f = __shfl_sync(FULL, flags, c & 31) >> (3 * (c >> 5));
        if (!(f & 3)) break;
        if (lane == w) myc = c;
        if (f & 2) r = has ? r + 1 : 0;           // deferred: neither takes nor gives a scale
        else if (f & 4) { r = 0; has = false; }
        else { r++; has = true; }
        w++;
    }
    const REC& q = rec[myc];
    const float x = q.b[0], y = q.b[1], z = q.b[2], wr = q.wr;
    const bool acc = lane < w && q.known == 1 && q.acc;
    const float need0 = fmaxf(q.rr, acc ? wr + pad : -1e30f) + margin;
    bool hit = false;
    for (unsigned m = __ballot_sync(FULL, acc && q.n > 0); m; m &= m - 1u) {
        const int k = __ffs(m) - 1;
        const float dx = wrapn(x - __shfl_sync(FULL, x, k), L, hL), dy = wrapn(y - __shfl_sync(FULL, y, k), L, hL),
                    dz = wrapn(z - __shfl_sync(FULL, z, k), L, hL);
        const float need = fmaxf(need0 + __shfl_sync(FULL, wr, k), 0.0f);
        hit = hit || (lane > k && lane < w && dx * dx + dy * dy + dz * dz < need * need);
    }
    const unsigned cm = __ballot_sync(FULL, hit);
    const int steps = cm ? __ffs(cm) - 1 : w;
    *taken = __any_sync(FULL, lane < steps && myc == mine);
    const unsigned dm = __ballot_sync(FULL, lane < steps && q.known == 1);
    if (dm) {
        const int last = 31 - __clz(dm);
        const double lam = __shfl_sync(FULL, q.lam, last);
        *carry = __shfl_sync(FULL, (int)acc, last) ? 0.0 : lam;
    }
    return steps;
}

// A_w = a0l / sqrt(n) rounded to binary32, a0l = A0 lam: the same float as rounding the quotient
// dvd(a0l, s), s = sqr_t(n), without its division (about 560 cycles on this part). With rs the rounded
// reciprocal of s, a0l rs lies within 3 units of the last binary64 place of the rounded quotient, so
// the two round to the same float unless the product is that close to the midpoint of two floats.
__device__ __forceinline__ float amp32(double a0l, double s, double rs) {
    const double q = mul(a0l, rs);
    const int low = (int)(__double_as_longlong(q) & 0x1fffffffLL) - 0x10000000;
    if (low >= -4 && low <= 4) return (float)dvd(a0l, s);
    return (float)q;
}

// ---- one warp's move ---------------------------------------------------------------------------
// The arithmetic of a move that one warp runs on beads in shared memory, for k_serial_smem (the whole
// periodic box, differences by minimum image) and k_colour_staged (a region in coordinates relative
// to its origin, no images). A move executes this code once, so its length is its cost as much as its
// arithmetic (instruction fetch): pair terms are first screened in binary32 into a short list, and one
// copy of the pair code, run for the new and the old distance, serves the list.
constexpr int kWarpMem = 48;         // support members a warp's move holds (a queue's first warp: n_cap)
constexpr int kWarpCand = 192;       // its candidates: beads within reach of the move outside the support
struct Box {
    const double* px;                // binary64 positions, axis a of bead t at a stride + t
    const float *hi, *lo;            // binary32 pairs of the (relative) coordinates
    int stride, count;               // beads
    double L, hL;
    float Lf, hLf;
};
struct WarpScr {
    double* nw;                      // 3 per member: new position (wrapped)
    float *nh, *nl;                  // ... as binary32 pair
    int* item;                       // screened pair terms (64)
    int* img;                        // packed image change per member
    unsigned short *mid, *cand;      // support and candidates, ascending
};
__host__ __device__ constexpr int warp_scr_bytes(int mem) {
    return (mem * (3 * 8 + 6 * 4 + 4 + 2) + 64 * 4 + kWarpCand * 2 + 7) & ~7;
}
__device__ __forceinline__ WarpScr warp_scr(char* p, int mem) {
    WarpScr W;
    W.nw = (double*)p;
    W.nh = (float*)(W.nw + 3 * mem);
    W.nl = W.nh + 3 * mem;
    W.item = (int*)(W.nl + 3 * mem);
    W.img = W.item + 64;
    W.mid = (unsigned short*)(W.img + mem);
    W.cand = W.mid + mem;
    return W;
}
struct WarpRec {
    double lam, du;
    float b[3], rr, wr;
    int n, acc, known, pe, re;       // known: 0 support beyond the scratch, 1 decided, 2 deferred
};

// New positions of the n members (Eqs. 21, 23) about the centre whose axis `lane % 3` is ba: lane = 3
// member + axis, so ten members share a binary64 instruction. p, pf: polarisation; lam, lamf, Aw, af:
// scale and amplitude in both precisions (mixed precision reads only the binary32 ones); ilam: 1 / lam.
template <int PREC, bool PERIODIC>
__device__ __forceinline__ void move_disp(const Box& B, const WarpScr& W, int n, double ba, const double* p, const float* pf,
                                          double lam, double ilam, float lamf, double Aw, float af, int lane) {
    const unsigned FULL = 0xffffffffu;
    const int mk = lane / 3, ax = lane - 3 * mk, base = lane - ax;
    const int a1 = ax == 2 ? 0 : ax + 1, a2 = ax == 0 ? 2 : ax - 1;
#pragma unroll 1
    for (int k0 = 0; k0 < n; k0 += 10) {
        const int k = k0 + mk;
        const bool on = lane < 30 && k < n;
        const int e = ax * B.stride + W.mid[on ? k : 0];
        const double o = B.px[e];
        const double d = mi_u(sub(o, ba), B.L, B.hL, FULL);
        double dl;
        float dlf;
        if (PREC == 0) {
            const double x = __shfl_sync(FULL, d, base), y = __shfl_sync(FULL, d, base + 1), z = __shfl_sync(FULL, d, base + 2);
            const double rho = div_by(sqr_t(norm2(x, y, z)), lam, ilam), sc = div_by(mul(Aw, sub(1.0, rho)), lam, ilam);
            const double d1 = a1 == 0 ? x : a1 == 1 ? y : z, d2 = a2 == 0 ? x : a2 == 1 ? y : z;
            dl = mul(sc, sub(mul(p[a1], d2), mul(p[a2], d1)));
            dlf = (float)dl;
        } else {
            const float df = (float)d;
            const float x = __shfl_sync(FULL, df, base), y = __shfl_sync(FULL, df, base + 1), z = __shfl_sync(FULL, df, base + 2);
            const float q2 = addf(addf(mulf(x, x), mulf(y, y)), mulf(z, z));
            const float rho = dvdf(sqrtf_(q2), lamf), sc = dvdf(mulf(af, subf(1.0f, rho)), lamf);
            const float d1 = a1 == 0 ? x : a1 == 1 ? y : z, d2 = a2 == 0 ? x : a2 == 1 ? y : z;
            dlf = mulf(sc, subf(mulf(pf[a1], d2), mulf(pf[a2], d1)));
            dl = (double)dlf;
        }
        int im = 0;
        const double nx = wrap_u(add(o, dl), B.L, FULL, &im);
        // old (hi, lo) plus the displacement by a binary32 two-sum, renormalised
        const float oh = B.hi[e], s1 = oh + dlf, bb = s1 - oh;
        const float l1 = B.lo[e] + ((oh - (s1 - bb)) + (dlf - bb));
        float h2 = s1 + l1, l2 = l1 - (h2 - s1);
        if (PERIODIC && __any_sync(FULL, im != 0) && im != 0) {   // wrapped across a face: split the binary64 value
            h2 = (float)nx;
            l2 = (float)(nx - (double)h2);
        }
        const int i1 = __shfl_sync(FULL, im, base + 1), i2 = __shfl_sync(FULL, im, base + 2);
        if (on) {
            W.nw[3 * k + ax] = nx;
            W.nh[3 * k + ax] = h2;
            W.nl[3 * k + ax] = l2;
            if (ax == 0) W.img[k] = pack_img(im, i1, i2);
        }
    }
    __syncwarp();
}

// The pair terms of a move: bonds of members to beads outside (partner(k, e): the bead on side e of
// member k's bead, or -1), pairs inside the support (bonded(k1, k2)), candidates outside: nsrc of them
// from W.cand, or (all) every bead but the members. Pairs that are not bonded are left out beyond rs
// (outside) or rs + disp (inside): the distance of the hi parts of the old positions at which neither
// the old nor the new pair can interact, one member's displacement being disp at most.
// pairs(m, a, b, inner, wca, bond): lane < m holds a term: member a, and member (inner) or bead b.
// *bond2: largest squared distance of a bonded partner from the point c, hi parts. One member after
// another with the lanes over its partners: no index is divided, and the terms are compacted so that
// the pair code, which is much longer than the screen, usually runs once.
template <bool PERIODIC, class PARTNER, class BONDED, class MEMBER, class PAIRS>
__device__ __forceinline__ void for_terms(const Box& B, const WarpScr& W, int n, int nc, bool all, bool bonds, bool wca,
                                          float rs, float disp, const float c[3], float* bond2, int lane, PARTNER&& partner,
                                          BONDED&& bonded, MEMBER&& member, PAIRS&& pairs) {
    const unsigned FULL = 0xffffffffu;
    const int nsrc = wca ? (all ? B.count : nc) : 0, end = n + nsrc;
    const float out2 = rs * rs, in2 = (rs + disp) * (rs + disp);
    auto dist2 = [&](int t, float x, float y, float z) {
        float dx = B.hi[t] - x, dy = B.hi[B.stride + t] - y, dz = B.hi[2 * B.stride + t] - z;
        if (PERIODIC) { dx = wrapn(dx, B.Lf, B.hLf); dy = wrapn(dy, B.Lf, B.hLf); dz = wrapn(dz, B.Lf, B.hLf); }
        return dx * dx + dy * dy + dz * dz;
    };
    // k = -1: the bonds, u over 2 n sides; then member k against members k + 1.. and the candidates, u
    // from k + 1 over both
    int cnt = 0, k = bonds ? -1 : 0, u = bonds ? 0 : 1;
    float far2 = 0.0f;
#pragma unroll 1
    while (true) {
#pragma unroll 1
        while (cnt < 32 && k < n) {
            int it = -1;                          // a | b << 8 | inner, wca, bond << 24..26
            const int w = u + lane;
            u += 32;
            if (k < 0) {
                if (w < 2 * n) {
                    const int q = partner(w >> 1, w & 1);
                    if (q >= 0 && !member(q)) {
                        it = (w >> 1) | q << 8 | 4 << 24;
                        far2 = fmaxf(far2, dist2(q, c[0], c[1], c[2]));
                    }
                }
                if (u >= 2 * n) { k = 0; u = 1; }
            } else {
                if (w < end) {
                    const bool inner = w < n;
                    const int t = W.mid[k], q = inner ? (int)W.mid[w] : all ? w - n : (int)W.cand[w - n];
                    const float d2 = dist2(q, B.hi[t], B.hi[B.stride + t], B.hi[2 * B.stride + t]);
                    if (inner) {
                        const int f = 1 | (wca && d2 <= in2 ? 2 : 0) | (bonded(k, w) ? 4 : 0);
                        if (f > 1) it = k | w << 8 | f << 24;
                    } else if (d2 <= out2 && !(all && member(q))) {
                        it = k | q << 8 | 2 << 24;
                    }
                }
                if (u >= end) { k++; u = k + 1; }
            }
            const unsigned v = __ballot_sync(FULL, it >= 0);
            if (it >= 0) W.item[cnt + __popc(v & ((1u << lane) - 1u))] = it;
            cnt += __popc(v);
        }
        if (cnt == 0) break;
        __syncwarp();
        const int m = min(cnt, 32);
        const int it = W.item[lane], rest = W.item[32 + lane];
        __syncwarp();
        if (lane < cnt - m) W.item[lane] = rest;
        pairs(m, it & 0xff, (it >> 8) & 0xffff, (it >> 24) & 1, (it >> 25) & 1, (it >> 26) & 1);
        cnt -= m;
    }
    *bond2 = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(far2)));
}

// Energy change of a move in binary32 with the magnitude sum, the summation depth (one lane's terms)
// and the pairs outside the support that carry a term.
template <bool PERIODIC, class TERMS>
__device__ __forceinline__ void move_energy32(const Box& B, const WarpScr& W, const Pot32& P32, int n, int lane,
                                              TERMS&& terms, float* d32, float* mag, int* T_out, int* pe) {
    const unsigned FULL = 0xffffffffu;
    float a32 = 0.0f, m32 = 0.0f;
    int T = 0, cnt = 0;
    if (P32.kappa_on)
        for (int k = lane; k < n; k += 32) {
            const int t = W.mid[k];
            float r[2] = {0.0f, 0.0f};
            for (int a = 0; a < 3; a++) {
                const float x = dif32(W.nw[3 * k + a], B.hL, B.L, B.hLf), y = dif32(B.px[a * B.stride + t], B.hL, B.L, B.hLf);
                r[0] += x * x;
                r[1] += y * y;
            }
            const float un = 0.5f * P32.kappa * r[0], uo = 0.5f * P32.kappa * r[1];
            a32 += un - uo; m32 += un + uo; T += 2;
        }
    terms([&](int m, int a, int b, bool inner, bool wca, bool bond) {
        if (lane >= m) return;
        bool some = false;
        // the new distance, then the old one
#pragma unroll 1
        for (int old = 0; old < 2; old++) {
            const int ta = old ? (int)W.mid[a] : 3 * a, sa = old ? B.stride : 1;
            const int tb = inner ? (old ? (int)W.mid[b] : 3 * b) : b, sb = inner && !old ? 1 : B.stride;
            const float *ha = old ? B.hi : W.nh, *la = old ? B.lo : W.nl, *hb = inner && !old ? W.nh : B.hi, *lb = inner && !old ? W.nl : B.lo;
            float r2 = 0.0f;
#pragma unroll
            for (int x = 0; x < 3; x++) {
                // the hi difference is rounded once relative to the result and the lo parts add the
                // rest, so a component carries about one ulp; one across a face of the box (rare for
                // pairs in range) from the binary64 positions
                const float dh = ha[ta + x * sa] - hb[tb + x * sb];
                float c = dh + (la[ta + x * sa] - lb[tb + x * sb]);
                if (PERIODIC && fabsf(dh) > B.hLf) {
                    const double e = sub((old ? B.px : W.nw)[ta + x * sa], (inner && !old ? W.nw : B.px)[tb + x * sb]);
                    c = (float)(e > 0.0 ? sub(e, B.L) : add(e, B.L));
                }
                r2 += c * c;
            }
            float u, mg;
            if (wca && r2 < P32.rc2) {
                wca32(P32, r2, u, mg);
                a32 += old ? -u : u; m32 += mg; T += 1;
                some = true;
            }
            if (bond) {
                bond32(P32, r2, u, mg);
                a32 += old ? -u : u; m32 += mg; T += 1;
            }
        }
        cnt += some && !inner;
    });
    T = (int)__reduce_max_sync(FULL, (unsigned)T);
    *d32 = 0.0f; *mag = 0.0f; *pe = 0;
    if (T) {
        for (int o = 16; o > 0; o >>= 1) {
            a32 += __shfl_xor_sync(FULL, a32, o);
            m32 += __shfl_xor_sync(FULL, m32, o);
        }
        *d32 = __shfl_sync(FULL, a32, 0);
        *mag = __shfl_sync(FULL, m32, 0);
        *pe = (int)__reduce_add_sync(FULL, (unsigned)cnt);
    }
    *T_out = T;
}
// The same in binary64.
template <class TERMS>
__device__ __forceinline__ double move_energy64(const Box& B, const WarpScr& W, const Pot& P, int n, int lane, TERMS&& terms, int* pe) {
    double a64 = 0.0;
    int cnt = 0;
    if (P.kappa != 0.0)
        for (int k = lane; k < n; k += 32) {
            const int t = W.mid[k];
            a64 += U_ext(P, W.nw[3 * k], W.nw[3 * k + 1], W.nw[3 * k + 2]) - U_ext(P, B.px[t], B.px[B.stride + t], B.px[2 * B.stride + t]);
        }
    terms([&](int m, int a, int b, bool inner, bool wca, bool bond) {
        if (lane >= m) return;
        bool some = false;
#pragma unroll 1
        for (int old = 0; old < 2; old++) {
            const int ta = old ? (int)W.mid[a] : 3 * a, sa = old ? B.stride : 1;
            const int tb = inner ? (old ? (int)W.mid[b] : 3 * b) : b, sb = inner && !old ? 1 : B.stride;
            const double *xa = old ? B.px : W.nw, *xb = inner && !old ? W.nw : B.px;
            const double r2 = norm2(mi(xa[ta] - xb[tb], B.L, B.hL), mi(xa[ta + sa] - xb[tb + sb], B.L, B.hL),
                                    mi(xa[ta + 2 * sa] - xb[tb + 2 * sb], B.L, B.hL));
            double u = 0.0;
            if (wca && r2 < P.rc2) { u = U_wca(P, r2); some = true; }
            if (bond) u += U_bond(P, r2);
            a64 += old ? -u : u;
        }
        cnt += some && !inner;
    });
    *pe = (int)__reduce_add_sync(0xffffffffu, (unsigned)cnt);
    return __shfl_sync(0xffffffffu, warp_sum(a64), 0);
}
// Decision of a move with members: binary32 outside the rigorous error band (per term 80 ulp of its
// magnitude, plus the summation: one lane's terms and the butterfly), binary64 inside it, in binary64
// mode, or (audit) both. terms(f) runs f over the move's pair terms.
template <int PREC, bool PERIODIC, class TERMS>
__device__ __forceinline__ void move_decide(const SimView& v, const Box& B, const WarpScr& W, const Pot32& P32, int n, float kT9,
                                            double thr, float thr32, int lane, TERMS&& terms, WarpRec& rec) {
    bool need64 = PREC == 0;
    float d32 = 0.0f, mag = 0.0f, band = 0.0f;
    if (PREC == 1) {
        int T;
        move_energy32<PERIODIC>(B, W, P32, n, lane, terms, &d32, &mag, &T, &rec.pe);
        band = 2.0f * (float)(80 + T + 5 + 6) * 5.9604645e-08f * mag + kT9 + 2.4e-7f * fabsf(thr32);
        need64 = !(isfinite(d32) && isfinite(band) && fabsf(d32 - thr32) > band);
        rec.acc = d32 <= thr32;
        rec.du = (double)d32;
    }
    if (need64 || (PREC == 1 && v.audit)) {
        int pe2 = 0;
        const double d64 = move_energy64(B, W, v.pot, n, lane, terms, &pe2);
        if (PREC == 1 && v.audit && lane == 0) audit_record(v, (double)d32, (double)band, (double)thr32, d64, thr);
        if (need64) { rec.acc = d64 <= thr; rec.du = d64; rec.re = PREC; }
        if (PREC == 0) rec.pe = pe2;
    }
}

// support lookup of the speculative form: bead id -> index in the support (open addressing, at most
// half full), in place of the marks in the bead records, which belong to one move at a time
constexpr int kSerialHash = 2 * kSerialMemCap;
// MODE of k_serial: one block in turn; speculative serial phase; speculative queues (see below)
enum SerialMode { ONE_BLOCK = 0, SPEC_SERIAL = 1, SPEC_QUEUES = 2 };
template <int PREC, int NT, int MODE> __host__ __device__ constexpr size_t serial_dyn_bytes() {
    return (size_t)serial_mem_cap<NT>() * (4 * sizeof(double) + sizeof(int)) + (size_t)serial_pair_cap<PREC, NT>() * sizeof(int2) +
           (size_t)serial_ent_cap<NT>() * 2 * sizeof(int) + (NT >= 512 ? (size_t)serial_mem_cap<NT>() * (sizeof(float) + sizeof(int)) + 16 : 0) + (MODE ? (size_t)kSerialHash * (sizeof(int) + sizeof(unsigned short)) : 0);
}
// One thread's polls of a grid barrier before it gives up (about ten seconds: far beyond any move), and the barrier of
// the nb blocks of a speculative serial launch: the phase-th arrival of every block. False (for every
// thread of the block) when it gave up.
constexpr int kSpecPolls = 1 << 24;
__device__ bool spec_barrier(unsigned* bar, unsigned target, int* sh_ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        int polls = 0;
        unsigned seen;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
        } while (seen < target && ++polls < kSpecPolls);
        __threadfence();
        *sh_ok = seen >= target;
    }
    __syncthreads();
    return *sh_ok != 0;
}
// SPEC: the moves of the phase are run ahead of their turn by the blocks of a cooperative launch.
// A serial move depends on the moves before it only through the recycled scale (a rejected move
// hands its lambda on) and through beads that an accepted move shifted. Block c = w(w+1)/2 + r
// evaluates the w-th move of the window on the assumption that the r moves before it are rejected
// (so it runs the scale they hand on) and the one before those is accepted; every outcome of the
// window's first moves is thus some block's hypothesis. After a grid barrier every block walks the
// window in schedule order along the outcomes that hold, up to the first move whose reads an
// accepted move of the window may have touched; the blocks on that path commit (their beads, cells
// and lists are disjoint), and the next window starts after it. Decisions and positions are those
// of the moves run one after another. One block per SM: a move keeps a block's barriers and list
// walks waiting, never a unit of the SM, so the moves run side by side at no cost to each other.
// (Times: at the launch, in launch_serial.)
// SPEC_QUEUES: the same for the queues of a colour phase whose regions hold more beads than shared
// memory stages: `group` blocks per queue, each group's queues one after another; a move that leaves
// the region, holds more than n_cap beads or bonds to a bead outside it is deferred (known 2).
template <int PREC, int NT, int MODE>
__global__ void __launch_bounds__(NT, 1) k_serial(const SimView* __restrict__ vs, int ls, int colour, int group, int ns_above) {
    constexpr bool SPEC = MODE != ONE_BLOCK, QUEUES = MODE == SPEC_QUEUES;
    const int l = QUEUES ? layer_real(ls) : ls;
    SIM_EXIT_IF(l >= gv.nL || gv.precision != PREC || (((gv.smem_layers | gv.big_layers) >> l) & 1) ||
                (QUEUES && (!sched_on(gv, ls) || colour >= gv.K * gv.K * gv.K)))
    SIM_PROLOGUE
    if (l >= v.nL || v.precision != PREC || (((v.smem_layers | v.big_layers) >> l) & 1)) return;
    if (!QUEUES && threadIdx.x == 0 && blockIdx.x == 0) *v.cl_stale = 0;   // rebuilt just before this launch if it was stale
    const int M = v.counts[l];
    const int use_list = QUEUES || v.layer[l].G > 0;
    int count = QUEUES ? 0 : use_list ? *v.serial_count : M;
    // this block's hypothesis (w, r) and the blocks that take part; audited runs evaluate each move once
    const int cb = QUEUES ? (int)blockIdx.x % group : SPEC ? (int)blockIdx.x : 0;
    int hw = 0;
    while (SPEC && (hw + 1) * (hw + 2) / 2 <= cb) hw++;
    const int hr = cb - hw * (hw + 1) / 2;
    const int nb = !SPEC || v.audit ? 1 : QUEUES ? group : (int)min((long long)gridDim.x, (long long)count * (count + 1) / 2);
    if (SPEC && ((!QUEUES && count == 0) || cb >= nb)) return;
    unsigned* const bar = SPEC ? v.spec_bar + (QUEUES ? 2 * ((int)blockIdx.x / group) : 0) : nullptr;
    SpecRec* const recs = SPEC ? v.spec_rec + (QUEUES ? (int)blockIdx.x - cb : 0) : nullptr;
    if (SPEC && (QUEUES || cb > 0)) {
        // this block's own scratch for the arrays indexed by support member
        __syncthreads();
        if (threadIdx.x == 0) {
            char* p = v.spec_mem + (size_t)blockIdx.x * v.spec_stride;
            const size_t cap = (size_t)v.spec_cap;
            sv_.s_new = (double*)p;
            sv_.s_box = (int*)(p + 24 * cap);
            sv_.s_changed = (int*)(p + 48 * cap);
            sv_.s_img = (int*)(p + 60 * cap);
            sv_.s_pre = (int*)(p + 64 * cap);
        }
        __syncthreads();
    }
    __shared__ double sh_b[3], sh_p[3], sh_carry, sh_awx[2];
    // dynamic shared memory: support offsets (4 per member) and ids of the first members, then
    // the pairs within the WCA cutoff (old or new) found by the binary32 pass, for a binary64
    // pass that then visits only those (more than the capacity: the full walk again)
    extern __shared__ __align__(16) double sh_dyn[];
    // occupied cells of the ball found by the row pass, walked one per thread afterwards (a row
    // of a dense region holds tens of beads: one thread walking it is the search's longest chain)
    constexpr int kCellCap = NT >= 512 ? 4096 : 1;
    __shared__ int sh_cells[kCellCap];
    __shared__ int sh_ncell;
    double* const sm_d = sh_dyn;
    int2* const sh_pairs = (int2*)(sh_dyn + 4 * serial_mem_cap<NT>());
    int* const sm_ids = (int*)(sh_pairs + serial_pair_cap<PREC, NT>());
    int* const ent_k = sm_ids + serial_mem_cap<NT>();
    int* const ent_c = ent_k + serial_ent_cap<NT>();
    __shared__ int sh_nent;
    // beads of an accepted move that change fine cell: (bead, old cell, new cell), relinked by
    // one thread per old cell and then one per new cell (a cell's beads in list order)
    constexpr int kChCap = NT >= 512 ? 1024 : 1;
    __shared__ int sc_m[kChCap], sc_oc[kChCap], sc_nc[kChCap];
    __shared__ int sh_np;
    __shared__ double sh_red[NT / 32];
    __shared__ int sh_n, sh_nch, sh_acc, sh_c0[3], sh_nc[3], sh_need64;
    __shared__ float sh_a32[3];                   // binary32 energy change, band, threshold (audit)
    __shared__ float sh_f32[NT / 32], sh_m32[NT / 32];
    __shared__ int sh_T[NT / 32];
    __shared__ int sh_scan[33];
    __shared__ uint32_t sh_tag;
    // the members' boxes as a prefix of their rows, and (mixed precision) the last displacement
    // component; the others take the place of the support offsets once the displacements are formed
    int* const sm_pre = ent_c + serial_ent_cap<NT>();
    float* const sm_dz = (float*)(sm_pre + (NT >= 512 ? serial_mem_cap<NT>() + 4 : 0));
    int* const sh_hkey = (int*)(sm_dz + (NT >= 512 ? serial_mem_cap<NT>() : 0));
    __shared__ int sh_ncx;                        // most cells along x of a member's partner box
    unsigned short* const sh_hval = (unsigned short*)(sh_hkey + kSerialHash);
    __shared__ SpecRec sh_rec[SPEC ? kSpecMax : 1];
    __shared__ float sh_bond;                     // farthest bonded partner read, from the centre
    __shared__ int sh_ok, sh_mine, sh_steps;
    __shared__ double sh_du;
    unsigned phase = 0;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const LayerDev& Ly = v.layer[l];
    const double L = v.L, hL = v.halfL;
    const Pot& P = v.pot;
    // trace flags of a serial move: 4 deferred by the colouring, 8 by its second colouring too (a queue
    // of the second colouring: 4)
    const int dflag = QUEUES ? (ls >= kLevel2 ? 4 : 0) : use_list ? (v.layer[l].G2 > 0 ? 12 : 4) : 0;
    const int* list = QUEUES ? nullptr : v.serial_list;
    __shared__ int sh_defer, sh_rlo[3], sh_rhi[3];   // a queue's deferral and the fine cells of its region
    int def = 0;
    long long att = 0, acc_n = 0, bu = 0, pe = 0, rechecks = 0, moved_n = 0;
    const float hLf = (float)hL, Lf = (float)L;
    const bool kappa_on = P.kappa != 0.0, eps_on = P.eps != 0.0;
    __shared__ double sh_lam, sh_lam2;
    __shared__ float sh_bf[3], sh_rl2f;
    // the binary64 values the whole block needs for a move are formed once, by thread 0, and
    // shared: on this part each binary64 instruction of every warp would occupy the pipe
    const LayerDev Ls = sched_layer(v, QUEUES ? ls : l);
    const int Gq = QUEUES ? Ls.G : 1, Q = Gq / v.K, nq = QUEUES ? Q * Q * Q : 1;
    bool gave_up = false;
    for (int q = QUEUES ? (int)blockIdx.x / group : 0; q < nq && !gave_up; q += QUEUES ? (int)gridDim.x / group : 1) {
    int start = 0, cell = 0;
    if (QUEUES) {
        count = v.q_count[colour * nq + q];
        if (count == 0 || v.rcount[q] <= ns_above) continue;
        start = v.q_start[colour * nq + q];
        list = v.q_slots + start;
        const int c[3] = {v.K * (q % Q) + colour % v.K, v.K * ((q / Q) % Q) + (colour / v.K) % v.K, v.K * (q / (Q * Q)) + colour / (v.K * v.K)};
        cell = c[0] + Gq * (c[1] + Gq * c[2]);
        __syncthreads();
        if (tid < 3) {
            const int e = tid == 0 ? c[0] : tid == 1 ? c[1] : c[2];
            sh_rlo[tid] = (int)ceildiv((2 * (int64_t)e - (v.K - 1)) * v.Gf, 2 * (int64_t)Gq);
            sh_rhi[tid] = (int)floordiv((2 * (int64_t)e + 2 + (v.K - 1)) * v.Gf, 2 * (int64_t)Gq) - 1;
        }
    }
    if (tid == 0) sh_carry = QUEUES ? v.carry_q[Ls.carry_off + cell] : v.carry_serial[l];
    __syncthreads();
    for (int t = 0; t < count;) {
        const int tw = t + hw;                    // the move this block evaluates
        const bool live = tw < count;
        const int j = !live ? 0 : use_list ? list[tw] : tw;
        int known = live;                         // 2: deferred
        int n = 0, pe_move = 0, re_move = 0;
        double lam = 0.0;
        auto evaluate = [&]() {
        const int i = v.slot_bead[j];
        if (tid < 3) {
            // the carried scale, or that of the slot the run of rejections started with; one axis a thread
            const int jl = SPEC ? (use_list ? list[tw - hr] : tw - hr) : j, a = tid;
            const double lam = (!SPEC || hr == hw) && sh_carry > 0.0 ? sh_carry : v.slot_lam[jl];
            const double ri = (&v.bead[i].x)[a], Va = v.slot_V[3 * j + a];
            const double ba = v.centring == 1 ? Va : wrap(add(ri, mul(lam, Va)), L, nullptr);
            sh_b[a] = ba;
            sh_p[a] = v.slot_p[3 * j + a];
            sh_bf[a] = (float)ba;
            const double eps = 1e-9;
            const int t0 = (int)floor(mul(sub(ba, lam + eps), v.invf));
            const int t1 = (int)floor(mul(add(ba, lam + eps), v.invf));
            sh_c0[a] = t0;
            sh_nc[a] = min(t1 - t0 + 1, v.Gf);
            bool in = true;
            if (QUEUES) {
                // the influence ball must lie in fine cells wholly inside the queue's region
                const double R = add(add(lam, rule_disp(v, lam)), v.r_reach);
                const int64_t r0 = (int64_t)floor(mul(sub(ba, R), v.invf));
                const int64_t r1 = (int64_t)floor(mul(add(ba, R), v.invf));
                in = range_inside(r0, r1, sh_rlo[a], sh_rhi[a], v.Gf);
            }
            in = __all_sync(7u, in);
            if (a == 0) {
                sh_defer = !in;
                sh_lam = lam;
                sh_lam2 = mul(lam, lam);
                const float rlf = (float)lam + (float)(8.0 * L * 5.9604644775390625e-8 + 1e-6);
                sh_rl2f = rlf * rlf * (1.0f + 9.5367431640625e-7f);
                sh_n = 0;
                sh_nch = 0;
                sh_np = 0;
                sh_ncell = 0;
                sh_nent = 0;
                sh_ncx = 1;
                sh_bond = 0.0f;
                if (!QUEUES && cb == 0) {
                    uint32_t tag = *v.serial_tag + 1u;
                    if (tag == 0u) tag = 1u;
                    *v.serial_tag = tag;
                    sh_tag = tag;
                }
            }
        }
        __syncthreads();
        lam = sh_lam;
        if (QUEUES && sh_defer) { known = 2; return; }
        const double lam2 = sh_lam2;
        const double b[3] = {sh_b[0], sh_b[1], sh_b[2]};
        // gather the support
        // binary32 screen on the shadow (margin 8 L 2^-24 + 1e-6 on the distance covers the rounding
        // of the shadow, of b and of the difference), then the binary64 test
        const float bxf = sh_bf[0], byf = sh_bf[1], bzf = sh_bf[2];
        const float rl2f = sh_rl2f;
        auto wrapg = [&](float f) { return fabsf(f) > hLf ? f - copysignf(Lf, f) : f; };
        auto screened = [&](const BeadF& f) {
            const float sx = wrapg(f.hx - bxf), sy = wrapg(f.hy - byf), sz = wrapg(f.hz - bzf);
            return sx * sx + sy * sy + sz * sz <= rl2f;
        };
        auto consider_exact = [&](int m, const Bead& bb) {
            double d0 = mi(sub(bb.x, b[0]), L, hL), d1 = mi(sub(bb.y, b[1]), L, hL), d2c = mi(sub(bb.z, b[2]), L, hL);
            double d2 = norm2(d0, d1, d2c);
            if (d2 < lam2) {
                int idx = atomicAdd(&sh_n, 1);
                int* ids = v.s_ids;
                double* dd = v.s_d;
                if (idx < serial_mem_cap<NT>()) { ids = sm_ids; dd = sm_d; }
                else if (SPEC && (QUEUES || cb > 0)) return;   // too large for this block's scratch: only counted
                ids[idx] = m;
                dd[4 * idx] = d0; dd[4 * idx + 1] = d1; dd[4 * idx + 2] = d2c; dd[4 * idx + 3] = d2;
            }
        };
        // four independent loads in flight per thread (the shadows of four beads, or the heads
        // of four cells) before any is used
        if ((int64_t)sh_nc[0] * sh_nc[1] * sh_nc[2] > v.N) {
            for (int64_t m0 = tid; m0 < v.N; m0 += 4 * (int64_t)NT) {
                BeadF f[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int64_t m = m0 + (int64_t)u * NT;
                    if (m < v.N) f[u] = v.bf[m];
                }
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int64_t m = m0 + (int64_t)u * NT;
                    if (m < v.N && screened(f[u])) consider_exact((int)m, v.bead[m]);
                }
            }
        } else if (v.occ) {
            // rows (y, z) of the ball's cell box over the threads; each row's x range read as
            // occupancy words, and only the lists of occupied cells walked
            const int c0[3] = {sh_c0[0], sh_c0[1], sh_c0[2]}, nc[3] = {sh_nc[0], sh_nc[1], sh_nc[2]};
            const int Gf = v.Gf, rows = nc[1] * nc[2];
            const int x0 = wrapi(c0[0], Gf);
            for (int r = tid; r < rows; r += NT) {
                const int y = wrapi(c0[1] + r % nc[1], Gf), z = wrapi(c0[2] + r / nc[1], Gf);
                const uint32_t* row = v.occ + ((size_t)y + (size_t)Gf * z) * v.occ_w;
                const int rowcell = Gf * (y + Gf * z);
                // the x range [x0, x0 + nc[0]) as at most two pieces inside [0, Gf)
                for (int piece = 0; piece < 2; piece++) {
                    const int a = piece == 0 ? x0 : 0;
                    const int b = piece == 0 ? min(x0 + nc[0], Gf) : x0 + nc[0] - Gf;
                    for (int wi = a >> 5; a < b && wi <= (b - 1) >> 5; wi++) {
                        uint32_t bits = row[wi];
                        const int lo = max(a - (wi << 5), 0), hi = min(b - (wi << 5), 32);
                        bits &= (hi >= 32 ? 0xffffffffu : ((1u << hi) - 1u)) & ~((1u << lo) - 1u);
                        for (; bits; bits &= bits - 1u) {
                            const int cell = rowcell + (wi << 5) + __ffs(bits) - 1;
                            const int slot = NT >= 512 ? atomicAdd(&sh_ncell, 1) : kCellCap;
                            if (slot < kCellCap) { sh_cells[slot] = cell; continue; }
                            int guard = 0;             // list full: walked here
                            for (int q = v.head[cell]; q >= 0;) {
                                const Bead bb = v.bead[q];
                                if (screened(v.bf[q])) consider_exact(q, bb);
                                q = bb.next;
                                if (++guard > kMaxWalk) { set_err(v, E_WALK); break; }
                            }
                        }
                    }
                }
            }
            if (NT >= 512) {
                __syncthreads();
                const int nlist = min(sh_ncell, kCellCap);
                // (the next cell's head is loaded before the current cell is walked)
                int hn = tid < nlist ? v.head[sh_cells[tid]] : -1;
                for (int i = tid; i < nlist; i += NT) {
                    int guard = 0;
                    const int h = hn;
                    if (i + NT < nlist) hn = v.head[sh_cells[i + NT]];
                    for (int q = h; q >= 0;) {
                        const Bead bb = v.bead[q];
                        if (screened(v.bf[q])) consider_exact(q, bb);
                        q = bb.next;
                        if (++guard > kMaxWalk) { set_err(v, E_WALK); break; }
                    }
                }
            }
        } else {
            const int c0[3] = {sh_c0[0], sh_c0[1], sh_c0[2]}, nc[3] = {sh_nc[0], sh_nc[1], sh_nc[2]};
            const int ncell = nc[0] * nc[1] * nc[2];
            for (int k0 = tid; k0 < ncell; k0 += 4 * NT) {
                int hd[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int k = k0 + u * NT;
                    hd[u] = -1;
                    if (k < ncell) {
                        const int kx = k % nc[0], ky = (k / nc[0]) % nc[1], kz = k / (nc[0] * nc[1]);
                        hd[u] = v.head[wrapi(c0[0] + kx, v.Gf) + v.Gf * (wrapi(c0[1] + ky, v.Gf) + v.Gf * wrapi(c0[2] + kz, v.Gf))];
                    }
                }
                for (int u = 0; u < 4; u++) {
                    int guard = 0;
                    for (int q = hd[u]; q >= 0;) {
                        const Bead bb = v.bead[q];
                        if (screened(v.bf[q])) consider_exact(q, bb);
                        q = bb.next;
                        if (++guard > kMaxWalk) { set_err(v, E_WALK); break; }
                    }
                }
            }
        }
        __syncthreads();
        n = sh_n;
        if (QUEUES && n > sched_ncap(v, ls)) { known = 2; return; }
        if (n == 0) {      // nothing inside: no motion, dU = 0 against the threshold
            if (tid == 0) { sh_acc = 0.0 <= v.slot_thr[j]; sh_du = 0.0; }
            __syncthreads();
            return;
        }
        // a support beyond the shared arrays runs through the simulation's own, in its turn only
        const bool small = n <= serial_mem_cap<NT>();
        if (SPEC && (QUEUES || cb > 0) && !small) { known = 0; return; }
        double* const mem_d = small ? sm_d : v.s_d;
        int* const mem_ids = small ? sm_ids : v.s_ids;
        const uint32_t tag = sh_tag;
        uint32_t hmask = 63u;                     // support lookup: by hash, or (large) by mark
        if (SPEC && small) {
            while (hmask + 1u < 2u * (uint32_t)n) hmask = 2u * hmask + 1u;
            for (uint32_t h = tid; h <= hmask; h += NT) sh_hkey[h] = -1;
        }
        auto find = [&](int q, const Bead& bq) -> int {
            if (SPEC && small) {
                for (uint32_t h = (uint32_t)q * 2654435761u >> 16 & hmask;; h = (h + 1u) & hmask) {
                    const int k = sh_hkey[h];
                    if (k == q) return sh_hval[h];
                    if (k < 0) return -1;
                }
            }
            return bq.mark == tag ? v.s_slot[q] : -1;
        };
        // A_w (Eq. 29) and the partner-box reach, formed once by thread 0: on this part every
        // binary64 instruction of a warp holds the unit for tens of cycles, so the division and
        // square root are not repeated in every warp that holds a member
        if (tid == 0) {
            const double aw = v.centring == 1 ? uniform_aw(v, lam) : dvd(mul(v.A0, lam), sqr_t((double)n));
            sh_awx[0] = aw;
            sh_awx[1] = add(v.rc, mul(0.25, aw)) + 1e-9;
        }
        __syncthreads();
        const double Aw = sh_awx[0];
        const double p[3] = {sh_p[0], sh_p[1], sh_p[2]};
        for (int k = tid; k < n; k += NT) {
            const bool in_sm = k < serial_mem_cap<NT>();
            const double* dd = in_sm ? sm_d : v.s_d;
            const int m = in_sm ? sm_ids[k] : v.s_ids[k];
            if (!small && in_sm) v.s_ids[k] = m;  // the later passes read the global arrays
            if (SPEC && small) {
                uint32_t h = (uint32_t)m * 2654435761u >> 16 & hmask;
                while (atomicCAS(&sh_hkey[h], -1, m) != -1) h = (h + 1u) & hmask;
                sh_hval[h] = (unsigned short)k;
            } else {
                v.bead[m].mark = tag;
                v.s_slot[m] = k;
            }
            double d[3] = {dd[4 * k], dd[4 * k + 1], dd[4 * k + 2]}, dl[3];
            if (PREC == 0) wavelet_disp64(d, dd[4 * k + 3], lam, Aw, p, dl);
            else wavelet_disp32(d, lam, Aw, p, dl);
            const double o[3] = {v.bead[m].x, v.bead[m].y, v.bead[m].z};
            int im[3] = {0, 0, 0};
            const unsigned am = __activemask();
            double nx[3] = {add(o[0], dl[0]), add(o[1], dl[1]), add(o[2], dl[2])};
            wrap3_u(nx, L, am, im);
            for (int a = 0; a < 3; a++) v.s_new[3 * k + a] = nx[a];
            v.s_img[k] = pack_img(im[0], im[1], im[2]);
            if (PREC == 1 && small) {
                // what the pair terms read of a member: shadow and displacement, in place of its offset
                const BeadF f = v.bf[m];
                float* const e = (float*)&sm_d[4 * k];
                e[0] = f.hx; e[1] = f.hy; e[2] = f.hz; e[3] = f.lx; e[4] = f.ly; e[5] = f.lz;
                e[6] = (float)dl[0]; e[7] = (float)dl[1];
                sm_dz[k] = (float)dl[2];
            } else {
                for (int a = 0; a < 3; a++) mem_d[4 * k + a] = dl[a];
            }
            // partner box: cells within reach of the old and the new position
            int cnt = 0;
            if (eps_on) {
                const double ext = sh_awx[1];
                double lo[3], hi[3];
                for (int a = 0; a < 3; a++) {
                    const double u = add(o[a], dl[a]);
                    lo[a] = sub(fmin(o[a], u), ext);
                    hi[a] = add(fmax(o[a], u), ext);
                }
                int c0[3], nc[3];
                cell_box(v, lo, hi, c0, nc);
                for (int a = 0; a < 3; a++) { v.s_box[6 * k + a] = c0[a]; v.s_box[6 * k + 3 + a] = nc[a]; }
                cnt = v.occ ? nc[1] * nc[2] : nc[0] * nc[1] * nc[2];   // rows (y, z), or cells
                if (nc[0] > 1) atomicMax(&sh_ncx, nc[0]);
            }
            (small && NT >= 512 ? sm_pre : v.s_pre)[k] = cnt;
        }
        __syncthreads();
        int* const pre = small && NT >= 512 ? sm_pre : v.s_pre;
        // shadow and displacement of member k (bead m)
        auto member_f = [&](int k, int m, float* h, float* lo, float* dl) {
            if (PREC == 1 && small) {
                const float* e = (const float*)&sm_d[4 * k];
                for (int a = 0; a < 3; a++) { h[a] = e[a]; lo[a] = e[3 + a]; }
                dl[0] = e[6]; dl[1] = e[7]; dl[2] = sm_dz[k];
            } else {
                const BeadF f = v.bf[m];
                h[0] = f.hx; h[1] = f.hy; h[2] = f.hz; lo[0] = f.lx; lo[1] = f.ly; lo[2] = f.lz;
                for (int a = 0; a < 3; a++) dl[a] = (float)mem_d[4 * k + a];
            }
        };
        auto member_d = [&](int k, float* dl) {
            if (PREC == 1 && small) {
                const float* e = (const float*)&sm_d[4 * k];
                dl[0] = e[6]; dl[1] = e[7]; dl[2] = sm_dz[k];
            } else {
                for (int a = 0; a < 3; a++) dl[a] = (float)mem_d[4 * k + a];
            }
        };
        // energy change: bonds and the external well per member; pair terms by one thread per
        // (member, fine cell of its partner box) item, so a small support still spreads its list
        // walks over the block. Mixed precision: a binary32 pass first (each difference of
        // binary64 positions rounded once, the new one formed from the old one and the binary32
        // displacements), deciding outside the rigorous error band; the binary64 pass decides
        // inside it and in binary64 mode.
        const double ext = sh_awx[1];
        const double thr = v.slot_thr[j];
        // old-position difference a - b, minimum image, rounded once to binary32
        auto d32 = [&](double a, double b) {
            const double e = sub(a, b);
            float f = (float)e;
            if (fabsf(f) > hLf) f = (float)(e > 0.0 ? sub(e, L) : add(e, L));
            return f;
        };
        auto wrapf = [&](float f) { return fabsf(f) > hLf ? f - copysignf(Lf, f) : f; };
        // the same difference from the binary32 shadows (hi, lo): no binary64 arithmetic unless
        // the pair straddles a face, where it is wrapped in binary64
        auto dsh = [&](float ha, float la, float hb, float lb, double a, double b) {
            const float dh = ha - hb;
            if (fabsf(dh) <= hLf) return dh + (la - lb);
            return d32(a, b);
        };
        // farthest bonded partner read (and, of a queue's move, whether one lies outside the region)
        if (SPEC) {
            for (int e2 = tid; e2 < 2 * n; e2 += NT) {
                const int m = mem_ids[e2 >> 1], q = e2 & 1 ? m + 1 : m - 1;
                if (q < 0 || q >= v.N || !(e2 & 1 ? v.bnext[m] : v.bnext[q])) continue;
                const BeadF f = v.bf[q];
                const float sx = wrapg(f.hx - bxf), sy = wrapg(f.hy - byf), sz = wrapg(f.hz - bzf);
                atomicMax((int*)&sh_bond, __float_as_int(sqrtf(sx * sx + sy * sy + sz * sz)));
                if (QUEUES) {
                    // bonded partners outside the support must lie in the region
                    const Bead bq = v.bead[q];
                    if (find(q, bq) >= 0) continue;
                    const int cq[3] = {fine_cell32(v, f.hx, bq.x), fine_cell32(v, f.hy, bq.y), fine_cell32(v, f.hz, bq.z)};
                    for (int a = 0; a < 3; a++)
                        if (!range_inside(cq[a], cq[a], sh_rlo[a], sh_rhi[a], v.Gf)) sh_defer = 1;
                }
            }
            if (QUEUES) {
                __syncthreads();
                if (sh_defer) { known = 2; return; }
            }
        }
        int W = 0;
        if (eps_on) {
            // exclusive prefix of the box sizes, NT members per pass
            for (int base = 0; base < n; base += NT) {
                const int k = base + tid;
                const int x = k < n ? pre[k] : 0;
                int total;
                const int px = W + block_excl_scan<NT / 32>(x, sh_scan, &total);
                if (k < n) pre[k] = px;
                W += total;
                if (base + NT < n) __syncthreads();   // sh_scan is rewritten by the next pass
            }
            if (tid == 0) pre[n] = W;
            __syncthreads();
        }
        // each thread takes a contiguous run of items, with one search for its first member and
        // member data reloaded only when the run crosses to the next member
        auto run_items = [&](int w0, int w1, auto&& item) {
            const int t0 = w0 + (int)((int64_t)tid * (w1 - w0) / NT), t1 = w0 + (int)((int64_t)(tid + 1) * (w1 - w0) / NT);
            if (t0 >= t1) return;
            int lo_k = 0, hi_k = n - 1;                 // last member with pre <= t0
            while (lo_k < hi_k) {
                const int mid = (lo_k + hi_k + 1) >> 1;
                if (pre[mid] <= t0) lo_k = mid; else hi_k = mid - 1;
            }
            int kn = lo_k, kn_start = pre[kn], kn_end = pre[kn + 1];
            int c0n[3] = {v.s_box[6 * kn], v.s_box[6 * kn + 1], v.s_box[6 * kn + 2]};
            int ncn[3] = {v.s_box[6 * kn + 3], v.s_box[6 * kn + 4], v.s_box[6 * kn + 5]};
            auto advance = [&](int t) {
                while (t >= kn_end) {
                    kn++;
                    kn_start = kn_end;
                    kn_end = pre[kn + 1];
                    for (int a = 0; a < 3; a++) { c0n[a] = v.s_box[6 * kn + a]; ncn[a] = v.s_box[6 * kn + 3 + a]; }
                }
            };
            item(t0, t1, advance, kn, kn_start, c0n, ncn);
        };
        auto walk = [&](auto&& visit, int h, int k, int m) {
            int guard = 0;
            for (int q = h; q >= 0;) {
                const Bead bq = v.bead[q];
                const int nx = bq.next;
                if (q != m) visit(k, m, q, bq);
                q = nx;
                if (++guard > kMaxWalk) { set_err(v, E_WALK); break; }
            }
        };
        // with occupancy bits an item is a row (y, z) of a member's partner box, whose x range is
        // read as occupancy words: cellfn(k, m, cell) for each occupied cell
        auto for_cells = [&](int w0, int w1, auto&& cellfn) {
            run_items(w0, w1, [&](int t0, int t1, auto& advance, int& kn, int& kn_start, int* c0n, int* ncn) {
                const int Gf = v.Gf;
                for (int t = t0; t < t1; t++) {
                    advance(t);
                    const int r = t - kn_start, m = mem_ids[kn];
                    const int y = wrapi(c0n[1] + r % ncn[1], Gf), z = wrapi(c0n[2] + r / ncn[1], Gf);
                    const uint32_t* row = v.occ + ((size_t)y + (size_t)Gf * z) * v.occ_w;
                    const int rowcell = Gf * (y + Gf * z), x0 = wrapi(c0n[0], Gf);
                    // the x range [x0, x0 + nc) as at most two pieces inside [0, Gf)
                    for (int piece = 0; piece < 2; piece++) {
                        const int xa = piece == 0 ? x0 : 0;
                        const int xb = piece == 0 ? min(x0 + ncn[0], Gf) : x0 + ncn[0] - Gf;
                        for (int wi = xa >> 5; xa < xb && wi <= (xb - 1) >> 5; wi++)
                            for (uint32_t bits = occ_masked(row[wi], xa, xb, wi); bits; bits &= bits - 1u)
                                cellfn(kn, m, rowcell + (wi << 5) + __ffs(bits) - 1);
                    }
                }
            });
        };
        // every (member, bead) pair of the partner boxes: visit(k, m, q, bead q)
        auto for_pairs = [&](auto&& visit) {
            if (v.occ && serial_ent_cap<NT>() > 0) {
                // the (member, occupied cell) entries of a range of rows listed, then walked one per thread
                // (a run of items in a dense region walked by one thread was the pass's longest chain), the
                // head of a thread's next entry loaded ahead; ranges of as many rows as fill the list with
                // half of their cells occupied (a fuller one is walked row by row)
                const int B = max(NT, 2 * serial_ent_cap<NT>() / sh_ncx);
                for (int w0 = 0; w0 < W; w0 += B) {
                    const int w1 = min(W, w0 + B);
                    if (w0 > 0) {
                        __syncthreads();
                        if (tid == 0) sh_nent = 0;
                        __syncthreads();
                    }
                    for_cells(w0, w1, [&](int k, int m, int cell) {
                        const int i = atomicAdd(&sh_nent, 1);
                        if (i < serial_ent_cap<NT>()) { ent_k[i] = k; ent_c[i] = cell; }
                    });
                    __syncthreads();
                    const int nent = sh_nent;
                    if (nent > serial_ent_cap<NT>()) {
                        for_cells(w0, w1, [&](int k, int m, int cell) { walk(visit, v.head[cell], k, m); });
                        continue;
                    }
                    int hn = tid < nent ? v.head[ent_c[tid]] : -1;
                    for (int i = tid; i < nent; i += NT) {
                        const int k = ent_k[i], h = hn;
                        if (i + NT < nent) hn = v.head[ent_c[i + NT]];
                        walk(visit, h, k, mem_ids[k]);
                    }
                }
                __syncthreads();
                if (tid == 0) sh_nent = 0;            // for another pass over the pairs
                return;
            }
            if (v.occ) {
                for_cells(0, W, [&](int k, int m, int cell) { walk(visit, v.head[cell], k, m); });
                return;
            }
            // an item is a cell; the head of the next item's cell is loaded before the current
            // cell is walked
            run_items(0, W, [&](int t0, int t1, auto& advance, int& kn, int& kn_start, int* c0n, int* ncn) {
                advance(t0);
                int h = v.head[box_cell(v, c0n, ncn, t0 - kn_start)];
                int cur_k = kn;
                for (int t = t0; t < t1; t++) {
                    int hn = -1, nk = cur_k;
                    if (t + 1 < t1) { advance(t + 1); hn = v.head[box_cell(v, c0n, ncn, t + 1 - kn_start)]; nk = kn; }
                    walk(visit, h, cur_k, mem_ids[cur_k]);
                    h = hn;
                    cur_k = nk;
                }
            });
        };
        bool need64 = PREC == 0;
        if (PREC == 1) {
            const Pot32 P32 = pot32(P);
            float a32 = 0.0f, m32 = 0.0f;
            int T = 0;
            for (int k = tid; k < n; k += NT) {
                const int m = mem_ids[k];
                const Bead bm = v.bead[m];
                const double o[3] = {bm.x, bm.y, bm.z};
                float dlm[3], mh[3], ml[3];
                member_f(k, m, mh, ml, dlm);
                if (kappa_on) {
                    float ro = 0.0f, rn = 0.0f;
                    for (int a = 0; a < 3; a++) {
                        const float c = d32(o[a], hL);
                        ro += c * c;
                        const float cn = wrapf(c + dlm[a]);
                        rn += cn * cn;
                    }
                    const float un = 0.5f * P32.kappa * rn, uo = 0.5f * P32.kappa * ro;
                    a32 += un - uo; m32 += un + uo; T += 2;
                }
                for (int e = 0; e < 2; e++) {
                    const int q = e ? m + 1 : m - 1;
                    if (q < 0 || q >= v.N || !(e ? v.bnext[m] : v.bnext[q])) continue;
                    const Bead bq = v.bead[q];
                    float dlq[3] = {0.0f, 0.0f, 0.0f};
                    const int sq = find(q, bq);
                    if (sq >= 0) {
                        if (q < m) continue;
                        member_d(sq, dlq);
                    }
                    const double qo[3] = {bq.x, bq.y, bq.z};
                    const BeadF fq = v.bf[q];
                    const float qh[3] = {fq.hx, fq.hy, fq.hz}, ql[3] = {fq.lx, fq.ly, fq.lz};
                    float ro = 0.0f, rn = 0.0f;
                    for (int a = 0; a < 3; a++) {
                        const float c = dsh(mh[a], ml[a], qh[a], ql[a], o[a], qo[a]);
                        ro += c * c;
                        const float cn = wrapf(c + dlm[a] - dlq[a]);
                        rn += cn * cn;
                    }
                    float un, mn, uo, mo;
                    bond32(P32, rn, un, mn);
                    bond32(P32, ro, uo, mo);
                    a32 += un - uo; m32 += mn + mo; T += 2;
                }
            }
            if (eps_on) {
                const float rc2p = P32.rc2 * 1.0001f;
                float dlm[3], mh[3], ml[3];
                for_pairs([&](int k, int m, int q, const Bead& bq) {
                    const BeadF fq = v.bf[q];
                    const int sq = find(q, bq);
                    const bool member = sq >= 0;
                    if (member && q < m) return;
                    member_f(k, m, mh, ml, dlm);
                    float dlq[3] = {0.0f, 0.0f, 0.0f};
                    if (member) member_d(sq, dlq);
                    const float qh[3] = {fq.hx, fq.hy, fq.hz}, ql[3] = {fq.lx, fq.ly, fq.lz};
                    float ro = 0.0f, rn = 0.0f;
                    for (int a = 0; a < 3; a++) {
                        const float dh = mh[a] - qh[a];
                        // across a face: wrapped in binary64 from the positions
                        const float c = fabsf(dh) <= hLf ? dh + (ml[a] - ql[a]) : d32((&v.bead[m].x)[a], (&bq.x)[a]);
                        ro += c * c;
                        const float cn = wrapf(c + dlm[a] - dlq[a]);
                        rn += cn * cn;
                    }
                    float un, mn, uo, mo;
                    wca32(P32, rn, un, mn);
                    wca32(P32, ro, uo, mo);
                    if (un != 0.0f || uo != 0.0f || mn != 0.0f || mo != 0.0f) {
                        a32 += un - uo; m32 += mn + mo; T += 2;
                        if (!member) pe_move++;
                    }
                    // within the cutoff with a margin far above the binary32 error of r^2
                    if (rn < rc2p || ro < rc2p) {
                        const int ip = atomicAdd(&sh_np, 1);
                        if (ip < serial_pair_cap<PREC, NT>()) sh_pairs[ip] = make_int2(k, q);
                    }
                });
            }
            for (int sft = 16; sft > 0; sft >>= 1) {
                a32 += __shfl_xor_sync(0xffffffffu, a32, sft);
                m32 += __shfl_xor_sync(0xffffffffu, m32, sft);
                T = max(T, __shfl_xor_sync(0xffffffffu, T, sft));
            }
            if (lane == 0) { sh_f32[wid] = a32; sh_m32[wid] = m32; sh_T[wid] = T; }
            __syncthreads();
            if (tid == 0) {
                float du = 0.0f, mm = 0.0f;
                int tt = 0;
                for (int w = 0; w < NT / 32; w++) { du += sh_f32[w]; mm += sh_m32[w]; tt = max(tt, sh_T[w]); }
                tt += 5 + NT / 32;     // summation depth: one thread's terms, the butterfly, the warp totals
                const float thr32 = (float)thr;
                const float band = 2.0f * (float)(80 + tt + 6) * 5.9604645e-08f * mm + 1e-9f * (float)v.kT +
                                   2.4e-7f * fabsf(thr32);
                sh_a32[0] = du; sh_a32[1] = band; sh_a32[2] = thr32;
                if (isfinite(du) && isfinite(band) && fabsf(du - thr32) > band) {
                    sh_acc = du <= thr32;
                    sh_need64 = v.audit ? 2 : 0;     // 2: the binary64 pass runs for the audit only
                    sh_du = (double)du;
                } else {
                    sh_need64 = 1;
                    re_move++;
                }
            }
            __syncthreads();
            need64 = sh_need64;
        }
        if (need64) {
            double dU = 0.0;
            for (int k = tid; k < n; k += NT) {
                const int m = mem_ids[k];
                const Bead bm = v.bead[m];
                const double o[3] = {bm.x, bm.y, bm.z};
                const double nw[3] = {v.s_new[3 * k], v.s_new[3 * k + 1], v.s_new[3 * k + 2]};
                dU += U_ext(P, nw[0], nw[1], nw[2]) - U_ext(P, o[0], o[1], o[2]);
                for (int e = 0; e < 2; e++) {
                    int q = e ? m + 1 : m - 1;
                    if (q < 0 || q >= v.N || !(e ? v.bnext[m] : v.bnext[q])) continue;
                    Bead bq = v.bead[q];
                    double qn[3] = {bq.x, bq.y, bq.z};
                    const int sq = find(q, bq);
                    if (sq >= 0) {
                        if (q < m) continue;
                        qn[0] = v.s_new[3 * sq]; qn[1] = v.s_new[3 * sq + 1]; qn[2] = v.s_new[3 * sq + 2];
                    }
                    double r2n = norm2(mi(nw[0] - qn[0], L, hL), mi(nw[1] - qn[1], L, hL), mi(nw[2] - qn[2], L, hL));
                    double r2o = norm2(mi(o[0] - bq.x, L, hL), mi(o[1] - bq.y, L, hL), mi(o[2] - bq.z, L, hL));
                    dU += U_bond(P, r2n) - U_bond(P, r2o);
                }
            }
            // the pairs the binary32 pass listed (mixed precision, list complete), else all pairs
            const int npairs = serial_pair_cap<PREC, NT>() > 0 ? sh_np : 1;
            if (eps_on && npairs <= serial_pair_cap<PREC, NT>()) {
                for (int ip = tid; ip < npairs; ip += NT) {
                    const int2 pr = sh_pairs[ip];
                    const int k = pr.x, m = mem_ids[k], q = pr.y;
                    const Bead bm = v.bead[m], bq = v.bead[q];
                    const double nw[3] = {v.s_new[3 * k], v.s_new[3 * k + 1], v.s_new[3 * k + 2]};
                    double qn[3] = {bq.x, bq.y, bq.z};
                    const int sq = find(q, bq);
                    if (sq >= 0) {
                        qn[0] = v.s_new[3 * sq]; qn[1] = v.s_new[3 * sq + 1]; qn[2] = v.s_new[3 * sq + 2];
                    }
                    const double r2n = norm2(mi(nw[0] - qn[0], L, hL), mi(nw[1] - qn[1], L, hL), mi(nw[2] - qn[2], L, hL));
                    const double r2o = norm2(mi(bm.x - bq.x, L, hL), mi(bm.y - bq.y, L, hL), mi(bm.z - bq.z, L, hL));
                    if (r2n < P.rc2 || r2o < P.rc2) dU += U_wca(P, r2n) - U_wca(P, r2o);
                }
            } else if (eps_on) {
                int mk = -1;
                double o[3] = {0.0, 0.0, 0.0}, nw[3] = {0.0, 0.0, 0.0};
                for_pairs([&](int k, int m, int q, const Bead& bq) {
                    const int sq = find(q, bq);
                    const bool member = sq >= 0;
                    if (member && q < m) return;
                    if (k != mk) {
                        mk = k;
                        const Bead bm = v.bead[m];
                        o[0] = bm.x; o[1] = bm.y; o[2] = bm.z;
                        nw[0] = v.s_new[3 * k]; nw[1] = v.s_new[3 * k + 1]; nw[2] = v.s_new[3 * k + 2];
                    }
                    double qn[3] = {bq.x, bq.y, bq.z};
                    if (member) {
                        qn[0] = v.s_new[3 * sq]; qn[1] = v.s_new[3 * sq + 1]; qn[2] = v.s_new[3 * sq + 2];
                    }
                    const double r2n = norm2(mi(nw[0] - qn[0], L, hL), mi(nw[1] - qn[1], L, hL), mi(nw[2] - qn[2], L, hL));
                    const double r2o = norm2(mi(o[0] - bq.x, L, hL), mi(o[1] - bq.y, L, hL), mi(o[2] - bq.z, L, hL));
                    if (r2n < P.rc2 || r2o < P.rc2) {
                        dU += U_wca(P, r2n) - U_wca(P, r2o);
                        if (!member && PREC == 0) pe_move++;
                    }
                });
            }
            dU = warp_sum(dU);
            if (lane == 0) sh_red[wid] = dU;
            __syncthreads();
            if (tid == 0) {
                double su = 0.0;
                for (int w = 0; w < NT / 32; w++) su += sh_red[w];
                if (PREC == 1 && v.audit) audit_record(v, (double)sh_a32[0], (double)sh_a32[1], (double)sh_a32[2], su, thr);
                if (PREC == 0 || sh_need64 != 2) {
                    sh_acc = su <= thr;
                    sh_du = su;
                }
            }
            __syncthreads();
        }
        };
        if (live) evaluate();
        bool mine = true;                         // this block's move runs
        int steps = 1;
        if (SPEC && nb > 1) {
            // the hypothesis' outcome with the balls it read and would write: every bead of the support
            // moves by at most A_w / 4 from within lambda of the centre; partners lie within r_c of an
            // old or new position; bonded partners where they were met
            if (tid == 0) {
                SpecRec rec;
                rec.known = known; rec.acc = known == 1 && sh_acc; rec.n = n; rec.lam = lam;
                for (int a = 0; a < 3; a++) rec.b[a] = sh_bf[a];
                const float far_ = (float)(n > 0 && known == 1 ? sh_awx[1] - v.rc : 0.0);
                rec.wr = (float)lam + far_;
                rec.rr = fmaxf(rec.wr + (float)v.rc, known ? sh_bond : 0.0f);
                recs[cb] = rec;
            }
            if (!spec_barrier(bar, nb * ++phase, &sh_ok)) { if (tid == 0) set_err(v, E_WALK); gave_up = true; break; }
            constexpr int RW = sizeof(SpecRec) / 4;
            for (int e = tid; e < nb * RW; e += NT) ((int*)sh_rec)[e] = __ldcg((const int*)recs + e);
            __syncthreads();
            if (wid == 0) {
                // two accepted moves must not share a fine cell either (their list changes run side by
                // side): its diagonal is added
                int taken;
                double carry = sh_carry;
                const int w = window_walk(sh_rec, nb, count - t, Lf, hLf, 1e-3f + 2e-6f * Lf, 1.7321f / (float)v.invf, cb, lane, &taken, &carry);
                if (lane == 0) { sh_mine = taken; sh_steps = w; sh_carry = carry; }
            }
            __syncthreads();
            mine = sh_mine != 0;
            steps = sh_steps;
        }
        else if (QUEUES) mine = live;
        const bool acc = mine && known == 1 && sh_acc;
        int* const mem_ids = n <= serial_mem_cap<NT>() ? sm_ids : v.s_ids;
        if (acc) {
            for (int k = tid; k < n; k += NT) {
                const int m = mem_ids[k];
                const Bead bm = v.bead[m];
                const int oc = cell_lin(v, bm.x, bm.y, bm.z);
                const double nw[3] = {v.s_new[3 * k], v.s_new[3 * k + 1], v.s_new[3 * k + 2]};
                const int ncl = cell_lin(v, nw[0], nw[1], nw[2]);
                put_bead(v.bead, v.bf, m, nw[0], nw[1], nw[2]);
                if (v.s_img[k] != pack_img(0, 0, 0)) {
                    int dd[3];
                    unpack_img(v.s_img[k], dd);
                    v.img[3 * m] += dd[0]; v.img[3 * m + 1] += dd[1]; v.img[3 * m + 2] += dd[2];
                }
                if (oc != ncl) {
                    int idx = atomicAdd(&sh_nch, 1);
                    v.s_changed[3 * idx] = m; v.s_changed[3 * idx + 1] = oc; v.s_changed[3 * idx + 2] = ncl;
                    if (idx < kChCap) { sc_m[idx] = m; sc_oc[idx] = oc; sc_nc[idx] = ncl; }
                }
            }
        }
        if (mine) pe += pe_move;
        __syncthreads();
        const int nch = acc ? sh_nch : 0;
        if (NT >= 512 && nch > 1 && nch <= kChCap) {
            grouped_relink(v, sc_m, sc_oc, sc_nc, nch, tid, NT);
        } else if (tid == 0) {
            for (int c = 0; c < nch; c++) {
                int m = v.s_changed[3 * c], oc = v.s_changed[3 * c + 1], ncl = v.s_changed[3 * c + 2];
                relink(v, m, oc, ncl);
            }
        }
        if (tid == 0 && mine && known == 2) {
            v.defer[start + tw] = 1;
            def++;
        } else if (tid == 0 && mine) {
            att++;
            bu += n;
            rechecks += re_move;
            if (acc) { acc_n++; moved_n += n; }
            v.tr_out[Ly.tr_off + j] = (uint8_t)((acc ? 1 : 2) | dflag);
            v.tr_n[Ly.tr_off + j] = n;
            v.tr_du[Ly.tr_off + j] = sh_du;
            if (nb == 1) sh_carry = acc ? 0.0 : lam;
        }
        __syncthreads();
        t += steps;
        // commits are in place before the next window's moves read
        if (SPEC && nb > 1 && (QUEUES || t < count) && !spec_barrier(bar, nb * ++phase, &sh_ok)) {
            if (tid == 0) set_err(v, E_WALK);
            gave_up = true;
            break;
        }
    }
    if (QUEUES && tid == 0 && cb == 0) v.carry_q[Ls.carry_off + cell] = sh_carry;
    }   // queues
    if (SPEC && nb > 1 && tid == 0) {
        // the last block to leave resets the barrier for the next launch
        if (atomicAdd(bar + 1, 1u) == (unsigned)nb - 1u) { bar[1] = 0u; bar[0] = 0u; }
    }
    // partner counts are per thread
    unsigned long long pe_all = (unsigned long long)pe;
    if (pe_all) atomicAdd(&v.ctr[C_PARTNER], pe_all);
    if (QUEUES && pe_all) atomicAdd(&v.ctr[C_CPE], pe_all);
    if (tid == 0) {
        if (!QUEUES && cb == 0) v.carry_serial[l] = sh_carry;
        if (QUEUES) {
            if (ls < kLevel2 && def) atomicAdd(&v.ctr[C_DEF + l], (unsigned long long)def);   // first deferrals only
            atomicAdd(&v.ctr[C_CBU], (unsigned long long)bu);
            atomicAdd(&v.ctr[C_CMOVED], (unsigned long long)moved_n);
        }
        atomicAdd(&v.ctr[C_ATT + l], (unsigned long long)att);
        atomicAdd(&v.ctr[C_ACC + l], (unsigned long long)acc_n);
        atomicAdd(&v.ctr[C_ACCTOT], (unsigned long long)acc_n);
        atomicAdd(&v.ctr[C_BU], (unsigned long long)bu);
        if (moved_n) atomicAdd(&v.ctr[C_MOVED], (unsigned long long)moved_n);
        if (rechecks) atomicAdd(&v.ctr[C_RECHECK], (unsigned long long)rechecks);
    }
}
// Serial phase of a small simulation whose layers are all serial: the whole simulation is staged in
// shared memory for the launch (positions in binary64 and as binary32 pairs), every slot of the
// layer runs on-chip, and the beads are written back at the end. The global cell lists are not
// updated here; they are marked stale and rebuilt before the next move that needs them.
//
// Every warp evaluates one hypothesis of a window of moves (see window_walk: a move depends on the
// ones before it only through the recycled scale and through beads they shifted), so a window costs
// two block barriers for several moves instead of seven for one. A move is one warp's own work:
//  - the beads are kept in groups of 32 consecutive ids with a bounding ball each (grown by accepted
//    moves); consecutive beads of a chain are close, so a move looks at the few groups its reach meets;
//  - binary64 steps hold this part's pipe ~64 cycles a warp instruction however few lanes need them,
//    so the three axes of up to ten members share one instruction (lane = 3 member + axis);
//  - binary32 energies with the rigorous band decide, binary64 inside the band (or in binary64 mode).
// (Cycles of a window by clock64(), 4 warps at 251 beads and 16 at 2,044: centre and scale 1.0k and 2.5k,
// search 1.8k and 3.2k, displacements 1.8k and 2.9k, pair terms 4.7k and 5.7k, wait for the slowest warp and
// walk 2.7k and 6.1k, for 2.4 and 5.3 moves; before the terms were found member by member, see for_terms.)
// A support beyond a warp's scratch, or a crowded one, is run by the whole block in its turn.
// Shared bytes: see smem_serial_bytes.
constexpr int kSmemChunk = 32;                     // slots prepared together
constexpr int kWarpScr = warp_scr_bytes(kWarpMem); // scratch bytes per warp
template <int PREC, int NT>
__global__ void __launch_bounds__(NT, 65536 / (NT * 128)) k_serial_smem(const SimView* __restrict__ vs, int l, int64_t nlo, int64_t nhi) {
    SIM_EXIT_IF(l >= gv.nL || gv.precision != PREC || !((gv.smem_layers >> l) & 1) || gv.counts[l] == 0 ||
                gv.N <= nlo || gv.N > nhi)
    SIM_PROLOGUE
    extern __shared__ __align__(16) char dsm[];
    if (l >= v.nL || v.precision != PREC || !((v.smem_layers >> l) & 1)) return;
    const int count = v.counts[l];
    if (count == 0) return;
    constexpr int NW = NT / 32;
    constexpr int NG = kSmemSerialMaxN / 32;
    const unsigned FULL = 0xffffffffu;
    const int N = (int)v.N;
    // 8-byte arrays first, then 4-, 2- and 1-byte ones, so every array is aligned for any N
    double* const px = (double*)dsm;             // binary64 positions, axis a of bead m at a N + m
    float* const fx = (float*)(px + 3 * (size_t)N);   // binary32 pairs: hi at a N + m, lo at (3 + a) N + m
    char* const scr = (char*)(fx + 6 * (size_t)N);
    double* const mnew = (double*)scr;           // a block's move: new positions, 3 per support member
    float* const mnf = (float*)(mnew + 3 * (size_t)N);   // ... hi
    float* const mnl = mnf + 3 * (size_t)N;              // ... and lo
    const size_t scr_bytes = max((size_t)N * 48, (size_t)NW * kWarpScr);
    short* const mid = (short*)(scr + scr_bytes);   // ... its support
    short* const sslot = mid + N;                // ... per bead: index in the support or -1
    short* const dimg = sslot + N;               // 3 per bead: image change over the launch
    uint8_t* const mimg = (uint8_t*)(dimg + 3 * (size_t)N);   // a block's move: packed image change per member
    uint8_t* const bn = mimg + N;                // bond to the next bead
    __shared__ float4 s_grp[NG];                 // bounding ball of beads 32 g .. 32 g + 31
    __shared__ WarpRec s_rec[NW];
    __shared__ double ch_lam[kSmemChunk], ch_V[3 * kSmemChunk], ch_p[3 * kSmemChunk], ch_thr[kSmemChunk], ch_A0l[kSmemChunk];
    __shared__ double ch_ilam[PREC == 0 ? kSmemChunk : 1];
    __shared__ float ch_lamf[kSmemChunk], ch_pf[3 * kSmemChunk], ch_thrf[kSmemChunk];
    __shared__ int ch_bead[kSmemChunk];
    __shared__ int sh_n, sh_acc, sh_stale, sh_need64;
    __shared__ double sh_b[3], sh_red[NW], sh_aw, sh_du;
    __shared__ float sh_f32[NW], sh_m32[NW], sh_a32[3];
    __shared__ int sh_T[NW];
    __shared__ double s_sqrt[kNCap + 1], s_rsq[kNCap + 1];   // sqrt(n), correctly rounded, and its reciprocal
    for (int i2 = threadIdx.x; i2 <= kNCap; i2 += NT) {
        s_sqrt[i2] = v.sq_tab[i2];
        s_rsq[i2] = v.sq_tab[kNCap + 1 + i2];
    }
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const LayerDev& Ly = v.layer[l];
    const double L = v.L, hL = v.halfL;
    const float Lf = (float)L, hLf = (float)hL;
    const Pot& P = v.pot;
    // binary32 screens: a distance error of the copies below 8 L 2^-24 (rounding of the copies,
    // of the difference and of the image shift), so screening at r + 8 L 2^-24 + 1e-6 and a
    // relative 2^-20 on the square keeps every bead the binary64 test accepts
    const float marg = (float)(8.0 * L * 5.9604644775390625e-8 + 1e-6);
    const float up20 = 1.0f + 9.5367431640625e-7f, dn20 = 1.0f - 9.5367431640625e-7f;
    for (int m = tid; m < N; m += NT) {
        const Bead b = v.bead[m];
        const double x[3] = {b.x, b.y, b.z};
        for (int a = 0; a < 3; a++) {
            const float h = (float)x[a];
            px[a * N + m] = x[a];
            fx[a * N + m] = h;
            fx[(3 + a) * N + m] = (float)(x[a] - (double)h);
            dimg[3 * m + a] = 0;
        }
        sslot[m] = -1;
        bn[m] = v.bnext[m];
    }
    if (tid == 0) sh_stale = 0;
    __syncthreads();
    // distance of bead m from a point, minimum image
    auto dist2 = [&](int m, float x, float y, float z) {
        const float dx = wrapn(fx[m] - x, Lf, hLf), dy = wrapn(fx[N + m] - y, Lf, hLf), dz = wrapn(fx[2 * N + m] - z, Lf, hLf);
        return dx * dx + dy * dy + dz * dz;
    };
    const int ngrp = (N + 31) / 32;
    for (int g = wid; g < ngrp; g += NW) {
        // about the middle bead of the group
        const int c = min(32 * g + 16, N - 1), m = min(32 * g + lane, N - 1);
        const float x = fx[c], y = fx[N + c], z = fx[2 * N + c];
        const float r2 = dist2(m, x, y, z);
        const unsigned far2 = __reduce_max_sync(FULL, __float_as_uint(r2));
        if (lane == 0) s_grp[g] = make_float4(x, y, z, __fsqrt_rn(__uint_as_float(far2)) * up20 + marg);
    }
    const Pot32 P32 = pot32(P);
    const bool kappa_on = P.kappa != 0.0, eps_on = P.eps != 0.0, uni = v.centring == 1;
    const float rcr = (float)v.rc, rcf = rcr + marg, rc2f = rcf * rcf * up20;
    const float A0f = (float)v.A0;
    long long att = 0, acc_n = 0, bu = 0, pe = 0, rechecks = 0, moved_n = 0;
    double carry = v.carry_serial[l];            // alike in every thread
    int hw = 0;                                  // this warp's hypothesis (hw, hr)
    while ((hw + 1) * (hw + 2) / 2 <= wid) hw++;
    const int hr = wid - hw * (hw + 1) / 2;
    const int nh = v.audit ? 1 : NW;             // audited runs evaluate each move once
    int wmax = 0;
    while (wmax * (wmax + 1) / 2 < nh) wmax++;   // moves a window can reach

    // ---- one warp's move: slot s of the chunk on scale lam (own: that of slot sl, whose binary32 forms
    // are at hand); the outcome into s_rec[wid] ----
    const Box B{px, fx, fx + 3 * (size_t)N, N, N, L, hL, Lf, hLf};
    const WarpScr W = warp_scr(scr + (size_t)wid * kWarpScr, kWarpMem);
    const int mk = lane / 3, ax = lane - 3 * mk;                    // this lane's member and axis of a pass
    const float kT9 = 1e-9f * (float)v.kT;
    auto warp_move = [&](int s, double lam, bool own, int sl) {
        WarpRec rec;
        rec.known = 1; rec.n = 0; rec.acc = 0; rec.pe = 0; rec.re = 0; rec.lam = lam; rec.du = 0.0;
        // centre: one axis per lane
        const double ba = uni ? ch_V[3 * s + ax]
                              : wrap_u(add(px[ax * N + ch_bead[s]], mul(lam, ch_V[3 * s + ax])), L, FULL, nullptr);
        const float baf = (float)ba, lamf = own ? ch_lamf[sl] : (float)lam;
        const double A0l = own ? ch_A0l[sl] : mul(v.A0, lam);
        const float bx = __shfl_sync(FULL, baf, 0), by = __shfl_sync(FULL, baf, 1), bz = __shfl_sync(FULL, baf, 2);
        rec.b[0] = bx; rec.b[1] = by; rec.b[2] = bz;
        // every WCA partner of a member, old or new position, lies within lam + A_w / 4 + r_c of the
        // centre (|displacement| <= A_w / 4); three margins cover the rounding of this screen and of
        // the energy pass's own
        const float far_ = 0.25f * (uni ? (float)uniform_aw(v, lam) : A0f * lamf) * up20;
        rec.wr = lamf + far_;
        const float rl = lamf + marg, rl2 = rl * rl * up20, ri = fmaxf(lamf - marg, 0.0f), ri2 = ri * ri * dn20;
        const float rR = rec.wr + rcr + 3.0f * marg, rR2 = rR * rR * up20;
        // the amplitude of every support size up to 32, one per lane, ahead of the search
        const float af_lane = PREC == 1 && !uni ? amp32(A0l, s_sqrt[lane + 1], s_rsq[lane + 1]) : 0.0f;
        int n = 0, nc = 0;
        for (int g0 = 0; g0 < ngrp; g0 += 32) {
            bool hit = false;
            if (g0 + lane < ngrp) {
                const float4 q = s_grp[g0 + lane];
                const float dx = wrapn(q.x - bx, Lf, hLf), dy = wrapn(q.y - by, Lf, hLf), dz = wrapn(q.z - bz, Lf, hLf);
                const float rg = rR + q.w + marg;
                hit = dx * dx + dy * dy + dz * dz <= rg * rg * up20;
            }
#pragma unroll 1
            for (unsigned bits = __ballot_sync(FULL, hit); bits; bits &= bits - 1u) {
                const int m = 32 * (g0 + __ffs(bits) - 1) + lane;
                const float d2 = m < N ? dist2(m, bx, by, bz) : 4.0f * rR2;
                bool in = d2 < ri2;
                const bool tie = !in && d2 <= rl2;
                if (__any_sync(FULL, tie)) {
                    double d[3] = {__shfl_sync(FULL, ba, 0), __shfl_sync(FULL, ba, 1), __shfl_sync(FULL, ba, 2)};
                    if (tie) {
                        for (int a = 0; a < 3; a++) d[a] = mi(sub(px[a * N + m], d[a]), L, hL);
                        in = norm2(d[0], d[1], d[2]) < mul(lam, lam);
                    }
                }
                const bool cd = !in && d2 <= rR2;
                const unsigned vi = __ballot_sync(FULL, in), vc = __ballot_sync(FULL, cd), below = (1u << lane) - 1u;
                if (in) { const int k = n + __popc(vi & below); if (k < kWarpMem) W.mid[k] = (unsigned short)m; }
                if (cd) { const int k = nc + __popc(vc & below); if (k < kWarpCand) W.cand[k] = (unsigned short)m; }
                n += __popc(vi);
                nc += __popc(vc);
            }
        }
        __syncwarp();
        rec.n = n;
        rec.rr = rR;
        if (n > kWarpMem || nc > kWarpCand) {
            rec.known = 0;
        } else if (n == 0) {
            rec.acc = 0.0 <= ch_thr[s];           // nothing inside: no motion, dU = 0 against the threshold
        } else {
            double Aw = 0.0;
            float af;
            if (uni) Aw = uniform_aw(v, lam);
            else if (PREC == 0) Aw = div_by(A0l, s_sqrt[n], s_rsq[n]);
            if (uni || PREC == 0) af = (float)Aw;
            else af = n <= 32 ? __shfl_sync(FULL, af_lane, n - 1) : amp32(A0l, s_sqrt[n], s_rsq[n]);
            const double ilam = PREC == 1 ? 0.0 : own ? ch_ilam[sl] : dvd(1.0, lam);
            move_disp<PREC, true>(B, W, n, ba, &ch_p[3 * s], &ch_pf[3 * s], lam, ilam, lamf, Aw, af, lane);
            const float disp = 0.25f * af * up20, rs = (rcr + disp + 2.0f * marg) * up20, c[3] = {bx, by, bz};
            float bond2 = 0.0f;                   // farthest bonded partner read, from the centre
            auto terms = [&](auto&& pairs) {
                for_terms<true>(B, W, n, nc, false, P.bond != 0, eps_on, rs, disp, c, &bond2, lane,
                    [&](int k, int e) {
                        const int m = W.mid[k], q = e ? m + 1 : m - 1;
                        if (q < 0 || q >= N || !(e ? bn[m] : bn[q])) return -1;
                        // members are in ascending order: a bonded neighbour inside the support is next to it
                        return (e ? (k + 1 < n && W.mid[k + 1] == q) : (k > 0 && W.mid[k - 1] == q)) ? -1 : q;
                    },
                    [&](int k1, int k2) { return W.mid[k2] == W.mid[k1] + 1 && bn[W.mid[k1]]; },
                    [&](int) { return false; }, pairs);
            };
            move_decide<PREC, true>(v, B, W, P32, n, kT9, ch_thr[s], ch_thrf[s], lane, terms, rec);
            rec.rr = fmaxf(rR, sqrtf(bond2) * up20 + marg);
        }
        if (lane == 0) s_rec[wid] = rec;
    };

    // squared distance of two points given as hi and lo parts (and as binary64 positions for a
    // component across a face, rare for pairs in range): the hi difference is rounded once relative
    // to the result and the lo parts add the rest, so a component carries about one ulp
    auto comp = [&](float ha, float la, float hb, float lb, double xa, double xb) {
        const float dh = ha - hb;
        if (fabsf(dh) <= hLf) return dh + (la - lb);
        const double e = sub(xa, xb);
        return (float)(e > 0.0 ? sub(e, L) : add(e, L));
    };

    // ---- a move of the whole block (any support): slot s of the chunk on its scale in turn ----
    auto block_move = [&](int s, int j) {
        const double lam = __double_as_longlong(carry) > 0 ? carry : ch_lam[s];
        if (tid < 3) {
            const double r0 = px[tid * N + ch_bead[s]];
            sh_b[tid] = uni ? ch_V[3 * s + tid] : wrap(add(r0, mul(lam, ch_V[3 * s + tid])), L, nullptr);
            if (tid == 0) sh_n = 0;
        }
        __syncthreads();
        const double b[3] = {sh_b[0], sh_b[1], sh_b[2]}, lam2 = mul(lam, lam);
        const float bx = (float)b[0], by = (float)b[1], bz = (float)b[2], lamf = (float)lam;
        const float rl = lamf + marg, rl2 = rl * rl * up20;
        for (int m = tid; m < N; m += NT) {
            if (dist2(m, bx, by, bz) > rl2) continue;
            const unsigned am = __activemask();
            double dd[3] = {sub(px[m], b[0]), sub(px[N + m], b[1]), sub(px[2 * N + m], b[2])};
            mi3_u(dd, L, hL, am);
            if (norm2(dd[0], dd[1], dd[2]) < lam2) mid[atomicAdd(&sh_n, 1)] = (short)m;
        }
        __syncthreads();
        const int n = sh_n;
        if (n == 0) {      // nothing inside: no motion, dU = 0 against the threshold
            if (tid == 0) { sh_acc = 0.0 <= ch_thr[s]; sh_du = 0.0; }
            __syncthreads();
            return lam;
        }
        if (tid == 0) sh_aw = uni ? uniform_aw(v, lam) : dvd(mul(v.A0, lam), n <= kNCap ? s_sqrt[n] : sqr_t((double)n));
        __syncthreads();
        const double Aw = sh_aw, p[3] = {ch_p[3 * s], ch_p[3 * s + 1], ch_p[3 * s + 2]};
        const float af = (float)Aw, pf[3] = {(float)p[0], (float)p[1], (float)p[2]};
        for (int k = tid; k < n; k += NT) {
            const unsigned am = __activemask();
            const int m = mid[k];
            const double o[3] = {px[m], px[N + m], px[2 * N + m]};
            double d[3] = {sub(o[0], b[0]), sub(o[1], b[1]), sub(o[2], b[2])}, dl[3];
            mi3_u(d, L, hL, am);
            if (PREC == 0) wavelet_disp64(d, norm2(d[0], d[1], d[2]), lam, Aw, p, dl);
            else wavelet_disp32f(d, lamf, af, pf, dl);
            int im[3] = {0, 0, 0};
            double nx[3] = {add(o[0], dl[0]), add(o[1], dl[1]), add(o[2], dl[2])};
            wrap3_u(nx, L, am, im);
            for (int a = 0; a < 3; a++) {
                mnew[3 * k + a] = nx[a];
                if (im[a] == 0) {
                    // old (hi, lo) plus the displacement by a binary32 two-sum, renormalised
                    const float oh = fx[a * N + m], dlf = (float)dl[a];
                    const float s1 = oh + dlf, bb = s1 - oh;
                    const float l1 = fx[(3 + a) * N + m] + ((oh - (s1 - bb)) + (dlf - bb));
                    const float h2 = s1 + l1;
                    mnf[3 * k + a] = h2;
                    mnl[3 * k + a] = l1 - (h2 - s1);
                } else {                       // wrapped across a face: split the binary64 value
                    mnf[3 * k + a] = (float)nx[a];
                    mnl[3 * k + a] = (float)(nx[a] - (double)mnf[3 * k + a]);
                }
            }
            mimg[k] = (uint8_t)pack_img(im[0], im[1], im[2]);
            sslot[m] = (short)k;
        }
        __syncthreads();
        // the (member, bead) pairs of the WCA sums: each member (one per warp) against the beads of the
        // groups whose balls its reach meets, each pair of members once. Pairs whose old distance by the
        // hi parts is beyond the cutoff and both displacements are passed over. (Every member against
        // every other and every candidate is n^2 work: 1.8 ms for a support of 1,000 beads.)
        const float rsc = (rcr + 0.5f * af * up20 + 2.0f * marg) * up20, rsc2 = rsc * rsc;
        auto for_wca_pairs = [&](auto&& f) {
            for (int k = wid; k < n; k += NW) {
                const int m = mid[k];
                const float x = fx[m], y = fx[N + m], z = fx[2 * N + m];
                for (int g0 = 0; g0 < ngrp; g0 += 32) {
                    bool hit = false;
                    if (g0 + lane < ngrp) {
                        const float4 q = s_grp[g0 + lane];
                        const float dx = wrapn(q.x - x, Lf, hLf), dy = wrapn(q.y - y, Lf, hLf), dz = wrapn(q.z - z, Lf, hLf);
                        const float rg = rsc + q.w + marg;
                        hit = dx * dx + dy * dy + dz * dz <= rg * rg * up20;
                    }
                    for (unsigned bits = __ballot_sync(FULL, hit); bits; bits &= bits - 1u) {
                        const int q = 32 * (g0 + __ffs(bits) - 1) + lane;
                        if (q >= N || q == m || dist2(q, x, y, z) > rsc2) continue;
                        const int sq = sslot[q];
                        if (!(sq >= 0 && q < m)) f(k, m, q, sq);
                    }
                }
            }
        };
        // squared distances of members and beads, new (through sq) and old
        auto o32 = [&](int m, int q) {
            const float x = comp(fx[m], fx[3 * N + m], fx[q], fx[3 * N + q], px[m], px[q]);
            const float y = comp(fx[N + m], fx[4 * N + m], fx[N + q], fx[4 * N + q], px[N + m], px[N + q]);
            const float z = comp(fx[2 * N + m], fx[5 * N + m], fx[2 * N + q], fx[5 * N + q], px[2 * N + m], px[2 * N + q]);
            return x * x + y * y + z * z;
        };
        auto n32 = [&](int k, int q, int sq) {
            float s2 = 0.0f;
            for (int a = 0; a < 3; a++) {
                const float c = sq >= 0 ? comp(mnf[3 * k + a], mnl[3 * k + a], mnf[3 * sq + a], mnl[3 * sq + a], mnew[3 * k + a], mnew[3 * sq + a])
                                        : comp(mnf[3 * k + a], mnl[3 * k + a], fx[a * N + q], fx[(3 + a) * N + q], mnew[3 * k + a], px[a * N + q]);
                s2 += c * c;
            }
            return s2;
        };
        auto o64 = [&](int m, int q) {
            return norm2(mi(px[m] - px[q], L, hL), mi(px[N + m] - px[N + q], L, hL), mi(px[2 * N + m] - px[2 * N + q], L, hL));
        };
        auto n64 = [&](int k, int q, int sq) {
            double d[3];
            for (int a = 0; a < 3; a++) d[a] = mi(mnew[3 * k + a] - (sq >= 0 ? mnew[3 * sq + a] : px[a * N + q]), L, hL);
            return norm2(d[0], d[1], d[2]);
        };
        // energy change. Mixed precision: a binary32 pass (with the magnitudes of its terms) decides
        // outside the rigorous error band; inside it, and in binary64 mode, the binary64 pass decides.
        const double thr = ch_thr[s];
        bool need64 = PREC == 0;
        int pe_move = 0;
        if (PREC == 1) {
            float a32 = 0.0f, m32 = 0.0f;
            int T = 0;
            for (int k = tid; k < n; k += NT) {
                const int m = mid[k];
                if (kappa_on) {
                    const float un = 0.5f * P32.kappa * norm2f(dif32(mnew[3 * k], hL, L, hLf), dif32(mnew[3 * k + 1], hL, L, hLf), dif32(mnew[3 * k + 2], hL, L, hLf));
                    const float uo = 0.5f * P32.kappa * norm2f(dif32(px[m], hL, L, hLf), dif32(px[N + m], hL, L, hLf), dif32(px[2 * N + m], hL, L, hLf));
                    a32 += un - uo; m32 += un + uo; T += 2;
                }
                for (int e = 0; e < 2; e++) {
                    const int q = e ? m + 1 : m - 1;
                    if (q < 0 || q >= N || !(e ? bn[m] : bn[q])) continue;
                    const int sq = sslot[q];
                    if (sq >= 0 && q < m) continue;
                    float un, mn, uo, mo;
                    bond32(P32, n32(k, q, sq), un, mn);
                    bond32(P32, o32(m, q), uo, mo);
                    a32 += un - uo; m32 += mn + mo; T += 2;
                }
            }
            if (eps_on) {
                for_wca_pairs([&](int k, int m, int q, int sq) {
                    const float rn = n32(k, q, sq), ro = o32(m, q);
                    if (rn <= rc2f || ro <= rc2f) {
                        float un, mn, uo, mo;
                        wca32(P32, rn, un, mn);
                        wca32(P32, ro, uo, mo);
                        a32 += un - uo; m32 += mn + mo; T += 2;
                        if (sq < 0 && (un != 0.0f || uo != 0.0f)) pe_move++;
                    }
                });
            }
            for (int o = 16; o > 0; o >>= 1) {
                a32 += __shfl_xor_sync(FULL, a32, o);
                m32 += __shfl_xor_sync(FULL, m32, o);
                T = max(T, __shfl_xor_sync(FULL, T, o));
            }
            if (lane == 0) { sh_f32[wid] = a32; sh_m32[wid] = m32; sh_T[wid] = T; }
            __syncthreads();
            if (tid == 0) {
                float d32 = 0.0f, mm = 0.0f;
                int tt = 0;
                for (int w = 0; w < NW; w++) { d32 += sh_f32[w]; mm += sh_m32[w]; tt = max(tt, sh_T[w]); }
                tt += 5 + NW;          // summation depth: one thread's terms, the butterfly, the warp totals
                const float thr32 = (float)thr;
                const float band = 2.0f * (float)(80 + tt + 6) * 5.9604645e-08f * mm + 1e-9f * (float)v.kT +
                                   2.4e-7f * fabsf(thr32);
                sh_a32[0] = d32; sh_a32[1] = band; sh_a32[2] = thr32;
                if (isfinite(d32) && isfinite(band) && fabsf(d32 - thr32) > band) {
                    sh_acc = d32 <= thr32;
                    sh_need64 = v.audit ? 2 : 0;     // 2: the binary64 pass runs for the audit only
                    sh_du = (double)d32;
                } else {
                    sh_need64 = 1;
                    rechecks++;
                }
            }
            __syncthreads();
            need64 = sh_need64;
        }
        if (need64) {
            double dU = 0.0;
            for (int k = tid; k < n; k += NT) {
                const int m = mid[k];
                dU += U_ext(P, mnew[3 * k], mnew[3 * k + 1], mnew[3 * k + 2]) - U_ext(P, px[m], px[N + m], px[2 * N + m]);
                for (int e = 0; e < 2; e++) {
                    const int q = e ? m + 1 : m - 1;
                    if (q < 0 || q >= N || !(e ? bn[m] : bn[q])) continue;
                    const int sq = sslot[q];
                    if (sq >= 0 && q < m) continue;
                    dU += U_bond(P, n64(k, q, sq)) - U_bond(P, o64(m, q));
                }
            }
            if (eps_on) {
                for_wca_pairs([&](int k, int m, int q, int sq) {
                    if (n32(k, q, sq) <= rc2f || o32(m, q) <= rc2f) {
                        const double rn = n64(k, q, sq), ro = o64(m, q);
                        if (rn < P.rc2 || ro < P.rc2) {
                            dU += U_wca(P, rn) - U_wca(P, ro);
                            if (sq < 0 && PREC == 0) pe_move++;
                        }
                    }
                });
            }
            dU = warp_sum(dU);
            if (lane == 0) sh_red[wid] = dU;
            __syncthreads();
            if (tid == 0) {
                double su = 0.0;
                for (int w = 0; w < NW; w++) su += sh_red[w];
                if (PREC == 1 && v.audit) audit_record(v, (double)sh_a32[0], (double)sh_a32[1], (double)sh_a32[2], su, thr);
                if (PREC == 0 || sh_need64 != 2) {
                    sh_acc = su <= thr;
                    sh_du = su;
                }
            }
            __syncthreads();
        }
        pe += pe_move;
        const bool acc = sh_acc;
        for (int k = tid; k < n; k += NT) {
            const int m = mid[k];
            if (acc) {
                int dd[3];
                unpack_img(mimg[k], dd);
                for (int a = 0; a < 3; a++) {
                    px[a * N + m] = mnew[3 * k + a];
                    fx[a * N + m] = mnf[3 * k + a];
                    fx[(3 + a) * N + m] = mnl[3 * k + a];
                    dimg[3 * m + a] += (short)dd[a];
                }
                const float4 q = s_grp[m >> 5];
                atomicMax((int*)&s_grp[m >> 5].w, __float_as_int(sqrtf(dist2(m, q.x, q.y, q.z)) * up20 + marg));
            }
            sslot[m] = -1;
        }
        return lam;
    };

    int c0 = 0, c1 = 0;                          // slots of the chunk
    bool alone = false;                          // the next move is run by the block at once
    for (int t = 0; t < count;) {
        if (min(t + wmax, count) > c1) {
            // slot parameters of the next slots (one read of global memory for many windows)
            __syncthreads();
            c0 = t;
            c1 = min(t + kSmemChunk, count);
            for (int e = tid; e < c1 - c0; e += NT) {
                const double lam = v.slot_lam[c0 + e];
                ch_lam[e] = lam;
                ch_lamf[e] = (float)lam;
                ch_A0l[e] = mul(v.A0, lam);
                if (PREC == 0) ch_ilam[e] = dvd(1.0, lam);
                ch_thr[e] = v.slot_thr[c0 + e];
                ch_thrf[e] = (float)ch_thr[e];
                ch_bead[e] = v.slot_bead[c0 + e];
            }
            for (int e = tid; e < 3 * (c1 - c0); e += NT) {
                ch_V[e] = v.slot_V[3 * c0 + e];
                ch_p[e] = v.slot_p[3 * c0 + e];
                ch_pf[e] = (float)ch_p[e];
            }
            __syncthreads();
        }
        int steps = 0;
        if (!alone) {
            const bool live = wid < nh && t + hw < count;
            if (live) {
                // the carried scale, or that of the slot the run of rejections started with
                const bool own = !(hr == hw && __double_as_longlong(carry) > 0);
                const int sl = t + hw - hr - c0;
                warp_move(t + hw - c0, own ? ch_lam[sl] : carry, own, sl);
            } else if (lane == 0) {
                s_rec[wid].known = 0;
            }
            __syncthreads();
            int mine;
            steps = window_walk(s_rec, nh, count - t, Lf, hLf, 1e-3f + 2e-6f * Lf, 0.0f, wid, lane, &mine, &carry);
            if (mine) {
                const WarpRec& q = s_rec[wid];
                if (q.acc) {
                    for (int k0 = 0; k0 < q.n; k0 += 10) {
                        const int k = k0 + mk;
                        if (lane < 30 && k < q.n) {
                            const int m = W.mid[k];
                            int dd[3];
                            unpack_img(W.img[k], dd);
                            px[ax * N + m] = W.nw[3 * k + ax];
                            fx[ax * N + m] = W.nh[3 * k + ax];
                            fx[(3 + ax) * N + m] = W.nl[3 * k + ax];
                            dimg[3 * m + ax] += (short)(ax == 0 ? dd[0] : ax == 1 ? dd[1] : dd[2]);
                        }
                    }
                    __syncwarp();
                    for (int k = lane; k < q.n; k += 32) {
                        const int m = W.mid[k];
                        const float4 s = s_grp[m >> 5];
                        atomicMax((int*)&s_grp[m >> 5].w, __float_as_int(sqrtf(dist2(m, s.x, s.y, s.z)) * up20 + marg));
                    }
                }
                if (lane == 0) {
                    const int j = t + hw;
                    att++;
                    bu += q.n;
                    pe += q.pe;
                    rechecks += q.re;
                    if (q.acc) { acc_n++; moved_n += q.n; }
                    v.tr_out[Ly.tr_off + j] = (uint8_t)(q.acc ? 1 : 2);
                    v.tr_n[Ly.tr_off + j] = q.n;
                    v.tr_du[Ly.tr_off + j] = q.du;
                }
            }
            __syncthreads();
        }
        if (steps == 0) {
            const int j = t;
            const double lam = block_move(t - c0, j);
            carry = sh_acc ? 0.0 : lam;
            alone = sh_n > kWarpMem / 2;
            if (tid == 0) {
                att++;
                bu += sh_n;
                if (sh_acc) { acc_n++; moved_n += sh_n; }
                v.tr_out[Ly.tr_off + j] = (uint8_t)(sh_acc ? 1 : 2);
                v.tr_n[Ly.tr_off + j] = sh_n;
                v.tr_du[Ly.tr_off + j] = sh_du;
            }
            steps = 1;
            __syncthreads();
        }
        t += steps;
    }
    // write back what moved; the cell lists go stale if a bead changed fine cell
    for (int m = tid; m < N; m += NT) {
        const Bead ob = v.bead[m];
        const double x = px[m], y = px[N + m], z = px[2 * N + m];
        if (ob.x == x && ob.y == y && ob.z == z) continue;
        put_bead(v.bead, v.bf, m, x, y, z);
        if (dimg[3 * m] | dimg[3 * m + 1] | dimg[3 * m + 2]) {
            v.img[3 * m] += dimg[3 * m]; v.img[3 * m + 1] += dimg[3 * m + 1]; v.img[3 * m + 2] += dimg[3 * m + 2];
        }
        if (cell_lin(v, ob.x, ob.y, ob.z) != cell_lin(v, x, y, z)) sh_stale = 1;
    }
    if (pe) atomicAdd(&v.ctr[C_PARTNER], (unsigned long long)pe);
    __syncthreads();
    if (lane == 0) {
        if (tid == 0) {
            if (sh_stale) *v.cl_stale = 1;
            v.carry_serial[l] = carry;
        }
        if (rechecks) atomicAdd(&v.ctr[C_RECHECK], (unsigned long long)rechecks);
        if (att) {
            atomicAdd(&v.ctr[C_ATT + l], (unsigned long long)att);
            atomicAdd(&v.ctr[C_ACC + l], (unsigned long long)acc_n);
            atomicAdd(&v.ctr[C_ACCTOT], (unsigned long long)acc_n);
            atomicAdd(&v.ctr[C_BU], (unsigned long long)bu);
            if (moved_n) atomicAdd(&v.ctr[C_MOVED], (unsigned long long)moved_n);
        }
    }
}

// shared bytes of a simulation of n beads in a block of nw warps
size_t smem_serial_bytes(int64_t n, int nw) {
    return (size_t)n * (3 * 8 + 6 * 4 + 2 + 2 + 3 * 2 + 1 + 1) + std::max((size_t)n * 48, (size_t)nw * kWarpScr) + 64;
}

int launch_serial(const SimView* d, const GroupDims& g, int l, cudaStream_t s, const ForkJoin* fj) {
    const int np = (g.prec_mask & 1) + ((g.prec_mask >> 1) & 1);
    int launched = g.any_global_serial ? np : 0;
    prepare_staged(g);
    // one launch per precision; each returns at once for simulations of the other precision
    const dim3 grid(1, g.S);
    if (g.smem_maxN > 0) {
        // one launch per size class, each with the shared memory of its largest simulation, so
        // small simulations pack many blocks per SM; with side streams the classes run side by side
        int ncls = 0;
        for (int c = 0; c < 3; c++) ncls += g.smem_cls[c] > 0;
        const bool fork = fj && fj->side[0] && ncls > 1;
        if (fork) {
            cudaEventRecord(fj->fork, s);
            cudaStreamWaitEvent(fj->side[0], fj->fork, 0);
            cudaStreamWaitEvent(fj->side[1], fj->fork, 0);
        }
        for (int c = 2; c >= 0; c--) {
            if (!g.smem_cls[c]) continue;
            cudaStream_t cs = fork ? (c == 2 ? s : fj->side[c]) : s;
            const size_t sm = smem_serial_bytes(g.smem_cls[c], 4 << c);
            const int64_t lo = c ? kSmemClassHi[c - 1] : 0, hi = kSmemClassHi[c];
            // threads per class: few for small simulations (several blocks share an SM), many
            // for large ones (one block per SM, whose warps must hide the latency of the scans)
            if (c == 0) {
                if (g.prec_mask & 1) k_serial_smem<0, 128><<<grid, 128, sm, cs>>>(d, l, lo, hi);
                if (g.prec_mask & 2) k_serial_smem<1, 128><<<grid, 128, sm, cs>>>(d, l, lo, hi);
            } else if (c == 1) {
                if (g.prec_mask & 1) k_serial_smem<0, 256><<<grid, 256, sm, cs>>>(d, l, lo, hi);
                if (g.prec_mask & 2) k_serial_smem<1, 256><<<grid, 256, sm, cs>>>(d, l, lo, hi);
            } else {
                if (g.prec_mask & 1) k_serial_smem<0, 512><<<grid, 512, sm, cs>>>(d, l, lo, hi);
                if (g.prec_mask & 2) k_serial_smem<1, 512><<<grid, 512, sm, cs>>>(d, l, lo, hi);
            }
            launched += np;
        }
        if (fork) {
            for (int c = 0; c < 2; c++) {
                cudaEventRecord(fj->join[c], fj->side[c]);
                cudaStreamWaitEvent(s, fj->join[c], 0);
            }
        }
    }
    if (!g.any_global_serial && !g.bigM[l]) return launched;
    if (g.smem_maxN > 0) {
        launch_cl_rebuild(d, g, s, 3 + l);
        launched += 3;
    }
    if (!g.any_global_serial) return launched;
    if (g.serial_threads <= 32) {
        if (g.prec_mask & 1) k_serial<0, 32, ONE_BLOCK><<<grid, 32, serial_dyn_bytes<0, 32, ONE_BLOCK>(), s>>>(d, l, 0, 1, 0);
        if (g.prec_mask & 2) k_serial<1, 32, ONE_BLOCK><<<grid, 32, serial_dyn_bytes<1, 32, ONE_BLOCK>(), s>>>(d, l, 0, 1, 0);
    } else if (g.serial_threads <= 128) {
        if (g.prec_mask & 1) k_serial<0, 128, ONE_BLOCK><<<grid, 128, serial_dyn_bytes<0, 128, ONE_BLOCK>(), s>>>(d, l, 0, 1, 0);
        if (g.prec_mask & 2) k_serial<1, 128, ONE_BLOCK><<<grid, 128, serial_dyn_bytes<1, 128, ONE_BLOCK>(), s>>>(d, l, 0, 1, 0);
    } else if (g.spec_blocks > 1) {
        // one simulation: a block for every hypothesis, no more than its moves can use. A sweep's serial
        // phases, one block against one per SM: 1M semi-dilute beads 473 -> 144 ms (7,100 deferred moves of
        // scale 8-16, neighbours in the list and often in conflict, and 1,800 of scale 16-32); 5M suspension
        // 92 -> 18 ms; a lone chain of 1,001 beads 2.3 -> 0.9 ms
        const int64_t M = g.Mmax[l];
        const dim3 gs((unsigned)std::min<int64_t>(g.spec_blocks, M * (M + 1) / 2), 1);
        int zero = 0, one = 1;
        void* args[] = {(void*)&d, (void*)&l, (void*)&zero, (void*)&one, (void*)&zero};
        if (g.prec_mask & 1)
            cudaLaunchCooperativeKernel((const void*)k_serial<0, 512, SPEC_SERIAL>, gs, dim3(512), args, serial_dyn_bytes<0, 512, SPEC_SERIAL>(), s);
        if (g.prec_mask & 2)
            cudaLaunchCooperativeKernel((const void*)k_serial<1, 512, SPEC_SERIAL>, gs, dim3(512), args, serial_dyn_bytes<1, 512, SPEC_SERIAL>(), s);
    } else {
        if (g.prec_mask & 1) k_serial<0, 512, ONE_BLOCK><<<grid, 512, serial_dyn_bytes<0, 512, ONE_BLOCK>(), s>>>(d, l, 0, 1, 0);
        if (g.prec_mask & 2) k_serial<1, 512, ONE_BLOCK><<<grid, 512, serial_dyn_bytes<1, 512, ONE_BLOCK>(), s>>>(d, l, 0, 1, 0);
    }
    return launched;
}

}  // namespace wmcd

namespace wmcd {

// ======================================================================================
// Plane-wave moves (Sec. VI, Appendix D): every bead moves by A_F cos(k.r + Phi) e.
// setup (1 thread) -> displacements (grid) -> energy change (grid, per-block partials)
// -> decision (1 block, fixed-order sum) -> commit (grid) -> cell-list rebuild if moved.
// ======================================================================================
// direct = 0: the m-th plane-wave slot of the current sweep (active if m < the sweep's count);
// direct = 1: the m-th move of a direct call. The counter is the sweep or the call index.
// inverse of the tabulated |k| CDF for u in (0, 1): the largest i with F_i <= u, then F^(1/3)
// linear between Q_i and Q_{i+1}; beyond the table the Q^-1 tail of 1 - F
__device__ double k_inverse(const double* F, double u) {
    if (u >= F[kKtN]) return mul((double)kKtN * kKtH, dvd(sub(1.0, F[kKtN]), sub(1.0, u)));
    int lo = 0, hi = kKtN;                 // F[lo] <= u < F[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (F[mid] <= u) lo = mid; else hi = mid;
    }
    const double a = cbrt(F[lo]), b = cbrt(F[lo + 1]);
    return add(mul((double)lo, kKtH), mul(kKtH, dvd(sub(cbrt(u), a), sub(b, a))));
}
// a nonzero point of the unit ball by rejection (kind, counter and first attempt as given); the
// unit vector along it
__device__ void unit_by_rejection(const SimView& v, uint32_t kind, uint64_t ctr, uint32_t m, uint32_t a0,
                                  double kh[3]) {
    double V[3] = {0.0, 0.0, 1.0};
    for (uint32_t b = 0; b < 64; b++) {
        const u4 d = draw(v.k0, v.k1, kind, 0, ctr, m, a0 + b);
        const double x = sym(d.x), y = sym(d.y), z = sym(d.z), q = norm2(x, y, z);
        if (q <= 1.0 && q > 0.0) { V[0] = x; V[1] = y; V[2] = z; break; }
    }
    const double r = sqr_t(norm2(V[0], V[1], V[2]));
    for (int c = 0; c < 3; c++) kh[c] = dvd(V[c], r);
}
// Fresh wave vector (Appendix D): the infinite system's |k| from the table and an isotropic
// direction; the quasi-continuous shell's snapped mode outside the discrete cube (up to 64
// attempts, the last standing); otherwise a mode of the table by its cumulative probability.
__device__ void pw_fresh_k(const SimView& v, uint32_t kshell, uint32_t kkdir, uint64_t ctr, uint32_t m, const u4& w1,
                           int lv[3], double kh[3], double* Q) {
    const double u_mode = u53(w1.x, w1.y);
    if (v.pw_mode == 3) {
        *Q = k_inverse(v.kF, u_open(w1.x, w1.y));
        unit_by_rejection(v, kkdir, ctr, m, 0u, kh);
        return;
    }
    if (v.pw_mode == 2 && !(u_mode < v.p_disc)) {
        const double lmax = v.layer[v.nL - 1].hi;
        for (uint32_t a = 0; a < 64; a++) {
            const u4 w = draw(v.k0, v.k1, kshell, 0, ctr, m, a);
            const double us = u_open(w.x, w.y);
            const double q = k_inverse(v.kF, add(v.kF0, mul(us, sub(1.0, v.kF0))));
            double d[3];
            unit_by_rejection(v, kkdir, ctr, m, 64u * a, d);
            const double sc = dvd(mul(q, v.L), mul(kTwoPi, lmax));
            int inside = 1;
            for (int c = 0; c < 3; c++) {
                lv[c] = (int)floor(add(mul(sc, d[c]), 0.5));
                if (abs(lv[c]) > v.pw_nl) inside = 0;
            }
            if (!inside) return;
        }
        return;
    }
    int lo = 0, hi = v.n_modes - 1;           // first mode with u < cdf
    while (lo < hi) { int mid = (lo + hi) >> 1; if (u_mode < v.mode_cdf[mid]) hi = mid; else lo = mid + 1; }
    for (int a = 0; a < 3; a++) lv[a] = v.modes[3 * lo + a];
}

__global__ void k_pw_setup(const SimView* __restrict__ vs, int direct, int m) {
    SIM_PROLOGUE
    if (threadIdx.x != 0) return;
    PWDev& P = *v.pw;
    *v.pw_rebuild = 0;
    P.active = direct ? 1 : (v.pw_on && m < v.counts[kMaxLayers]);
    if (!P.active) return;
    const uint64_t ctr = v.step[direct ? 1 : 0];
    const int kmode = direct ? K_DPWMODE : K_PWMODE, kdir = direct ? K_DPWDIR : K_PWDIR;
    const uint32_t kshell = direct ? K_DPWSHELL : K_PWSHELL, kkdir = direct ? K_DPWKDIR : K_PWKDIR;
    const bool cont = v.pw_mode == 3;
    const int trace_index = m;
    u4 w1 = draw(v.k0, v.k1, (uint32_t)kmode, 0, ctr, (uint32_t)m, 0);
    u4 w2 = draw(v.k0, v.k1, (uint32_t)kdir, 0, ctr, (uint32_t)m, 0);
    const double phi = u53(w1.z, w1.w), psi = u53(w2.x, w2.y);
    const int perm = (int)(((uint64_t)w2.z * 6u) >> 32);
    const uint32_t signs = w2.w & 7u;
    const int PERM[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
    int lv[3] = {0, 0, 0};
    double kh[3] = {0.0, 0.0, 1.0}, Q = 0.0;
    if (P.carry && !cont) {
        // recycle |k| after a rejection: permute the components, flip each sign with prob 1/2
        for (int a = 0; a < 3; a++) {
            int x = P.carry_l[PERM[perm][a]];
            lv[a] = ((signs >> a) & 1u) ? -x : x;
        }
    } else {
        pw_fresh_k(v, kshell, kkdir, ctr, (uint32_t)m, w1, lv, kh, &Q);
        if (P.carry && cont) Q = P.carry_Q;     // the same |k|, a new direction
    }
    const double lmax = v.layer[v.nL - 1].hi;
    for (int a = 0; a < 3; a++) P.lv[a] = lv[a];
    P.cont = cont;
    P.Q = Q;
    const bool fits = abs(lv[0]) <= 127 && abs(lv[1]) <= 127 && abs(lv[2]) <= 127;
    P.mode_packed = (cont || !fits) ? -1 : (lv[0] + 128) | ((lv[1] + 128) << 8) | ((lv[2] + 128) << 16);
    P.phi = phi;
    P.null_move = !cont && (lv[0] == 0 && lv[1] == 0 && lv[2] == 0);
    P.accept = 0;
    atomicAdd(&v.ctr[C_PWATT], 1ull);
    if (trace_index >= 0 && trace_index < v.tr_pw_cap) {
        v.tr_pw_mode[trace_index] = P.mode_packed;
        const double sc = cont ? dvd(mul(Q, v.L), mul(kTwoPi, lmax)) : 0.0;
        for (int a = 0; a < 3; a++) v.tr_pw_k[3 * trace_index + a] = cont ? mul(sc, kh[a]) : (double)lv[a];
    }
    if (P.null_move) {
        // k = 0 moves nothing and is accepted (Sec. VI.A)
        P.accept = 1;
        P.carry = 0;
        atomicAdd(&v.ctr[C_PWACC], 1ull);
        atomicAdd(&v.ctr[C_ACCTOT], 1ull);
        if (trace_index >= 0 && trace_index < v.tr_pw_cap) v.tr_pw_out[trace_index] = 1;
        return;
    }
    double u1[3], u2[3];
    if (cont) {
        // infinite system: A_F = (2/k) sqrt(dU_est/(mu N)) with k = Q / lambda_max (Eq. 48), the
        // polarisation about the continuous direction kh, the phase in turns per unit length
        const double kmag = dvd(Q, lmax);
        P.AF = dvd(mul(2.0, v.A0), mul(kmag, sqr_t(mul(5.0, (double)v.N))));
        P.kappa = dvd(Q, mul(kTwoPi, lmax));
        for (int a = 0; a < 3; a++) P.kh[a] = kh[a];
        if (kh[0] == 0.0 && kh[1] == 0.0) { u1[0] = 1.0; u1[1] = 0.0; u1[2] = 0.0; }
        else {
            const double nr = sqr_t(add(mul(kh[0], kh[0]), mul(kh[1], kh[1])));
            u1[0] = dvd(kh[1], nr); u1[1] = dvd(-kh[0], nr); u1[2] = 0.0;
        }
    } else {
        // A_F = (2/k) sqrt(dU_est/(mu N)), dU_est/mu = M6 A0^2/(2 pi)^3 = A0^2/5 (Eq. 48)
        const int l2 = lv[0] * lv[0] + lv[1] * lv[1] + lv[2] * lv[2];
        const double lm = sqr_t((double)l2);
        const double kmag = dvd(mul(kTwoPi, lm), v.L);
        P.AF = dvd(mul(2.0, v.A0), mul(kmag, sqr_t(mul(5.0, (double)v.N))));
        // polarisation e perpendicular to k: e = cos(psi) u1 + sin(psi) u2, u1 = k x z / |k x z|
        kh[0] = dvd((double)lv[0], lm); kh[1] = dvd((double)lv[1], lm); kh[2] = dvd((double)lv[2], lm);
        if (lv[0] == 0 && lv[1] == 0) { u1[0] = 1.0; u1[1] = 0.0; u1[2] = 0.0; }
        else {
            double nr = sqr_t((double)(lv[0] * lv[0] + lv[1] * lv[1]));
            u1[0] = dvd((double)lv[1], nr); u1[1] = dvd((double)(-lv[0]), nr); u1[2] = 0.0;
        }
    }
    u2[0] = sub(mul(kh[1], u1[2]), mul(kh[2], u1[1]));
    u2[1] = sub(mul(kh[2], u1[0]), mul(kh[0], u1[2]));
    u2[2] = sub(mul(kh[0], u1[1]), mul(kh[1], u1[0]));
    const double cp = cos2pi(psi), sp = sin2pi(psi);
    for (int a = 0; a < 3; a++) P.e[a] = add(mul(cp, u1[a]), mul(sp, u2[a]));
    P.reach = v.rc + 2.0 * fabs(P.AF) + 1e-9;
}

// squared binary32 distance of two wrapped points, minimum image (coordinates and side rounded first: the
// distance is within 2.1e-7 L and a few units of its own last place)
__device__ __forceinline__ float near32(const double* a, const double* b, float L, float hL) {
    const float x = wrapn((float)a[0] - (float)b[0], L, hL), y = wrapn((float)a[1] - (float)b[1], L, hL), z = wrapn((float)a[2] - (float)b[2], L, hL);
    return x * x + y * y + z * z;
}
__global__ void k_pw_disp(const SimView* __restrict__ vs) {
    SIM_EXIT_IF(!gv.pw->active || gv.pw->null_move)
    SIM_PROLOGUE
    const PWDev& P = *v.pw;
    if (!P.active || P.null_move) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) *v.cl_stale = 0;   // rebuilt just before, if it was stale
    const double lx = (double)P.lv[0], ly = (double)P.lv[1], lz = (double)P.lv[2];
    // x / L as div_by, from the rounded reciprocal formed once per block (not for a significand of ones)
    __shared__ double sh_rL;
    if (threadIdx.x == 0) sh_rL = (__double_as_longlong(v.L) & 0xfffffffffffffLL) == 0xfffffffffffffLL ? 0.0 : dvd(1.0, v.L);
    __syncthreads();
    const double rL = sh_rL;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < v.N; i += (int64_t)gridDim.x * blockDim.x) {
        const Bead b = v.bead[i];
        const double r[3] = {b.x, b.y, b.z};
        double t;
        if (P.cont) {
            // infinite system: the field at the unwrapped position
            double X[3];
            for (int a = 0; a < 3; a++) X[a] = add(r[a], mul((double)v.img[3 * i + a], v.L));
            t = add(mul(P.kappa, add(add(mul(P.kh[0], X[0]), mul(P.kh[1], X[1])), mul(P.kh[2], X[2]))), P.phi);
        } else {
            const double lr = add(add(mul(lx, r[0]), mul(ly, r[1])), mul(lz, r[2]));
            t = add(rL != 0.0 ? div_by(lr, v.L, rL) : dvd(lr, v.L), P.phi);
        }
        double dl[3];
        if (v.precision == 0) {
            const double amp = mul(P.AF, cos2pi(t));
            for (int a = 0; a < 3; a++) dl[a] = mul(amp, P.e[a]);
        } else {
            const float amp = mulf((float)P.AF, cos2pi_f(t));
            for (int a = 0; a < 3; a++) dl[a] = (double)mulf(amp, (float)P.e[a]);
        }
        int im[3] = {0, 0, 0};
        for (int a = 0; a < 3; a++) v.pw_new[3 * i + a] = wrap(add(r[a], dl[a]), v.L, &im[a]);
        v.pw_imgd[i] = pack_img(im[0], im[1], im[2]);
    }
}

// Energy change of a plane wave: one thread per bead finds its partners (higher ids within reach) by a
// binary32 screen on the old positions and lists the pairs; the block then takes the listed pairs in
// binary64, spread over its threads. The binary64 pipe is the bound (a warp instruction holds it ~64
// cycles): with each thread taking its own pairs, a warp ran for its busiest lane (a chain bead has
// several partners, a free sphere none) and formed the cell boxes in binary64 as well. 628,000 beads
// of the dilute suspension: 858 us a move through the heads of all cells, 755 through the occupancy
// words, about 250 with a list behind a shared counter, 227 with its prefix.
// The sum has a fixed order: a thread lists its partners in a column of its own, the columns are closed up
// behind a prefix of their lengths, each in ascending partner id, and entry e goes to thread e mod 256. (An
// atomic counter in place of the prefix let the scheduling of the warps choose the order, so equal runs
// formed other last bits.) Only partners beyond a full column are summed as the cell lists hold them.
constexpr int kPwCol = 16;           // listed partners of a bead (more: taken by their finder)
__global__ void __launch_bounds__(256) k_pw_energy(const SimView* __restrict__ vs) {
    SIM_EXIT_IF(!gv.pw->active || (int)blockIdx.x >= gv.pw_blocks)
    SIM_PROLOGUE
    __shared__ double red[8];
    __shared__ int pq[kPwCol * 256];                    // partner k of bead t of the block at 256 k + t
    __shared__ unsigned short ord[kPwCol * 256];        // the entries of pq that hold a pair, in order
    __shared__ int s_w[33];
    const PWDev& P = *v.pw;
    if (!P.active || blockIdx.x >= v.pw_blocks) return;
    double dU = 0.0;
    long long pe = 0;
    if (!P.null_move) {
        const double L = v.L, hL = v.halfL;
        const Pot& Po = v.pot;
        const int tid = threadIdx.x;
        const int64_t i0 = blockIdx.x * (int64_t)blockDim.x, i = i0 + tid;
        int found = 0;
        auto pair = [&](int64_t a, int64_t b, bool bond) {
            const Bead x = v.bead[a], y = v.bead[b];
            const double *xn = &v.pw_new[3 * a], *yn = &v.pw_new[3 * b];
            const double r2n = norm2(mi(xn[0] - yn[0], L, hL), mi(xn[1] - yn[1], L, hL), mi(xn[2] - yn[2], L, hL));
            const double r2o = norm2(mi(x.x - y.x, L, hL), mi(x.y - y.y, L, hL), mi(x.z - y.z, L, hL));
            if (bond) dU += U_bond(Po, r2n) - U_bond(Po, r2o);
            else if (r2n < Po.rc2 || r2o < Po.rc2) { dU += U_wca(Po, r2n) - U_wca(Po, r2o); pe++; }
        };
        if (i < v.N) {
            if (Po.kappa != 0.0) {
                const Bead b = v.bead[i];
                dU += U_ext(Po, v.pw_new[3 * i], v.pw_new[3 * i + 1], v.pw_new[3 * i + 2]) - U_ext(Po, b.x, b.y, b.z);
            }
            if (i + 1 < v.N && v.bnext[i]) pair(i, i + 1, true);
            if (Po.eps != 0.0) {
                // partners lie within reach of the old position (r_c and both displacements); the margin
                // covers the rounding of coordinates to binary32 and of the cell quotients below
                const Bead b = v.bead[i];
                const float Lf = (float)L, hLf = (float)hL, x[3] = {(float)b.x, (float)b.y, (float)b.z};
                const float reach = (float)P.reach * (1.0f + 1e-6f) + 1e-6f * Lf, r2 = reach * reach, inv = (float)v.invf;
                const float slack = 5e-7f * (float)v.Gf + 1e-6f;
                int c0[3], nc[3];
                for (int a = 0; a < 3; a++) {
                    c0[a] = (int)floorf((x[a] - reach) * inv - slack);
                    nc[a] = min((int)floorf((x[a] + reach) * inv + slack) - c0[a] + 1, v.Gf);
                }
                for_occupied(v, c0, nc, [&](int cell) {
                    int guard = 0;
                    for (int q = v.head[cell]; q >= 0;) {
                        const Bead bq = v.bead[q];
                        if (q > i) {
                            const float dx = wrapn((float)bq.x - x[0], Lf, hLf), dy = wrapn((float)bq.y - x[1], Lf, hLf),
                                        dz = wrapn((float)bq.z - x[2], Lf, hLf);
                            if (dx * dx + dy * dy + dz * dz <= r2) {
                                if (found < kPwCol) pq[256 * found++ + tid] = q;
                                else pair(i, q, false);
                            }
                        }
                        q = bq.next;
                        if (++guard > kMaxWalk) { set_err(v, E_WALK); break; }
                    }
                });
            }
        }
        int np;
        const int at = block_excl_scan<8>(found, s_w, &np);
        for (int k = 0; k < found; k++) {
            const int q = pq[256 * k + tid];
            int r = 0;
            for (int j = 0; j < found; j++) r += pq[256 * j + tid] < q;
            ord[at + r] = (unsigned short)(256 * k + tid);
        }
        __syncthreads();
        for (int e = tid; e < np; e += 256) pair(i0 + (ord[e] & 255), pq[ord[e]], false);
    }
    dU = warp_sum(dU);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = dU;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < 8; w++) s += red[w];
        v.pw_part[blockIdx.x] = s;
    }
    if (pe) atomicAdd(&v.ctr[C_PARTNER], (unsigned long long)pe);
}

__global__ void __launch_bounds__(256) k_pw_decide(const SimView* __restrict__ vs, int direct, int m) {
    SIM_EXIT_IF(!gv.pw->active || gv.pw->null_move)
    SIM_PROLOGUE
    __shared__ double red[8];
    PWDev& P = *v.pw;
    if (!P.active || P.null_move) return;
    const uint64_t ctr = v.step[direct ? 1 : 0];
    const int kacc = direct ? K_DPWACC : K_PWACC;
    const int trace_index = m;
    double s = 0.0;
    for (int b = threadIdx.x; b < v.pw_blocks; b += 256) s += v.pw_part[b];
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double dU = 0.0;
    for (int w = 0; w < 8; w++) dU += red[w];
    u4 w = draw(v.k0, v.k1, (uint32_t)kacc, 0, ctr, (uint32_t)m, 0);
    const double thr = accept_threshold(v, w);
    const bool acc = dU <= thr;
    P.accept = acc;
    atomicAdd(&v.ctr[C_BU], (unsigned long long)v.N);
    if (acc) {
        P.carry = 0;
        atomicAdd(&v.ctr[C_PWACC], 1ull);
        atomicAdd(&v.ctr[C_ACCTOT], 1ull);
        atomicAdd(&v.ctr[C_MOVED], (unsigned long long)v.N);
    } else {
        P.carry = 1;
        for (int a = 0; a < 3; a++) P.carry_l[a] = P.lv[a];
        P.carry_Q = P.Q;
    }
    if (trace_index >= 0 && trace_index < v.tr_pw_cap) v.tr_pw_out[trace_index] = (uint8_t)(acc ? 1 : 2);
}

__global__ void k_pw_commit(const SimView* __restrict__ vs) {
    SIM_EXIT_IF(!(gv.pw->active && gv.pw->accept && !gv.pw->null_move))
    SIM_PROLOGUE
    const PWDev& P = *v.pw;
    const bool moved = P.active && P.accept && !P.null_move;
    if (blockIdx.x == 0 && threadIdx.x == 0) *v.pw_rebuild = moved;
    if (!moved) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < v.N; i += (int64_t)gridDim.x * blockDim.x) {
        put_bead(v.bead, v.bf, i, v.pw_new[3 * i], v.pw_new[3 * i + 1], v.pw_new[3 * i + 2]);
        const int pk = v.pw_imgd[i];
        if (pk != pack_img(0, 0, 0)) {
            int dd[3];
            unpack_img(pk, dd);
            v.img[3 * i] += dd[0]; v.img[3 * i + 1] += dd[1]; v.img[3 * i + 2] += dd[2];
        }
    }
}

int launch_planewave(const SimView* d, const GroupDims& g, int direct, int m, cudaStream_t s) {
    const int nb = g.pw_blocks;
    const int gb = (int)gx(nb, g.S);
    k_pw_setup<<<dim3(1, g.S), 32, 0, s>>>(d, direct, m);
    launch_cl_rebuild(d, g, s, 2);
    k_pw_disp<<<dim3(gb, g.S), 256, 0, s>>>(d);
    k_pw_energy<<<dim3(nb, g.S), 256, 0, s>>>(d);
    k_pw_decide<<<dim3(1, g.S), 256, 0, s>>>(d, direct, m);
    k_pw_commit<<<dim3(gb, g.S), 256, 0, s>>>(d);
    launch_cl_rebuild(d, g, s, 1);
    return 11;
}

}  // namespace wmcd

namespace wmcd {

// ======================================================================================
// Serial moves of a large-scale layer on the whole GPU (Sec. VIII: a single large wavelet
// move executed in parallel). One move is a short sequence of launches over all beads or
// all support members: centre and slot parameters (one thread), support by a scan of all
// beads, displacements, energy change with per-block partial sums, the decision (fixed-order
// sum of the partials), the commit, and a cell-list rebuild if the move was accepted. The
// arithmetic of every step is that of the one-block serial kernel, so decisions agree.
// ======================================================================================
__global__ void k_big_setup(const SimView* __restrict__ vs, int l, int t) {
    SIM_PROLOGUE
    if (threadIdx.x != 0) return;
    *v.pw_rebuild = 0;                          // every simulation: the rebuild below is only for this move
    if (l >= v.nL || !((v.big_layers >> l) & 1)) return;
    BigMove& B = *v.big;
    B.active = t < v.counts[l];
    if (!B.active) return;
    const int j = t;
    const double carry = v.carry_serial[l];
    const double lam = carry > 0.0 ? carry : v.slot_lam[j];
    const Bead bi = v.bead[v.slot_bead[j]];
    const double ri[3] = {bi.x, bi.y, bi.z};
    for (int a = 0; a < 3; a++) {
        B.b[a] = v.centring == 1 ? v.slot_V[3 * j + a] : wrap(add(ri[a], mul(lam, v.slot_V[3 * j + a])), v.L, nullptr);
        B.p[a] = v.slot_p[3 * j + a];
    }
    B.lam = lam;
    B.j = j;
    B.thr = v.slot_thr[j];
    B.n = 0;
    B.acc = 0;
    B.nch = 0;
    uint32_t tag = *v.serial_tag + 1u;
    if (tag == 0u) tag = 1u;
    *v.serial_tag = tag;
    B.tag = tag;
}

// support: every bead strictly inside the ball (minimum image), in no particular order
__global__ void k_big_gather(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(l >= gv.nL || !((gv.big_layers >> l) & 1) || !gv.big->active)
    SIM_PROLOGUE
    BigMove* B = v.big;
    const double b[3] = {B->b[0], B->b[1], B->b[2]};
    const double lam = B->lam, lam2 = mul(lam, lam);
    const double L = v.L, hL = v.halfL;
    // binary32 screen on the shadows (margin 8 L 2^-24 + 1e-6 on the distance, as in the serial kernel):
    // most beads are far outside the ball and cost no binary64 step
    const float Lf = (float)L, hLf = (float)hL, bx = (float)b[0], by = (float)b[1], bz = (float)b[2];
    const float rl = (float)lam + (float)(8.0 * L * 5.9604644775390625e-8 + 1e-6), rl2 = rl * rl * (1.0f + 9.5367431640625e-7f);
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < v.N; m += (int64_t)gridDim.x * blockDim.x) {
        const BeadF f = v.bf[m];
        const float sx = wrapn(f.hx - bx, Lf, hLf), sy = wrapn(f.hy - by, Lf, hLf), sz = wrapn(f.hz - bz, Lf, hLf);
        if (sx * sx + sy * sy + sz * sz > rl2) continue;
        const Bead bb = v.bead[m];
        const double d0 = mi(sub(bb.x, b[0]), L, hL), d1 = mi(sub(bb.y, b[1]), L, hL), d2c = mi(sub(bb.z, b[2]), L, hL);
        const double d2 = norm2(d0, d1, d2c);
        if (d2 < lam2) {
            const int idx = atomicAdd(&B->n, 1);
            v.s_ids[idx] = (int)m;
            v.s_d[4 * idx] = d0; v.s_d[4 * idx + 1] = d1; v.s_d[4 * idx + 2] = d2c; v.s_d[4 * idx + 3] = d2;
        }
    }
}

__global__ void k_big_disp(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(l >= gv.nL || !((gv.big_layers >> l) & 1) || !gv.big->active || gv.big->n == 0)
    SIM_PROLOGUE
    const BigMove& B = *v.big;
    const int n = B.n;
    const double lam = B.lam;
    // formed by one thread of a block and shared: a binary64 division and square root of every warp
    // would hold the pipe for thousands of cycles
    __shared__ double sh_aw;
    if (threadIdx.x == 0) {
        sh_aw = v.centring == 1 ? uniform_aw(v, lam) : dvd(mul(v.A0, lam), sqr_t((double)n));
        if (blockIdx.x == 0) v.big->ext = add(v.rc, mul(0.25, sh_aw)) + 1e-9;
    }
    __syncthreads();
    const double Aw = sh_aw;
    const double p[3] = {B.p[0], B.p[1], B.p[2]};
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int m = v.s_ids[k];
        v.bead[m].mark = B.tag;
        v.s_slot[m] = k;
        double d[3] = {v.s_d[4 * k], v.s_d[4 * k + 1], v.s_d[4 * k + 2]}, dl[3];
        if (v.precision == 0) wavelet_disp64(d, v.s_d[4 * k + 3], lam, Aw, p, dl);
        else wavelet_disp32(d, lam, Aw, p, dl);
        const Bead bm = v.bead[m];
        const double o[3] = {bm.x, bm.y, bm.z};
        int im[3] = {0, 0, 0};
        for (int a = 0; a < 3; a++) {
            v.s_new[3 * k + a] = wrap(add(o[a], dl[a]), v.L, &im[a]);
            v.s_d[4 * k + a] = dl[a];          // the displacement, for the partner box
        }
        v.s_img[k] = pack_img(im[0], im[1], im[2]);
    }
}

// energy change, eight lanes per member: external well, bonds, WCA with every bead in the member's
// partner box, whose rows (y, z) the lanes share; per-block partial sums in pw_part. A support of a few
// thousand beads is only a few blocks of one thread per member, each walking its ~27-64 cells one after
// another: 250 us at 4,000 members (one thread) before.
constexpr int kBigLanes = 8;
__global__ void __launch_bounds__(256) k_big_energy(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(l >= gv.nL || !((gv.big_layers >> l) & 1) || !gv.big->active ||
                (int)(blockIdx.x * (blockDim.x / kBigLanes)) >= gv.big->n || (int)blockIdx.x >= gv.pw_blocks)
    SIM_PROLOGUE
    __shared__ double red[8];
    const BigMove& B = *v.big;
    const int n = B.n;
    const uint32_t tag = B.tag;
    const double L = v.L, hL = v.halfL;
    const Pot& P = v.pot;
    const int sub_ = threadIdx.x % kBigLanes;
    // binary32 screen of the pairs at the cutoff widened by five times the rounding of near32
    const float rcm = (float)v.rc * (1.0f + 1e-6f) + 1e-6f * (float)L, rcm2 = rcm * rcm * (1.0f + 1e-6f);
    double dU = 0.0;
    long long pe = 0;
    // over this simulation's own blocks (a batch's grid is that of its largest member)
    const int stride = min((int)gridDim.x, v.pw_blocks) * (256 / kBigLanes);
    for (int k0 = blockIdx.x * (256 / kBigLanes); k0 < n; k0 += stride) {
        const int k = k0 + (int)threadIdx.x / kBigLanes;
        if (k >= n) continue;
        const int m = v.s_ids[k];
        const Bead bm = v.bead[m];
        const double o[3] = {bm.x, bm.y, bm.z};
        const double nw[3] = {v.s_new[3 * k], v.s_new[3 * k + 1], v.s_new[3 * k + 2]};
        if (sub_ == 0) dU += U_ext(P, nw[0], nw[1], nw[2]) - U_ext(P, o[0], o[1], o[2]);
        if (sub_ < 2) {
            const int q = sub_ ? m + 1 : m - 1;
            if (q >= 0 && q < v.N && (sub_ ? v.bnext[m] : v.bnext[q])) {
                const Bead bq = v.bead[q];
                double qn[3] = {bq.x, bq.y, bq.z};
                const bool member = bq.mark == tag;
                if (!(member && q < m)) {
                    if (member) {
                        const int sq = v.s_slot[q];
                        qn[0] = v.s_new[3 * sq]; qn[1] = v.s_new[3 * sq + 1]; qn[2] = v.s_new[3 * sq + 2];
                    }
                    const double r2n = norm2(mi(nw[0] - qn[0], L, hL), mi(nw[1] - qn[1], L, hL), mi(nw[2] - qn[2], L, hL));
                    const double r2o = norm2(mi(o[0] - bq.x, L, hL), mi(o[1] - bq.y, L, hL), mi(o[2] - bq.z, L, hL));
                    dU += U_bond(P, r2n) - U_bond(P, r2o);
                }
            }
        }
        if (P.eps != 0.0) {
            const double ext = B.ext;
            double lo[3], hi[3];
            for (int a = 0; a < 3; a++) {
                const double u = add(o[a], v.s_d[4 * k + a]);
                lo[a] = sub(fmin(o[a], u), ext);
                hi[a] = add(fmax(o[a], u), ext);
            }
            int c0[3], nc[3];
            cell_box(v, lo, hi, c0, nc);
            // this lane's rows
            const int rows = nc[1] * nc[2];
            for (int r = sub_; r < rows; r += kBigLanes) {
                const int c1[3] = {c0[0], c0[1] + r % nc[1], c0[2] + r / nc[1]}, one[3] = {nc[0], 1, 1};
                for_occupied(v, c1, one, [&](int cell) {
                    int guard = 0;
                    for (int q = v.head[cell]; q >= 0;) {
                        const Bead bq = v.bead[q];
                        const int nx = bq.next;
                        if (q != m) {
                            const bool member = bq.mark == tag;
                            if (!(member && q < m)) {
                                const double qo[3] = {bq.x, bq.y, bq.z};
                                double qn[3] = {qo[0], qo[1], qo[2]};
                                if (member) {
                                    const int sq = v.s_slot[q];
                                    qn[0] = v.s_new[3 * sq]; qn[1] = v.s_new[3 * sq + 1]; qn[2] = v.s_new[3 * sq + 2];
                                }
                                const float fn = near32(nw, qn, (float)L, (float)hL), fo = near32(o, qo, (float)L, (float)hL);
                                if (fn < rcm2 || fo < rcm2) {
                                    const double r2n = norm2(mi(nw[0] - qn[0], L, hL), mi(nw[1] - qn[1], L, hL), mi(nw[2] - qn[2], L, hL));
                                    const double r2o = norm2(mi(o[0] - qo[0], L, hL), mi(o[1] - qo[1], L, hL), mi(o[2] - qo[2], L, hL));
                                    if (r2n < P.rc2 || r2o < P.rc2) { dU += U_wca(P, r2n) - U_wca(P, r2o); if (!member) pe++; }
                                }
                            }
                        }
                        q = nx;
                        if (++guard > kMaxWalk) { set_err(v, E_WALK); break; }
                    }
                });
            }
        }
    }
    dU = warp_sum(dU);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = dU;
    __syncthreads();
    if (threadIdx.x == 0) {
        double su = 0.0;
        for (int w = 0; w < 8; w++) su += red[w];
        v.pw_part[blockIdx.x] = su;
    }
    if (pe) atomicAdd(&v.ctr[C_PARTNER], (unsigned long long)pe);
}

// decision: the partials of the blocks that held members, summed in a fixed order
__global__ void __launch_bounds__(256) k_big_decide(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(l >= gv.nL || !((gv.big_layers >> l) & 1) || !gv.big->active)
    SIM_PROLOGUE
    __shared__ double red[8];
    BigMove& B = *v.big;
    const int n = B.n;
    const int nb = min((n + 256 / kBigLanes - 1) / (256 / kBigLanes), v.pw_blocks);   // the blocks that held members
    double su = 0.0;
    for (int b = threadIdx.x; b < nb; b += 256) su += v.pw_part[b];
    su = warp_sum(su);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = su;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double dU = 0.0;
    for (int w = 0; w < 8; w++) dU += red[w];
    const LayerDev& Ly = v.layer[l];
    const bool acc = (n == 0 ? 0.0 : dU) <= B.thr;   // an empty support moves nothing: dU = 0
    B.acc = acc;
    v.tr_out[Ly.tr_off + B.j] = (uint8_t)(acc ? 1 : 2);
    v.tr_n[Ly.tr_off + B.j] = n;
    v.tr_du[Ly.tr_off + B.j] = n == 0 ? 0.0 : dU;
    v.carry_serial[l] = acc ? 0.0 : B.lam;
    atomicAdd(&v.ctr[C_ATT + l], 1ull);
    atomicAdd(&v.ctr[C_BU], (unsigned long long)n);
    if (acc) {
        atomicAdd(&v.ctr[C_ACC + l], 1ull);
        atomicAdd(&v.ctr[C_ACCTOT], 1ull);
        if (n) atomicAdd(&v.ctr[C_MOVED], (unsigned long long)n);
    }
}

__global__ void k_big_commit(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(l >= gv.nL || !((gv.big_layers >> l) & 1) || !gv.big->active || !gv.big->acc || gv.big->n == 0)
    SIM_PROLOGUE
    const int n = v.big->n;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int m = v.s_ids[k];
        const Bead ob = v.bead[m];
        const int oc = cell_lin(v, ob.x, ob.y, ob.z), ncl = cell_lin(v, v.s_new[3 * k], v.s_new[3 * k + 1], v.s_new[3 * k + 2]);
        if (oc != ncl) {
            // the cell changes, relinked next (or, beyond what one block relinks, a rebuild)
            const int idx = atomicAdd(&v.big->nch, 1);
            v.s_changed[3 * idx] = m; v.s_changed[3 * idx + 1] = oc; v.s_changed[3 * idx + 2] = ncl;
        }
        put_bead(v.bead, v.bf, m, v.s_new[3 * k], v.s_new[3 * k + 1], v.s_new[3 * k + 2]);
        const int pk = v.s_img[k];
        if (pk != pack_img(0, 0, 0)) {
            int dd[3];
            unpack_img(pk, dd);
            v.img[3 * m] += dd[0]; v.img[3 * m + 1] += dd[1]; v.img[3 * m + 2] += dd[2];
        }
    }
}

// the cell changes of an accepted whole-GPU move relinked by one block, or (more than it holds,
// or lists left stale) the cell lists rebuilt by the launches after it
constexpr int kBigRelinkCap = 3072;
__global__ void __launch_bounds__(1024) k_big_relink(const SimView* __restrict__ vs, int l) {
    SIM_EXIT_IF(l >= gv.nL || !((gv.big_layers >> l) & 1) || !gv.big->active || !gv.big->acc || gv.big->n == 0)
    SIM_PROLOGUE
    const int nch = v.big->nch;
    // lists a shared-memory serial phase left stale cannot be relinked: rebuilt instead
    if (nch > kBigRelinkCap || *v.cl_stale) {
        if (threadIdx.x == 0) *v.pw_rebuild = 1;
        return;
    }
    __shared__ int cm[kBigRelinkCap], co[kBigRelinkCap], cn[kBigRelinkCap];
    for (int c = threadIdx.x; c < nch; c += blockDim.x) {
        cm[c] = v.s_changed[3 * c]; co[c] = v.s_changed[3 * c + 1]; cn[c] = v.s_changed[3 * c + 2];
    }
    __syncthreads();
    grouped_relink(v, cm, co, cn, nch, threadIdx.x, blockDim.x);
}
int launch_big(const SimView* d, const GroupDims& g, int l, int t, cudaStream_t s) {
    const int gb = (int)gx((g.maxN + 255) / 256, g.S);
    k_big_setup<<<dim3(1, g.S), 32, 0, s>>>(d, l, t);
    k_big_gather<<<dim3(gb, g.S), 256, 0, s>>>(d, l);
    k_big_disp<<<dim3(gb, g.S), 256, 0, s>>>(d, l);
    k_big_energy<<<dim3(g.pw_blocks, g.S), 256, 0, s>>>(d, l);
    k_big_decide<<<dim3(1, g.S), 256, 0, s>>>(d, l);
    k_big_commit<<<dim3(gb, g.S), 256, 0, s>>>(d, l);
    k_big_relink<<<dim3(1, g.S), 1024, 0, s>>>(d, l);
    launch_cl_rebuild(d, g, s, 1);
    return 10;
}

}  // namespace wmcd

namespace wmcd {

// ======================================================================================
// Staged concurrent wavelet moves. In a colour phase every queue owns the beads in the fine
// cells wholly inside its region (no other queue reads or writes them), so its warp copies
// them into shared memory once, runs all its moves there and writes them back at the end.
// Beads are assigned to regions by a counting sort over all beads before each colour phase.
// ======================================================================================
// The fine cells come from the binary32 shadows (the binary64 quotients of the definition made the
// count a binary64-bound pass: 150 us for 5 million beads), and the count's own atomics give each bead
// its rank in its queue (kept in s_slot, free between moves), so the placement needs none.
// With at most kRegionPriv queues per colour (coarse layers, whose regions hold thousands of
// beads each) the counts are kept per block in shared memory and added to the global ones once
// per block and queue: one global counter per queue would otherwise take an atomic per bead.
constexpr int kRegionPriv = 8192;
__global__ void k_region_count(const SimView* __restrict__ vs, int l, int colour) {
    SIM_EXIT_IF(!sched_on(gv, l) || colour >= gv.K * gv.K * gv.K)
    SIM_PROLOGUE
    if (!sched_on(v, l) || colour >= v.K * v.K * v.K) return;
    const int K = v.K, Gf = v.Gf, Q = sched_layer(v, l).G / K, nq = Q * Q * Q;
    const int ox = colour % K, oy = (colour / K) % K, oz = colour / (K * K);
    const int* tab = v.axis_tab + (size_t)l * K * Gf;
    __shared__ int sh[kRegionPriv];
    const bool priv = nq <= kRegionPriv;
    if (priv) {
        for (int i = threadIdx.x; i < nq; i += blockDim.x) sh[i] = 0;
        __syncthreads();
    }
    const int64_t m0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, ms = (int64_t)gridDim.x * blockDim.x;
    for (int64_t m = m0; m < v.N; m += ms) {
        const BeadF f = v.bf[m];
        const Bead* const b = &v.bead[m];            // read only near a cell face
        const int qx = tab[ox * Gf + fine_cell32(v, f.hx, &b->x)];
        const int qy = tab[oy * Gf + fine_cell32(v, f.hy, &b->y)];
        const int qz = tab[oz * Gf + fine_cell32(v, f.hz, &b->z)];
        const int key = (qx < 0 || qy < 0 || qz < 0) ? -1 : qx + Q * (qy + Q * qz);
        v.rkey[m] = key;
        if (key >= 0) v.s_slot[m] = atomicAdd(priv ? &sh[key] : &v.rcount[key], 1);
    }
    if (priv) {
        __syncthreads();
        for (int i = threadIdx.x; i < nq; i += blockDim.x)
            if (sh[i]) sh[i] = atomicAdd(&v.rcount[i], sh[i]);
        __syncthreads();
        for (int64_t m = m0; m < v.N; m += ms) {
            const int key = v.rkey[m];
            if (key >= 0) v.s_slot[m] += sh[key];
        }
    }
}
// Bead ids grouped by queue (the order within a queue is immaterial: a staged region is
// searched as a set).
__global__ void k_region_scatter(const SimView* __restrict__ vs, int l, int colour) {
    SIM_EXIT_IF(!sched_on(gv, l) || colour >= gv.K * gv.K * gv.K)
    SIM_PROLOGUE
    if (!sched_on(v, l) || colour >= v.K * v.K * v.K) return;
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < v.N; m += (int64_t)gridDim.x * blockDim.x) {
        const int key = v.rkey[m];
        if (key >= 0) v.rlist[v.rstart[key] + v.s_slot[m]] = (int)m;
    }
}

// What a move needs of its queue's region: fine cells of the interior, origin (also as a binary32
// pair) and side per axis.
struct Region {
    int64_t lo[3], hi[3];
    double org[3];
    float oh[3], ol[3], side[3], maxside;
};
// Shared memory of one queue. A lane addresses an axis of a bead at a cap + t.
struct Stage {
    Region* reg;
    double* px;                      // staged positions (binary64, wrapped)
    float* hi;                       // position relative to the region origin: hi part ...
    float* lo;                       // ... and lo part (hi + lo carries the binary64 value)
    float4* grp;                     // bounding ball of the staged beads 32 g .. 32 g + 31
    int *sid, *sdim;                 // bead id; image change | dirty
    short *up, *dn;                  // staged index of the bonded neighbours: -1 no bond, -2 not staged
    double *clam, *cV, *cp, *cthr;   // slot chunk: scale, centre offset, polarisation, threshold
    double *cA0l, *cilam;            // ... A0 lam and 1 / lam for the slot's own scale
    float *cpf, *cthrf, *clamf;      // ... binary32 forms of p, the threshold and the scale
    int *cj, *cti;                   // ... slot id, staged index of the picked bead (-1: not staged)
    char* scr;                       // per-warp scratch: warp 0's, then the others'
    int cap;                         // staged beads
};
constexpr int kQueueMem = 32;        // support members of the warps beyond a queue's first
constexpr int kLightChunk = 16;      // slots prepared together by a light warp (a queue has about three)
__host__ __device__ constexpr int stage_chunk(bool light) { return light ? kLightChunk : kSlotChunk; }
// bytes of one queue's shared memory: `warps` warps run it, the first with room for ncap members
__host__ __device__ inline size_t stage_bytes(int cap, int ncap, int warps, bool light) {
    const size_t groups = light ? 0 : (size_t)((cap + 31) / 32) * 16;
    return (((size_t)cap * (3 * 8 + 6 * 4 + 4 + 4 + 2 + 2) + 15) & ~(size_t)15) + groups +
           (size_t)stage_chunk(light) * (8 + 24 + 24 + 8 + 8 + 8 + 12 + 4 + 4 + 4 + 4) + warp_scr_bytes(ncap) + sizeof(Region) +
           (size_t)(warps - 1) * warp_scr_bytes(kQueueMem) + 48;
}
__device__ inline Stage stage_carve(char* base, int cap, bool light) {
    Stage S;
    S.cap = cap;
    const int ch = stage_chunk(light);
    char* p = base;
    auto take = [&](size_t bytes) { char* q = p; p += bytes; return q; };
    S.reg = (Region*)take((sizeof(Region) + 15) & ~(size_t)15);
    if (!light) S.grp = (float4*)take((size_t)((cap + 31) / 32) * 16);
    S.px = (double*)take((size_t)24 * cap);
    S.clam = (double*)take(8 * ch); S.cV = (double*)take(24 * ch); S.cp = (double*)take(24 * ch); S.cthr = (double*)take(8 * ch);
    S.cA0l = (double*)take(8 * ch); S.cilam = (double*)take(8 * ch);
    S.hi = (float*)take((size_t)12 * cap); S.lo = (float*)take((size_t)12 * cap);
    S.sid = (int*)take((size_t)4 * cap); S.sdim = (int*)take((size_t)4 * cap);
    S.cpf = (float*)take(12 * ch); S.cthrf = (float*)take(4 * ch); S.clamf = (float*)take(4 * ch);
    S.cj = (int*)take(4 * ch); S.cti = (int*)take(4 * ch);
    S.up = (short*)take((size_t)2 * cap); S.dn = (short*)take((size_t)2 * cap);
    S.scr = base + (((p - base) + 7) & ~7);
    return S;
}
// Coordinate (h, lo as the shadow holds it) relative to o = oh + ol, brought into [0, L), as a
// binary32 pair: exact differences of the hi parts (two-sum), the lo parts added, about 2^-48 of the
// box off, without binary64 arithmetic
__device__ __forceinline__ void local32(float h, float lo, float oh, float ol, float Lh, float Ll, float& hi, float& low) {
    auto plus = [](float& s, float& t, float bh, float bl) {     // (s, t) + (bh, bl)
        const float x = s + bh, bp = x - s;
        t += ((s - (x - bp)) + (bh - bp)) + bl;
        s = x;
    };
    float s = h, t = lo;
    plus(s, t, -oh, -ol);
    if (s + t < 0.0f) plus(s, t, Lh, Ll);
    else if (s + t >= Lh) plus(s, t, -Lh, -Ll);
    hi = s + t;
    low = t - (hi - s);
}
// coordinate relative to the region origin o, brought into [0, L), as a binary32 pair hi + lo
__device__ __forceinline__ void local_split(double x, double o, double L, float& hi, float& lo) {
    double t = sub(x, o);
    if (lt_zero(t)) t = add(t, L);
    else if (ge_pos(t, L)) t = sub(t, L);
    hi = (float)t;
    lo = (float)sub(t, (double)hi);
}

// What the warps of a queue's block share besides its Stage.
struct QueueSh {
    WarpRec rec[8];
    int item, nch;
    int cnt[512];                    // counting sort of the staged beads by cell of the region
    int scan[33];
};
// binary32 constants of a launch
struct Stage32 {
    float A0, reach, rcs, kT9;
};
// One move of a staged queue by one warp: slot c of the chunk on scale lam (own: that of slot sl, whose
// other forms are at hand), into rec.
template <int PREC, bool GROUPS>
__device__ __forceinline__ void stage_move(const SimView& v, const Stage& S, const Stage32& C, const Pot32& P32, int ns,
                                           int ls, int c, double lam, bool own, int sl, const WarpScr& W, int mem, int lane,
                                           WarpRec& rec) {
    const unsigned FULL = 0xffffffffu;
    const double L = v.L, hL = v.halfL;
    const int cap = S.cap, ax = lane % 3;
    const bool uni = v.centring == 1;
    const Region& Rg = *S.reg;
    const Box B{S.px, S.hi, S.lo, cap, ns, L, hL, 0.0f, 0.0f};
    rec.known = 2; rec.n = 0; rec.acc = 0; rec.pe = 0; rec.re = 0; rec.lam = lam; rec.du = 0.0;
    rec.wr = 0.0f; rec.rr = -1e30f;
    rec.b[0] = rec.b[1] = rec.b[2] = 0.0f;
    const int ti = S.cti[c];
    if (ti < 0 && !uni) return;                   // the picked bead lies outside the region interior
    // centre b = r_i + lam V (Appendix D), wrapped; binary64 because the region rule and the support
    // must match the sequential definition exactly; one axis per lane. Relative to the region origin
    // in binary32 (from the picked bead's staged coordinates) its error, a few 1e-7 of the region
    // side plus lam, is far inside the margins of the screens below.
    const double lV = uni ? 0.0 : mul(lam, S.cV[3 * c + ax]);
    const double ba = uni ? S.cV[3 * c + ax] : wrap_u(add(S.px[ax * cap + ti], lV), L, FULL, nullptr);
    const float lamf = own ? S.clamf[sl] : (float)lam;
    float bl;
    if (uni) {
        float h_, l_;
        local_split(ba, Rg.org[ax], L, h_, l_);
        bl = h_ + l_;
    } else {
        bl = (S.hi[ax * cap + ti] + S.lo[ax * cap + ti]) + (float)lV;
    }
    const float bx = __shfl_sync(FULL, bl, 0), by = __shfl_sync(FULL, bl, 1), bz = __shfl_sync(FULL, bl, 2);
    rec.b[0] = bx; rec.b[1] = by; rec.b[2] = bz;
    const float eps = 1e-6f * (Rg.maxside + lamf) + 1e-9f;
    // region rule: a binary32 screen proves most balls well inside the region's interior; the others
    // take the binary64 cell indices of the definition
    double Aw = 0.0;
    float Rf = lamf * (1.0f + 0.25f * C.A0) + C.reach;
    if (uni) {
        Aw = uniform_aw(v, lam);
        Rf = lamf + (float)rule_disp(v, lam, Aw) + C.reach;
    }
    rec.rr = lamf + 2.0f * eps;
    bool inside = true;
    {
        const float side = Rg.side[ax], dm = 2e-6f * (side + Rf) + 1e-6f;
        const bool sure = bl - Rf >= dm && bl + Rf <= side - dm;
        if (!__all_sync(FULL, sure)) {
            const double R = add(add(lam, rule_disp(v, lam, Aw)), v.r_reach);
            const int64_t t0 = (int64_t)floor(mul(sub(ba, R), v.invf));
            const int64_t t1 = (int64_t)floor(mul(add(ba, R), v.invf));
            inside = range_inside(t0, t1, Rg.lo[ax], Rg.hi[ax], v.Gf);
        }
    }
    if (!__all_sync(FULL, inside)) return;
    // support and candidates in one binary32 pass over the staged beads (hi parts, with a margin
    // eps for their rounding); ties within eps of the sphere decided in binary64
    const float li = fmaxf(lamf - eps, 0.0f), lin = li * li, lout = (lamf + eps) * (lamf + eps);
    const float Rc = Rf + 2.0f * eps, rcand = Rc * Rc;
    // the amplitude of every support size up to 32, one per lane, ahead of the search
    const double A0l = own ? S.cA0l[sl] : mul(v.A0, lam);
    const float af_lane = PREC == 1 && !uni ? amp32(A0l, v.sq_tab[lane + 1], v.sq_tab[kNCap + 2 + lane]) : 0.0f;
    int n = 0, nc = 0;
    auto scan32 = [&](int t) {
        float d2 = 4.0f * rcand + 1.0f;
        if (t < ns) {
            const float dx = S.hi[t] - bx, dy = S.hi[cap + t] - by, dz = S.hi[2 * cap + t] - bz;
            d2 = dx * dx + dy * dy + dz * dz;
        }
        bool in = d2 < lin;
        const bool tie = !in && d2 <= lout;
        if (__any_sync(FULL, tie)) {
            double d[3] = {__shfl_sync(FULL, ba, 0), __shfl_sync(FULL, ba, 1), __shfl_sync(FULL, ba, 2)};
            if (tie) {
                for (int a = 0; a < 3; a++) d[a] = mi(sub(S.px[a * cap + t], d[a]), L, hL);
                in = norm2(d[0], d[1], d[2]) < mul(lam, lam);
            }
        }
        const bool cd = !in && d2 < rcand;
        const unsigned vi = __ballot_sync(FULL, in), vc = __ballot_sync(FULL, cd), below = (1u << lane) - 1u;
        if (in) { const int k = n + __popc(vi & below); if (k < mem) W.mid[k] = (unsigned short)t; }
        if (cd) { const int k = nc + __popc(vc & below); if (k < kWarpCand) W.cand[k] = (unsigned short)t; }
        n += __popc(vi);
        nc += __popc(vc);
    };
    if (GROUPS) {
        const int ngrp = (ns + 31) >> 5;
        for (int g0 = 0; g0 < ngrp; g0 += 32) {
            bool hit = false;
            if (g0 + lane < ngrp) {
                const float4 q = S.grp[g0 + lane];
                const float dx = q.x - bx, dy = q.y - by, dz = q.z - bz, rg = Rc + q.w;
                hit = dx * dx + dy * dy + dz * dz <= rg * rg;
            }
#pragma unroll 1
            for (unsigned bits = __ballot_sync(FULL, hit); bits; bits &= bits - 1u) scan32(32 * (g0 + __ffs(bits) - 1) + lane);
        }
    } else {
#pragma unroll 1
        for (int t0 = 0; t0 < ns; t0 += 32) scan32(t0 + lane);
    }
    __syncwarp();                                 // support and candidate lists are read by every lane
    rec.n = n;
    if (n > sched_ncap(v, ls)) return;            // deferred
    if (n > mem) { rec.known = 0; return; }
    if (n == 0) { rec.known = 1; rec.acc = 0.0 <= S.cthr[c]; return; }   // no bead moves: dU = 0 against the threshold
    // bonded partners: staged (inside the region) or the move is deferred
    bool bad = false;
    for (int k = lane; k < n; k += 32) bad = bad || S.up[W.mid[k]] == -2 || S.dn[W.mid[k]] == -2;
    if (__any_sync(FULL, bad)) return;
    rec.known = 1;
    // displacement (Sec. V.A) with A_w = A0 lam / sqrt(n) (Eq. 29)
    float af;
    if (!uni && n > kNCap) Aw = dvd(A0l, sqr_t((double)n));
    else if (!uni && PREC == 0) Aw = div_by(A0l, v.sq_tab[n], v.sq_tab[kNCap + 1 + n]);
    if (uni || PREC == 0 || n > kNCap) af = (float)Aw;
    else af = n <= 32 ? __shfl_sync(FULL, af_lane, n - 1) : amp32(A0l, v.sq_tab[n], v.sq_tab[kNCap + 1 + n]);
    const double ilam = PREC == 1 ? 0.0 : own ? S.cilam[sl] : dvd(1.0, lam);
    move_disp<PREC, false>(B, W, n, ba, &S.cp[3 * c], &S.cpf[3 * c], lam, ilam, lamf, Aw, af, lane);
    rec.wr = lamf + 0.25f * af * 1.00001f;
    const float disp = 0.25f * af * 1.00001f, rs = C.rcs + disp + 2.0f * eps, b3[3] = {bx, by, bz};
    float bond2 = 0.0f;                           // farthest bonded partner read, from the centre
    auto member = [&](int t) {
        int lo_ = 0, hi_ = n - 1;
        while (lo_ <= hi_) {
            const int m = (lo_ + hi_) >> 1, x = W.mid[m];
            if (x == t) return true;
            if (x < t) lo_ = m + 1; else hi_ = m - 1;
        }
        return false;
    };
    auto terms = [&](auto&& pairs) {
        for_terms<false>(B, W, n, nc, nc > kWarpCand, P32.bond != 0, P32.eps_on, rs, disp, b3, &bond2, lane,
            [&](int k, int e) { return (int)(e ? S.up[W.mid[k]] : S.dn[W.mid[k]]); },
            [&](int k1, int k2) { return S.up[W.mid[k1]] == W.mid[k2] || S.up[W.mid[k2]] == W.mid[k1]; }, member, pairs);
    };
    move_decide<PREC, false>(v, B, W, P32, n, C.kT9, S.cthr[c], S.cthrf[c], lane, terms, rec);
    rec.rr = fmaxf(rec.wr + C.rcs, sqrtf(bond2)) + 2.0f * eps;
}
// the accepted move q of a warp's scratch takes place in the staged region
template <bool GROUPS>
__device__ __forceinline__ void stage_commit(const Stage& S, const WarpScr& W, int n, int lane) {
    const int cap = S.cap, mk = lane / 3, ax = lane - 3 * mk;
    for (int k0 = 0; k0 < n; k0 += 10) {
        const int k = k0 + mk;
        if (lane < 30 && k < n) {
            const int t = W.mid[k];
            S.px[ax * cap + t] = W.nw[3 * k + ax];
            S.hi[ax * cap + t] = W.nh[3 * k + ax];
            S.lo[ax * cap + t] = W.nl[3 * k + ax];
            if (ax == 0) {
                // accumulate the image change (3 fields of 8 bits, offset 128) and mark dirty (bit 24)
                int dd[3];
                const int cur = S.sdim[t];
                unpack_img(W.img[k], dd);
                const int x = ((cur & 0xff) - 128) + dd[0], y = (((cur >> 8) & 0xff) - 128) + dd[1], z = (((cur >> 16) & 0xff) - 128) + dd[2];
                S.sdim[t] = (x + 128) | ((y + 128) << 8) | ((z + 128) << 16) | (1 << 24);
            }
        }
    }
    if (GROUPS) {
        __syncwarp();
        for (int k = lane; k < n; k += 32) {
            const int t = W.mid[k];
            const float4 q = S.grp[t >> 5];
            const float dx = S.hi[t] - q.x, dy = S.hi[cap + t] - q.y, dz = S.hi[2 * cap + t] - q.z;
            atomicMax((int*)&S.grp[t >> 5].w, __float_as_int(sqrtf(dx * dx + dy * dy + dz * dz) * 1.000001f + 1e-6f));
        }
    }
}

// Write staged bead t (bead m) back: position, shadow, image counters; its fine cell before (from its
// record) and after.
__device__ __forceinline__ void stage_write(const SimView& v, const Stage& S, int t, int m, int* oldcell, int* newcell) {
    const int dm = S.sdim[t];
    const Bead ob = v.bead[m];
    const BeadF of = v.bf[m];
    *oldcell = fine_cell32(v, of.hx, ob.x) + v.Gf * (fine_cell32(v, of.hy, ob.y) + v.Gf * fine_cell32(v, of.hz, ob.z));
    const double x = S.px[t], y = S.px[S.cap + t], z = S.px[2 * S.cap + t];
    BeadF f;
    f.hx = (float)x; f.hy = (float)y; f.hz = (float)z;
    f.lx = (float)(x - (double)f.hx); f.ly = (float)(y - (double)f.hy); f.lz = (float)(z - (double)f.hz);
    f.pad0 = 0.0f; f.pad1 = 0.0f;
    v.bead[m].x = x; v.bead[m].y = y; v.bead[m].z = z;
    v.bf[m] = f;
    const int ax = (dm & 0xff) - 128, ay = ((dm >> 8) & 0xff) - 128, az = ((dm >> 16) & 0xff) - 128;
    if (ax | ay | az) { v.img[3 * m] += ax; v.img[3 * m + 1] += ay; v.img[3 * m + 2] += az; }
    *newcell = fine_cell32(v, f.hx, x) + v.Gf * (fine_cell32(v, f.hy, y) + v.Gf * fine_cell32(v, f.hz, z));
}

// One colour phase, split by the beads of a queue's region into launches of disjoint queues (so the
// split changes nothing in the results):
// VAR 1 (light, up to kLightCap beads): one warp per queue, several queues per block, moves in turn.
// VAR 2 or, in a phase of few queues, VAR 3 with twice the warps (middle, up to kMidCap) and VAR 0 (the rest): a block per queue, taken from the phase's list of
// dense regions until it is done (list = 1 or 2), or queue blockIdx.x (list = 0). Its warps evaluate
// the queue's next moves ahead of their turn (window_walk; hypothesis = warp), and the staged beads are
// sorted by cell of the region in groups of 32 with a bounding ball each, so a move looks at the few
// groups its reach meets. VAR 0 has eight warps, the most staging a block
// can have, and a path through the global cell lists for regions beyond that.
template <bool LIGHT>
__device__ __forceinline__ auto* queue_scratch() {
    struct None { int item, nch, cnt[1], scan[1]; WarpRec rec[1]; };   // a light warp shares nothing
    __shared__ std::conditional_t<LIGHT, None, QueueSh> s;
    return &s;
}
template <int VAR> __host__ __device__ constexpr int stage_threads() { return VAR == 0 || VAR == 3 ? 256 : 128; }
template <int PREC, int VAR>
__global__ void __launch_bounds__(stage_threads<VAR>(), VAR == 0 ? 1 : VAR == 3 ? 2 : 4) k_colour_staged(const SimView* __restrict__ vs, int l, int colour,
                                                                                  int cap, int qpb, int ncap, int stride,
                                                                                  int max_slots, int ns_lo, int ns_hi, int list) {
    SIM_EXIT_IF(!sched_on(gv, l) || gv.precision != PREC || colour >= gv.K * gv.K * gv.K ||
                (list ? (int)blockIdx.x >= gv.hq_ctl[list == 2 ? 2 : 0]
                      : ((int)(blockIdx.x * qpb) >= (sched_layer(gv, l).G / gv.K) * (sched_layer(gv, l).G / gv.K) * (sched_layer(gv, l).G / gv.K))))
    SIM_PROLOGUE
    extern __shared__ __align__(16) char dsm[];
    if (!sched_on(v, l) || v.precision != PREC || colour >= v.K * v.K * v.K) return;
    constexpr bool LIGHT = VAR == 1;
    constexpr int NT = stage_threads<VAR>(), NW = NT / 32, CH = stage_chunk(LIGHT);
    auto& X = *queue_scratch<LIGHT>();
    __shared__ Stage32 C;
    if (threadIdx.x == 0) {
        C.A0 = (float)v.A0;
        C.reach = (float)v.r_reach;
        C.rcs = (float)(v.rc * (1.0 + 1e-6) + 1e-6);
        C.kT9 = 1e-9f * (float)v.kT;
    }
    __syncthreads();
    const uint64_t sweep = v.step[0];
    const int wid = (int)(threadIdx.x >> 5), lane = threadIdx.x & 31, tid = threadIdx.x;
    const unsigned FULL = 0xffffffffu;
    const LayerDev Ly = sched_layer(v, l);
    // random draws, counters and trace are the layer's own; a second colouring's moves carry flag 4
    const int lr = layer_real(l);
    const uint8_t tflag = l >= kLevel2 ? 4 : 0;
    const int G = Ly.G, K = v.K, Q = G / K, nq = Q * Q * Q;
    const Pot32 P32 = pot32(v.pot);
    // an upper bound of the side of a region (K cells of the grid, rounded to fine cells)
    const float Gside = (float)(v.L * K / G) * 1.00001f;
    const float Lh = (float)v.L, Ll = (float)(v.L - (double)Lh);
    // this warp's hypothesis (hw, hr) and the moves a window can reach
    int hw = 0, wmax = 0;
    const int nh = LIGHT || v.audit ? 1 : NW;
    if (!LIGHT) while ((hw + 1) * (hw + 2) / 2 <= wid) hw++;
    while (wmax * (wmax + 1) / 2 < nh) wmax++;
    const int hr = LIGHT ? 0 : wid - hw * (hw + 1) / 2;
    // threads of the queue: a warp (light) or the block
    const int ql = LIGHT ? lane : tid, qn = LIGHT ? 32 : NT;
    auto qsync = [&]() { if (LIGHT) __syncwarp(); else __syncthreads(); };
    for (int it = 0;; it++) {
        int q;
        if (list) {
            // list 1: the front of hq_list (regions up to the middle size), list 2: its back
            const int lc = list == 2 ? 2 : 0;
            if (tid == 0) X.item = atomicAdd(&v.hq_ctl[lc + 1], 1);
            __syncthreads();
            const int i = X.item;
            __syncthreads();                          // read by all before the next item is taken
            if (i >= v.hq_ctl[lc]) break;
            q = v.hq_list[list == 2 ? nq - 1 - i : i];
        } else {
            // (a block of the light launch goes on to further queues: its view and constants are copied once)
            q = (blockIdx.x + it * gridDim.x) * qpb + (LIGHT ? wid : 0);
            if (q >= nq) break;
        }
        const int key = colour * nq + q;
        const int start = v.q_start[key], cnt = v.q_count[key];
        const int rs = v.rstart[q], ns = v.rcount[q];
        if (cnt == 0 || cnt > max_slots || ns < ns_lo || ns > ns_hi) continue;   // no slots, or another launch runs the queue
        const Stage S = stage_carve(dsm + (LIGHT ? (size_t)wid * (size_t)stride : 0), cap, LIGHT);
        // the region, one axis per lane
        if (ql < 3) {
            const int e = ql == 0 ? K * (q % Q) + colour % K : ql == 1 ? K * ((q / Q) % Q) + (colour / K) % K : K * (q / (Q * Q)) + colour / (K * K);
            // ceil((2 e - (K - 1)) Gf / 2G) and floor((2 e + 2 + (K - 1)) Gf / 2G) - 1; Gf < 1291 and
            // G <= 256, so 32 bits hold them (the first numerator may be negative: 2 G Gf is added)
            const int lo = (int)((unsigned)((2 * e - (K - 1)) * v.Gf + 2 * G * v.Gf + 2 * G - 1) / (2u * G)) - v.Gf;
            const int hi = (int)((unsigned)((2 * e + 2 + (K - 1)) * v.Gf) / (2u * G)) - 1;
            const double hf = v.L / v.Gf, o = (double)lo * hf;
            S.reg->lo[ql] = lo;
            S.reg->hi[ql] = hi;
            S.reg->org[ql] = o;
            S.reg->oh[ql] = (float)o;
            S.reg->ol[ql] = (float)(o - (double)(float)o);
            S.reg->side[ql] = (float)((double)(hi - lo + 1) * hf);
            if (ql == 0) S.reg->maxside = Gside;
        }
        qsync();
        const Region& Rg = *S.reg;
        const int cell = K * (q % Q) + colour % K + G * (K * ((q / Q) % Q) + (colour / K) % K + G * (K * (q / (Q * Q)) + colour / (K * K)));
        double carry = v.carry_q[Ly.carry_off + cell];      // alike in every thread of the queue
        int att = 0, acc = 0, def = 0, pe = 0, rechecks = 0;
        long long bu = 0, moved = 0;
        if (VAR == 0 && ns > cap) {
            // region too full for shared memory: the global-memory path
            if (wid == 0) {
                // (its scratch takes the place of the staged region)
                const int64_t rlo[3] = {Rg.lo[0], Rg.lo[1], Rg.lo[2]}, rhi[3] = {Rg.hi[0], Rg.hi[1], Rg.hi[2]};
                __syncwarp();
                WarpSmem& sm = *(WarpSmem*)dsm;
                for (int t = 0; t < cnt; t++) {
                    const int j = v.q_slots[start + t];
                    const double lam = carry > 0.0 ? carry : v.slot_lam[j];
                    int n = 0;
                    double du = 0.0;
                    int r = warp_attempt<PREC>(v, sm, l, j, v.slot_bead[j], lam, sweep, rlo, rhi, lane, &n, &pe, &rechecks, &du);
                    __syncwarp();
                    if (r == DEFER) { if (lane == 0) v.defer[start + t] = 1; def++; continue; }
                    att++; bu += n;
                    if (r == ACCEPT) { acc++; moved += n; }
                    if (lane == 0) {
                        v.tr_out[Ly.tr_off + j] = (uint8_t)((r == ACCEPT ? 1 : 2) | tflag);
                        v.tr_n[Ly.tr_off + j] = n;
                        v.tr_du[Ly.tr_off + j] = du;
                    }
                    carry = (r == ACCEPT) ? 0.0 : lam;
                }
            }
        } else {
            const int mem = LIGHT || wid == 0 ? ncap : kQueueMem;
            const WarpScr W = warp_scr(S.scr + (LIGHT || wid == 0 ? 0 : warp_scr_bytes(ncap) + (wid - 1) * warp_scr_bytes(kQueueMem)), mem);
            auto stage_bead = [&](int t, int m) {
                const Bead bb = v.bead[m];
                const BeadF f = v.bf[m];
                S.px[t] = bb.x; S.px[cap + t] = bb.y; S.px[2 * cap + t] = bb.z;
                local32(f.hx, f.lx, Rg.oh[0], Rg.ol[0], Lh, Ll, S.hi[t], S.lo[t]);
                local32(f.hy, f.ly, Rg.oh[1], Rg.ol[1], Lh, Ll, S.hi[cap + t], S.lo[cap + t]);
                local32(f.hz, f.lz, Rg.oh[2], Rg.ol[2], Lh, Ll, S.hi[2 * cap + t], S.lo[2 * cap + t]);
                S.sid[t] = m;
                S.sdim[t] = 128 | (128 << 8) | (128 << 16);
                v.s_slot[m] = t;                            // free between the moves of the serial phases
            };
            if (LIGHT) {
                for (int t = lane; t < ns; t += 32) stage_bead(t, v.rlist[rs + t]);
            } else {
                // counting sort by cell of the region, 8 per axis in Morton order, so that 32 consecutive
                // beads are close together
                auto part = [](float x, float o, float side, float Lb) {
                    float d = x - o;
                    if (d < 0.0f) d += Lb;
                    else if (d >= Lb) d -= Lb;
                    return max(0, min(7, (int)(8.0f * d / side)));
                };
                auto spread = [](int x) { return (x & 1) | ((x & 2) << 2) | ((x & 4) << 4); };
                for (int i = tid; i < 512; i += NT) X.cnt[i] = 0;
                __syncthreads();
                for (int t = tid; t < ns; t += NT) {
                    const BeadF f = v.bf[v.rlist[rs + t]];
                    const int k = spread(part(f.hx, Rg.oh[0], Rg.side[0], Lh)) | (spread(part(f.hy, Rg.oh[1], Rg.side[1], Lh)) << 1) |
                                  (spread(part(f.hz, Rg.oh[2], Rg.side[2], Lh)) << 2);
                    S.up[t] = (short)k;
                    atomicAdd(&X.cnt[k], 1);
                }
                __syncthreads();
                {
                    constexpr int PER = 512 / NT;
                    int x[PER], sum = 0, total;
                    for (int u = 0; u < PER; u++) { x[u] = X.cnt[PER * tid + u]; sum += x[u]; }
                    int pre = block_excl_scan<NW>(sum, X.scan, &total);
                    for (int u = 0; u < PER; u++) { X.cnt[PER * tid + u] = pre; pre += x[u]; }
                }
                __syncthreads();
                for (int t = tid; t < ns; t += NT) S.sid[atomicAdd(&X.cnt[S.up[t]], 1)] = v.rlist[rs + t];
                __syncthreads();
                for (int t = tid; t < ns; t += NT) stage_bead(t, S.sid[t]);
            }
            qsync();
            // staged indices of the bonded neighbours
            for (int t = ql; t < ns; t += qn) {
                const int m = S.sid[t];
                S.up[t] = !v.bnext[m] ? -1 : v.rkey[m + 1] == q ? (short)v.s_slot[m + 1] : -2;
                S.dn[t] = !(m > 0 && v.bnext[m - 1]) ? -1 : v.rkey[m - 1] == q ? (short)v.s_slot[m - 1] : -2;
            }
            if (!LIGHT) {
                const int ngrp = (ns + 31) / 32;
                for (int g = wid; g < ngrp; g += NW) {
                    // about the middle of the group's extent
                    const int t = min(32 * g + lane, ns - 1);
                    float mid[3], d2 = 0.0f;
                    for (int a = 0; a < 3; a++) {
                        const float x = S.hi[a * cap + t];   // not negative beyond rounding: order of the bits
                        const float hi_ = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(fmaxf(x, 0.0f))));
                        const float lo_ = __uint_as_float(__reduce_min_sync(FULL, __float_as_uint(fmaxf(x, 0.0f))));
                        mid[a] = 0.5f * (lo_ + hi_);
                        d2 += (x - mid[a]) * (x - mid[a]);
                    }
                    const float far_ = sqrtf(__uint_as_float(__reduce_max_sync(FULL, __float_as_uint(d2))));
                    if (lane == 0) S.grp[g] = make_float4(mid[0], mid[1], mid[2], far_ * 1.000001f + 1e-6f);
                }
            }
            int c0 = 0, c1 = 0;                       // slots of the chunk
            for (int t = 0; t < cnt;) {
                if (min(t + wmax, cnt) > c1) {
                    // slot parameters of the next slots: V (with uniform centres: the centre itself), p and
                    // the acceptance threshold as the slot kernel drew them (Appendix D, Eq. 20)
                    qsync();
                    c0 = t;
                    c1 = min(t + CH, cnt);
                    for (int e = ql; e < c1 - c0; e += qn) {
                        const int j = v.q_slots[start + c0 + e], i = v.slot_bead[j];
                        S.cj[e] = j;
                        const double lam = v.slot_lam[j];
                        S.clam[e] = lam;
                        S.clamf[e] = (float)lam;
                        S.cA0l[e] = mul(v.A0, lam);
                        if (PREC == 0) S.cilam[e] = dvd(1.0, lam);
                        S.cthr[e] = v.slot_thr[j];
                        for (int a = 0; a < 3; a++) {
                            S.cV[3 * e + a] = v.slot_V[3 * j + a];
                            S.cp[3 * e + a] = v.slot_p[3 * j + a];
                            S.cpf[3 * e + a] = (float)S.cp[3 * e + a];
                        }
                        S.cthrf[e] = (float)S.cthr[e];
                        S.cti[e] = v.rkey[i] == q ? v.s_slot[i] : -1;
                    }
                    qsync();
                }
                WarpRec rec;
                int steps = 1;
                bool mine = true;
                if (LIGHT) {
                    const bool own = !(__double_as_longlong(carry) > 0);
                    stage_move<PREC, false>(v, S, C, P32, ns, l, t - c0, own ? S.clam[t - c0] : carry, own, t - c0, W, mem, lane, rec);
                    if (rec.known == 1) carry = rec.acc ? 0.0 : rec.lam;
                } else {
                    rec.known = 0;
                    if (wid < nh && t + hw < cnt) {
                        // the carried scale, or that of the slot the run of rejections started with
                        const bool own = !(hr == hw && __double_as_longlong(carry) > 0);
                        const int sl = t + hw - hr - c0;
                        stage_move<PREC, true>(v, S, C, P32, ns, l, t + hw - c0, own ? S.clam[sl] : carry, own, sl, W, mem, lane, rec);
                    }
                    if (lane == 0) X.rec[wid] = rec;
                    __syncthreads();
                    int taken;
                    steps = window_walk(X.rec, nh, cnt - t, 1e30f, 1e29f, 1e-3f + 2e-6f * Rg.maxside, 0.0f, wid, lane, &taken, &carry);
                    mine = taken != 0;
                }
                if (mine) {
                    const int j = S.cj[t + hw - c0];
                    if (rec.known == 2) {
                        if (lane == 0) v.defer[start + t + hw] = 1;
                        def++;
                    } else {
                        att++;
                        bu += rec.n;
                        pe += rec.pe;
                        rechecks += rec.re;
                        if (rec.acc) {
                            acc++;
                            moved += rec.n;
                            if (rec.n) stage_commit<!LIGHT>(S, W, rec.n, lane);
                        }
                        if (lane == 0) {
                            v.tr_out[Ly.tr_off + j] = (uint8_t)((rec.acc ? 1 : 2) | tflag);
                            v.tr_n[Ly.tr_off + j] = rec.n;
                            v.tr_du[Ly.tr_off + j] = rec.du;
                        }
                    }
                }
                qsync();
                t += steps;
            }
            // write back the moved beads; the fine cell of each before and after (the old one from the
            // bead's record, which nothing else writes during the phase)
            if (LIGHT) {
                for (int base = 0; base < ns; base += 32) {
                    const int t = base + lane;
                    int newcell = -1, oldcell = -1, m = 0;
                    if (t < ns && (S.sdim[t] & (1 << 24))) {
                        m = S.sid[t];
                        stage_write(v, S, t, m, &oldcell, &newcell);
                    }
                    // cell-list moves one after another, in staged order
                    for (unsigned bits = __ballot_sync(FULL, newcell != oldcell); bits; bits &= bits - 1u) {
                        if (lane == __ffs(bits) - 1) relink(v, m, oldcell, newcell);
                        __syncwarp();
                    }
                }
            } else {
                // cell-list moves by one thread per cell, as many at a time as the scratch lists hold
                int* const cm = (int*)S.scr;
                constexpr int LC = 256;
                for (int base = 0; base < ns; base += LC) {
                    if (tid == 0) X.nch = 0;
                    __syncthreads();
                    for (int t = base + tid; t < min(ns, base + LC); t += NT) {
                        if (!(S.sdim[t] & (1 << 24))) continue;
                        const int m = S.sid[t];
                        int oldcell, newcell;
                        stage_write(v, S, t, m, &oldcell, &newcell);
                        if (oldcell != newcell) {
                            const int e = atomicAdd(&X.nch, 1);
                            cm[e] = m; cm[LC + e] = oldcell; cm[2 * LC + e] = newcell;
                        }
                    }
                    __syncthreads();
                    if (X.nch) grouped_relink(v, cm, cm + LC, cm + 2 * LC, X.nch, tid, NT);
                    __syncthreads();
                }
            }
        }
        if (lane == 0 && (att | def)) {
            atomicAdd(&v.ctr[C_ATT + lr], (unsigned long long)att);
            atomicAdd(&v.ctr[C_ACC + lr], (unsigned long long)acc);
            if (l < kLevel2 && def) atomicAdd(&v.ctr[C_DEF + lr], (unsigned long long)def);   // first deferrals only
            atomicAdd(&v.ctr[C_ACCTOT], (unsigned long long)acc);
            atomicAdd(&v.ctr[C_BU], (unsigned long long)bu);
            atomicAdd(&v.ctr[C_CBU], (unsigned long long)bu);
            atomicAdd(&v.ctr[C_CMOVED], (unsigned long long)moved);
            atomicAdd(&v.ctr[C_MOVED], (unsigned long long)moved);
            if (pe) { atomicAdd(&v.ctr[C_PARTNER], (unsigned long long)pe); atomicAdd(&v.ctr[C_CPE], (unsigned long long)pe); }
            if (rechecks) atomicAdd(&v.ctr[C_RECHECK], (unsigned long long)rechecks);
        }
        if (lane == 0 && (LIGHT || wid == 0)) v.carry_q[Ly.carry_off + cell] = carry;
        qsync();                                      // the next queue reuses the shared memory
    }   // queues
}

// the launch of ordinary regions: regions of at most kLightCap beads, up to kMaxStageWarps queues per block
// the dense regions: up to kMidCap beads by blocks of four warps, three or more per SM; the larger ones
// by blocks of eight with the most shared memory
constexpr int kMidCap = 640;
// (a light warp's supports are at most its region's kLightCap beads)
static int light_ncap(int ncap) { return ncap < kLightCap ? ncap : kLightCap; }
static size_t light_stride(int ncap) { return (stage_bytes(kLightCap, light_ncap(ncap), 1, true) + 15) & ~(size_t)15; }
static size_t mid_bytes(int ncap, int warps) { return stage_bytes(kMidCap, ncap, warps, false); }
// largest support of schedule index l's concurrent moves over the group
static int sched_ncap_g(const GroupDims& g, int l) { return l >= kLevel2 ? kNCapMax : g.ncap; }
// most beads a block of one queue can stage: dynamic shared memory + the static view copy, tables and
// queue scratch within the 227 KB of a block (and the global-memory path's scratch, which is smaller)
static size_t heavy_bytes(int cap, int ncap) {
    const size_t b = stage_bytes(cap, ncap, stage_threads<0>() / 32, false);
    return b > sizeof(WarpSmem) ? b : sizeof(WarpSmem);
}
int staged_cap_max(int ncap) {
    int cap = 256;
    while (heavy_bytes(cap + 32, ncap) + sizeof(SimView) + sizeof(QueueSh) + 512 <= 227u * 1024u) cap += 32;
    return cap;
}

// The largest dynamic shared memory each kernel was opened for, per device: raised before a launch needs
// more, so that launches recorded into a graph set nothing.
static RaisedLimit g_staged_smem[64][2][3], g_serial_smem[64][2], g_serial_opened[64];
template <class... K> static bool open_smem(int bytes, K... kernels) {
    bool ok = true;
    ((ok = cudaFuncSetAttribute(kernels, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess && ok), ...);
    return ok;
}
void prepare_staged(const GroupDims& g) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    g_serial_opened[dev].raise(1, [](int) {
        return open_smem((int)serial_dyn_bytes<1, 512, ONE_BLOCK>(), k_serial<1, 512, ONE_BLOCK>) &&
               open_smem((int)serial_dyn_bytes<0, 512, ONE_BLOCK>(), k_serial<0, 512, ONE_BLOCK>) &&
               open_smem((int)serial_dyn_bytes<1, 512, SPEC_SERIAL>(), k_serial<1, 512, SPEC_SERIAL>) &&
               open_smem((int)serial_dyn_bytes<0, 512, SPEC_SERIAL>(), k_serial<0, 512, SPEC_SERIAL>) &&
               open_smem((int)serial_dyn_bytes<1, 512, SPEC_QUEUES>(), k_serial<1, 512, SPEC_QUEUES>) &&
               open_smem((int)serial_dyn_bytes<0, 512, SPEC_QUEUES>(), k_serial<0, 512, SPEC_QUEUES>);
    });
    if (g.smem_maxN > 0) {
        const int sm = (int)smem_serial_bytes(g.smem_maxN, 16);
        if (g.prec_mask & 1)
            g_serial_smem[dev][0].raise(sm, [](int b) { return open_smem(b, k_serial_smem<0, 128>, k_serial_smem<0, 256>, k_serial_smem<0, 512>); });
        if (g.prec_mask & 2)
            g_serial_smem[dev][1].raise(sm, [](int b) { return open_smem(b, k_serial_smem<1, 128>, k_serial_smem<1, 256>, k_serial_smem<1, 512>); });
    }
    int smem = 0, smemL = 0, smemM = 0;
    for (int i = 0; i < 2 * g.maxL; i++) {
        const int l = i < g.maxL ? i : kLevel2 + i - g.maxL;
        if (!g.coloured[l]) continue;
        const int ncap = sched_ncap_g(g, l);
        smemL = std::max(smemL, (int)(kMaxStageWarps * light_stride(ncap)));
        smemM = std::max(smemM, (int)mid_bytes(ncap, stage_threads<3>() / 32));
        smem = std::max(smem, (int)heavy_bytes(staged_cap_max(ncap), ncap));
    }
    if (g.prec_mask & 1) {
        g_staged_smem[dev][0][0].raise(smem, [](int b) { return open_smem(b, k_colour_staged<0, 0>); });
        g_staged_smem[dev][0][1].raise(smemL, [](int b) { return open_smem(b, k_colour_staged<0, 1>); });
        g_staged_smem[dev][0][2].raise(smemM, [](int b) { return open_smem(b, k_colour_staged<0, 2>, k_colour_staged<0, 3>); });
    }
    if (g.prec_mask & 2) {
        g_staged_smem[dev][1][0].raise(smem, [](int b) { return open_smem(b, k_colour_staged<1, 0>); });
        g_staged_smem[dev][1][1].raise(smemL, [](int b) { return open_smem(b, k_colour_staged<1, 1>); });
        g_staged_smem[dev][1][2].raise(smemM, [](int b) { return open_smem(b, k_colour_staged<1, 2>, k_colour_staged<1, 3>); });
    }
}

// Blocks a speculative serial launch can have resident at once (all of them wait for one another).
static int sm_count();
int spec_blocks_max() {
    prepare_staged(GroupDims());
    int most = kSpecMax / sm_count() + 1;
    auto fits = [&](const void* k, size_t dyn) {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, 512, dyn) != cudaSuccess) { cudaGetLastError(); per = 0; }
        most = std::min(most, per);
    };
    fits((const void*)k_serial<0, 512, SPEC_SERIAL>, serial_dyn_bytes<0, 512, SPEC_SERIAL>());
    fits((const void*)k_serial<1, 512, SPEC_SERIAL>, serial_dyn_bytes<1, 512, SPEC_SERIAL>());
    fits((const void*)k_serial<0, 512, SPEC_QUEUES>, serial_dyn_bytes<0, 512, SPEC_QUEUES>());
    fits((const void*)k_serial<1, 512, SPEC_QUEUES>, serial_dyn_bytes<1, 512, SPEC_QUEUES>());
    return std::max(1, std::min(kSpecMax, most * sm_count()));
}

// multiprocessors of the current device (cached per device)
static int sm_count() {
    static std::atomic<int> cache[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    int n = cache[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 1;
        cache[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

int launch_colour_staged(const SimView* d, const GroupDims& g, int l, int colour, cudaStream_t s, const ForkJoin* fj) {
    const int nq = g.nq[l];
    const int gb = (int)gx((g.maxN + 255) / 256, g.S);
    const int ncap = sched_ncap_g(g, l);
    const bool split = fj && fj->side[0];
    // which queues go to blocks, and how many warps these have
    const PhaseShape shape = phase_shape(nq, g.S, g.maxN, sm_count());
    const bool wide = shape.wide;
    const int slots = shape.slots;
    k_zero<<<dim3(gx((nq + 255) / 256, g.S), g.S), 256, 0, s>>>(d, 1, l);
    k_region_count<<<dim3(gb, g.S), 256, 0, s>>>(d, l, colour);
    const int scans = launch_scan(d, g, nq, 1, l, colour, split ? kLightCap : -1, slots, kMidCap, s);
    k_region_scatter<<<dim3(gb, g.S), 256, 0, s>>>(d, l, colour);
    prepare_staged(g);
    const int np = (g.prec_mask & 1) + ((g.prec_mask >> 1) & 1);
    const int capH = staged_cap_max(ncap), big = 1 << 30;
    const size_t smemH = heavy_bytes(capH, ncap);
    constexpr int NH = stage_threads<0>(), NM = stage_threads<2>(), NM8 = stage_threads<3>();
    // one launch per precision; each returns at once for simulations of the other precision
    if (!split) {
        const dim3 grid(nq, g.S);
        if (g.prec_mask & 1) k_colour_staged<0, 0><<<grid, NH, smemH, s>>>(d, l, colour, capH, 1, ncap, 0, big, 0, big, 0);
        if (g.prec_mask & 2) k_colour_staged<1, 0><<<grid, NH, smemH, s>>>(d, l, colour, capH, 1, ncap, 0, big, 0, big, 0);
        return 3 + scans + np;
    }
    // A layer whose average region is beyond half of what a block stages: the regions beyond it run
    // after the others by groups of blocks through the global cell lists (a lone simulation, all of
    // whose blocks fit the device at once); elsewhere a rare region of that size takes the dense
    // regions' own global-memory path (one warp: 50-250 us a move against about 30 in a block, several
    // moves at a time). 65k semi-dilute beads, layer 1's eight queues: 13 ms a phase -> 1.0 ms; 1M, layer
    // 2's 27 queues: 4.7 -> 1.1 ms.
    const bool queues = g.spec_blocks > 1 && g.S == 1 && (double)g.maxN / nq > 0.5 * capH;
    // Ordinary regions (at most kLightCap beads) on the stream, one warp per queue; the dense regions
    // (a chain's worth of beads, the longest queues of the phase) at the same time on side streams,
    // persistently over the lists the region scan made.
    const int qL = light_queues(g.block_warps), ncL = light_ncap(ncap);
    const dim3 gridL(std::min((nq + qL - 1) / qL, std::max(1, 16 * sm_count() / g.S)), g.S);
    const size_t strideL = light_stride(ncap), smemM = mid_bytes(ncap, NM / 32), smemM8 = mid_bytes(ncap, NM8 / 32);
    const dim3 gridH(std::min(nq, sm_count()), g.S), gridM(std::min(nq, 4 * sm_count()), g.S);
    cudaStream_t sm_ = fj->side[0], sh_ = fj->side[1] ? fj->side[1] : fj->side[0];
    cudaEventRecord(fj->fork, s);
    cudaStreamWaitEvent(sm_, fj->fork, 0);
    if (sh_ != sm_) cudaStreamWaitEvent(sh_, fj->fork, 0);
    if (g.prec_mask & 1) {
        if (wide) k_colour_staged<0, 3><<<gridM, NM8, smemM8, sm_>>>(d, l, colour, kMidCap, 1, ncap, 0, big, 0, kMidCap, 1);
        else k_colour_staged<0, 2><<<gridM, NM, smemM, sm_>>>(d, l, colour, kMidCap, 1, ncap, 0, big, 0, kMidCap, 1);
        k_colour_staged<0, 0><<<gridH, NH, smemH, sh_>>>(d, l, colour, capH, 1, ncap, 0, big, kMidCap + 1, queues ? capH : big, 2);
    }
    if (g.prec_mask & 2) {
        if (wide) k_colour_staged<1, 3><<<gridM, NM8, smemM8, sm_>>>(d, l, colour, kMidCap, 1, ncap, 0, big, 0, kMidCap, 1);
        else k_colour_staged<1, 2><<<gridM, NM, smemM, sm_>>>(d, l, colour, kMidCap, 1, ncap, 0, big, 0, kMidCap, 1);
        k_colour_staged<1, 0><<<gridH, NH, smemH, sh_>>>(d, l, colour, capH, 1, ncap, 0, big, kMidCap + 1, queues ? capH : big, 2);
    }
    if (g.prec_mask & 1) k_colour_staged<0, 1><<<gridL, qL * 32, qL * strideL, s>>>(d, l, colour, kLightCap, qL, ncL, (int)strideL, slots, 0, kLightCap, 0);
    if (g.prec_mask & 2) k_colour_staged<1, 1><<<gridL, qL * 32, qL * strideL, s>>>(d, l, colour, kLightCap, qL, ncL, (int)strideL, slots, 0, kLightCap, 0);
    cudaEventRecord(fj->join[0], sm_);
    cudaStreamWaitEvent(s, fj->join[0], 0);
    if (sh_ != sm_) {
        cudaEventRecord(fj->join[1], sh_);
        cudaStreamWaitEvent(s, fj->join[1], 0);
    }
    if (queues) {
        // blocks per queue: all of the device's over the queues of the phase, at most 21 (six moves ahead);
        // one where the caller chose a serial phase of one block: such a program shares the SMs with other
        // work, and blocks that wait for one another start only when all of them have room (65k semi-dilute
        // beads with it: 114 ms a sweep in groups, 127 with one block a queue, 208 with one warp)
        int group = g.serial_threads > 128 ? std::max(1, std::min(21, g.spec_blocks / nq)) : 1, above = capH;
        auto launch = [&](const void* k, dim3 grid, void** args, size_t dyn) {
            if (group > 1) cudaLaunchCooperativeKernel(k, grid, dim3(512), args, dyn, s);
            else cudaLaunchKernel(k, grid, dim3(512), args, dyn, s);
        };
        const dim3 gq((unsigned)(group * std::min(nq, g.spec_blocks / group)));
        void* args[] = {(void*)&d, (void*)&l, (void*)&colour, (void*)&group, (void*)&above};
        if (g.prec_mask & 1)
            launch((const void*)k_serial<0, 512, SPEC_QUEUES>, gq, args, serial_dyn_bytes<0, 512, SPEC_QUEUES>());
        if (g.prec_mask & 2)
            launch((const void*)k_serial<1, 512, SPEC_QUEUES>, gq, args, serial_dyn_bytes<1, 512, SPEC_QUEUES>());
    }
    return 3 + scans + 3 * np + (queues ? np : 0);
}

}  // namespace wmcd
