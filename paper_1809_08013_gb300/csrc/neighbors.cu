// neighbors.cu -- Algorithm 1 step 2: the neighbours and the smoothing length.
//
// Pair test. The definition is the FP64 test r_ij^2 < (2h)^2 with
// r^2 = (dx dx + dy dy) + dz dz, each operation rounded on its own (minimum
// image along z when periodic). GB300 issues FP64 at 1/64 of the FP32 rate,
// so candidates are classified in FP32 from float copies of the positions:
//   r2f < Tin   -> certainly inside,   r2f > Tout -> certainly outside,
//   otherwise   -> the exact FP64 test above decides.
// Tin/Tout come from a rigorous bound on the FP32 error evaluated with
// directed-rounding FP32 operations (thresholds()), so every decision equals
// the FP64 one and the neighbour sets are exact.
//
// h search (reading of the Section 3 footnote: h follows a target neighbour
// count): bracketing search using only correctly rounded * and +,
//   n < target - tol: lo = h; h = (hi == inf) ? 1.25 h : (lo + hi) / 2
//   n > target + tol: hi = h; h = (lo == 0)   ? 0.8 h  : (lo + hi) / 2
// for at most max_h_iter counts; the result is the last h counted.
//
// Symmetric set S_i = { j != i : r_ij < 2h_i or r_ij < 2h_j } as CSR: row i
// holds N_i (r_ij < 2h_i) first, then the rest.
//
// Work decomposition: a first count at the h a particle comes with, 32
// consecutive particles at a time, one lane each (k_h_count; ~98% of them need
// no more in a running simulation); those that go on, one warp per particle
// (k_h_iterate), which takes 32 candidates at a time with ballots and ballot
// prefix counts, so that a particle's own iteration count never stalls the
// others. A large instance of which much goes on (a first step) first takes
// further counts 32 particles at a time (k_h_union).
#include <math_constants.h>

#include <algorithm>
#include <type_traits>

#include "df.cuh"
#include "sph_internal.cuh"

namespace sph {

constexpr unsigned kFull = 0xffffffffu;

struct Thr {
    float tin, tout;
};

// FP32 classification thresholds for radius R = 2h (R > 0).
// The FP32 norm of a pair differs from the norm of the FP64 difference vector
// by at most d = sqrt(3) e, e = eC + eR R (see k_grid_setup); the FP32 sum of
// squares adds at most 3 * 2^-24 relative; the FP64 square differs from the
// FP64 norm squared by < 2^-50 relative. All operations round outward.
__device__ __forceinline__ Thr thresholds(double R, const Grid* __restrict__ g) {
    float Rl, Rh;
    f32_bounds(R, Rl, Rh);
    const float e = __fmaf_ru(g->eR, Rh, g->eC);
    const float d = __fmul_ru(1.7320525f, e);
    Thr t;
    const float a = __fsub_rd(__fmul_rd(Rl, 0.99999905f), d);  // Rl (1 - 2^-20) - d
    t.tin = a > 0.0f ? __fmul_rd(__fmul_rd(a, a), 0.9999997f) : -1.0f;
    const float b = __fadd_ru(__fmul_ru(Rh, 1.00000096f), d);   // Rh (1 + 2^-20) + d
    t.tout = __fmul_ru(__fmul_ru(b, b), 1.0000003f);
    if (g->periodic_z && Rh > 0.25f * g->lzf) {  // wrap decisions may differ: exact path only
        t.tin = -1.0f;
        t.tout = CUDART_INF_F;
    }
    return t;
}

__device__ __forceinline__ float f_r2(const float4& a, const float4& b, const Grid* __restrict__ g) {
    const float dx = a.x - b.x, dy = a.y - b.y;
    float dz = a.z - b.z;
    if (g->periodic_z) {
        if (dz > g->halflzf) dz -= g->lzf;
        else if (dz < -g->halflzf) dz += g->lzf;
    }
    return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}

// The defining FP64 squared distance, operation by operation.
__device__ __forceinline__ double exact_r2(const double4_32a& a, const double4_32a& b,
                                           const Grid* __restrict__ g) {
    return exact_r2_def(a, b, g->periodic_z != 0, g->lz);
}

__device__ __forceinline__ int wrapi(int k, int n) {
    int r = k % n;
    return r < 0 ? r + n : r;
}

// Cell index range overlapping [v - R, v + R] along axis d (clamped); along the
// periodic z axis an unclamped range (wrapped by the caller) or the whole axis.
// A non-finite v or R (a particle outside the geometry range) gets no cells;
// a periodic range far from the box (|index| >= 2^30) takes the whole axis,
// so the callers' int loops never come near overflow.
__device__ __forceinline__ void axis_range(float v, float R, const Grid* __restrict__ g, int d,
                                           int& k0, int& k1) {
    const float inv = g->invwf[d], s = g->slop[d];
    const int n = g->n[d];
    if (!(fabsf(v) < CUDART_INF_F) || !(R < CUDART_INF_F)) {
        k0 = 0;
        k1 = -1;
        return;
    }
    if (d == 2 && g->periodic_z) {
        const float fa = floorf((v - R - s + g->halflzf) * inv);
        const float fb = floorf((v + R + s + g->halflzf) * inv);
        if (!(fb - fa + 1.0f < (float)n) || !(fabsf(fa) < 1.0e9f && fabsf(fb) < 1.0e9f)) {
            k0 = 0;
            k1 = n - 1;
            return;
        }
        k0 = (int)fa;
        k1 = (int)fb;
        return;
    }
    const float lo = g->lof[d];
    float fa = floorf((v - R - s - lo) * inv);
    float fb = floorf((v + R + s - lo) * inv);
    fa = fminf(fmaxf(fa, 0.0f), (float)n);
    fb = fmaxf(fminf(fb, (float)(n - 1)), -1.0f);
    k0 = (int)fa;
    k1 = (int)fb;
}

// Distance from v to the slab of cell k along axis d (0 inside), inflated by slop.
__device__ __forceinline__ float axis_gap(float v, int k, const Grid* __restrict__ g, int d) {
    const float a = g->lof[d] + (float)k * g->wf[d] - g->slop[d];
    const float b = g->lof[d] + (float)(k + 1) * g->wf[d] + g->slop[d];
    return fmaxf(0.0f, fmaxf(a - v, v - b));
}

// Cell index range overlapping [a, b] along axis d (clamped); along the
// periodic z axis an unclamped range (wrapped by the caller) or the whole axis.
// Non-finite bounds and far periodic ranges as in axis_range.
__device__ __forceinline__ void box_range(float a, float b, const Grid* __restrict__ g, int d,
                                          int& k0, int& k1) {
    const float inv = g->invwf[d], s = g->slop[d];
    const int n = g->n[d];
    if (!(fabsf(a) < CUDART_INF_F) || !(fabsf(b) < CUDART_INF_F)) {
        k0 = 0;
        k1 = -1;
        return;
    }
    if (d == 2 && g->periodic_z) {
        const float fa = floorf((a - s + g->halflzf) * inv);
        const float fb = floorf((b + s + g->halflzf) * inv);
        if (!(fb - fa + 1.0f < (float)n) || !(fabsf(fa) < 1.0e9f && fabsf(fb) < 1.0e9f)) {
            k0 = 0;
            k1 = n - 1;
            return;
        }
        k0 = (int)fa;
        k1 = (int)fb;
        return;
    }
    const float lo = g->lof[d];
    float fa = floorf((a - s - lo) * inv);
    float fb = floorf((b + s - lo) * inv);
    fa = fminf(fmaxf(fa, 0.0f), (float)n);
    fb = fmaxf(fminf(fb, (float)(n - 1)), -1.0f);
    k0 = (int)fa;
    k1 = (int)fb;
}

__device__ __forceinline__ float wmin(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}
__device__ __forceinline__ float wmax(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

// A flat list of the particles of up to 32 cells, one cell per lane (num
// particles from slot start on): place t of the list is slot t + delta[k] of
// the k-th occupied cell. The warp's 32 places t0 .. t0 + 31 find their cells
// from the number of cells that start before t0 and a word of the places where
// cells start after it, both by warp votes: no search in memory.
struct FlatCells {
    int pl, total;  // place of this lane's cell (INT_MAX: empty), length of the list
    __device__ __forceinline__ FlatCells(int num, int start, int* delta) {
        const int lane = threadIdx.x & 31;
        int inc = num;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += v;
        }
        total = __shfl_sync(kFull, inc, 31);
        const int place = inc - num;
        const unsigned occ = __ballot_sync(kFull, num > 0);
        if (num > 0) delta[__popc(occ & ((1u << lane) - 1u))] = start - place;
        pl = num > 0 ? place : 0x7fffffff;
        __syncwarp();
    }
    // slot of place t0 + lane, -1 from place `end` on (t0 < total)
    __device__ __forceinline__ int slot(int t0, int end, const int* delta) const {
        const int lane = threadIdx.x & 31;
        const unsigned before = __ballot_sync(kFull, pl < t0);
        unsigned bit;  // (shl gives 0 for a shift of 32 or more, as of a negative one)
        asm("shl.b32 %0, 1, %1;" : "=r"(bit) : "r"(pl - t0));
        const unsigned starts = __reduce_or_sync(kFull, bit);
        const int k = __popc(before) + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
        return t0 + lane < end ? t0 + lane + delta[k] : -1;
    }
};

// One warp, one particle: enumerate the candidates of every cell overlapping
// the box [q - R, q + R] as one flat list, the cells 32 at a time. The list is
// handed out 32 candidates at a time: chunk(valid, j, f) is called by all
// lanes together, lane l receiving candidate j at f = fpos[j] (valid = false
// past the end); the next candidates load meanwhile. PRUNE = 1 drops a cell whose box lies farther than R from the
// particle; PRUNE = 2 drops it unless its box lies within
// 2 max(h_i, max h of the cell) of the particle (hib = bits of h_i).
template <int PRUNE, class Chunk>
__device__ __forceinline__ void particle_pass(const Grid* __restrict__ g,
                                              const int2* __restrict__ cells,
                                              const unsigned long long* cell_hmax,
                                              const float4* fpos, const float4& q,
                                              float R, long long hib, int* delta, Chunk&& chunk) {
    const int lane = threadIdx.x & 31;
    int x0, x1, y0, y1, z0, z1;
    axis_range(q.x, R, g, 0, x0, x1);
    axis_range(q.y, R, g, 1, y0, y1);
    axis_range(q.z, R, g, 2, z0, z1);
    const int nxr = x1 - x0 + 1, nyr = y1 - y0 + 1, nzr = z1 - z0 + 1;
    if (nxr <= 0 || nyr <= 0 || nzr <= 0) return;
    const int C = nxr * nyr * nzr;
    const int nx = g->n[0], ny = g->n[1], nz = g->n[2];
    const bool per = g->periodic_z != 0;
    for (int c0 = 0; c0 < C; c0 += 32) {
        const int c = c0 + lane;
        int start = 0, cnt = 0;
        if (c < C) {
            const int kx = x0 + c % nxr;
            const int rr = c / nxr;
            const int ky = y0 + rr % nyr;
            const int kz = z0 + rr / nyr;
            const int cz = per ? wrapi(kz, nz) : kz;
            const long long lin = ((long long)cz * ny + ky) * nx + kx;
            const int2 se = __ldg(&cells[lin]);
            start = se.x;
            cnt = max(se.y - se.x, 0);
            if (PRUNE && cnt > 0) {
                float reach = R;
                if (PRUNE == 2) {
                    const long long hcb = (long long)cell_hmax[lin];
                    reach = reach_f32(__longlong_as_double(hcb > hib ? hcb : hib));
                }
                const float gx = axis_gap(q.x, kx, g, 0), gy = axis_gap(q.y, ky, g, 1);
                const float gz = per ? 0.0f : axis_gap(q.z, kz, g, 2);
                if (fmaf(gz, gz, fmaf(gy, gy, gx * gx)) >= reach * reach) cnt = 0;
            }
        }
        const FlatCells F(cnt, start, delta);
        // (PRUNE = 2: cell_hmax and fpos.w were written by this same kernel)
        auto load = [&](int j) { return PRUNE == 2 ? fpos[j] : __ldg(&fpos[j]); };
        int jn = F.total > 0 ? F.slot(0, F.total, delta) : -1;
        float4 fn = jn >= 0 ? load(jn) : make_float4(0.f, 0.f, 0.f, 0.f);
        for (int t0 = 0; t0 < F.total; t0 += 32) {
            const int j = jn;
            const float4 f = fn;
            if (t0 + 32 < F.total) {
                jn = F.slot(t0 + 32, F.total, delta);
                if (jn >= 0) fn = load(jn);
            }
            chunk(j >= 0, j, f);
        }
        __syncwarp();
    }
}

// A cluster of a warp's lanes (the first remaining lane and every remaining
// lane whose cell is within one cell of it: a warp whose particles straddle a
// jump of the Morton curve searches two compact boxes instead of one spanning
// both places): the box around its particles, with centre o and half extents
// e, the largest reach Rm of its lanes, and the cells within reach of the box.
struct Cluster {
    float x0, x1, y0, y1, z0, z1;  // the box (z in the first lane's periodic image)
    float ox, oy, oz, ex, ey, ez;
    float Rm, reach, L;  // reach: of the box, with slop; L >= |p|, |q| from the centre
    float D;             // bound on the norm of (q - p) in floats minus in FP64
    int kx0, ky0, kz0, nxr, nyr, C;
    bool ok, wraps, zgap;
};

// mine: the lanes of the cluster; z in the image of its first lane; Rq >= 2 h
// of the lane's search (widened, reach_f32).
// Per component q - p differs from its FP64 value by u |x| (u = 2^-24) from
// each conversion to float, u L from each subtraction of the centre, and along
// z, where the box's reach crosses the end of a periodic axis (wraps), the
// shifts of both by lz: u (|x| + lz) and the error of lz as a float each.
__device__ __forceinline__ Cluster make_cluster(bool mine, float x, float y, float z, float Rq,
                                                const Grid* __restrict__ g) {
    Cluster K;
    const float inf = CUDART_INF_F;
    const bool per = g->periodic_z != 0;
    const float lzf = g->lzf, hlz = g->halflzf;
    const float sl = fmaxf(g->slop[0], fmaxf(g->slop[1], g->slop[2]));
    K.x0 = wmin(mine ? x : inf);
    K.x1 = wmax(mine ? x : -inf);
    K.y0 = wmin(mine ? y : inf);
    K.y1 = wmax(mine ? y : -inf);
    K.z0 = wmin(mine ? z : inf);
    K.z1 = wmax(mine ? z : -inf);
    K.Rm = wmax(mine ? Rq : 0.0f);
    K.ox = 0.5f * K.x0 + 0.5f * K.x1;
    K.oy = 0.5f * K.y0 + 0.5f * K.y1;
    K.oz = 0.5f * K.z0 + 0.5f * K.z1;
    K.ex = fmaxf(K.x1 - K.ox, K.ox - K.x0);
    K.ey = fmaxf(K.y1 - K.oy, K.oy - K.y0);
    K.ez = fmaxf(K.z1 - K.oz, K.oz - K.z0);
    K.reach = (K.Rm + sl) * 1.0001f;
    K.L = sqrtf(fmaf(K.ez, K.ez, fmaf(K.ey, K.ey, K.ex * K.ex))) * 1.0001f + K.reach;
    // Not ok: scales whose squares leave the normal floats, and a periodic
    // axis so short that a candidate within reach of a lane might not be at its
    // image nearest the centre (R + ez < lz/2 is needed), or that the wrap could
    // decide differently in FP32 (R > lz/4).
    K.ok = K.L < 4.0e18f && K.Rm > 1.0e-15f &&
           !(per && (K.Rm > 0.25f * lzf || K.Rm + K.ez > 0.49f * lzf));
    K.wraps = per && (K.z0 - K.reach < -hlz || K.z1 + K.reach > hlz);
    const float dxy = 1.2e-7f * (g->Xf + K.L);
    const float dz = dxy + (K.wraps ? 1.2e-7f * (g->Xf + lzf) + 2.0f * g->lzerr : 0.0f);
    K.D = sqrtf(fmaf(dz, dz, 2.0f * dxy * dxy)) * 1.0001f;
    int kx1, ky1, kz1;
    box_range(K.x0 - K.Rm, K.x1 + K.Rm, g, 0, K.kx0, kx1);
    box_range(K.y0 - K.Rm, K.y1 + K.Rm, g, 1, K.ky0, ky1);
    box_range(K.z0 - K.Rm, K.z1 + K.Rm, g, 2, K.kz0, kz1);
    K.nxr = kx1 - K.kx0 + 1;
    K.nyr = ky1 - K.ky0 + 1;
    const int nzr = kz1 - K.kz0 + 1;
    K.C = K.nxr > 0 && K.nyr > 0 && nzr > 0 ? K.nxr * K.nyr * nzr : 0;
    K.zgap = !per || nzr < g->n[2];  // (the whole periodic axis: no distance along z)
    return K;
}

// Particles of cell c of the cluster's range, 0 if the cell is out of its reach.
__device__ __forceinline__ int cluster_cell(const Cluster& K, const Grid* __restrict__ g,
                                            const int2* __restrict__ cells, int c, int& start) {
    start = 0;
    if (c >= K.C) return 0;
    const int kx = K.kx0 + c % K.nxr, rr = c / K.nxr;
    const int ky = K.ky0 + rr % K.nyr, kz = K.kz0 + rr / K.nyr;
    const int cz = g->periodic_z ? wrapi(kz, g->n[2]) : kz;
    const int2 se = __ldg(&cells[((long long)cz * g->n[1] + ky) * g->n[0] + kx]);
    start = se.x;
    auto gap = [&](int k, int d, float v0, float v1) {
        const float c0 = g->lof[d] + (float)k * g->wf[d] - g->slop[d];
        const float c1 = g->lof[d] + (float)(k + 1) * g->wf[d] + g->slop[d];
        return fmaxf(0.0f, fmaxf(c0 - v1, v0 - c1));
    };
    const float gx = gap(kx, 0, K.x0, K.x1), gy = gap(ky, 1, K.y0, K.y1);
    const float gz = K.zgap ? gap(kz, 2, K.z0, K.z1) : 0.0f;
    return fmaf(gz, gz, fmaf(gy, gy, gx * gx)) < K.Rm * K.Rm ? max(se.y - se.x, 0) : 0;
}

// The places [first, last) of the cluster's flat list of candidates, 32 at a
// time: f(ok, q, j) is called by all lanes together, lane l with candidate j at
// q from the centre (q.w = |q|^2), ok when it lies within reach of the box. The
// next candidates load while these are worked on.
template <class F>
__device__ __forceinline__ void cluster_walk(const Cluster& K, const Grid* __restrict__ g,
                                             const int2* __restrict__ cells,
                                             const float4* __restrict__ fpos, int* delta,
                                             int first, int last, F&& f) {
    const int lane = threadIdx.x & 31;
    const float lzf = g->lzf, hlz = g->halflzf;
    int seen = 0;  // candidates before this batch of cells
    for (int c0 = 0; c0 < K.C; c0 += 32) {
        int start;
        const int num = cluster_cell(K, g, cells, c0 + lane, start);
        const FlatCells cl(num, start, delta);
        const int ta = max(first - seen, 0), tb = min(last - seen, cl.total);
        int jn = ta < tb ? cl.slot(ta, tb, delta) : -1;
        float4 qn = jn >= 0 ? __ldg(&fpos[jn]) : make_float4(0.f, 0.f, 0.f, 0.f);
        for (int t0 = ta; t0 < tb; t0 += 32) {
            const int j = jn;
            float4 q = qn;
            if (t0 + 32 < tb) {
                jn = cl.slot(t0 + 32, tb, delta);
                if (jn >= 0) qn = __ldg(&fpos[jn]);
            }
            if (K.wraps) {
                const float d = q.z - K.oz;
                if (d > hlz) q.z -= lzf;
                else if (d < -hlz) q.z += lzf;
            }
            q.x -= K.ox;
            q.y -= K.oy;
            q.z -= K.oz;
            const float gx = fmaxf(fabsf(q.x) - K.ex, 0.0f), gy = fmaxf(fabsf(q.y) - K.ey, 0.0f);
            const float gz = fmaxf(fabsf(q.z) - K.ez, 0.0f);
            const bool ok = j >= 0 && fmaf(gz, gz, fmaf(gy, gy, gx * gx)) <= K.reach * K.reach;
            q.w = fmaf(q.z, q.z, fmaf(q.y, q.y, q.x * q.x));
            f(ok, q, j);
        }
        seen += cl.total;
        __syncwarp();
    }
}

// (2 h)^2 in the length unit of the double-float pair kernels, as a float within
// 2^-22 (integer and FP32 operations only), for the spare float of the position
// pack; NaN (the exact test alone decides) where the periodic wrap could decide
// differently, or for an h whose exponent cannot be moved.
__device__ __forceinline__ float pair_reach2(double h, const Grid* __restrict__ g) {
    const long long b = __double_as_longlong(h);
    if (b == 0) return 0.0f;
    if (b < (64ll << 52) || b > kHMaxBits) return CUDART_NAN_F;
    float lo, hi;
    f32_bounds(h, lo, hi);
    if (g->periodic_z && 2.0f * hi > 0.2499f * g->lzf) return CUDART_NAN_F;
    f32_bounds(__longlong_as_double(b + ((long long)(1 - g->uL) << 52)), lo, hi);
    return lo * lo;
}

// What a finished search leaves in the pack of particle i (precision 0).
__device__ __forceinline__ void write_reach2(float4* __restrict__ xpk, int64_t i, double h,
                                             const Grid* __restrict__ g, const KParams& kp) {
    if (kp.precision == PREC_FP64) xpk[3 * i + 2].w = pair_reach2(h, g);
}

// ------------------------------------------------------------ h search
// Groups (union_group, k_h_union): one warp per 32 consecutive (Morton-sorted)
// particles, one lane per particle, for the groups left with more than
// defer_lanes searching lanes by the first count (k_h_count; with candidate
// lists the search starts here). Each pass counts N_i(h) for every
// still-searching lane over the union of their query boxes (candidates staged
// once for the warp) and records the gather set in the slab. While more than
// defer_lanes lanes are still searching the warp keeps going; the stragglers
// are then handed, with their bisection state, to the per-particle kernel
// below through a worklist.

// Cell index of a (float) coordinate along axis d, clamped to the grid; only
// used to cluster the lanes of a warp, so FP32 rounding is harmless.
__device__ __forceinline__ int lane_cell(float v, const Grid* __restrict__ g, int d) {
    const float lo = (d == 2 && g->periodic_z) ? -g->halflzf : g->lof[d];
    const int k = (int)floorf((v - lo) * g->invwf[d]);
    return min(max(k, 0), g->n[d] - 1);
}

// Test the 32 staged candidates of a warp against every lane's particle and
// fold the outcome into that lane's count and gather slab. Candidates are
// (float x, y, z) already moved to the lane's periodic image; sidx holds
// their particle indices. Padding slots sit far away.
// rec: instead of counting, record (r^2 in FP32, j) of every candidate that
// may lie within the thresholds' radius (r2 <= Tout) in recb (up to kRec),
// except those with r2 < tin_lo, certainly within 2 lo (lo the bisection's
// lower bound, so within 2 h for every h still to be tried): those go to the
// gather slab and the count c at once.
// BL: also append to the lane's candidate list (slots, entries 32 apart from
// lrow on; nl of them) every staged candidate with r^2 <= tL. Padding slots
// (sidx -1) are never counted, recorded or listed.
template <bool BL>
__device__ __forceinline__ void union_chunk(const float4* __restrict__ st, const int* __restrict__ sidx,
                                            const float4& fi, const Thr& t, bool active, bool rec,
                                            float tin_lo, int64_t i, double h, double& R2,
                                            const double4_32a* posh, const Grid* __restrict__ g,
                                            int32_t* slab, int& c, int2* recb, int& nrec,
                                            float tL, int32_t* __restrict__ lrow, int& nl) {
    unsigned in = 0u, bd = 0u, lb = 0u;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const float4 q = st[k];
        const float dx = fi.x - q.x, dy = fi.y - q.y, dz = fi.z - q.z;
        const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
        if (r2 < t.tin) in |= 1u << k;
        if (r2 <= t.tout) bd |= 1u << k;
        if (BL && r2 <= tL) lb |= 1u << k;
    }
    if (!active) return;
    if (BL) {
        while (lb) {
            const int k = __ffs(lb) - 1;
            lb &= lb - 1u;
            const int j = sidx[k];
            if (j == i || j < 0) continue;
            if (nl < kList) lrow[nl * 32] = j;
            ++nl;
        }
    }
    if (rec) {
        while (bd) {
            const int k = __ffs(bd) - 1;
            bd &= bd - 1u;
            const int j = sidx[k];
            if (j == i || j < 0) continue;
            const float4 q = st[k];
            const float dx = fi.x - q.x, dy = fi.y - q.y, dz = fi.z - q.z;
            const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
            if (r2 < tin_lo) {
                if (c < kGSlab) slab[c] = j;
                ++c;
                continue;
            }
            if (nrec < kRec) recb[nrec] = make_int2(__float_as_int(r2), j);
            ++nrec;
        }
        return;
    }
    bd &= ~in;
    while (bd) {  // the ~1e-5-wide border band: exact FP64 test (rare: reloads p_i)
        const int k = __ffs(bd) - 1;
        bd &= bd - 1u;
        const int j = sidx[k];
        if (j == i || j < 0) continue;
        if (R2 < 0.0) {
            const double R = 2.0 * h;
            R2 = __dmul_rn(R, R);
        }
        if (exact_r2(posh[i], posh[j], g) < R2) in |= 1u << k;
    }
    while (in) {
        const int k = __ffs(in) - 1;
        in &= in - 1u;
        const int j = sidx[k];
        if (j == i || j < 0) continue;
        if (c < kGSlab) slab[c] = j;
        ++c;
    }
}

// N_i(h) from a candidate list (slots, ln entries 32 apart from L on): the
// same FP32 decisions with the exact FP64 band as a cell walk, the members
// written to the slab in list order. The list must hold every j within 2 h of
// i (the caller checks that it still does).
__device__ __forceinline__ int list_count(const int32_t* __restrict__ L, int ln,
                                          const float4* __restrict__ fpos, const float4& fi,
                                          const Thr& t, int64_t i, double h,
                                          const double4_32a* posh, const Grid* __restrict__ g,
                                          int32_t* slab) {
    int c = 0;
    double R2 = -1.0;
    constexpr int G = 4;  // entries in flight per group (loads first, then the tests)
    for (int e0 = 0; e0 < ln; e0 += G) {
        int j[G];
        float4 f[G];
#pragma unroll
        for (int k = 0; k < G; ++k) j[k] = e0 + k < ln ? __ldg(&L[(e0 + k) * 32]) : -1;
#pragma unroll
        for (int k = 0; k < G; ++k) f[k] = j[k] >= 0 ? __ldg(&fpos[j[k]]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < G; ++k) {
            if (j[k] < 0) continue;
            const float r2 = f_r2(fi, f[k], g);
            bool in = r2 < t.tin;
            if (!in && r2 <= t.tout) {
                if (R2 < 0.0) {
                    const double R = 2.0 * h;
                    R2 = __dmul_rn(R, R);
                }
                in = exact_r2(posh[i], posh[j[k]], g) < R2;
            }
            if (in) {
                if (c < kGSlab) slab[c] = j[k];
                ++c;
            }
        }
    }
    return c;
}

// |N_i(hh)| from the c0 neighbours certainly within 2 lo <= 2 hh (already in
// the slab) and the records of a record pass made at a radius >= 2 hh, with
// the same decisions as a counting pass (FP32 thresholds, exact FP64 test in
// the band between them); with slab, the recorded members of N_i(hh) are
// appended after the first c0, in record order.
__device__ int count_records(const int2* recb, int nrec, double hh, const Grid* __restrict__ g,
                             const double4_32a* posh, int64_t i, int32_t* slab, int c0) {
    const double R = 2.0 * hh;
    const Thr t = thresholds(R, g);
    double R2 = -1.0;
    int c = c0;
    for (int q = 0; q < nrec; ++q) {
        const int2 e = recb[q];
        const float r2 = __int_as_float(e.x);
        bool in = r2 < t.tin;
        if (!in && r2 <= t.tout) {
            if (R2 < 0.0) R2 = __dmul_rn(R, R);
            in = exact_r2(posh[i], posh[e.y], g) < R2;
        }
        if (in) {
            if (slab && c < kGSlab) slab[c] = e.y;
            ++c;
        }
    }
    return c;
}

// The 32 particles i0 .. i0 + 31 (one per lane; all of one instance).
// LISTS: the batch has instances with candidate lists; the search starts here.
// Else k_h_count has made the first count, and the lanes with hs_it > 0 go on
// from the bracket it left.
template <bool LISTS>
__device__ __forceinline__ void union_group(
    int64_t i0, int64_t n, const Batch& B, double4_32a* posh, const float4* __restrict__ fpos,
    const int2* __restrict__ cells, int32_t* __restrict__ nnb, int32_t* __restrict__ ngather,
    int32_t* __restrict__ rslab, double* __restrict__ hs_lo, double* __restrict__ hs_hi,
    int32_t* __restrict__ hs_it, int32_t* __restrict__ wl, unsigned* __restrict__ status,
    float4* st, int* sidx, int2* recb, const int32_t* __restrict__ order,
    int32_t* __restrict__ lst, LMeta* __restrict__ lmeta, float4* __restrict__ xpk) {
    const int lane = threadIdx.x & 31;
    const int64_t i = i0 + lane;
    const int inst = slot_inst(B, i0);
    const Grid* __restrict__ g = B.grid + inst;
    const KParams& kp = B.kp[inst];
    cells += g->cbase;
    const bool inb = i < n;
    const bool valid = inb && slot_real(B, inst, i);
    float4 fi = make_float4(0.f, 0.f, 0.f, 0.f);
    double h = 1.0, lo = 0.0, hi = CUDART_INF;
    if (valid) {
        h = posh[i].w;
        fi = fpos[i];
    }
    // a particle outside the geometry range (reported by the bounding box)
    // does not search: no neighbours, h unchanged
    const bool geo = valid && isfinite(fi.x) && isfinite(fi.y) && isfinite(fi.z) && h_ok(h);
    const int lowb = kp.n_target - kp.n_tol, highb = kp.n_target + kp.n_tol;
    const int max_it = kp.max_h_iter;
    const int defer = kp.defer_lanes;
    int cnt = 0, it = 0;
    bool active = geo && max_it > 0, conv = false, deferred = false;
    if (!LISTS) {
        it = valid ? hs_it[i] : -1;
        active = it > 0;
        if (active) {
            lo = hs_lo[i];
            hi = hs_hi[i];
        }
    }
    const bool entered = LISTS || active;
    int32_t* slab = rslab + (valid ? i : 0) * kRSlab;
    const bool per = g->periodic_z != 0;
    const int nx = g->n[0], ny = g->n[1], nz = g->n[2];
    const unsigned lt = (1u << lane) - 1u;
    // Candidate lists: a lane with a kept list was served by k_h_lists. A
    // build step walks every lane, recording its list (every candidate within
    // 2 h (1 + skin)) in the first walk.
    const bool build = LISTS && kp.list_skin > 0.0 && g->lbuild != 0;
    const int32_t id = LISTS && valid && kp.list_skin > 0.0 ? __ldg(&order[i]) : 0;
    int32_t* lrow = lst + (i >> 5) * (int64_t)kList * 32 + (i & 31);
    int nl = 0;
    bool listed = false;
    if (build && valid) {  // the list build's record of the particle (its list comes with the walk)
        const double4_32a p = posh[i];
        reinterpret_cast<float4*>(lmeta)[2 * id] =
            make_float4(dfl::from_double(p.x).hi, dfl::from_double(p.y).hi,
                        dfl::from_double(p.z).hi, 0.0f);
        lmeta[id].stamp = g->lstamp;  // (the cell code was recorded by the sort)
        lmeta[id].cnt = 0;
    } else if (LISTS && kp.list_skin > 0.0 && active && lmeta[id].cnt > 0) {
        listed = true;
        active = false;
    }
    for (int pass = LISTS ? 0 : 1;; ++pass) {  // warp-uniform; it (per lane) stops at convergence
        const unsigned am = __ballot_sync(kFull, active);
        if (!am) break;
        // Pass 0 counts N_i(h). Later passes record every candidate within 2 hs,
        // hs = the largest h the bisection can still test without growing (hi, or
        // h while hi is unbounded), and resolve the following counts from the
        // records: a search from a poor initial h takes ~2 passes, not ~8.
        const bool rec = pass > 0;
        const double hs = rec && !isinf(hi) ? hi : h;
        const Thr t = thresholds(2.0 * hs, g);
        const float tin_lo = rec && lo > 0.0 ? thresholds(2.0 * lo, g).tin : -1.0f;
        const bool blist = build && pass == 0;  // list radius RL = 2 hs (1 + skin)
        const double RL = blist ? 2.0 * hs * (1.0 + kp.list_skin) : 0.0;
        const float tL = blist ? thresholds(RL, g).tout : 0.0f;
        const float Rq = blist ? reach_f32(0.5 * RL) : reach_f32(hs);
        const float lzz = wmin(active ? fi.z - Rq : CUDART_INF_F), hzz = wmax(active ? fi.z + Rq : -CUDART_INF_F);
        // Periodic z: candidates are moved to the image nearest a reference lane's
        // z, which is each lane's minimum image while the lanes' z span S and
        // reach R satisfy R + S < lz/2 (a candidate within R of lane i is then
        // within lz/2 of the reference lane). A warp with S + 2R > lz/4 hands
        // its particles to the per-particle kernel: correct up to ~lz/2, but
        // measured faster there (27k periodic patch: 0.47 ms per step at lz/4,
        // 0.52 at 0.45 lz; the 1M patch the same within 1%).
        const bool wide = per && (hzz - lzz > 0.25f * g->lzf);
        if ((pass > 0 && __popc(am) <= defer) || wide) {
            if (active) {
                deferred = true;
                active = false;
                posh[i].w = h;
                hs_lo[i] = lo;
                hs_hi[i] = hi;
                hs_it[i] = it;
                wl[atomicAdd(&status[3], 1u)] = (int32_t)i;
            }
            break;
        }
        // The active lanes are served in clusters: the first remaining lane and
        // every remaining lane whose cell is within one cell of it. A warp whose
        // particles straddle a jump of the Morton curve thus searches two
        // compact boxes instead of one box spanning both places.
        const int mcx = lane_cell(fi.x, g, 0), mcy = lane_cell(fi.y, g, 1);
        const int mcz = lane_cell(fi.z, g, 2);
        double R2 = -1.0;
        int c = 0, nrec = 0;
        unsigned todo = am;
        while (todo) {
            const int a = __ffs(todo) - 1;
            const int ax = __shfl_sync(kFull, mcx, a), ay = __shfl_sync(kFull, mcy, a);
            const int az = __shfl_sync(kFull, mcz, a);
            int dzc = abs(mcz - az);
            if (per) dzc = min(dzc, nz - dzc);
            const bool mine = ((todo >> lane) & 1u) && abs(mcx - ax) <= 1 && abs(mcy - ay) <= 1 &&
                              dzc <= 1;
            todo &= ~__ballot_sync(kFull, mine);
            const float sx0 = wmin(mine ? fi.x - Rq : CUDART_INF_F), sx1 = wmax(mine ? fi.x + Rq : -CUDART_INF_F);
            const float sy0 = wmin(mine ? fi.y - Rq : CUDART_INF_F), sy1 = wmax(mine ? fi.y + Rq : -CUDART_INF_F);
            const float sz0 = wmin(mine ? fi.z - Rq : CUDART_INF_F), sz1 = wmax(mine ? fi.z + Rq : -CUDART_INF_F);
            const float zc = __shfl_sync(kFull, fi.z, a);
            int x0, x1, y0, y1, z0, z1;
            box_range(sx0, sx1, g, 0, x0, x1);
            box_range(sy0, sy1, g, 1, y0, y1);
            box_range(sz0, sz1, g, 2, z0, z1);
            int fill = 0;  // staged candidates (warp-uniform)
            const float Rq2 = Rq * Rq;
            // Query box of the cluster: a candidate within 2h_i (FP64) of one of its
            // lanes lies inside it. The slop (>= 1e-3 cell widths + 1.2e-7 X)
            // covers the FP32 rounding of both coordinates and of the periodic shift.
            const float bx0 = sx0 - g->slop[0], bx1 = sx1 + g->slop[0];
            const float by0 = sy0 - g->slop[1], by1 = sy1 + g->slop[1];
            const float bz0 = sz0 - g->slop[2], bz1 = sz1 + g->slop[2];
            // and in a ball around the cluster's centre o: |q - o| <= |q - p_i| + |p_i - o|
            // <= Rq_i + |p_i - o| for a candidate q within reach of lane i
            const float ox = 0.5f * (wmin(mine ? fi.x : CUDART_INF_F) + wmax(mine ? fi.x : -CUDART_INF_F));
            const float oy = 0.5f * (wmin(mine ? fi.y : CUDART_INF_F) + wmax(mine ? fi.y : -CUDART_INF_F));
            const float oz = 0.5f * (wmin(mine ? fi.z : CUDART_INF_F) + wmax(mine ? fi.z : -CUDART_INF_F));
            float rb = 0.0f;
            if (mine) {
                const float ex = fi.x - ox, ey = fi.y - oy, ez = fi.z - oz;
                rb = sqrtf(fmaf(ez, ez, fmaf(ey, ey, ex * ex))) + Rq;
            }
            rb = wmax(rb) * 1.00001f + fmaxf(g->slop[0], fmaxf(g->slop[1], g->slop[2]));
            const float rb2 = rb * rb;
            for (int kz = z0; kz <= z1; ++kz) {
                const int cz = per ? wrapi(kz, nz) : kz;
                const float gz = per ? 0.0f : axis_gap(fi.z, kz, g, 2);
                for (int ky = y0; ky <= y1; ++ky) {
                    const long long row = ((long long)cz * ny + ky) * nx;
                    const float gy = axis_gap(fi.y, ky, g, 1);
                    for (int kx = x0; kx <= x1; ++kx) {
                        const int2 se = __ldg(&cells[row + kx]);
                        if (se.y <= se.x) continue;
                        const float gx = axis_gap(fi.x, kx, g, 0);
                        if (!__any_sync(kFull, mine && fmaf(gz, gz, fmaf(gy, gy, gx * gx)) < Rq2))
                            continue;
                        // append the cell's particles that lie in the query box to the
                        // staging buffer (ballot-compacted, so the order of the kept
                        // candidates is unchanged); run full chunks
                        for (int s0 = se.x; s0 < se.y; s0 += 32) {
                            const int j = s0 + lane;
                            bool ok = j < se.y;
                            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (ok) {
                                f = __ldg(&fpos[j]);
                                if (per) {
                                    const float d = f.z - zc;
                                    if (d > g->halflzf) f.z -= g->lzf;
                                    else if (d < -g->halflzf) f.z += g->lzf;
                                }
                                const float qx = f.x - ox, qy = f.y - oy, qz = f.z - oz;
                                ok = f.x >= bx0 && f.x <= bx1 && f.y >= by0 && f.y <= by1 &&
                                     f.z >= bz0 && f.z <= bz1 &&
                                     fmaf(qz, qz, fmaf(qy, qy, qx * qx)) <= rb2;
                            }
                            const unsigned m = __ballot_sync(kFull, ok);
                            if (!m) continue;
                            const int r = __popc(m & lt), cnt = __popc(m), room = 32 - fill;
                            if (ok && r < room) {
                                st[fill + r] = f;
                                sidx[fill + r] = j;
                            }
                            if (cnt < room) {
                                fill += cnt;
                                continue;
                            }
                            __syncwarp();
                            if (blist)
                                union_chunk<true>(st, sidx, fi, t, mine, rec, tin_lo, i, h, R2,
                                                  posh, g, slab, c, recb, nrec, tL, lrow, nl);
                            else
                                union_chunk<false>(st, sidx, fi, t, mine, rec, tin_lo, i, h, R2,
                                                   posh, g, slab, c, recb, nrec, tL, lrow, nl);
                            __syncwarp();
                            if (ok && r >= room) {
                                st[r - room] = f;
                                sidx[r - room] = j;
                            }
                            fill = cnt - room;
                        }
                    }
                }
            }
            if (fill > 0) {  // last partial chunk: pad with far-away slots
                if (lane >= fill) {
                    st[lane] = make_float4(3.0e30f, 3.0e30f, 3.0e30f, 0.0f);
                    sidx[lane] = -1;
                }
                __syncwarp();
                if (blist)
                    union_chunk<true>(st, sidx, fi, t, mine, rec, tin_lo, i, h, R2, posh, g, slab,
                                      c, recb, nrec, tL, lrow, nl);
                else
                    union_chunk<false>(st, sidx, fi, t, mine, rec, tin_lo, i, h, R2, posh, g, slab,
                                       c, recb, nrec, tL, lrow, nl);
                __syncwarp();
            }
        }
        if (blist && active) {  // the list of this walk, complete unless it overflowed
            float lo_r, hi_r;
            f32_bounds(RL, lo_r, hi_r);
            lmeta[id].rad = lo_r * 0.999999f;
            lmeta[id].cnt = nl <= kList ? nl : 0;
        }
        if (active && rec && nrec > kRec) {  // too many to record: one warp of its own
            deferred = true;
            active = false;
            posh[i].w = h;
            hs_lo[i] = lo;
            hs_hi[i] = hi;
            hs_it[i] = it;
            wl[atomicAdd(&status[3], 1u)] = (int32_t)i;
        }
        // counts of this pass (or from its records) and the bisection updates
        const int cbase = rec ? c : 0;  // a record pass: the neighbours within 2 lo
        for (bool counted = !rec; active;) {
            if (rec) {
                if (h > hs) break;  // beyond the recorded radius: another pass
                c = count_records(recb, nrec, h, g, posh, i, nullptr, cbase);
            } else if (counted) {
                counted = false;  // c holds this pass's count
            } else {
                break;
            }
            cnt = c;
            ++it;
            if (cnt >= lowb && cnt <= highb) {
                conv = true;
                active = false;
            } else if (it >= max_it) {
                active = false;
            } else if (cnt < lowb) {
                lo = h;
                h = isinf(hi) ? __dmul_rn(h, 1.25) : __dmul_rn(0.5, __dadd_rn(lo, hi));
            } else {
                hi = h;
                h = (lo == 0.0) ? __dmul_rn(h, 0.8) : __dmul_rn(0.5, __dadd_rn(lo, hi));
            }
            if (!rec) break;
            if (!active) count_records(recb, nrec, h, g, posh, i, slab, cbase);  // N_i(final h)
        }
    }
    if (!entered) return;
    if (!valid) {
        if (inb) {  // empty slot: empty row
            nnb[i] = 0;
            ngather[i] = 0;
        }
        return;
    }
    if (deferred || listed) return;
    posh[i].w = h;
    write_reach2(xpk, i, h, g, kp);
    nnb[i] = cnt;
    ngather[i] = cnt;
    if (cnt > kGSlab) atomicOr(&status[2], (unsigned)IF_SLAB_OVF);
    if (!conv) {
        atomicOr(&status[0], (unsigned)ST_HNOCONV);
        atomicAdd(&status[1], 1u);
    }
}

// The first count of the particles with a kept candidate list (one thread
// per slot; the others are left to k_h_union): one scan of the list at the
// current h, while the list still covers 2h (its radius at the build minus
// twice the largest displacement since), with the cell walk's decisions. A
// particle that converges is done; one that must go on bisecting (or whose
// list does not cover 2h) is handed, with its bisection state, to
// k_h_iterate, which takes its records from the list while it covers them:
// the same sequence of h and the same neighbour set as the cell walk.
__global__ void __launch_bounds__(kThreads)
k_h_lists(int64_t n, Batch B, double4_32a* posh, const float4* __restrict__ fpos,
          int32_t* __restrict__ nnb, int32_t* __restrict__ ngather, int32_t* __restrict__ rslab,
          double* __restrict__ hs_lo, double* __restrict__ hs_hi, int32_t* __restrict__ hs_it,
          int32_t* __restrict__ wl, unsigned* __restrict__ status,
          const int32_t* __restrict__ order, const int32_t* __restrict__ lst,
          const LMeta* __restrict__ lmeta, float4* __restrict__ xpk) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int inst = slot_inst(B, i);
    if (!slot_real(B, inst, i)) return;
    const KParams& kp = B.kp[inst];
    const Grid* __restrict__ g = B.grid + inst;
    if (!(kp.list_skin > 0.0) || g->lbuild || kp.max_h_iter < 1) return;
    const int32_t id = order[i];
    const int ln = lmeta[id].cnt;
    if (ln <= 0) return;
    double h = posh[i].w;
    const float4 fi = fpos[i];
    if (!(isfinite(fi.x) && isfinite(fi.y) && isfinite(fi.z) && h_ok(h))) return;
    const float lrad = lmeta[id].rad, dm2 = g->dm2;
    const int lowb = kp.n_target - kp.n_tol, highb = kp.n_target + kp.n_tol;
    const int max_it = kp.max_h_iter;
    const int32_t* L = lst + (i >> 5) * (int64_t)kList * 32 + (i & 31);
    int32_t* slab = rslab + i * kRSlab;
    double lo = 0.0, hi = CUDART_INF;
    int cnt = 0, it = 0;
    bool conv = false;
    // one count at the current h, from the list if it still covers 2h; a
    // particle that has to go on bisecting (or whose list no longer covers
    // 2h) continues in k_h_iterate, which records its candidates once
    const bool covered = reach_f32(h) + dm2 <= lrad;
    if (covered) {
        cnt = list_count(L, ln, fpos, fi, thresholds(2.0 * h, g), i, h, posh, g, slab);
        it = 1;
        conv = cnt >= lowb && cnt <= highb;
    }
    if (!covered || (!conv && it < max_it)) {
        if (covered) {
            if (cnt < lowb) {
                lo = h;
                h = __dmul_rn(h, 1.25);  // no upper bound yet
            } else {
                hi = h;
                h = __dmul_rn(h, 0.8);  // no lower bound yet
            }
        }
        posh[i].w = h;
        hs_lo[i] = lo;
        hs_hi[i] = hi;
        hs_it[i] = it;
        wl[atomicAdd(&status[3], 1u)] = (int32_t)i;
        return;
    }
    posh[i].w = h;
    write_reach2(xpk, i, h, g, kp);
    nnb[i] = cnt;
    ngather[i] = cnt;
    if (cnt > kGSlab) atomicOr(&status[2], (unsigned)IF_SLAB_OVF);
    if (!conv) {
        atomicOr(&status[0], (unsigned)ST_HNOCONV);
        atomicAdd(&status[1], 1u);
    }
}

// ------------------------------------------------------------ first count
// The first count of every particle (without candidate lists): N_i(h) at the
// h the particle comes with, which is the last one needed for ~98% of the
// particles of a running simulation. One block of W warps per 32 consecutive
// (Morton-sorted) particles, one lane per particle in every warp; the
// candidates of a cluster of lanes (as in union_group) are split between the
// W warps in W contiguous parts.
//
// A warp takes the cells around the cluster 32 at a time (one per lane), lists
// their particles flat, 32 at a time, and keeps those within reach of the box
// around the cluster's particles. Every lane tests every kept candidate: with
// positions q, p relative to the box's centre, the sign of
//     d = |q|^2 - 2 p.q + (|p|^2 - t)        (one addition, three FMAs)
// tells r^2 < t, t the middle of the FP32 thresholds of (2h)^2; a neighbour is
// appended to the lane's column in shared memory. A chunk of 32 candidates
// whose smallest |d| is within the band w, a bound on every rounding of d
// (below), is done again with the candidates in the band decided by the
// defining FP64 test: the sets are exact. The columns go to the rows four
// entries at a time, in the order of the candidates, which does not depend on
// W.
//
// Bound: instruction issue. Against testing, collecting bits and appending bit
// by bit in one loop (the record passes of k_h_union), a candidate costs ~10
// instead of ~16 instructions, the appends do not diverge chunk by chunk, and
// a row takes a quarter of the stores. Measured (ncu, a steady step): 17.1k
// warp instructions a group on the 70^3 patch (24.7k before); 1M patch 641 us
// (940), 1M sphere 848 us (1,227), 8,191-particle sphere 46 us (232). Tried:
// sign bits of a chunk shifted into a word and walked bit by bit at the end
// (825 us: the walk diverges); columns of 96 or 128 entries with 16-bit places
// and 16 to 22 warps resident (701 to 757 us; more warps beat fewer writes).
//
// The band. With D the bound of make_cluster on the float error of q - p, T_out
// = (2h + D)^2 rounded up and T_in = (2h - D)^2 rounded down, |q - p|^2 >= T_out
// is out and < T_in is in. d rounds by at most u (21 L^2 + 8 t) (|q|^2: 3 L^2;
// |p|^2 - t: 4 L^2 + 4 t; the sum: 2 L^2 + t; the FMAs: 3 (4 L^2 + t)), so with t
// the middle of T_in and T_out, w = half their difference plus that.
// Per warp, for W warps: chunks of 32 candidates kept, entries of a column.
template <int W>
constexpr int kCountChunks = W == 1 || W == 8 ? 8 : (W == 2 ? 24 : 16);
template <int W>
constexpr int kCountCap = W == 1 ? 96 : kGSlab;
constexpr int kCountWarps = 28;  // W = 1: resident warps per SM

// (the places of 256 candidates fit a byte)
template <int W>
using CountPlace = typename std::conditional<(kCountChunks<W> <= 8), uint8_t, uint16_t>::type;

template <int W>
struct CountSmem {  // per warp
    float4 st[32];                        // the chunk being filled: q and |q|^2
    int idx[kCountChunks<W> * 32];        // the candidates kept
    int delta[32];                        // cells of the walk: first slot - place in the list
    int self[32];                         // place in the open chunk of particle i0 + l
    CountPlace<W> col[kCountCap<W>][32];  // per lane: its neighbours' places in idx
};

template <int W>
__global__ void __launch_bounds__(32 * W, W == 1 ? kCountWarps : 16 / W)
k_h_count(int64_t n, Batch B, double4_32a* posh, const float4* __restrict__ fpos,
          const int2* __restrict__ cells, int32_t* __restrict__ nnb, int32_t* __restrict__ ngather,
          int32_t* __restrict__ rslab, double* __restrict__ hs_lo, double* __restrict__ hs_hi,
          int32_t* __restrict__ hs_it, int32_t* __restrict__ wl, int32_t* __restrict__ gwl,
          unsigned* __restrict__ status, unsigned long long* __restrict__ wctr,
          float4* __restrict__ xpk) {
    constexpr int kCh = kCountChunks<W>, kCap = kCountCap<W>;
    __shared__ CountSmem<W> s_w[W];
    __shared__ int s_cnt[W][32];
    const int lane = threadIdx.x & 31, warp = W > 1 ? (int)(threadIdx.x >> 5) : 0;
    CountSmem<W>& S = s_w[warp];
    const int64_t i0 = (int64_t)blockIdx.x * 32, i = i0 + lane;
    const int inst = slot_inst(B, i0);
    const Grid* __restrict__ g = B.grid + inst;
    const KParams& kp = B.kp[inst];
    cells += g->cbase;
    const bool inb = i < n;
    const bool valid = inb && slot_real(B, inst, i);
    float4 fi = make_float4(0.f, 0.f, 0.f, 0.f);
    double h = 1.0, lo = 0.0, hi = CUDART_INF;
    if (valid) {
        h = posh[i].w;
        fi = fpos[i];
    }
    // a particle outside the geometry range (reported by the bounding box)
    // does not search: no neighbours, h unchanged
    const bool geo = valid && isfinite(fi.x) && isfinite(fi.y) && isfinite(fi.z) && h_ok(h);
    const int max_it = kp.max_h_iter;
    bool active = geo && max_it > 0;  // still searching
    bool conv = false, handed = false;
    int cnt = 0, it = 0;
    int32_t* row = rslab + (valid ? i : 0) * kRSlab;
    const bool per = g->periodic_z != 0;
    const float lzf = g->lzf, hlz = g->halflzf;
    const int nz = g->n[2];
    const unsigned lt = (1u << lane) - 1u;
    const int i0s = (int)i0;
    const int mcx = lane_cell(fi.x, g, 0), mcy = lane_cell(fi.y, g, 1), mcz = lane_cell(fi.z, g, 2);
    const float Rq = active ? reach_f32(h) : 0.0f;
    unsigned todo = __ballot_sync(kFull, active);
    while (todo) {  // clusters of lanes, as in union_group
        const int a = __ffs(todo) - 1;
        const int acx = __shfl_sync(kFull, mcx, a), acy = __shfl_sync(kFull, mcy, a);
        const int acz = __shfl_sync(kFull, mcz, a);
        const float fza = __shfl_sync(kFull, fi.z, a);
        int dzc = abs(mcz - acz);
        if (per) dzc = min(dzc, nz - dzc);
        const bool mine = ((todo >> lane) & 1u) && abs(mcx - acx) <= 1 && abs(mcy - acy) <= 1 &&
                          dzc <= 1;
        todo &= ~__ballot_sync(kFull, mine);
        // z in the periodic image of the first lane
        float pz = fi.z;
        if (per) {
            const float d = pz - fza;
            if (d > hlz) pz -= lzf;
            else if (d < -hlz) pz += lzf;
        }
        const Cluster K = make_cluster(mine, fi.x, fi.y, pz, Rq, g);
        if (!K.ok) {
            if (mine) {
                handed = true;
                active = false;
            }
            continue;
        }
        float ax = 0.0f, ay = 0.0f, az = 0.0f, b = 1.0e38f, w = -1.0f;  // (finds nothing)
        if (mine) {
            const float px = fi.x - K.ox, py = fi.y - K.oy, pzr = pz - K.oz;
            float Rl, Rh;
            f32_bounds(2.0 * h, Rl, Rh);
            const float ro = __fadd_ru(__fmul_ru(Rh, 1.00000024f), K.D);
            const float ri = __fsub_rd(__fmul_rd(Rl, 0.99999976f), K.D);
            const float To = __fmul_ru(__fmul_ru(ro, ro), 1.0000003f);
            const float Ti = ri > 0.0f ? __fmul_rd(__fmul_rd(ri, ri), 0.9999997f) : -To;
            const float t = 0.5f * (Ti + To);
            ax = -2.0f * px;
            ay = -2.0f * py;
            az = -2.0f * pzr;
            b = fmaf(pzr, pzr, fmaf(py, py, px * px)) - t;
            w = 0.50001f * (To - Ti) + 1.3e-6f * (K.L * K.L) + 6.0e-7f * To;
        }
        int flat = 0;  // W > 1: length of the flat list
        if (W > 1) {
            for (int c0 = 0; c0 < K.C; c0 += 32) {
                int st;
                flat += cluster_cell(K, g, cells, c0 + lane, st);
            }
            flat = __reduce_add_sync(kFull, flat);
        }
        int nch = 0, fill = 0;  // chunks kept, candidates in the open one
        int e = 0;              // entries of this lane's column (past kCap: only counted)
        int written = 0;        // entries written to the row
        bool own = false;       // the open chunk holds some of the 32 particles themselves
        constexpr unsigned kRow = sizeof S.col[0];
        const unsigned col0 = (unsigned)__cvta_generic_to_shared(&S.col[0][lane]);
        // test the open chunk (its slots past `count` padded) and close it
        auto close = [&](int count) {
            const int id = nch * 32;
            if (lane >= count) {
                S.st[lane] = make_float4(0.0f, 0.0f, 0.0f, 3.0e38f);
                S.idx[id + lane] = -1;
            }
            __syncwarp();
            bool again = own || (W > 1 && __any_sync(kFull, e > kCap - 32));
            if (!again) {
                float mn = CUDART_INF_F;
                unsigned at = col0 + (unsigned)e * kRow;
#pragma unroll
                for (int k0 = 0; k0 < 32; k0 += 8) {  // eight tests in flight, then their appends
                    float d[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float4 q = S.st[k0 + k];
                        d[k] = fmaf(az, q.z, fmaf(ay, q.y, fmaf(ax, q.x, q.w + b)));
                    }
#pragma unroll
                    for (int k = 0; k < 8; k += 2) mn = fminf(mn, fminf(fabsf(d[k]), fabsf(d[k + 1])));
                    // (predicated instructions: left to the compiler, each was a branch)
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        if (sizeof(CountPlace<W>) == 2)
                            asm volatile("{.reg .pred p; setp.lt.f32 p, %1, 0f00000000;\n\t"
                                         "@p st.shared.u16 [%0], %2;\n\t@p add.u32 %0, %0, %3;}"
                                         : "+r"(at) : "f"(d[k]), "r"(id + k0 + k), "n"(kRow) : "memory");
                        else
                            asm volatile("{.reg .pred p; setp.lt.f32 p, %1, 0f00000000;\n\t"
                                         "@p st.shared.u8 [%0], %2;\n\t@p add.u32 %0, %0, %3;}"
                                         : "+r"(at) : "f"(d[k]), "r"(id + k0 + k), "n"(kRow) : "memory");
                    }
                }
                again = __any_sync(kFull, !(mn > w));  // a candidate in some lane's band
                if (!again) e = (int)((at - col0) / kRow);
            }
            if (again) {
                // the signs of d and of |d| - w as bits (candidate k: bit 31 - k); the
                // band decided in FP64, the particle itself taken out, the rest appended
                unsigned in = 0u, bd = 0u;
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                    const float4 q = S.st[k];
                    const float d = fmaf(az, q.z, fmaf(ay, q.y, fmaf(ax, q.x, q.w + b)));
                    in = __funnelshift_l((unsigned)__float_as_int(d), in, 1);
                    bd = __funnelshift_l((unsigned)__float_as_int(fabsf(d) - w), bd, 1);
                }
                S.self[lane] = 32;
                __syncwarp();
                const int js = S.idx[id + lane];
                if (js >= 0 && (unsigned)(js - i0s) < 32u) S.self[js - i0s] = lane;
                __syncwarp();
                while (bd) {
                    const int k = __clz((int)bd);
                    const unsigned bit = 0x80000000u >> k;
                    bd ^= bit;
                    const double R = 2.0 * h;
                    if (exact_r2(posh[i], posh[S.idx[id + k]], g) < __dmul_rn(R, R)) in |= bit;
                    else in &= ~bit;
                }
                const int sp = S.self[lane];
                if (sp < 32) in &= ~(0x80000000u >> sp);
                if (!mine) in = 0u;
                while (in) {
                    const int k = __clz((int)in);
                    in ^= 0x80000000u >> k;
                    if (W == 1 || e < kCap) S.col[e][lane] = (CountPlace<W>)(id + k);
                    ++e;
                }
            }
            ++nch;
            own = false;
            __syncwarp();
        };
        // the first `num` entries of the column to entries from, from + 1, ... of the row
        auto put = [&](int from, int num) {
            auto entry = [&](int p) { return S.idx[S.col[p][lane]]; };
            int p = 0;
            for (const int head = min((4 - (from & 3)) & 3, num); p < head; ++p)
                if (from + p < kGSlab) row[from + p] = entry(p);
            for (; p + 4 <= num; p += 4) {
                const int4 v = make_int4(entry(p), entry(p + 1), entry(p + 2), entry(p + 3));
                if (from + p + 4 <= kGSlab) *reinterpret_cast<int4*>(row + from + p) = v;
            }
            for (; p < num; ++p)
                if (from + p < kGSlab) row[from + p] = entry(p);
        };
        // One warp takes the whole list. Several take it in rounds of at most
        // as many candidates as they can keep, each warp a contiguous part of
        // the round; all but the last round write their entries at once (a row
        // holds kGSlab gather entries, so a column needs no more).
        constexpr int kRound = W * kCh * 32;
        for (int base = 0;; base += kRound) {
            const bool final_round = W == 1 || base + kRound >= flat;
            int first = 0, last = 0x7fffffff;  // this warp's part of the flat list
            if (W > 1) {
                const int len = min(kRound, flat - base);
                first = base + len * warp / W;
                last = base + len * (warp + 1) / W;
                e = nch = fill = 0;
            }
            cluster_walk(K, g, cells, fpos, S.delta, first, last, [&](bool ok, const float4& q, int j) {
                const unsigned m = __ballot_sync(kFull, ok);
                if (!m) return;
                const int r = __popc(m & lt), room = 32 - fill, got = __popc(m);
                const bool self = ok && (unsigned)(j - i0s) < 32u;
                if (ok && r < room) {
                    S.st[fill + r] = q;
                    S.idx[nch * 32 + fill + r] = j;
                }
                own = own || __any_sync(kFull, self && r < room);
                if (got < room) {
                    fill += got;
                    return;
                }
                close(32);
                // (a round of several warps has no more than they keep)
                if (W == 1 && (nch == kCh || __any_sync(kFull, e > kCap - 32))) {
                    put(written, e);
                    written += e;
                    e = nch = 0;
                    __syncwarp();
                }
                if (ok && r >= room) {
                    S.st[r - room] = q;
                    S.idx[nch * 32 + r - room] = j;
                }
                own = __any_sync(kFull, self && r >= room);
                fill = got - room;
            });
            if (fill > 0) close(fill);
            int tot = written + e, from = written;
            if (W > 1) {
                s_cnt[warp][lane] = e;
                __syncthreads();
                tot = written;
#pragma unroll
                for (int v = 0; v < W; ++v) {
                    if (v == warp) from = tot;
                    tot += s_cnt[v][lane];
                }
            }
            if (mine && final_round) {
                cnt = tot;
                it = 1;
                if (cnt >= kp.n_target - kp.n_tol && cnt <= kp.n_target + kp.n_tol) {
                    conv = true;
                    active = false;
                } else if (it >= max_it) {
                    active = false;
                } else if (cnt < kp.n_target - kp.n_tol) {
                    lo = h;
                    h = __dmul_rn(h, 1.25);  // no upper bound yet
                } else {
                    hi = h;
                    h = __dmul_rn(h, 0.8);  // no lower bound yet
                }
            }
            if (mine && !(final_round && active)) put(from, W == 1 ? e : min(e, kCap));
            if (W > 1) __syncthreads();  // the counts and the columns are reused
            else __syncwarp();
            if (final_round) break;
            written = tot;
        }
    }
    if (warp != 0) return;
    // searches to go on with: few in a warp, or of a small instance, one warp
    // each (k_h_iterate); else the group together (k_h_union)
    const unsigned am = __ballot_sync(kFull, active);
    const bool few = __popc(am) <= kp.defer_lanes || __ldg(&B.icnt[inst]) < kGroupSearchN;
    if (handed || active) {
        posh[i].w = h;
        hs_lo[i] = lo;
        hs_hi[i] = hi;
        if (handed || few) {
            hs_it[i] = it;
            wl[atomicAdd(&status[3], 1u)] = (int32_t)i;
        }
    }
    if (!few) {
        if (inb && !handed) hs_it[i] = active ? it : -1;
        if (lane == 0) gwl[atomicAdd(&wctr[1], 1ull)] = (int32_t)blockIdx.x;
    }
    if (!inb || handed || active) return;
    nnb[i] = cnt;
    ngather[i] = cnt;
    if (!valid) return;
    write_reach2(xpk, i, h, g, kp);
    if (cnt > kGSlab) atomicOr(&status[2], (unsigned)IF_SLAB_OVF);
    if (!conv) {
        atomicOr(&status[0], (unsigned)ST_HNOCONV);
        atomicAdd(&status[1], 1u);
    }
}

// Persistent: warps take groups of 32 particles from a counter, so a group
// whose particles straddle far-apart cells (a jump of the Morton curve: a
// large query box, many candidates) delays one warp, not a whole wave.
template <bool LISTS>
__global__ void __launch_bounds__(kThreads, kUnionBlocksPerSM)
k_h_union(int64_t n, Batch B, double4_32a* posh, const float4* __restrict__ fpos,
          const int2* __restrict__ cells,
          int32_t* __restrict__ nnb, int32_t* __restrict__ ngather, int32_t* __restrict__ rslab,
          double* __restrict__ hs_lo, double* __restrict__ hs_hi, int32_t* __restrict__ hs_it,
          int32_t* __restrict__ wl, unsigned* __restrict__ status,
          unsigned long long* __restrict__ wctr, int2* __restrict__ recs,
          const int32_t* __restrict__ order, int32_t* __restrict__ lst,
          LMeta* __restrict__ lmeta, const int32_t* __restrict__ gwl, float4* __restrict__ xpk) {
    __shared__ float4 s_f[kThreads / 32][32];
    __shared__ int s_i[kThreads / 32][32];
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const long long ngroups = LISTS ? (n + 31) / 32 : (long long)wctr[1];
    for (;;) {
        long long gi = 0;
        if (lane == 0) gi = (long long)atomicAdd(wctr, 1ull);
        gi = __shfl_sync(kFull, gi, 0);
        if (gi >= ngroups) break;
        if (!LISTS) gi = gwl[gi];
        union_group<LISTS>(gi * 32, n, B, posh, fpos, cells, nnb, ngather, rslab, hs_lo, hs_hi, hs_it,
                    wl, status, s_f[warp], s_i[warp],
                    recs + ((int64_t)(blockIdx.x * (kThreads / 32) + warp) * 32 + lane) * kRec,
                    order, lst, lmeta, xpk);
    }
}

// The candidates of a list (ln entries 32 apart from L on), 32 at a time:
// chunk(valid, j, f) is called by all lanes together, lane l receiving entry
// e0 + l (valid = false past the end), as particle_pass hands out a walk's.
template <class Chunk>
__device__ __forceinline__ void list_pass(const int32_t* __restrict__ L, int ln,
                                          const float4* __restrict__ fpos, Chunk&& chunk) {
    const int lane = threadIdx.x & 31;
    for (int e0 = 0; e0 < ln; e0 += 32) {
        const int e = e0 + lane;
        const int j = e < ln ? __ldg(&L[e * 32]) : -1;
        chunk(j >= 0, j, j >= 0 ? __ldg(&fpos[j]) : make_float4(0.f, 0.f, 0.f, 0.f));
    }
}

// One warp per particle that goes on searching (persistent grid over the
// worklist), from the bracket its first count left. hs, the largest h the
// bisection can still test without growing (hi once bracketed; before, h, or
// 1.25 h for a first count), bounds the counts: one walk over the cells writes
// the candidates certainly within 2 lo to the row and records those that may
// lie within 2 hs in shared memory; the counts at every h <= hs come from the
// records, with a walk's FP32 / exact FP64 decisions. Every bracket update
// takes records out: those within 2 lo join the row, those beyond 2 hi are
// dropped; 32 or fewer are held one per lane. Only growth beyond hs walks the
// cells again, and more candidates than the buffer holds are counted by
// walking. Bound: issue (72% in a first step) and, with one particle per warp
// in flight, latency (issue 52% in a steady step). Measured: a steady step of
// the 1M patch 144 us (293 when the records kept everything within 1.25 times
// the next h and the row was written with every count), 27,000 particles from a
// poor h 172 us (300).
constexpr int kRecW = 512;  // records per warp

// h / 2 and 2 h of a normal h by its exponent (exact; no FP64 pipe, which
// serves one warp instruction in 16 cycles an SM)
__device__ __forceinline__ double scale_exp(double v, int e) {
    return __longlong_as_double(__double_as_longlong(v) + ((long long)e << 52));
}

// non-negative doubles order like their bits
__device__ __forceinline__ long long dbits(double v) { return __double_as_longlong(v); }
constexpr long long kInfBits = 0x7ff0000000000000LL;
constexpr long long kTinyBits = 0x0020000000000000LL;  // 2^-1021: halves and doubles are normal

// (a + b) / 2, both operations rounded
__device__ __forceinline__ double half_sum(double a, double b) {
    const double s = __dadd_rn(a, b);
    return dbits(s) > kTinyBits && dbits(s) < kInfBits ? scale_exp(s, -1) : __dmul_rn(0.5, s);
}

template <bool LISTS>
__global__ void __launch_bounds__(kThreads, 4)
k_h_iterate(Batch B, double4_32a* posh, const float4* __restrict__ fpos,
            const int2* __restrict__ cells,
            int32_t* __restrict__ nnb, int32_t* __restrict__ ngather,
            int32_t* __restrict__ rslab, const double* __restrict__ hs_lo,
            const double* __restrict__ hs_hi, const int32_t* __restrict__ hs_it,
            const int32_t* __restrict__ wl, unsigned* __restrict__ status,
            const int32_t* __restrict__ order, const int32_t* __restrict__ lst,
            const LMeta* __restrict__ lmeta, float4* __restrict__ xpk) {
    __shared__ int s_delta[kThreads / 32][32];
    __shared__ int2 s_rec[kThreads / 32][kRecW];  // (FP32 r^2 bits, j)
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const unsigned count = *(volatile unsigned*)&status[3];
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const unsigned lt = (1u << lane) - 1u;
    int2* rec = s_rec[warp];
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < count; w += nwarps) {
        const int i = wl[w];
        const int inst = slot_inst(B, i);
        const Grid* __restrict__ g = B.grid + inst;
        const KParams& kp = B.kp[inst];
        const int2* __restrict__ cl = cells + g->cbase;
        const int lowb = kp.n_target - kp.n_tol, highb = kp.n_target + kp.n_tol;
        const int max_it = kp.max_h_iter;
        const float4 fi = fpos[i];
        double h = posh[i].w, lo = hs_lo[i], hi = hs_hi[i];
        int cnt = 0;
        bool conv = false;
        int32_t* slab = rslab + (int64_t)i * kRSlab;
        long long hsb = -1;  // bits of hs, radius / 2 the records cover (-1: none)
        int nrec = 0;      // records: in shared memory, or one per lane (in_regs)
        int base = 0;      // row entries: certain neighbours at every h still to come
        bool in_regs = false;
        int2 own = make_int2(0x7f800000, -1);  // this lane's record (in_regs): r^2 = inf if none
        // the particle's kept candidate list, while it covers a radius 2 hq
        // (then it replaces the cell walk: the same candidates within 2 hq)
        const bool lists = LISTS && kp.list_skin > 0.0 && !g->lbuild;
        const int ln = lists ? lmeta[order[i]].cnt : 0;
        const float lrad = ln > 0 ? lmeta[order[i]].rad : 0.0f;
        const int32_t* L = lst + (i >> 5) * (int64_t)kList * 32 + (i & 31);
        auto list_covers = [&](double hq) { return ln > 0 && reach_f32(hq) + g->dm2 <= lrad; };
        // append j of the lanes with `in` to the row after its first c entries
        auto append = [&](bool in, int j, int c) {
            const unsigned m = __ballot_sync(kFull, in);
            const int q = c + __popc(m & lt);
            if (in && q < kGSlab) slab[q] = j;
            return __popc(m);
        };
        for (int it = hs_it[i]; it < max_it; ++it) {
            const double R = dbits(h) > kTinyBits ? scale_exp(h, 1) : 2.0 * h;
            const Thr t = thresholds(R, g);
            // r < 2h, decided as by a walk
            auto within = [&](float r2f, int j) {
                bool in = r2f < t.tin;
                const bool bd = !in && r2f <= t.tout && j >= 0;
                if (__any_sync(kFull, bd) && bd)
                    in = exact_r2(posh[i], posh[j], g) < __dmul_rn(R, R);
                return in;
            };
            int c = 0;
            unsigned bits = 0u;  // the decisions of this count: bit q / 32 of lane q % 32
            static_assert(kRecW <= 32 * 32, "one bit per word of records");
            if (!(dbits(h) <= hsb)) {
                // walk the cells once more: what is certainly within 2 lo to the
                // row, what may lie within 2 hs to the records
                const double hs = dbits(hi) != kInfBits ? hi : (dbits(lo) > 0 ? h : __dmul_rn(h, 1.25));
                hsb = dbits(hs);
                const float tout_s = thresholds(2.0 * hs, g).tout;
                const float tin_lo = dbits(lo) > 0 ? thresholds(2.0 * lo, g).tin : -1.0f;
                nrec = base = 0;
                in_regs = false;
                auto record = [&](bool valid, int j, const float4& f) {
                    const float r2f = valid && j != i ? f_r2(fi, f, g) : CUDART_INF_F;
                    base += append(r2f < tin_lo, j, base);
                    const bool keep = r2f >= tin_lo && r2f <= tout_s && valid && j != i;
                    const unsigned m = __ballot_sync(kFull, keep);
                    const int q = nrec + __popc(m & lt);
                    if (keep && q < kRecW) rec[q] = make_int2(__float_as_int(r2f), j);
                    nrec += __popc(m);
                };
                if (list_covers(hs)) list_pass(L, ln, fpos, record);
                else particle_pass<1>(g, cl, nullptr, fpos, fi, reach_f32(hs), 0, s_delta[warp], record);
                __syncwarp();
                if (nrec > kRecW) hsb = -1;  // too many to keep: count by walking
            }
            const bool kept = dbits(h) <= hsb;
            if (kept) {
                c = base;
                if (!in_regs && nrec <= 32) {
                    in_regs = true;
                    own = lane < nrec ? rec[lane] : make_int2(0x7f800000, -1);
                    __syncwarp();
                }
                if (in_regs) {
                    bits = within(__int_as_float(own.x), own.y) ? 1u : 0u;
                    c += __popc(__ballot_sync(kFull, bits != 0u));
                } else {
                    for (int q0 = 0; q0 < nrec; q0 += 32) {
                        const int2 e = q0 + lane < nrec ? rec[q0 + lane] : make_int2(0x7f800000, -1);
                        const bool in = within(__int_as_float(e.x), e.y);
                        bits |= in ? 1u << (q0 >> 5) : 0u;
                        c += __popc(__ballot_sync(kFull, in));
                    }
                }
            } else {
                auto walk = [&](bool valid, int j, const float4& f) {
                    const float r2f = valid && j != i ? f_r2(fi, f, g) : CUDART_INF_F;
                    c += append(within(r2f, valid && j != i ? j : -1) && valid && j != i, j, c);
                };
                if (list_covers(h)) list_pass(L, ln, fpos, walk);
                else particle_pass<1>(g, cl, nullptr, fpos, fi, reach_f32(h), 0, s_delta[warp], walk);
            }
            cnt = c;
            conv = cnt >= lowb && cnt <= highb;
            const bool last = conv || it == max_it - 1, low = cnt < lowb;
            if (kept) {
                // members join the row when this is the last count or lo rises to h;
                // the rest of the records stay while they lie between lo and hi
                if (in_regs) {
                    const bool in = bits != 0u;
                    if (last || low) base += append(in, own.y, base);
                    if (in == low) own = make_int2(0x7f800000, -1);
                } else {
                    int keep = 0;
                    for (int q0 = 0; q0 < nrec; q0 += 32) {
                        const int2 e = q0 + lane < nrec ? rec[q0 + lane] : make_int2(0x7f800000, -1);
                        const bool in = (bits >> (q0 >> 5)) & 1u;
                        if (last || low) base += append(in, e.y, base);
                        const bool stay = in != low && e.y >= 0;
                        const unsigned m = __ballot_sync(kFull, stay);
                        __syncwarp();  // (keep <= q0: the places written have been read)
                        if (stay) rec[keep + __popc(m & lt)] = e;
                        keep += __popc(m);
                    }
                    nrec = keep;
                    __syncwarp();
                }
            }
            if (last) break;
            if (low) {
                lo = h;
                h = dbits(hi) == kInfBits ? __dmul_rn(h, 1.25) : half_sum(lo, hi);
            } else {
                hi = h;
                h = dbits(lo) == 0 ? __dmul_rn(h, 0.8) : half_sum(lo, hi);
            }
        }
        __syncwarp();  // the records are reused by this warp's next particle
        if (lane == 0) {
            posh[i].w = h;
            write_reach2(xpk, i, h, g, kp);
            nnb[i] = cnt;
            ngather[i] = cnt;
            if (cnt > kGSlab) atomicOr(&status[2], (unsigned)IF_SLAB_OVF);
            if (!conv) {
                atomicOr(&status[0], (unsigned)ST_HNOCONV);
                atomicAdd(&status[1], 1u);
            }
        }
    }
}

// FP32 thresholds of particle i at its final h, for the kernels that look at
// pairs from both sides (k_outer, the CSR fallback).
__device__ __forceinline__ void write_thresholds(int64_t i, const Batch& B,
                                                 const double4_32a* __restrict__ posh,
                                                 float4* __restrict__ fpos, float* __restrict__ tin) {
    const int inst = slot_inst(B, i);
    if (!slot_real(B, inst, i)) return;
    const Thr t = thresholds(2.0 * posh[i].w, B.grid + inst);
    fpos[i].w = t.tout;
    tin[i] = t.tin;
}

__global__ void __launch_bounds__(kThreads)
k_thresholds(int64_t n, Batch B, const double4_32a* __restrict__ posh, float4* __restrict__ fpos,
             float* __restrict__ tin) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) write_thresholds(i, B, posh, fpos, tin);
}

// ------------------------------------------------------------ CSR
// Slab path (normal case). The h search left N_i at the start of row i of the
// row slab. The rest of S_i is the transpose of the non-mutual gather pairs:
// S_j \ N_j = { i : j in N_i and i not in N_j }: k_outer scans the gather
// sets and appends such i after N_j (atomic slot, so unordered),
// k_rowlen_sort sorts each outer part by index (deterministic rows) and forms
// |S_i|; k_compose copies the rows into a CSR when a caller asks for the
// neighbour list.
__global__ void __launch_bounds__(kThreads)
k_outer(int64_t n, Batch B, const double4_32a* __restrict__ posh,
        const float4* __restrict__ fpos, const float* __restrict__ tin,
        const int32_t* __restrict__ ngather, int32_t* __restrict__ rslab,
        int32_t* __restrict__ ocnt, unsigned* __restrict__ status) {
    const int lane = threadIdx.x & 31;
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n || (status[2] & IF_SLAB_OVF)) return;
    const int inst = slot_inst(B, i);
    if (!slot_real(B, inst, i)) return;
    const Grid* __restrict__ g = B.grid + inst;
    const int ng = ngather[i];
    const float4 fi = fpos[i];
    // the slab row is read up front so the dependent loads of the entries overlap
    constexpr int kPer = kGSlab / 32;
    int jj[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int s = k * 32 + lane;
        jj[k] = s < ng ? rslab[i * kRSlab + s] : -1;
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int j = jj[k];
        if (j < 0) continue;
        const float4 fj = __ldg(&fpos[j]);
        const float r2f = f_r2(fi, fj, g);
        bool in_j;
        if (r2f < __ldg(&tin[j])) {
            in_j = true;
        } else if (r2f > fj.w) {
            in_j = false;
        } else {
            const double4_32a pj = posh[j];
            const double Rj = 2.0 * pj.w;
            in_j = exact_r2(posh[i], pj, g) < __dmul_rn(Rj, Rj);
        }
        if (!in_j) {  // i joins the outer part of row j, after j's gather set
            const int q = __ldg(&ngather[j]) + atomicAdd(&ocnt[j], 1);
            if (q < kRSlab) rslab[(int64_t)j * kRSlab + q] = (int32_t)i;
            else atomicOr(&status[2], (unsigned)IF_SLAB_OVF);
        }
    }
}

// Row lengths, and the outer part of each row (appended in atomic order)
// sorted by index in place: the rows, and every sum over them, become
// deterministic. One warp per rw rows (4 to 32): the lengths are read and
// written coalesced, one row per lane, and the rows with something to sort (two
// outer entries or more) are taken four at a time, eight lanes each. A row's entries
// are read once, into shared memory; the rank of an entry (the indices of a
// row are distinct) is the number of smaller ones, and each is stored at its
// rank. Bounded by memory latency: there is no chain of dependent memory
// steps, as there was in the one-thread-per-row insertion sort this replaces.
constexpr int kSortLanes = 8;
constexpr int kSortRows = 32 / kSortLanes;  // rows a warp sorts at a time

__global__ void __launch_bounds__(kThreads)
k_rowlen_sort(int64_t n, const int32_t* __restrict__ ngather, const int32_t* __restrict__ ocnt,
              int32_t* __restrict__ rowlen, int32_t* rslab, const unsigned* __restrict__ status,
              unsigned mask, int rw) {
    if (status[2] & mask) return;
    __shared__ int pick[kThreads / 32][32];
    __shared__ int32_t ents[kThreads / kSortLanes][kRSlab];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane % kSortLanes;
    const int64_t i = ((int64_t)blockIdx.x * (kThreads / 32) + warp) * rw + lane;
    int ng = 0, no = 0;
    if (lane < rw && i < n) {
        ng = ngather[i];
        no = ocnt[i];
        rowlen[i] = ng + no;
    }
    const unsigned m = __ballot_sync(kFull, no > 1);
    if (no > 1) pick[warp][__popc(m & ((1u << lane) - 1u))] = lane;
    __syncwarp();
    const int rows = __popc(m);
    int32_t* e = ents[threadIdx.x / kSortLanes];
    for (int r = 0; r < rows; r += kSortRows) {
        const int at = r + lane / kSortLanes;
        const int src = at < rows ? pick[warp][at] : 0;
        const int rng = __shfl_sync(kFull, ng, src);
        const int rno = __shfl_sync(kFull, no, src);
        const int cnt = at < rows ? rno : 0;
        int32_t* row = rslab + (i - lane + src) * kRSlab + rng;
        for (int k = l; k < cnt; k += kSortLanes) e[k] = row[k];
        __syncwarp();
        for (int k = l; k < cnt; k += kSortLanes) {
            const int32_t v = e[k];
            int rank = 0;
            for (int q = 0; q < cnt; ++q) rank += e[q] < v ? 1 : 0;
            row[rank] = v;
        }
        __syncwarp();  // e is rewritten by the next rows
    }
}

// The rows as a CSR (for callers of the neighbour list): a copy of each row.
__global__ void __launch_bounds__(kThreads)
k_compose(int64_t n, const int32_t* __restrict__ rowlen, const int32_t* __restrict__ rslab,
          const int64_t* __restrict__ offsets, int32_t* __restrict__ idx, int64_t nnzcap,
          unsigned* __restrict__ status) {
    const int lane = threadIdx.x & 31;
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (status[2] & (IF_SLAB_OVF | IF_OUTER_OVF)) return;  // the fallback wrote the CSR
    if (offsets[n] > nnzcap) {
        if (i == 0 && lane == 0) atomicOr(&status[0], (unsigned)ST_CAPACITY);
        return;
    }
    if (i >= n) return;
    const int64_t off = offsets[i];
    const int len = rowlen[i];
    for (int s = lane; s < len; s += 32) idx[off + s] = __ldg(&rslab[i * kRSlab + s]);
}

// Fallback (a row overflowed a slab): the full two-pass build below. One warp,
// row i of an instance with grid g:
// FILL = false: rowlen[i] = |S_i|, ngather[i] = |N_i|; returns |S_i|.
// FILL = true : write the row (of rowlen[i] entries) at idx + first, N_i first,
//               with ballot-compacted, coalesced stores.
// A cell is visited when its box lies within 2 max(h_i, max h of the cell).
template <bool FILL>
__device__ __forceinline__ int csr_row(int64_t i, const Batch& B,
                                       const double4_32a* __restrict__ posh, const float4* fpos,
                                       const float* tin, const int2* __restrict__ cells,
                                       const unsigned long long* cell_hmax, int32_t* rowlen,
                                       int32_t* ngather, int64_t first, int32_t* __restrict__ idx,
                                       int* delta) {
    const int lane = threadIdx.x & 31;
    const int inst = slot_inst(B, i);
    if (!slot_real(B, inst, i)) {
        if (!FILL && lane == 0) {
            rowlen[i] = 0;
            ngather[i] = 0;
        }
        return 0;
    }
    const Grid* __restrict__ g = B.grid + inst;
    const int2* __restrict__ cl = cells + g->cbase;
    const unsigned long long* chm = cell_hmax + g->cbase;
    const double4_32a pi = posh[i];
    const float4 fi = fpos[i];
    const float tin_i = tin[i];
    const long long hib = __double_as_longlong(pi.w);
    const long long hgb = (long long)*(volatile const unsigned long long*)&g->hmax_bits;
    const float Rbig = reach_f32(__longlong_as_double(hgb > hib ? hgb : hib));
    double R2i = -1.0;
    const unsigned lt = (1u << lane) - 1u;
    int64_t pg = 0, po = 0, po_end = 0;
    if (FILL) {
        pg = first;
        po = pg + ngather[i];
        po_end = pg + rowlen[i];
    }
    int cg = 0, co = 0;
    particle_pass<2>(g, cl, chm, fpos, fi, Rbig, hib, delta,
                        [&](bool valid, int j, const float4& fj) {
        bool in_i = false, in_j = false;
        if (valid && j != i) {
            const float r2f = f_r2(fi, fj, g);
            bool bd_i = false;
            if (r2f < tin_i) in_i = true;
            else if (r2f <= fi.w) bd_i = true;
            double er2 = -1.0;
            if (bd_i) {
                if (R2i < 0.0) R2i = __dmul_rn(2.0 * pi.w, 2.0 * pi.w);
                er2 = exact_r2(pi, posh[j], g);
                in_i = er2 < R2i;
            }
            if (!in_i && r2f <= fj.w) {
                if (r2f < tin[j]) {
                    in_j = true;
                } else {
                    const double4_32a pj = posh[j];
                    if (er2 < 0.0) er2 = exact_r2(pi, pj, g);
                    const double Rj = 2.0 * pj.w;
                    in_j = er2 < __dmul_rn(Rj, Rj);
                }
            }
        }
        const unsigned gm = __ballot_sync(kFull, in_i);
        const unsigned om = __ballot_sync(kFull, in_j);
        if (FILL) {
            if (in_i) {
                const int64_t q = pg + cg + __popc(gm & lt);
                if (q < po) idx[q] = j;
            } else if (in_j) {
                const int64_t q = po + co + __popc(om & lt);
                if (q < po_end) idx[q] = j;
            }
        }
        cg += __popc(gm);
        co += __popc(om);
    });
    if (!FILL && lane == 0) {
        rowlen[i] = cg + co;
        ngather[i] = cg;
    }
    return cg + co;
}

// Wait, all threads of the block together, until *done items are done. False
// when kCsrIdle looks in a row (half a microsecond apart on average, so some 15 s)
// found no progress: reported (SPH_E_TIMEOUT), and the rows count as over
// capacity, so that nothing reads them.
constexpr int kCsrIdle = 1 << 25;
__device__ __forceinline__ bool csr_wait(const unsigned* done, unsigned target, int64_t* total,
                                         int64_t nnzcap, unsigned* status) {
    __shared__ bool s_ok;
    if (threadIdx.x == 0) {
        unsigned seen = 0u;
        bool ok = false;
        for (int idle = 0; idle < kCsrIdle; ++idle) {
            const unsigned v = *(volatile const unsigned*)done;
            ok = v >= target;
            if (ok) break;
            if (v != seen) idle = 0;
            seen = v;
            __nanosleep(500);
        }
        if (!ok) {
            atomicOr(&status[0], (unsigned)ST_TIMEOUT);
            *(volatile int64_t*)total = nnzcap + 1;
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok;
}

// An item of a phase is done (all threads together); the number done before it,
// valid in every thread.
__device__ __forceinline__ unsigned csr_done(unsigned* done) {
    __shared__ unsigned s_before;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_before = atomicAdd(done, 1u);
        __threadfence();
    }
    __syncthreads();
    return s_before;
}

// Rows of an item, of the 8 warps of a block in turn: the most while that leaves
// kCsrItems items for every block, else fewer, down to one a warp. A step of
// 90,003 particles with rows of 140 entries takes 1,988 us at two items a block
// (the last ones leave blocks idle), 1,886 at four, 1,915 at eight.
constexpr int kCsrWarps = kThreads / 32;
constexpr int kCsrRowsMax = 8, kCsrItems = 4;
__device__ __forceinline__ int csr_rows_per_item(int64_t n, int blocks) {
    const int64_t r = n / (kCsrItems * (int64_t)kCsrWarps * blocks);
    return kCsrWarps * (r < 1 ? 1 : (r > kCsrRowsMax ? kCsrRowsMax : (int)r));
}

// The whole fallback in one kernel. Without the flag every block returns at
// once: a step launches this twice, where the passes and the scan as kernels of
// their own made ten launches that did nothing (and two more kernels prepared in
// every step what only they read). Three phases of items: thresholds and the
// cells' max h; row lengths, summed per item, the sums scanned by whoever counts
// the last; offsets and rows. Blocks draw their items from one counter, in the
// order of the phases, and an item waits only for earlier phases, whose items all
// belong to blocks that run already: it ends for any number of resident blocks. (A
// cooperative launch with grid barriers, which needs all its blocks resident
// together, held back the work of other contexts: two contexts of 4,096
// particles on two streams took 251 us a step of both, now 186; eight of 27,000
// 1,303 and 1,070.)
__global__ void __launch_bounds__(kThreads)
k_csr_fallback(int64_t n, Batch B, Grid* gw_, const double4_32a* __restrict__ posh, float4* fpos,
               float* tin, const int2* __restrict__ cells, unsigned long long* cell_hmax,
               int32_t* rowlen, int32_t* ngather, int64_t* offsets, int64_t* part,
               int32_t* __restrict__ idx, int64_t nnzcap, unsigned* status, unsigned mask,
               CsrSync* Y) {
    if (!(*(volatile unsigned*)&status[2] & mask)) return;  // the slab path built the list
    __shared__ int s_delta[kCsrWarps][32];
    __shared__ int64_t s_sum[kCsrWarps];
    __shared__ int64_t s_off[kCsrWarps * kCsrRowsMax];
    __shared__ unsigned s_item;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rows = csr_rows_per_item(n, (int)gridDim.x);
    const unsigned nprep = (unsigned)((n + kThreads - 1) / kThreads);
    const unsigned nrow = (unsigned)((n + rows - 1) / rows);
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(&Y->next, 1u);
        __syncthreads();
        unsigned t = s_item;
        if (t < nprep) {  // 256 slots, of one instance, and their share of its cells
            const int64_t i = (int64_t)t * kThreads + threadIdx.x;
            const int inst = slot_inst(B, (int64_t)t * kThreads);
            if (i < n) write_thresholds(i, B, posh, fpos, tin);
            const int64_t all = (__ldg(&B.icnt[inst]) + kThreads - 1) / kThreads * kThreads;
            const long long nc = B.grid[inst].ncells, cb = B.grid[inst].cbase;
            long long most = 0;  // bits of positive doubles order like their values
            for (long long c = i - __ldg(&B.ioff[inst]); c < nc; c += all) {
                const int2 se = cells[cb + c];
                long long m = 0;
                for (int q = se.x; q < se.y; ++q) {
                    const long long hb = __double_as_longlong(posh[q].w);
                    m = (hb > m && hb <= kHMaxBits) ? hb : m;  // (h outside the geometry range: not counted)
                }
                cell_hmax[cb + c] = (unsigned long long)m;
                most = m > most ? m : most;
            }
            if (most > 0) atomicMax(&gw_[inst].hmax_bits, (unsigned long long)most);
            csr_done(&Y->prepared);
            continue;
        }
        t -= nprep;
        if (t < nrow) {
            if (!csr_wait(&Y->prepared, nprep, offsets + n, nnzcap, status)) return;
            const int64_t i0 = (int64_t)t * rows;
            int64_t sum = 0;
            for (int r = warp; r < rows && i0 + r < n; r += kCsrWarps)
                sum += csr_row<false>(i0 + r, B, posh, fpos, tin, cells, cell_hmax, rowlen, ngather,
                                      0, idx, s_delta[warp]);
            if (lane == 0) s_sum[warp] = sum;
            __syncthreads();
            if (threadIdx.x == 0) {
                int64_t a = 0;
                for (int w = 0; w < kCsrWarps; ++w) a += s_sum[w];
                part[t] = a;
            }
            if (csr_done(&Y->counted) + 1 != nrow) continue;
            // the last item counted: exclusive scan of the items' sums
            int64_t before = 0;
            for (unsigned q0 = 0; q0 < nrow; q0 += kThreads) {
                const unsigned q = q0 + threadIdx.x;
                const int64_t v = q < nrow ? part[q] : 0;
                int64_t inc = v;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int64_t u = __shfl_up_sync(kFull, inc, o);
                    if (lane >= o) inc += u;
                }
                __syncthreads();
                if (lane == 31) s_sum[warp] = inc;
                __syncthreads();
                int64_t off = before;
                for (int w = 0; w < kCsrWarps; ++w) {
                    off += w < warp ? s_sum[w] : 0;
                    before += s_sum[w];
                }
                if (q < nrow) part[q] = off + inc - v;
            }
            if (threadIdx.x == 0) {
                *(volatile int64_t*)&offsets[n] = before;
                if (before > nnzcap) atomicOr(&status[0], (unsigned)ST_CAPACITY);
            }
            csr_done(&Y->scanned);
            continue;
        }
        t -= nrow;
        if (t >= nrow || !csr_wait(&Y->scanned, 1u, offsets + n, nnzcap, status)) return;
        const int64_t i0 = (int64_t)t * rows;
        if (warp == 0) {  // offsets of the item's rows (at most two a lane)
            static_assert(kCsrWarps * kCsrRowsMax == 64, "two rows a lane");
            const int64_t ia = i0 + 2 * lane;
            const int64_t a = 2 * lane < rows && ia < n ? rowlen[ia] : 0;
            const int64_t b = 2 * lane + 1 < rows && ia + 1 < n ? rowlen[ia + 1] : 0;
            int64_t inc = a + b;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t u = __shfl_up_sync(kFull, inc, o);
                if (lane >= o) inc += u;
            }
            const int64_t off = part[t] + inc - (a + b);
            s_off[2 * lane] = off;
            s_off[2 * lane + 1] = off + a;
            if (2 * lane < rows && ia < n) offsets[ia] = off;
            if (2 * lane + 1 < rows && ia + 1 < n) offsets[ia + 1] = off + a;
        }
        __syncthreads();
        if (*(volatile int64_t*)&offsets[n] > nnzcap) continue;
        for (int r = warp; r < rows && i0 + r < n; r += kCsrWarps)
            csr_row<true>(i0 + r, B, posh, fpos, tin, cells, cell_hmax, rowlen, ngather, s_off[r],
                          idx, s_delta[warp]);
    }
}

// Blocks of the fallback, and the items of at most n rows: of kCsrRowsMax rows a
// warp, or of r < kCsrRowsMax, and then n < (r + 1) kCsrItems kCsrWarps blocks.
int csr_fallback_blocks(int nsm) { return 4 * nsm; }
int64_t csr_fallback_parts(int64_t n, int nsm) {
    return n / (kCsrWarps * kCsrRowsMax) + 2 * kCsrItems * (int64_t)csr_fallback_blocks(nsm) + 2;
}

void launch_h_search(sph_ctx* c, cudaStream_t s) {
    const int64_t n = c->n;
    if (n == 0) return;
    const unsigned nb = (unsigned)((n + kThreads - 1) / kThreads);
    double4_32a* posh = c->posh[c->cur];
    const Batch B = batch_of(c);
    c->launches += 2;  // the first count, k_h_iterate
    if (c->any_lists) {
        c->launches += 1;
        k_h_lists<<<nb, kThreads, 0, s>>>(n, B, posh, c->fpos, c->nnb, c->ngather, c->rslab,
                                          c->hs_lo, c->hs_hi, c->hs_it, c->wl, c->status,
                                          c->order[c->cur], c->lst, c->lmeta, c->xpk);
    }
    const int64_t nbu = std::min<int64_t>((int64_t)c->nsm * kUnionBlocksPerSM, ((n + 31) / 32 + 7) / 8);
    if (c->any_lists) {
        k_h_union<true><<<(unsigned)nbu, kThreads, 0, s>>>(
            n, B, posh, c->fpos, c->cells, c->nnb, c->ngather, c->rslab, c->hs_lo, c->hs_hi,
            c->hs_it, c->wl, c->status, c->wctr, c->recs, c->order[c->cur], c->lst, c->lmeta, c->gwl, c->xpk);
        k_h_iterate<true><<<kReduceBlocks * 4, kThreads, 0, s>>>(
            B, posh, c->fpos, c->cells, c->nnb, c->ngather, c->rslab, c->hs_lo, c->hs_hi,
            c->hs_it, c->wl, c->status, c->order[c->cur], c->lst, c->lmeta, c->xpk);
    } else {
        const int64_t groups = (n + 31) / 32;
        auto count = [&](auto fn, int warps) {
            fn<<<(unsigned)groups, 32 * warps, 0, s>>>(n, B, posh, c->fpos, c->cells, c->nnb,
                                                       c->ngather, c->rslab, c->hs_lo, c->hs_hi,
                                                       c->hs_it, c->wl, c->gwl, c->status, c->wctr,
                                                       c->xpk);
        };
        // Warps per group: as many as fill the chip once. Measured (first count,
        // us, with 8 / 4 / 2 / 1 warps): 4,096 particles 24 / 31 / 48 / 86, the
        // 8,191-particle sphere 45 / 51 / 71 / 126, 27,000 45 / 38 / 38 / 80, 104k
        // 174 / 129 / 122 / 118, the 200k sphere 446 / 321 / 289 / 270.
        const int64_t room = (int64_t)c->nsm * 24;
        if (groups * 2 > room) count(k_h_count<1>, 1);
        else if (groups * 4 > room) count(k_h_count<2>, 2);
        else if (groups * 8 > room) count(k_h_count<4>, 4);
        else count(k_h_count<8>, 8);
        if (c->group_search) {
            c->launches += 1;
            k_h_union<false><<<(unsigned)nbu, kThreads, 0, s>>>(
                n, B, posh, c->fpos, c->cells, c->nnb, c->ngather, c->rslab, c->hs_lo, c->hs_hi,
                c->hs_it, c->wl, c->status, c->wctr, c->recs, c->order[c->cur], c->lst, c->lmeta,
                c->gwl, c->xpk);
        }
        k_h_iterate<false><<<kReduceBlocks * 4, kThreads, 0, s>>>(
            B, posh, c->fpos, c->cells, c->nnb, c->ngather, c->rslab, c->hs_lo, c->hs_hi,
            c->hs_it, c->wl, c->status, c->order[c->cur], c->lst, c->lmeta, c->xpk);
    }
}

// The two-pass CSR build, for the rows flagged in status[2] & mask (launched
// every step; without the flag it returns at once). The step's two launches
// have their own counters (CsrSync, cleared with every build).
static void csr_fallback(sph_ctx* c, cudaStream_t s, unsigned mask) {
    c->launches += 1;
    k_csr_fallback<<<(unsigned)csr_fallback_blocks(c->nsm), kThreads, 0, s>>>(
        c->n, batch_of(c), c->grid, c->posh[c->cur], c->fpos, c->tin, c->cells, c->cell_hmax,
        c->rowlen, c->ngather, c->offsets, c->row_part, c->idx, c->nnzcap, c->status, mask,
        c->csync + (mask == (unsigned)IF_OUTER_OVF ? 1 : 0));
}

static void rowlen_sort(sph_ctx* c, cudaStream_t s, unsigned mask) {
    // a warp's rows are sorted four at a time, one round of memory latency each:
    // fewer rows per warp while the warps do not fill the chip (measured: 4,096
    // particles 7 us at 4 rows and 19 at 32, the 8,191-particle sphere 13 and 50;
    // the one-thread-per-row sort took 39 and 140). At 32: 1M patch 43 us (84
    // before), 1M sphere 78 us (182 before).
    int rw = kSortRows;
    while (rw < 32 && c->n >= (int64_t)c->nsm * 32 * 2 * rw) rw *= 2;
    const int64_t per = (int64_t)(kThreads / 32) * rw;
    k_rowlen_sort<<<(unsigned)((c->n + per - 1) / per), kThreads, 0, s>>>(
        c->n, c->ngather, c->ocnt, c->rowlen, c->rslab, c->status, mask, rw);
}

void launch_csr(sph_ctx* c, cudaStream_t s, bool outer_later) {
    const int64_t n = c->n;
    c->csr_ready = false;
    if (n == 0) {
        c->launches += 1;
        cudaMemsetAsync(c->offsets, 0, sizeof(int64_t), s);
        return;
    }
    const unsigned nbw = (unsigned)((n * 32 + kThreads - 1) / kThreads);
    double4_32a* posh = c->posh[c->cur];
    const Batch B = batch_of(c);
    if (!outer_later) {
        c->launches += 3;
        k_thresholds<<<(unsigned)((n + kThreads - 1) / kThreads), kThreads, 0, s>>>(
            n, B, posh, c->fpos, c->tin);
        k_outer<<<nbw, kThreads, 0, s>>>(n, B, posh, c->fpos, c->tin, c->ngather, c->rslab,
                                         c->ocnt, c->status);
        rowlen_sort(c, s, (unsigned)IF_SLAB_OVF);
    }
    // fallback (a row did not fit its slab): the full two-pass build into the CSR
    csr_fallback(c, s, (unsigned)IF_SLAB_OVF);
}

// After a density kernel that appended the outer entries: sort them, and build the CSR instead if one of them overflowed its slab.
void launch_rows_finish(sph_ctx* c, cudaStream_t s) {
    const int64_t n = c->n;
    if (n == 0) return;
    c->launches += 1;
    rowlen_sort(c, s, (unsigned)(IF_SLAB_OVF | IF_OUTER_OVF));
    csr_fallback(c, s, (unsigned)IF_OUTER_OVF);
}

void launch_compose(sph_ctx* c, cudaStream_t s) {
    const int64_t n = c->n;
    c->csr_ready = true;
    if (n == 0) return;
    const unsigned nbw = (unsigned)((n * 32 + kThreads - 1) / kThreads);
    c->launches += 4;
    // row offsets of the slab rows (the steps scan them only for the fallback)
    launch_scan_i32_i64(c->rowlen, n, c->offsets, c->row_part, s);
    k_compose<<<nbw, kThreads, 0, s>>>(n, c->rowlen, c->rslab, c->offsets, c->idx, c->nnzcap,
                                       c->status);
}

}  // namespace sph
