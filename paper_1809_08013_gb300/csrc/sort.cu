// sort.cu -- Algorithm 1 step 1 (the tree build), done as Morton-sorted cell
// lists: bounding box and cell grid on the device, 24-bit Morton key of each
// particle's cell, a stable LSD radix sort (3 passes of 8 bits, one more for
// the instance id of a batch; one kernel per pass), the permutation of the
// particle state into sorted order with the [start, end) range of every
// occupied cell.
//
// The keys are sorted in caller order (each particle at its "rank" roff[k] +
// its index within its instance), not in the order the previous step left,
// so particles of one cell always end up ordered by caller index: the
// internal order -- and with it every summation order -- depends only on the
// positions, and a run split into several calls gives the same bits as one.
#include <math_constants.h>

#include "df.cuh"
#include "sph_internal.cuh"

namespace sph {

// ------------------------------------------------------------------ state I/O
// Caller arrays (instances back to back) into the slot layout: instance k's
// particle r goes to slot ioff[k] + r; empty slots get an inert state and
// order = -1.
__global__ void __launch_bounds__(kThreads)
k_load_state(int64_t n, Batch B, const int64_t* __restrict__ coff, const double* __restrict__ x,
             const double* __restrict__ y, const double* __restrict__ z,
             const double* __restrict__ h, const double* __restrict__ vx,
             const double* __restrict__ vy, const double* __restrict__ vz,
             const double* __restrict__ m, const double* __restrict__ u,
             double4_32a* __restrict__ posh, double4_32a* __restrict__ velm,
             double* __restrict__ ue, int32_t* __restrict__ order, double4_32a* __restrict__ posh2,
             double4_32a* __restrict__ velm2, double* __restrict__ ue2, int32_t* __restrict__ order2,
             int32_t* __restrict__ ocnt) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int inst = slot_inst(B, k);
    const int64_t r = k - __ldg(&B.ioff[inst]);
    if (r >= __ldg(&B.icnt[inst])) {  // empty slot, inert in both buffers (never permuted)
        posh[k] = posh2[k] = make_double4_32a(0.0, 0.0, 0.0, 1.0);
        velm[k] = velm2[k] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
        ue[k] = ue2[k] = 0.0;
        order[k] = order2[k] = -1;
        ocnt[k] = 0;
        return;
    }
    const int64_t c = __ldg(&coff[inst]) + r;
    posh[k] = make_double4_32a(x[c], y[c], z[c], h[c]);
    velm[k] = make_double4_32a(vx ? vx[c] : 0.0, vy ? vy[c] : 0.0, vz ? vz[c] : 0.0, m ? m[c] : 0.0);
    ue[k] = u ? u[c] : 0.0;
    order[k] = (int32_t)c;
}

void launch_load_state(sph_ctx* c, const sph_particles* P, cudaStream_t s) {
    const int64_t n = c->n;
    if (n == 0) return;
    const int b = c->cur;
    c->launches += 1;
    k_load_state<<<(unsigned)((n + kThreads - 1) / kThreads), kThreads, 0, s>>>(
        n, batch_of(c), c->coff, P->x, P->y, P->z, P->h, P->vx, P->vy, P->vz, P->m, P->u,
        c->posh[b], c->velm[b], c->ue[b], c->order[b], c->posh[1 - b], c->velm[1 - b],
        c->ue[1 - b], c->order[1 - b], c->ocnt);
}

// Pack of the double-float pair kernels for particle k: the fixed-point chunks
// of its position (dfl::to_fx, exponents of its instance) and its mass, both
// in the pair kernels' units of the instance,
//   xpk[3k] = (x.c2, y.c2, z.c2, m.hi), xpk[3k+1] = (x.c1, y.c1, z.c1, m.lo),
//   xpk[3k+2] = (x.c0, y.c0, z.c0, 0).
__device__ __forceinline__ void write_xpk(float4* __restrict__ xpk, int64_t k, const double4_32a& p,
                                          double mass, const Grid& g) {
    const int f = g.fxk + g.uL;
    const dfl::fx3 X = dfl::to_fx(p.x, g.fxk, f), Y = dfl::to_fx(p.y, g.fxk, f);
    const dfl::fx3 Z = dfl::to_fx(p.z, g.fxk, f);
    const dfl::df m = dfl::from_double_fp64(mass * p2d(-g.uM));
    xpk[3 * k + 0] = make_float4(X.c2, Y.c2, Z.c2, m.hi);
    xpk[3 * k + 1] = make_float4(X.c1, Y.c1, Z.c1, m.lo);
    xpk[3 * k + 2] = make_float4(X.c0, Y.c0, Z.c0, 0.0f);
}

// Velocity of particle k as float pairs in the velocity unit 2^uV of its
// instance (the double-float force kernels' view of it).
__device__ __forceinline__ void write_vpk(float4* __restrict__ vpa, float2* __restrict__ vpb,
                                          int64_t k, const double4_32a& v, const Grid& g) {
    const double sv = p2d(-g.uV);
    const dfl::df x = dfl::from_double_fp64(v.x * sv), y = dfl::from_double_fp64(v.y * sv);
    const dfl::df z = dfl::from_double_fp64(v.z * sv);
    vpa[k] = make_float4(x.hi, x.lo, y.hi, y.lo);
    vpb[k] = make_float2(z.hi, z.lo);
}

// Re-read the caller's arrays into the sorted order of the last build and
// derive the per-particle quantities the pair kernels load for j.
__global__ void __launch_bounds__(kThreads)
k_gather_state(int64_t n, int what, int precision, double alpha, const int32_t* __restrict__ order,
               const double* __restrict__ x, const double* __restrict__ y,
               const double* __restrict__ z, const double* __restrict__ h,
               const double* __restrict__ vx, const double* __restrict__ vy,
               const double* __restrict__ vz, const double* __restrict__ m,
               const double* __restrict__ rho, const double* __restrict__ p,
               const double* __restrict__ cs, double4_32a* __restrict__ posh,
               double4_32a* __restrict__ velm, double4_32a* __restrict__ therm,
               double2* __restrict__ kern, double* __restrict__ cint, float4* __restrict__ dpk,
               float4* __restrict__ xpk, float4* __restrict__ vpa, float2* __restrict__ vpb,
               const Grid* __restrict__ grid, unsigned* status) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int64_t o = order[k];
    if (o < 0) return;  // empty slot
    const double hh = h[o];
    const double4_32a ps = make_double4_32a(x[o], y[o], z[o], hh);
    posh[k] = ps;
    const double mm = m[o];
    const Grid& g = grid[0];  // a single problem: instance 0
    write_xpk(xpk, k, ps, mm, g);
    if (what == GATHER_DENSITY) {
        velm[k] = make_double4_32a(0.0, 0.0, 0.0, mm);
    } else {
        const double4_32a vv = make_double4_32a(vx[o], vy[o], vz[o], mm);
        velm[k] = vv;
        if (precision == PREC_FP64) write_vpk(vpa, vpb, k, vv, g);
        const double r = rho[o], c = cs[o];
        const double hinv = 1.0 / hh;
        const double h2 = hinv * hinv;
        const double A = p[o] / (r * r);
        therm[k] = make_double4_32a(0.5 * r, A, 0.5 * alpha * c, 0.5 * hh);
        kern[k] = make_double2(hinv, h2 * h2);
        if (precision == PREC_FP64)  // the double-float kernels' pack
            dfl::write_pack(dpk, k, hinv, A, hh, r, alpha, c, dfl::pair_units(g.uL, g.uM, g.uV),
                            status, ST_RANGE);
        cint[k] = c;
    }
}

void launch_gather_state(sph_ctx* c, const sph_particles* P, const KParams& kp, int what,
                         cudaStream_t s) {
    const int64_t n = c->n;
    if (n == 0) return;
    const int b = c->cur;
    c->launches += 1;
    k_gather_state<<<(unsigned)((n + kThreads - 1) / kThreads), kThreads, 0, s>>>(
        n, what, kp.precision, kp.alpha, c->order[b], P->x, P->y, P->z, P->h, P->vx, P->vy, P->vz, P->m,
        P->rho, P->p, P->c, c->posh[b], c->velm[b], c->therm, c->kern, c->cint, c->dpk, c->xpk,
        c->vpa, c->vpb, c->grid, c->status);
}

// ------------------------------------------------------------ bbox and grid
// Min / max of doubles as signed 64-bit integer min / max of order-preserving
// keys (GB300's FP64 pipe is narrow; integer compares are not on it).
__device__ __forceinline__ long long okey(double x) {
    const long long b = __double_as_longlong(x);
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double okey_inv(long long k) {
    return __longlong_as_double(k >= 0 ? k : (k ^ 0x7fffffffffffffffLL));
}

constexpr long long kKeyMax = 0x7fffffffffffffffLL, kKeyMin = -kKeyMax - 1;

// Bounding-box partials: min x, y, z and max x, y, z, h, m, |v| (largest
// component), u (as keys) and the sum of h over the particles of each group
// of kSlotAlign slots (one instance), one block of kSlotAlign / kBoxWarpSlots
// warps per group, reduced in a fixed
// order; with candidate lists also the largest displacement since the last
// list build, the smallest list slack (list radius - 2h), and the largest and
// smallest build stamp. Stored as kBoxStride doubles per group: mn[3],
// mx[11], hs.
constexpr int kBoxMax = 11;
enum { BX_D = 7, BX_NSLACK = 8, BX_STAMP = 9, BX_NSTAMP = 10 };

struct BoxPart {
    long long mn[3], mx[kBoxMax];
    double hs;
};

__device__ __forceinline__ void box_init(BoxPart& b) {
    for (int d = 0; d < 3; ++d) b.mn[d] = kKeyMax;
    for (int d = 0; d < kBoxMax; ++d) b.mx[d] = kKeyMin;
    b.hs = 0.0;
}

// Fixed-order warp reduction of the first NMAX maxima (the others untouched).
template <int NMAX = kBoxMax>
__device__ __forceinline__ void box_warp_reduce(BoxPart& b) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const long long v = __shfl_xor_sync(0xffffffffu, b.mn[d], o);
            b.mn[d] = v < b.mn[d] ? v : b.mn[d];
        }
#pragma unroll
        for (int d = 0; d < NMAX; ++d) {
            const long long v = __shfl_xor_sync(0xffffffffu, b.mx[d], o);
            b.mx[d] = v > b.mx[d] ? v : b.mx[d];
        }
        b.hs += __shfl_xor_sync(0xffffffffu, b.hs, o);
    }
}

static_assert(kSlotAlign % kBoxWarpSlots == 0 && kBoxWarpSlots % 32 == 0, "bbox groups");
constexpr int kBoxThreads = kSlotAlign / kBoxWarpSlots * 32;  // one block per group

// LISTS: some instance keeps candidate lists (their statistics are gathered).
template <bool LISTS>
__global__ void __launch_bounds__(kBoxThreads)
k_bbox(int64_t n, Batch B, const double4_32a* __restrict__ posh,
       const double4_32a* __restrict__ velm, const double* __restrict__ ue,
       const int32_t* __restrict__ order, const LMeta* __restrict__ lmeta,
       double* __restrict__ part, unsigned* __restrict__ status, uint32_t* __restrict__ hist,
       int64_t nhist) {
    // the digit counts of the sort that follows, cleared for k_keys and its passes
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nhist;
         t += (int64_t)gridDim.x * blockDim.x)
        hist[t] = 0u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t grp = blockIdx.x;  // group of kSlotAlign slots (< n: one block per group)
    const int64_t w0 = grp * kSlotAlign + (int64_t)warp * kBoxWarpSlots;
    const int inst = slot_inst(B, grp * kSlotAlign);
    const int64_t end = __ldg(&B.ioff[inst]) + __ldg(&B.icnt[inst]);
    const KParams& kp = B.kp[inst];
    const bool lists = LISTS && kp.list_skin > 0.0;
    const bool per = kp.periodic_z != 0;
    const float lzf = (float)kp.lz, hlzf = 0.5f * lzf;
    BoxPart b;
    box_init(b);
    bool bad = false;
#pragma unroll
    for (int q = 0; q < kBoxWarpSlots / 32; ++q) {
        const int64_t k = w0 + q * 32 + lane;
        if (k < end) {
            // a particle outside the geometry range (NaN, infinity, beyond the
            // FP32 range) is reported and kept out of the box and the means:
            // the cells, the search and the units stay those of the others
            const double4_32a p = posh[k];
            const double4_32a v = velm[k];
            const double uk = ue[k];
            const bool geo = coord_ok(p.x) && coord_ok(p.y) && coord_ok(p.z) && h_ok(p.w);
            const bool fin = finite_bits(v.x) && finite_bits(v.y) && finite_bits(v.z) &&
                             finite_bits(v.w) && finite_bits(uk);
            if (lists && geo) {
                // since the last list build: the displacement (truncated floats,
                // the minimum image along a periodic z), the list's slack at the
                // current h, the build stamp
                const int32_t id = order[k];
                const float4 m0 = __ldg(reinterpret_cast<const float4*>(lmeta) + 2 * id);
                const int4 m1 = __ldg(reinterpret_cast<const int4*>(lmeta) + 2 * id + 1);
                const float dx = dfl::from_double(p.x).hi - m0.x;
                const float dy = dfl::from_double(p.y).hi - m0.y;
                float dz = dfl::from_double(p.z).hi - m0.z;
                if (per) {
                    if (dz > hlzf) dz -= lzf;
                    else if (dz < -hlzf) dz += lzf;
                }
                const long long kd = __float_as_int(sqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx))));
                b.mx[BX_D] = kd > b.mx[BX_D] ? kd : b.mx[BX_D];  // NaN keys above +inf
                if (m1.z > 0) {
                    const long long ks = fkey(reach_f32(p.w) - m0.w);
                    b.mx[BX_NSLACK] = ks > b.mx[BX_NSLACK] ? ks : b.mx[BX_NSLACK];
                }
                b.mx[BX_STAMP] = m1.x > b.mx[BX_STAMP] ? m1.x : b.mx[BX_STAMP];
                b.mx[BX_NSTAMP] = -(long long)m1.x > b.mx[BX_NSTAMP] ? -(long long)m1.x : b.mx[BX_NSTAMP];
            }
            bad |= !(geo && fin);
            if (!(geo && fin)) continue;
            const long long kx = okey(p.x), ky = okey(p.y), kz = okey(p.z), kh = okey(p.w);
            b.mn[0] = kx < b.mn[0] ? kx : b.mn[0];
            b.mn[1] = ky < b.mn[1] ? ky : b.mn[1];
            b.mn[2] = kz < b.mn[2] ? kz : b.mn[2];
            b.mx[0] = kx > b.mx[0] ? kx : b.mx[0];
            b.mx[1] = ky > b.mx[1] ? ky : b.mx[1];
            b.mx[2] = kz > b.mx[2] ? kz : b.mx[2];
            b.mx[3] = kh > b.mx[3] ? kh : b.mx[3];
            b.hs += p.w;
            const long long km = okey(v.w), ku = okey(uk);
            const long long kv = okey(fmax(fabs(v.x), fmax(fabs(v.y), fabs(v.z))));
            b.mx[4] = km > b.mx[4] ? km : b.mx[4];
            b.mx[5] = kv > b.mx[5] ? kv : b.mx[5];
            b.mx[6] = ku > b.mx[6] ? ku : b.mx[6];
        }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, (unsigned)ST_NONFINITE);
    // without lists the list fields are neither reduced nor written (nothing reads them)
    constexpr int NMAX = LISTS ? kBoxMax : BX_D;
    box_warp_reduce<NMAX>(b);
    __shared__ BoxPart wb[kBoxThreads / 32];
    if (lane == 0) wb[warp] = b;
    __syncthreads();
    if (threadIdx.x == 0) {  // the block's warps in order: a fixed summation order
        BoxPart a = wb[0];
        for (int w = 1; w < kBoxThreads / 32; ++w) {
            for (int d = 0; d < 3; ++d) a.mn[d] = wb[w].mn[d] < a.mn[d] ? wb[w].mn[d] : a.mn[d];
            for (int d = 0; d < NMAX; ++d) a.mx[d] = wb[w].mx[d] > a.mx[d] ? wb[w].mx[d] : a.mx[d];
            a.hs += wb[w].hs;
        }
        double* o = part + grp * kBoxStride;
        for (int d = 0; d < 3; ++d) o[d] = __longlong_as_double(a.mn[d]);
        for (int d = 0; d < NMAX; ++d) o[3 + d] = __longlong_as_double(a.mx[d]);
        o[3 + kBoxMax] = a.hs;
    }
}

__device__ __forceinline__ int grid_count(double ext, double w, double* wout) {
    double c = floor(ext / w) + 1.0;
    if (c > (double)kMaxCellsPerAxis) c = (double)kMaxCellsPerAxis;
    if (!(c >= 1.0)) c = 1.0;  // also a NaN extent: never an empty axis
    double ww = w;
    if (c * ww <= ext) ww = ext / (c - 0.5);
    *wout = ww;
    return (int)c;
}

// One block per instance: reduce the instance's bbox partials (fixed order:
// thread t takes partials t, t + 1024, ..., then a fixed tree) and derive its
// cell grid. The cell width is 2 <h> cell_scale (<h> the mean smoothing
// length), widened while the grid would exceed the instance's cell budget;
// the neighbour sets do not depend on it, only the candidates visited do.
constexpr int kGridThreads = 1024;

__global__ void __launch_bounds__(kGridThreads)
k_grid_setup(const double* __restrict__ part, Batch B, Grid* __restrict__ grid,
             unsigned* __restrict__ status, unsigned long long* __restrict__ wctr,
             unsigned* __restrict__ lctr, CsrSync* __restrict__ csync) {
    const int inst = blockIdx.x;
    const int64_t n = B.icnt[inst];
    const int64_t b0 = B.ioff[inst] / kSlotAlign;
    const int64_t nbk = (n + kSlotAlign - 1) / kSlotAlign;
    // field f = t % 16 of every 64th partial from partial t / 16 on: each
    // load instruction of a warp reads two whole partials. Fields 0-2 are
    // minima, 3 .. 3 + kBoxMax - 1 maxima, 3 + kBoxMax the sum of h.
    static_assert(kBoxStride == 16 && 3 + kBoxMax < kBoxStride, "bbox partial layout");
    const int f = threadIdx.x & 15;
    const bool fmin_ = f < 3, fsum = f == 3 + kBoxMax;
    long long acc = fmin_ ? kKeyMax : kKeyMin;
    double hsum = 0.0;
    const double* base = part + b0 * kBoxStride + f;
    for (int64_t b = threadIdx.x >> 4; b < nbk; b += kGridThreads / 16) {
        const double v = base[b * kBoxStride];
        const long long k = __double_as_longlong(v);
        if (fmin_) acc = k < acc ? k : acc;
        else acc = k > acc ? k : acc;
        if (fsum) hsum += v;
    }
    // lanes l and l + 16 hold the same field: combine, lower lane first (a
    // fixed order), then the warps in order
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    {
        const long long ok = __shfl_xor_sync(0xffffffffu, acc, 16);
        const double oh = __shfl_xor_sync(0xffffffffu, hsum, 16);
        acc = fmin_ ? (ok < acc ? ok : acc) : (ok > acc ? ok : acc);
        hsum = lane < 16 ? hsum + oh : oh + hsum;
    }
    static_assert(kGridThreads / 32 == 32, "one lane per warp's partial below");
    __shared__ long long wk[kGridThreads / 32][16];
    __shared__ double wh[kGridThreads / 32];
    if (lane < 16) wk[warp][lane] = acc;
    if (lane == 3 + kBoxMax) wh[warp] = hsum;
    __syncthreads();
    // warp f combines field f over the warps by shuffles (one thread combining
    // all of them in turn took half of this kernel's time at small sizes); the
    // sum of h in the order of the warps
    __shared__ long long fk[3 + kBoxMax];
    __shared__ double hs;
    if (warp < 3 + kBoxMax) {
        long long v = wk[lane][warp];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long u = __shfl_xor_sync(0xffffffffu, v, o);
            v = warp < 3 ? (u < v ? u : v) : (u > v ? u : v);
        }
        if (lane == 0) fk[warp] = v;
    } else if (warp == 3 + kBoxMax && lane == 0) {
        double a = 0.0;
        for (int w = 0; w < kGridThreads / 32; ++w) a += wh[w];
        hs = a;
    }
    __syncthreads();
    if (warp != 0) return;
    // The rest is one warp: lane d (0 to 2) takes axis d, the others repeat
    // axis 2; the divisions of the three axes and of the mean run side by side.
    const int d = lane < 2 ? lane : 2;
    const long long* lk = fk + 3 + BX_D;  // list keys: displacement, -slack, stamp, -stamp
    const KParams& kp = B.kp[inst];
    Grid* g = grid + inst;
    const bool per = kp.periodic_z != 0;
    const double lz = kp.lz;
    double mn = okey_inv(fk[d]), mx = okey_inv(fk[3 + d]);
    // no particle, or none inside the geometry range
    if (n == 0 || !__all_sync(0xffffffffu, mn <= mx)) {
        if (n == 0 || !(mn <= mx)) { mn = 0.0; mx = 0.0; }
    }
    if (inst == 0 && lane == 0) {
        status[2] = 0u;
        status[3] = 0u;
        wctr[0] = 0ull;
        wctr[1] = 0ull;
        csync[0] = csync[1] = CsrSync{0u, 0u, 0u, 0u};
    }
    const double hmean = n > 0 ? hs / (double)n : 1.0;
    double w = 2.0 * hmean * kp.cell_scale;
    if (!(w > 0.0) || !isfinite(w)) w = 1.0;
    double X = fmax(fabs(mn), fabs(mx));
    X = fmax(X, __shfl_xor_sync(0xffffffffu, X, 1));
    X = fmax(__shfl_sync(0xffffffffu, X, 0), __shfl_sync(0xffffffffu, X, 2));
    if (per) X = fmax(X, 0.5 * lz);
    // Candidate lists of the h search. The instance keeps its lists while
    // every particle carries the same build stamp and twice the largest
    // displacement since that build (bounded with the truncation errors of
    // both positions) is below every list's slack at the current h: then any
    // j within 2 h of i now was within the list radius at the build, and is
    // listed. Otherwise this step rebuilds them under a new stamp. While they
    // are kept, so are the build's cell geometry and (through the sort keys)
    // its cells, whose walks then reach further by the displacement bound.
    bool keep = false;
    float dm2 = CUDART_INF_F;
    int stamp = 0;
    if (kp.list_skin > 0.0 && n > 0) {
        const long long smax = lk[2], smin = -lk[3];
        const bool epoch = smax == smin && smin > 0;
        const float D = lk[0] == kKeyMin ? 0.0f : __int_as_float((int)lk[0]);
        const double Dm = (double)D * (1.0 + 0x1p-20) + 0x1p-20 * (X + (double)D);
        dm2 = (float)(2.0 * Dm * (1.0 + 0x1p-20));
        const float slack = lk[1] == kKeyMin ? CUDART_INF_F : -fkey_inv(lk[1]);
        keep = epoch && g->gvalid && dm2 < slack;  // false for a NaN displacement
        if (keep) stamp = (int)smin;
        else if (lane == 0) stamp = (int)((atomicAdd(lctr, 1u) & 0x3fffffffu) + 1u);
    }
    int cnt = 1;
    double ww = 1.0, lo = mn;
    if (!keep) {
        const long long cellcap = g->cap;
        long long cells = 1;
        for (int tries = 0; tries < 200; ++tries) {
            if (per && d == 2) {
                double c = floor(lz / w);
                if (c < 1.0) c = 1.0;
                if (c > (double)kMaxCellsPerAxis) c = (double)kMaxCellsPerAxis;
                cnt = (int)c;
                lo = -0.5 * lz;
                ww = lz / c;
            } else {
                cnt = grid_count(mx - mn, w, &ww);
            }
            cells = (long long)__shfl_sync(0xffffffffu, cnt, 0) *
                    __shfl_sync(0xffffffffu, cnt, 1) * __shfl_sync(0xffffffffu, cnt, 2);
            if (cells <= cellcap) break;
            w *= 1.25;
        }
        if (lane < 3) {
            const double inv = 1.0 / ww;
            g->lo[d] = lo;
            g->w[d] = ww;
            g->inv_w[d] = inv;
            g->n[d] = cnt;
            g->lof[d] = (float)lo;
            g->wf[d] = (float)ww;
            g->invwf[d] = (float)inv;
        }
        if (lane == 0) {
            // (an empty instance has no cells: no block clears or marks them)
            g->ncells = n > 0 ? cells : 0;
            g->gvalid = 1;
        }
    } else {
        ww = g->w[d];
    }
    if (lane < 3)
        g->slop[d] = (float)(1e-3 * ww + 1.2e-7 * X + (keep ? 0.5 * 1.001 * dm2 : 0.0));
    if (lane != 0) return;
    g->lstamp = stamp;
    g->lbuild = kp.list_skin > 0.0 && n > 0 && !keep ? 1 : 0;
    g->dm2 = dm2;
    g->periodic_z = per ? 1 : 0;
    g->lz = lz;
    g->lzf = (float)lz;
    g->halflzf = (float)(0.5 * lz);
    g->X = X;
    g->Xf = __double2float_ru(X);
    g->lzerr = __double2float_ru(fabs(lz - (double)(float)lz));
    // |fl32 difference - FP64 difference| <= 2^-24 (4X + 2.02R + 2 lz) per
    // component (conversions of both coordinates, the FP32 subtraction, the
    // periodic shift); 1.0001 and the upward rounding keep it an upper bound
    const double u24 = 5.9604644775390625e-08;
    g->eC = __double2float_ru(u24 * (4.0 * X + (per ? 2.0 * lz : 0.0)) * 1.0001 + 1e-37);
    g->eR = __double2float_ru(u24 * 2.02 * 1.0001);
    // Units of the pair kernels (Grid::uL, uM, uV): the power of two at or
    // just above the mean h, the largest mass and a velocity scale (the
    // largest |v| component, or the sound speed the parameters imply if that
    // is larger: c0 for Tait, sqrt(gamma (gamma - 1) max u) for an ideal gas).
    // The exponents come from the bits (v < 2^e; a subnormal ends at the
    // clamp).
    auto exp2_of = [](double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7ff) - 1022; };
    auto unit_exp = [&](double v) {
        if (!(v > 0.0) || !isfinite(v)) return 0;
        const int e = exp2_of(v);
        return e < -300 ? -300 : (e > 300 ? 300 : e);
    };
    const double umax = okey_inv(fk[3 + 6]);
    double vs = n > 0 ? okey_inv(fk[3 + 5]) : 0.0;
    if (kp.eos == 0) vs = fmax(vs, fabs(kp.c0));
    else if (n > 0 && umax > 0.0) vs = fmax(vs, sqrt(kp.gamma * (kp.gamma - 1.0) * umax));
    const int uL = unit_exp(hmean);
    g->uL = uL;
    g->uM = unit_exp(n > 0 ? okey_inv(fk[3 + 4]) : 0.0);
    g->uV = unit_exp(vs);
    // fixed-point exponent of the coordinate chunks (dfl::to_fx): |x| 2^k < 2^61,
    // and the chunks' float exponent k + uL must keep them normal floats
    int k = X > 0.0 && isfinite(X) ? 61 - exp2_of(X) : 61;
    k = k < -1000 ? -1000 : (k > 1000 ? 1000 : k);
    if (k + uL > 100 || k + uL < -60) {  // coordinates out of all proportion to h
        k = k + uL > 100 ? 100 - uL : -60 - uL;
        if (kp.precision == PREC_FP64) atomicOr(&status[0], (unsigned)ST_RANGE);
    }
    g->fxk = k;
    const dfl::fx3 L = dfl::to_fx(per ? lz : 0.0, k, k + uL);
    g->lzc[0] = L.c2;
    g->lzc[1] = L.c1;
    g->lzc[2] = L.c0;
    g->hlzc = (float)(0.5 * lz * p2d(-uL));
    g->hmean = hmean;
    g->hmax_bits = 0ull;
}

// ----------------------------------------------------------- Morton keys
__device__ __forceinline__ uint32_t spread3(uint32_t v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

__device__ __forceinline__ uint32_t compact3(uint32_t v) {
    v &= 0x09249249u;
    v = (v | (v >> 2)) & 0x030c30c3u;
    v = (v | (v >> 4)) & 0x0300f00fu;
    v = (v | (v >> 8)) & 0x030000ffu;
    v = (v | (v >> 16)) & 0x000003ffu;
    return v;
}

// Cell index along one axis, in FP32 from the truncated float of v (integer
// operations, no FP64 pipe). The neighbour search widens every query box by
// the grid's slop (>= 1e-3 cell widths), far more than these roundings, so
// any particle within reach of a query lies in a cell the query visits.
__device__ __forceinline__ int cell_coord(double v, float lo, float inv, int n) {
    const float f = floorf((dfl::from_double(v).hi - lo) * inv);
    const int top = n > 1 ? n - 1 : 0;
    if (!(f >= 0.0f)) return 0;  // also catches NaN
    if (f > (float)top) return top;
    return (int)f;
}

// key = instance (top 8 bits) | 24-bit Morton code of the particle's cell in
// its instance's grid, stored at the particle's rank roff[k] + (caller index
// - coff[k]) with its current slot as the value.
// While the instance keeps its candidate lists, the code is the particle's
// code at the list build, so the sort gives every particle its slot of then;
// a build step records the codes it sorts by.
// Also counts the keys' first digits (a chained sort) and clears the cells.
__global__ void __launch_bounds__(kThreads)
k_keys(int64_t n, Batch B, const int64_t* __restrict__ coff, const int64_t* __restrict__ roff,
       const double4_32a* __restrict__ posh, const int32_t* __restrict__ order,
       uint32_t* __restrict__ keys, int32_t* __restrict__ vals, LMeta* __restrict__ lmeta,
       RadixGeom R, uint32_t* __restrict__ hist, int2* __restrict__ cells) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int inst = slot_inst(B, (int64_t)blockIdx.x * blockDim.x);
    const Grid* g = B.grid + inst;
    {
        const int64_t all = (__ldg(&B.icnt[inst]) + kThreads - 1) / kThreads * kThreads;
        const long long nc = g->ncells, cb = g->cbase;
        for (long long c = k - __ldg(&B.ioff[inst]); c < nc; c += all) cells[cb + c] = make_int2(0, 0);
    }
    if (k >= n) return;
    if (!slot_real(B, inst, k)) return;
    const bool lists = B.kp[inst].list_skin > 0.0;
    const int32_t id = order[k];
    uint32_t code;
    if (lists && !g->lbuild) {
        code = lmeta[id].code;
    } else {
        const double4_32a p = posh[k];
        const int kx = cell_coord(p.x, g->lof[0], g->invwf[0], g->n[0]);
        const int ky = cell_coord(p.y, g->lof[1], g->invwf[1], g->n[1]);
        const int kz = cell_coord(p.z, g->lof[2], g->invwf[2], g->n[2]);
        code = spread3(kx) | (spread3(ky) << 1) | (spread3(kz) << 2);
        if (lists) lmeta[id].code = code;
    }
    const int64_t q = __ldg(&roff[inst]) + ((int64_t)id - __ldg(&coff[inst]));
    keys[q] = ((uint32_t)inst << 24) | code;
    vals[q] = (int32_t)k;
    if (R.chained) R.count(hist, q >> R.tile_shift, code & 255u, 1u);
}

// --------------------------------------------------------- stable radix sort
// The blocks of a pass need, for every digit, the number of keys with a
// smaller digit and of keys with that digit in earlier tiles; both come from
// counts per tile and per group of tiles. Small sorts (RadixGeom::chained) are
// one kernel per pass: whoever writes a key to its place for a pass (k_keys,
// or the pass before) knows the tile it lands in and its next digit, and
// counts it by atomic additions (integers: the order does not matter). Large
// ones, where those additions cost more than reading the keys once more
// (measured at 1M: 35 us a pass against 8), count in a kernel of their own.
// Either way no scan kernels: a histogram kernel and the three kernels of a
// scan in each pass made 15 launches of 3-7 us each in a 27k-particle step.
__global__ void __launch_bounds__(kThreads)
k_radix_hist(const uint32_t* __restrict__ keys, int64_t n, int shift, RadixGeom R,
             uint32_t* __restrict__ hist) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kThreads * kRadixItems;
#pragma unroll
    for (int k = 0; k < kRadixItems; ++k) {
        const int64_t i = base + k * kThreads + threadIdx.x;
        if (i < n) atomicAdd(&h[(keys[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    R.count(hist, blockIdx.x, threadIdx.x, h[threadIdx.x]);
}

// Each warp ranks a contiguous run of keys in (iteration, lane) order, so the
// rank of a key among equal digits follows its input position: stable.
template <int ITEMS, bool NEXT>
__global__ void __launch_bounds__(kThreads)
k_radix_scatter(const uint32_t* __restrict__ kin, const int32_t* __restrict__ vin, int64_t n,
                int shift, RadixGeom R, const uint32_t* __restrict__ hist,
                uint32_t* __restrict__ next, uint32_t* __restrict__ kout,
                int32_t* __restrict__ vout) {
    __shared__ uint32_t cnt[kThreads / 32][256];
    __shared__ uint32_t wtot[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * (kThreads * ITEMS) + warp * (32 * ITEMS);
    uint32_t key[ITEMS];
    int32_t val[ITEMS];
    uint32_t rank[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int64_t i = base + it * 32 + lane;
        key[it] = i < n ? kin[i] : 0u;
        val[it] = i < n ? vin[i] : 0;
    }
    // thread d: keys of digit d in all tiles, and in the tiles before this one
    uint32_t total = 0, before = 0;
    {
        static_assert(kThreads == 256 && kRadixThreads == kThreads, "one digit per thread");
        const int d = threadIdx.x;
        const int tile = (int)blockIdx.x;
        if (R.groups == 1) {
#pragma unroll 8
            for (int t = 0; t < R.tiles; ++t) {
                const uint32_t v = __ldg(&hist[t * 256 + d]);
                total += v;
                before += t < tile ? v : 0u;
            }
        } else {
            const int grp = tile >> R.group_shift;
            const uint32_t* groups = hist + (int64_t)R.tiles * 256;
#pragma unroll 8
            for (int g = 0; g < R.groups; ++g) {
                const uint32_t v = __ldg(&groups[g * 256 + d]);
                total += v;
                before += g < grp ? v : 0u;
            }
#pragma unroll 8
            for (int t = grp << R.group_shift; t < tile; ++t)
                before += __ldg(&hist[(int64_t)t * 256 + d]);
        }
    }
    uint32_t inc = total;  // inclusive scan of the totals over the digits
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) wtot[warp] = inc;
    for (int q = threadIdx.x; q < (kThreads / 32) * 256; q += kThreads) (&cnt[0][0])[q] = 0;
    __syncthreads();
    uint32_t start = before + inc - total;  // place of this tile's first key of digit d
    for (int w = 0; w < warp; ++w) start += wtot[w];
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const bool ok = base + it * 32 + lane < n;
        const uint32_t d = ok ? ((key[it] >> shift) & 255u) : 256u;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t b = ok ? cnt[warp][d] : 0u;
        __syncwarp();
        if (ok && lane == __ffs(peers) - 1) cnt[warp][d] = b + __popc(peers);
        __syncwarp();
        rank[it] = b + __popc(peers & lt);
    }
    __syncthreads();
    {
        const int d = threadIdx.x;
        uint32_t run = start;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            const uint32_t c = cnt[w][d];
            cnt[w][d] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        if (base + it * 32 + lane < n) {
            const uint32_t pos = cnt[warp][(key[it] >> shift) & 255u] + rank[it];
            kout[pos] = key[it];
            vout[pos] = val[it];
            if (NEXT) R.count(next, pos >> R.tile_shift, (key[it] >> (shift + 8)) & 255u, 1u);
        }
    }
}

// ------------------------------------------------------ permute and cells
// Sorted rank p of instance i goes to slot ioff[i] + (p - roff[i]); the first
// and the last particle of a cell write its range (in slots).
__global__ void __launch_bounds__(kThreads)
k_permute(int64_t ntot, Batch B, const int64_t* __restrict__ roff,
          const uint32_t* __restrict__ keys, const int32_t* __restrict__ perm,
          const double4_32a* __restrict__ posh_in,
          const double4_32a* __restrict__ velm_in, const double* __restrict__ u_in,
          const int32_t* __restrict__ order_in, double4_32a* __restrict__ posh_out,
          double4_32a* __restrict__ velm_out, double* __restrict__ u_out,
          int32_t* __restrict__ order_out, float4* __restrict__ fpos, float4* __restrict__ xpk,
          float4* __restrict__ vpa, float2* __restrict__ vpb, int2* __restrict__ cells,
          int32_t* __restrict__ ocnt) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= ntot) return;
    const int64_t o = perm[r];
    const uint32_t key = keys[r];
    const int inst = (int)(key >> 24);
    const int64_t a = __ldg(&roff[inst]), e = a + __ldg(&B.icnt[inst]);
    const int64_t k = __ldg(&B.ioff[inst]) + (r - a);
    const bool first = (r == a) || keys[r - 1] != key;
    const bool last = (r == e - 1) || keys[r + 1] != key;
    if (first || last) {
        const Grid* g = B.grid + inst;
        const uint32_t code = key & 0xffffffu;
        const int kx = compact3(code), ky = compact3(code >> 1), kz = compact3(code >> 2);
        const long long lin = g->cbase + ((long long)kz * g->n[1] + ky) * g->n[0] + kx;
        if (first) cells[lin].x = (int)k;
        if (last) cells[lin].y = (int)(k + 1);
    }
    const double4_32a p = posh_in[o];
    posh_out[k] = p;
    const double4_32a v = velm_in[o];
    velm_out[k] = v;
    write_xpk(xpk, k, p, v.w, B.grid[inst]);
    if (B.kp[inst].precision == PREC_FP64) write_vpk(vpa, vpb, k, v, B.grid[inst]);
    u_out[k] = u_in[o];
    order_out[k] = order_in[o];
    fpos[k] = make_float4((float)p.x, (float)p.y, (float)p.z, 0.0f);
    ocnt[k] = 0;  // outer entries of the row, to be appended
}

void launch_build_cells(sph_ctx* c, cudaStream_t s) {
    const int64_t n = c->n;
    const unsigned nb = (unsigned)((n + kThreads - 1) / kThreads);
    const Batch B = batch_of(c);
    const int64_t nt = c->ntot;
    const RadixGeom R = radix_geom(nt);
    const int passes = c->ninst > 1 ? 4 : 3;
    c->launches += 1;
    if (nb > 0) {  // one block per group of kSlotAlign slots
        c->launches += 1;
        const unsigned gb = (unsigned)((n + kSlotAlign - 1) / kSlotAlign);
        if (c->any_lists)
            k_bbox<true><<<gb, kBoxThreads, 0, s>>>(n, B, c->posh[c->cur], c->velm[c->cur],
                                                 c->ue[c->cur], c->order[c->cur], c->lmeta,
                                                 c->red_part, c->status, c->hist,
                                                 passes * R.counts());
        else
            k_bbox<false><<<gb, kBoxThreads, 0, s>>>(n, B, c->posh[c->cur], c->velm[c->cur],
                                                  c->ue[c->cur], c->order[c->cur], c->lmeta,
                                                  c->red_part, c->status, c->hist,
                                                  passes * R.counts());
    }
    k_grid_setup<<<c->ninst, kGridThreads, 0, s>>>(c->red_part, B, c->grid, c->status, c->wctr,
                                                    c->lctr, c->csync);
    if (n == 0) return;
    if (nt == 0) return;
    const unsigned nbt = (unsigned)((nt + kThreads - 1) / kThreads);
    c->launches += 2 + passes;
    k_keys<<<nb, kThreads, 0, s>>>(n, B, c->coff, c->roff, c->posh[c->cur], c->order[c->cur],
                                   c->keys[0], c->vals[0], c->lmeta, R, c->hist, c->cells);
    int src = 0;
    for (int pass = 0; pass < passes; ++pass) {
        const uint32_t* h = c->hist + pass * R.counts();
        auto go = [&](auto fn) {
            fn<<<(unsigned)R.tiles, kThreads, 0, s>>>(c->keys[src], c->vals[src], nt, 8 * pass, R, h,
                                                      c->hist + (pass + 1) * R.counts(),
                                                      c->keys[1 - src], c->vals[1 - src]);
        };
        if (!R.chained) {
            c->launches += 1;
            k_radix_hist<<<(unsigned)R.tiles, kThreads, 0, s>>>(
                c->keys[src], nt, 8 * pass, R, c->hist + pass * R.counts());
            go(k_radix_scatter<kRadixItems, false>);
        } else if (pass + 1 < passes) {
            go(k_radix_scatter<kRadixItemsSmall, true>);
        } else {
            go(k_radix_scatter<kRadixItemsSmall, false>);
        }
        src = 1 - src;
    }
    // sorted keys / permutation now in keys[src], vals[src]
    const int a = c->cur, b = 1 - c->cur;
    k_permute<<<nbt, kThreads, 0, s>>>(nt, B, c->roff, c->keys[src], c->vals[src], c->posh[a],
                                        c->velm[a], c->ue[a], c->order[a], c->posh[b], c->velm[b],
                                        c->ue[b], c->order[b], c->fpos, c->xpk, c->vpa, c->vpb,
                                        c->cells, c->ocnt);
    c->cur = b;
}

}  // namespace sph
