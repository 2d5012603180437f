// Master problem (Eq. 6): min F(DA y) subject to lo <= y <= hi, by
// Barzilai-Borwein steps (Eq. 7-8, used alternately) with the subspace scheme
// of Eq. 9-10 and the stopping rules of Section 2.1.
//
// The paper runs four steps per iteration on one GPU (aperture gradient, step
// length with cuBLAS dot products, subspace update, dose update).  Here one
// persistent cooperative kernel runs a whole solve.  DA is kept in a warp-tile
// layout: blocks of 32 voxels, each block a 128-byte head holding the 32 voxels'
// structure labels, then the apertures in groups of four with the four values
// of a voxel side by side,
//     DA(i, k) = DA[(i / 32) * wstride + 32 + (k / 4) * 128 + (i % 32) * 4 + k % 4],
// so the labels and the first n columns of a block are one contiguous run of
// 128 + 512 ceil(n / 4) bytes.  Every warp streams its own blocks into shared
// memory with one bulk copy each (several in flight on the warp's own mbarrier
// ring, continuing across iterations; no CTA-wide barrier in the loop); each
// lane owns a voxel, reads its four-aperture groups with 128-bit shared loads,
// forms z = DA y with four independent chains, the objective term and
// g = -grad F, and adds DA_ik g_i to its register-resident shares of
// G = grad_y F = -DA^T g.  DA is read from HBM (or L2, when it fits there) once
// per iteration.  Objective terms w d^2 are formed in FP32 and summed per lane
// with compensation (Kahan), then as float pairs across lanes and CTAs: the
// voxel loop runs no FP64 instruction (FP64 issues at a small fraction of the
// FP32 rate on this GPU).  The CTA partials of every column are then summed in a
// fixed order by one CTA each and the sums sent to all (exchange_columns: tagged
// words, no barrier), and every CTA takes the same step in shared memory: the
// Eq. 9-10 freeze, the stopping tests, the BB step length (FP64) and the projected
// update.  The first iteration's Cauchy
// step needs DA G and one more pass.
//
// Readings (where the paper is silent): G is the gradient of F, so both BB
// step lengths are positive and Eq. 9-10 freeze at lo when G > 0 and at hi when
// G < 0; y is projected onto the box after each step; BB1 on even and BB2 on
// odd iterations; s.r <= 0 takes the largest step; steps are clamped to
// [delta_min, delta_max] times the Cauchy step.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "internal.cuh"

namespace vmat {

constexpr int MP_THREADS = 256; // voxels per tile of the fallback and Cauchy kernels
constexpr int MP_NW = MP_THREADS / 32;
constexpr int MP_WT = 32;       // voxels per warp tile
constexpr int MP_HEAD = 32;     // floats of a warp tile's label head (128 bytes)
constexpr int MP_CHUNK = 8;     // iterations launched between host polls
constexpr size_t MP_SMEM_LIMIT = 220 * 1024;
constexpr int RES_COPIES = 32; // copies of the reduced columns (a lane of the owner's warp writes each)
constexpr int MP_NMAX = 96; // register-resident gradient shares: up to 96 apertures

struct BBState {
    double F_hist[6];
    double F;
    double delta0;
    double gg;
    int32_t t;
    int32_t done;
    int32_t stop;
    int32_t iters;
    int32_t need_cauchy;
    uint32_t ticket;  // CTAs of the current pass that have written their partials
    int32_t started;  // elastic batched solver: the state below t was saved by a previous epoch
};

struct MPArgs {
    const float *DA; // warp-tile layout (see above)
    int64_t wstride; // floats per 32-voxel warp tile (32 + 128 * groups)
    int32_t V, n;
    const uint8_t *sid;
    const float *T, *wo, *wu;
    int32_t n_struct;
    float *y;
    float *z;
    const float *lo, *hi; // may be null
    double *G, *Gprev;
    float *yprev;
    double *part;  // fallback solver: [P][n + 1] doubles
    double *cpart; // fallback solver: [P]
    // exchange of the persistent solvers (see exchange_columns): tagged float pairs
    ulonglong2 *slots; // [n + 1][pstride]: column k of CTA c at k * pstride + c
    ulonglong2 *res;   // [RES_COPIES][rstride]: the reduced columns, then the elastic solver's epoch
    int32_t rstride;
    unsigned *tag;     // tags up to this one have been used in slots and res
    int32_t pstride;   // CTAs a column of slots has room for
    int32_t n_tiles;  // 256-voxel tiles (fallback and Cauchy kernels)
    int64_t n_wtiles; // 32-voxel warp tiles
    BBState *st;
    const int32_t *skip;           // when non-null and set, the solve is skipped (device-driven plans)
    int32_t *iters_acc;            // when non-null, the persistent solver adds its iteration count
    double *bytes_acc;             // when non-null, the persistent solver adds the bytes its passes moved
    int32_t *status;
    vmat_bb_opts opts;
    double F_offset;
    // Live-tile solves (tiles may be null: every tile): only the warp tiles
    // tiles[0 .. *n_live) of DA are in the problem (the tiles some placed aperture
    // reaches), and *F_off_dev, the constant penalty of the others, is added to F.
    const int32_t *tiles;
    const int32_t *n_live;
    const double *F_off_dev;
    // Packed live tiles (null: read DA's tiles whole): list entry i at 128-byte unit poff[i] of
    // packed, its head (labels, group mask at byte 32) then its marked groups.
    const float *packed;
    const int32_t *poff;
};

// A value that is the same in the whole warp, in a form the compiler knows to be so: branches
// and loops on it are then uniform.  Inside a branch on threadIdx.x / 32, or a loop to a
// bound read from shared memory, it cannot rule out a diverged warp, and every shuffle and
// vote there took 230 cycles instead of 31.
__device__ __forceinline__ int warp_uniform(int x) { return __shfl_sync(0xffffffffu, x, 0); }
__device__ __forceinline__ int warp_index() { return warp_uniform((int)(threadIdx.x >> 5)); }

__device__ __forceinline__ int64_t min64(int64_t x, int64_t y) { return x < y ? x : y; }

// Offset of DA(voxel i, aperture k) in the warp-tile layout.
__device__ __forceinline__ int64_t da_at(const MPArgs &a, int64_t i, int k) {
    return (i >> 5) * a.wstride + MP_HEAD + (int64_t)(k >> 2) * 128 + ((i & 31) << 2) + (k & 3);
}

__device__ __forceinline__ float lo_of(const MPArgs &a, int k) { return a.lo ? a.lo[k] : 0.f; }
__device__ __forceinline__ float hi_of(const MPArgs &a, int k) { return a.hi ? a.hi[k] : INFINITY; }

__global__ void mp_init_kernel(MPArgs a) {
    if (a.skip && *a.skip) return;
    for (int k = threadIdx.x; k < a.n; k += blockDim.x) a.y[k] = fminf(fmaxf(a.y[k], lo_of(a, k)), hi_of(a, k));
    if (threadIdx.x == 0) {
        BBState s = {};
        *a.st = s;
    }
}

// Fixed-order block reductions (result valid in every thread).
__device__ double block_reduce_sum(double v, double *sh) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < MP_NW; ++w) t += sh[w];
    return t;
}

__device__ void finish(BBState *st, int reason, int t) {
    st->done = 1;
    st->stop = reason;
    st->iters = t + 1;
}

// Projected update y <- clamp(y - delta G) after saving (y, G) as the previous iterate.
__device__ void take_step(const MPArgs &a, double delta) {
    for (int k = threadIdx.x; k < a.n; k += MP_THREADS) {
        const float yk = a.y[k];
        a.yprev[k] = yk;
        a.Gprev[k] = a.G[k];
        const double yn = (double)yk - delta * a.G[k];
        a.y[k] = fminf(fmaxf((float)yn, lo_of(a, k)), hi_of(a, k));
    }
}

// G_k = -sum_b part[b][k] and F = sum_b part[b][n] + offset.  One warp per column;
// lane l sums blocks l, l + 32, ... in order, then a fixed butterfly.
__device__ void reduce_partials(const MPArgs &a, int P) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = a.n;
    for (int k = wid; k <= n; k += MP_NW) {
        double s = 0.0;
        // other CTAs' writes: bypass L1; 8 loads in flight per lane
#pragma unroll 8
        for (int b = lane; b < P; b += 32) s += __ldcg(a.part + (int64_t)b * (n + 1) + k);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if (lane == 0) {
            if (k < n) a.G[k] = -s;
            else a.st->F = s + a.F_offset + (a.F_off_dev ? __ldcg(a.F_off_dev) : 0.0);
        }
    }
    __syncthreads();
}

// Eq. 9-10 freeze, stopping tests, BB step length and projected update (one block).
__device__ void bb_step(const MPArgs &a) {
    BBState *st = a.st;
    __shared__ double sh[MP_NW];
    __shared__ int decided;
    __shared__ double delta_s;
    const int t = st->t;
    const int n = a.n;
    for (int k = threadIdx.x; k < n; k += MP_THREADS) {
        const float yk = a.y[k], l = lo_of(a, k), h = hi_of(a, k);
        const double g = a.G[k];
        if (yk <= l && g > 0.0) {
            a.y[k] = l;
            a.G[k] = 0.0;
        } else if (yk >= h && g < 0.0) {
            a.y[k] = h;
            a.G[k] = 0.0;
        }
    }
    __syncthreads();
    const double F = st->F;
    double dy = 0.0, ymax = 0.0, gg = 0.0, ss = 0.0, sr = 0.0, rr = 0.0;
    for (int k = threadIdx.x; k < n; k += MP_THREADS) {
        const double yk = a.y[k], g = a.G[k];
        ymax = fmax(ymax, fabs(yk));
        gg += g * g;
        if (t > 0) {
            const double s = yk - (double)a.yprev[k], r = g - a.Gprev[k];
            dy = fmax(dy, fabs(s));
            ss += s * s;
            sr += s * r;
            rr += r * r;
        }
    }
    { // one combined block reduction of the six quantities (two maxima, four sums)
        __shared__ double red[MP_NW][6];
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            dy = fmax(dy, __shfl_down_sync(0xffffffffu, dy, d));
            ymax = fmax(ymax, __shfl_down_sync(0xffffffffu, ymax, d));
            gg += __shfl_down_sync(0xffffffffu, gg, d);
            ss += __shfl_down_sync(0xffffffffu, ss, d);
            sr += __shfl_down_sync(0xffffffffu, sr, d);
            rr += __shfl_down_sync(0xffffffffu, rr, d);
        }
        if (lane == 0) {
            red[wid][0] = dy;
            red[wid][1] = ymax;
            red[wid][2] = gg;
            red[wid][3] = ss;
            red[wid][4] = sr;
            red[wid][5] = rr;
        }
        __syncthreads();
        dy = red[0][0];
        ymax = red[0][1];
        gg = red[0][2];
        ss = red[0][3];
        sr = red[0][4];
        rr = red[0][5];
        for (int w = 1; w < MP_NW; ++w) {
            dy = fmax(dy, red[w][0]);
            ymax = fmax(ymax, red[w][1]);
            gg += red[w][2];
            ss += red[w][3];
            sr += red[w][4];
            rr += red[w][5];
        }
    }
    if (threadIdx.x == 0) {
        decided = 1;
        st->F_hist[t % 6] = F;
        if (t >= 5 && fabs(st->F_hist[(t - 5) % 6] - F) <= a.opts.rel_tol5 * F) finish(st, VMAT_STOP_REL, t);
        else if (t >= 1 && dy <= a.opts.step_tol * fmax(1.0, ymax)) finish(st, VMAT_STOP_STEP, t);
        else if (t == a.opts.max_iter - 1) finish(st, VMAT_STOP_MAXIT, t);
        else if (t == 0) {
            if (gg == 0.0) finish(st, VMAT_STOP_GRAD0, t);
            else {
                st->gg = gg;
                st->need_cauchy = 1; // the step length needs DA G
            }
        } else {
            double delta;
            if (sr <= 0.0) delta = a.opts.delta_max * st->delta0;
            else if (t & 1) delta = sr / rr;
            else delta = ss / sr;
            delta = fmin(fmax(delta, a.opts.delta_min * st->delta0), a.opts.delta_max * st->delta0);
            delta_s = delta;
            decided = 0;
        }
    }
    __syncthreads();
    if (!decided) {
        take_step(a, delta_s);
        if (threadIdx.x == 0) st->t = t + 1;
    }
}

// Per-voxel part of an iteration for voxel i with dose zi (fallback kernel):
// returns g_i, adds F_i to facc.
__device__ __forceinline__ float voxel_terms(const float *sT, const float *sO, const float *sU, int s, float zi,
                                             double &facc) {
    const float d = zi - sT[s];
    const float w = d > 0.f ? sO[s] : sU[s];
    facc += (double)((w * d) * d);
    return -2.f * w * d; // g = -grad F: -2 w+ (z - T) above, +2 w- (T - z) below
}

// Ends a pass: write this CTA's partials; the last of the n_cta CTAs reduces them and steps.
__device__ void pass_epilogue(const MPArgs &a, const double *accG, double facc, int cta, int n_cta) {
    __shared__ double sh[MP_NW];
    __shared__ bool last;
    const int tid = threadIdx.x;
    const double fb = block_reduce_sum(facc, sh);
    double *out = a.part + (int64_t)cta * (a.n + 1);
    for (int k = tid; k < a.n; k += MP_THREADS) out[k] = accG[k];
    if (tid == 0) out[a.n] = fb;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&a.st->ticket, 1u) == (unsigned)n_cta - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    reduce_partials(a, n_cta);
    bb_step(a);
    if (tid == 0) a.st->ticket = 0u;
}

// Bytes one bulk copy brings for n apertures: a warp tile's label head and its first ceil(n/4) groups.
__host__ __device__ constexpr size_t wt_copy_bytes(int n) { return 128 + (size_t)((n + 3) / 4) * 512; }

// ---------------------------------------------------------------------------
// Persistent solver: one cooperative launch runs the whole BB loop.  Every
// iteration is a pass over DA (each warp streams its own tiles), the exchange of
// the CTA partials' sums, and the step, which every CTA computes identically in
// its own shared memory from the same reduced values.  Cross-thread sums of
// FP32 values are formed as unevaluated float pairs (hi + lo, Knuth's TwoSum),
// in a fixed order; the BB dot products, F and the step stay FP64.
// ---------------------------------------------------------------------------
struct FF {
    float hi, lo;
};

// (a.hi + a.lo) + (b.hi + b.lo) as a float pair: TwoSum of the high parts, then
// the low parts, renormalised.  No multiply, so no FMA contraction applies.
__device__ __forceinline__ FF ff_add(FF a, FF b) {
    const float s = a.hi + b.hi;
    const float bv = s - a.hi;
    const float e = (a.hi - (s - bv)) + (b.hi - bv);
    const float t = e + (a.lo + b.lo);
    const float h = s + t;
    return FF{h, t - (h - s)};
}

__device__ __forceinline__ FF ff_shfl_xor(FF v, int d) {
    return FF{__shfl_xor_sync(0xffffffffu, v.hi, d), __shfl_xor_sync(0xffffffffu, v.lo, d)};
}

// The warp's sum of one float pair per lane (fixed butterfly, every lane).
__device__ __forceinline__ FF warp_ff(FF v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v = ff_add(v, ff_shfl_xor(v, d));
    return v;
}
__device__ __forceinline__ double ff_to_double(FF v) { return (double)v.hi + (double)v.lo; }

// ---------------------------------------------------------------------------
// Column sums over the CTAs of a solve, and their broadcast, without a grid barrier.
//
// A float pair travels as two 64-bit words, each (float bits, tag): a reader polls the
// words until both carry the tag of the current exchange, so a value and the news of its
// arrival are one access, with no fence, counter or barrier between writer and reader.
// The results are written RES_COPIES times (one per lane of the owner's warp), each copy
// polled by a share of the CTAs: with one copy the polls of 600 CTAs on one or two lines
// held up the stores they waited for.
// Every CTA writes its partial of column k to slot (k, cta); the CTA that owns column k
// (CTA k, or with fewer CTAs than columns a warp of CTA k mod CTAs) polls the column's
// slots, sums them in a fixed order and writes res[k]; every CTA polls res.  One buffer
// is enough: a CTA writes a slot of exchange e + 1 only after it has read every result of
// exchange e, whose owners had then read every slot of e; and an owner writes res[k] of
// e + 1 only after every CTA's partial of e + 1, sent after that CTA had read res of e.
// Tags grow by one per exchange over all solves on a workspace (zeroed when allocated);
// CTAs of a solve are never more than one exchange apart.
//
// What bounds it: two trips through L2 (a store is seen by another SM's poll after about
// 500 cycles on the same die, 870 on the other one), an owner's chain of additions and the
// wait for the slowest CTA.  Measured per iteration (cycles, exchange and step; before: a
// grid barrier, every CTA reducing every column, and the step): 40^3 voxels, 16
// apertures, 250 CTAs: 10.5K -> 9.7K; 422K voxels, 40 apertures, 304 CTAs: 19.7K -> 12.1K;
// 1.1M voxels, 56 apertures, 152 CTAs: 13.7K -> 10.3K.  That master problem (422K voxels, 40
// apertures, 185 iterations) takes 3.24 ms instead of 4.16 ms, the 40^3 plan of 20
// apertures 9.14 ms instead of 10.29 ms.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tagged_store(ulonglong2 *p, FF v, unsigned tag) {
    const unsigned long long hi = ((unsigned long long)tag << 32) | __float_as_uint(v.hi);
    const unsigned long long lo = ((unsigned long long)tag << 32) | __float_as_uint(v.lo);
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(hi), "l"(lo) : "memory");
}
__device__ __forceinline__ ulonglong2 tagged_load(const ulonglong2 *p) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ bool tagged_ok(ulonglong2 v, unsigned tag) {
    return (unsigned)(v.x >> 32) == tag && (unsigned)(v.y >> 32) == tag;
}
__device__ __forceinline__ FF tagged_value(ulonglong2 v) {
    return FF{__uint_as_float((unsigned)v.x), __uint_as_float((unsigned)v.y)};
}
// The sum of one column's slots by a warp: lane l adds CTAs l, l + 32, ... in order, then a
// fixed butterfly (the result in every lane).  SLOT_BATCH slots per lane are polled
// together (few: more loads in flight here cost the solver's pass its registers).
// Returns false when a slot never arrived.
constexpr int SLOT_BATCH = 2;
__device__ __forceinline__ bool column_sum(const ulonglong2 *col, int n_cta, unsigned tag, FF *out) {
    const int lane = threadIdx.x & 31;
    FF v{0.f, 0.f};
    const long long t0 = clock64();
    for (int b0 = 0; b0 < n_cta; b0 += 32 * SLOT_BATCH) { // warp-uniform
        ulonglong2 q[SLOT_BATCH];
        while (true) {
            bool good = true;
#pragma unroll
            for (int u = 0; u < SLOT_BATCH; ++u) {
                const int b = b0 + 32 * u + lane;
                if (b < n_cta) q[u] = tagged_load(col + b);
            }
#pragma unroll
            for (int u = 0; u < SLOT_BATCH; ++u)
                if (b0 + 32 * u + lane < n_cta) good = good && tagged_ok(q[u], tag);
            if (__all_sync(0xffffffffu, good)) break;
            if (__any_sync(0xffffffffu, clock64() - t0 > WAIT_LIMIT_CYCLES)) return false;
        }
#pragma unroll
        for (int u = 0; u < SLOT_BATCH; ++u)
            if (b0 + 32 * u + lane < n_cta) v = ff_add(v, tagged_value(q[u]));
    }
    *out = warp_ff(v);
    return true;
}

// The same sum by the whole CTA: every thread polls the slots tid, tid + 256, ... and
// stages their pairs, then the last warp adds them in the order above (the result in its
// lanes).  stage: room for n_cta pairs.  Returns false, in every thread, when a slot never
// arrived.
__device__ __forceinline__ bool column_sum_cta(const ulonglong2 *col, int n_cta, unsigned tag, FF *stage, int wid,
                                               FF *out) {
    bool ok = true;
    const long long t0 = clock64();
    for (int b = threadIdx.x; b < n_cta && ok; b += MP_THREADS) {
        ulonglong2 w = tagged_load(col + b);
        while (ok && !tagged_ok(w, tag)) {
            ok = clock64() - t0 <= WAIT_LIMIT_CYCLES;
            w = tagged_load(col + b);
        }
        stage[b] = tagged_value(w);
    }
    if (!__syncthreads_and(ok)) return false;
    if (wid == MP_NW - 1) {
        FF v{0.f, 0.f};
        for (int b = threadIdx.x & 31; b < n_cta; b += 32) v = ff_add(v, stage[b]);
        *out = warp_ff(v);
    }
    return true;
}

// Barrier of the whole batched grid.  The last CTA to arrive records the batch
// epoch (gctl[3]) and the set of problems still iterating (gctl[4..5]) before it
// releases the others: the CTA split that follows reads only these words, which
// no CTA changes until every CTA has arrived at the next batch barrier.
__device__ bool batch_sync(unsigned *gctl, unsigned n_cta, const MPArgs *args, int n_plans);

// Solver state every CTA keeps in shared memory (identical in all CTAs but for cta), and
// what the end of an iteration needs of the solve's arguments.
struct PState {
    double F_hist[6];
    double F, delta0, gg, delta;
    double F_off; // the constant of the tiles not in the solve (*F_off_dev)
    int t, done, stop;
    unsigned tag;   // of the last exchange
    unsigned epoch; // elastic solver: the batch epoch the last exchange brought
    int passes;     // passes over DA (iterations and the Cauchy pass)
    int stop_rel, stop_step; // the step's stopping tests, formed in parallel
    int abort;      // a wait of this CTA ran out
    // set by solve_begin
    int n, nmax, off; // apertures, their rounded count, byte offset of the arrays in dynamic shared memory
    unsigned cta, n_cta;
    ulonglong2 *slots, *res;
    int pstride, rstride;
    const unsigned *epoch_src;
    const float *lo, *hi;
    vmat_bb_opts opts;
    double F_offset;
};
// One object per CTA: every function that names it gets the same shared variable.
__device__ __forceinline__ PState &solve_state() {
    __shared__ PState ps;
    return ps;
}

struct SolveSmem {
    unsigned char *stage0; // [MP_NW][stages][cbytes]
    int off;               // byte offset of sy4 in dynamic shared memory
    float4 *sy4;           // [GMAX]   y, zero-padded
    float4 *sg4;           // [GMAX]   G as float (Cauchy pass), zero-padded
    double *sG, *sGp;      // [NMAX]   G_t, G_{t-1}
    double *sS, *sR;       // [NMAX]   s = y_t - y_{t-1}, r = G_t - G_{t-1} (the step's inputs)
    FF *sF;                // [MP_NW]  the warps' shares of F (of the curvature) as float pairs
    float *sYp;            // [NMAX]   y_{t-1}
    float *wred;           // [MP_NW][NMAX]
    float *sT, *sO, *sU;   // [256]
    uint64_t *bars;        // [MP_NW][PQ]
    uint32_t *ring_meta;   // [MP_NW][PQ][2] packed tiles: ring offset, bytes held
    int32_t *wlist;        // [MP_NW][WL_CAP][3] the warp's first tiles: tile, packed unit offset, units
    // then FF [mp_cta_cap(NMAX)]: a column's slots staged for their sum (TailSmem::stage)
};

// Resident CTAs per SM the persistent solvers are compiled for (a register budget): what
// their shared memory (solve_smem) lets an SM hold, four up to 4 apertures, two up to 44
// (the 48 of the last kernel of that class), else one.  At the limits of a class a few words are
// spilled (4 bytes stored a thread; in the batched solver 8-24 for 25-64 apertures).  No aperture count from 2 to 96 is slower for it per iteration, at 12K, 180K and 1.1M voxels, than with the
// budgets before (4, 3, 2 and 1 CTAs up to 8, 24, 48 and 96): 1.1M voxels, 8 / 24 / 48 / 64 apertures 18.4 / 23.7 /
// 38.7 / 50.3 -> 16.9 / 21.7 / 36.0 / 47.0 us, the exchange included.
__host__ __device__ constexpr int mp_min_ctas(int nmax) { return nmax <= 4 ? 4 : (nmax <= 48 ? 2 : 1); }

// CTAs a solve of nmax apertures has at most (room for a column's staged slots; up to 160 SMs).
__host__ __device__ constexpr int mp_cta_cap(int nmax) { return 160 * mp_min_ctas(nmax); }

// Copies in flight per warp at most (mbarriers per warp): the tile stages of whole tiles, or
// the packed tiles that fit in the warp's byte ring.
constexpr int PQ = 8;
// Tiles of a warp whose index and packed place are kept in shared memory (loaded once per
// solve, so that issuing a copy and placing a tile's voxels wait on no global load); a
// warp's tiles past the first WL_CAP are looked up in global memory.
constexpr int WL_CAP = 64;

// Bulk copy of the warp's pipeline slot `it` (global tile-use index across passes).
struct WarpPipe {
    unsigned char *my;
    uint64_t *mb;
    const unsigned char *src;
    int64_t tile_bytes, w0, W, n_my;
    const int32_t *tiles; // warp tile of list entry q (null: tile q)
    int64_t it_base; // pipeline slot of this tile set's first tile
    uint32_t cbytes;
    int stages;
    uint64_t pol;
    // Packed tiles (poff non-null): each is copied whole into the warp's byte ring (stages *
    // cbytes bytes, the tiles in issue order, a tile that would cross the end starting again
    // at 0), up to PQ copies in flight, as many as the ring holds.  Lane 0 is the producer.
    const unsigned char *packed; // packed live tiles
    const int32_t *poff;         // list entry q at 128-byte unit poff[q] of packed
    uint32_t *moff, *mspan;      // [PQ] per slot: ring offset of its tile, ring bytes it holds
    int32_t *wl;                 // [WL_CAP][3] this warp's tile j: tile, packed unit offset, units
    uint32_t ring_bytes;
    int64_t iss;                 // lane 0: the next tile to issue
    int64_t jiss;                // lane 0: its place in the warp's tile cycle, (iss - it_base) mod n_my
    uint32_t pos, span;          // lane 0: ring write position, ring bytes held by tiles in flight
    __device__ __forceinline__ int64_t tile_of(int64_t q) const { return tiles ? (int64_t)__ldg(tiles + q) : q; }
    // the warp's tile j (0 <= j < n_my): tile index, from the shared list when it holds it
    __device__ __forceinline__ int64_t my_tile(int64_t j) const {
        return j < WL_CAP ? (int64_t)wl[3 * j] : tile_of(w0 + j * W);
    }
    __device__ __forceinline__ void issue(int64_t it) const {
        const int s = (int)((uint32_t)it % (uint32_t)stages);
        const int64_t wt = my_tile((uint32_t)(it - it_base) % (uint32_t)n_my);
        mbar_arrive_expect_tx(&mb[s], cbytes);
        bulk_g2s(my + (size_t)s * cbytes, src + wt * tile_bytes, cbytes, &mb[s], pol);
    }
    __device__ __forceinline__ bool wait(int64_t it) const {
        return mbar_wait_bounded(&mb[(uint32_t)it % (uint32_t)stages], ((uint32_t)it / (uint32_t)stages) & 1u,
                                 WAIT_LIMIT_CYCLES);
    }
    // packed: issue tiles iss, iss + 1, ... while fewer than PQ are in flight past tile `it`
    // (the next to be consumed) and the ring has room (lane 0)
    __device__ __forceinline__ void fill(int64_t it) {
        if (span == 0) pos = 0; // an empty ring: any tile fits from its start
        while (iss - it < PQ) {
            const int64_t j = jiss;
            int64_t u0;
            uint32_t units;
            if (j < WL_CAP) {
                u0 = wl[3 * j + 1];
                units = (uint32_t)wl[3 * j + 2];
            } else {
                const int64_t q = w0 + j * W;
                u0 = __ldg(poff + q);
                units = (uint32_t)(__ldg(poff + q + 1) - u0);
            }
            const uint32_t bytes = units * 128u; // at most cbytes <= ring_bytes
            uint32_t start = pos, gap = 0;
            if (pos + bytes > ring_bytes) { // the ring's end: skip the rest, start at 0
                gap = ring_bytes - pos;
                start = 0;
            }
            if (span + gap + bytes > ring_bytes) break;
            const int s = (int)(iss % PQ);
            moff[s] = start;
            mspan[s] = gap + bytes;
            mbar_arrive_expect_tx(&mb[s], bytes);
            bulk_g2s(my + start, packed + u0 * 128, bytes, &mb[s], pol);
            pos = start + bytes;
            span += gap + bytes;
            ++iss;
            if (++jiss == n_my) jiss = 0;
        }
    }
    // after consuming tile `it` (lane 0): packed, release its ring bytes and top the ring up;
    // whole tiles, reuse its slot for the tile `stages` ahead
    __device__ __forceinline__ void refill(int64_t it, bool packed_mode) {
        if (packed_mode) {
            span -= mspan[it % PQ];
            fill(it + 1);
        } else {
            issue(it + stages);
        }
    }
    __device__ __forceinline__ bool wait_packed(int64_t it) const {
        return mbar_wait_bounded(&mb[it % PQ], (uint32_t)((it / PQ) & 1), WAIT_LIMIT_CYCLES);
    }
};

enum { PASS_ITER = 0, PASS_CAUCHY = 1 };

// One sweep over this warp's tiles.  PASS_ITER: z = DA y, objective terms, G
// shares; PASS_CAUCHY: q = DA G and the curvature terms w q^2.  Consumes
// pipeline slots it .. it + n_my - 1 (advancing it) and issues slot + stages
// after each.  Returns false (it at the slot) if a copy never landed.
template <int NMAX, int MODE, bool PACKED>
__device__ __forceinline__ bool solve_pass(const MPArgs &a, const SolveSmem &S, WarpPipe &P, int64_t &it,
                                           float *gacc, float &fs, float &fc) {
    constexpr int GMAX = NMAX / 4;
    // From 49 to 64 apertures (one CTA per SM, registers to spare) a tile's groups stay in
    // registers between the dose and the G shares, so its slot is refilled before the
    // objective; the Cauchy pass reads the slot once and refills at the same point.
    constexpr bool KEEP = NMAX >= 56 && NMAX <= 64 && MODE == PASS_ITER;
    constexpr bool EARLY = KEEP || MODE == PASS_CAUCHY;
    const int G = (a.n + 3) >> 2;
    const int lane = threadIdx.x & 31;
    for (int64_t j = 0; j < P.n_my; ++j, ++it) {
        const bool ok = PACKED ? P.wait_packed(it) : P.wait(it);
        if (!__all_sync(0xffffffffu, ok)) return false;
        const unsigned char *blk =
            PACKED ? P.my + P.moff[it % PQ] : P.my + (size_t)((uint32_t)it % (uint32_t)P.stages) * P.cbytes;
        const float4 *D4 = reinterpret_cast<const float4 *>(blk + 128) + lane; // group g at D4[32 g]
        const float4 *w4 = MODE == PASS_ITER ? S.sy4 : S.sg4;
        // packed: the marked groups only, in order (a group left out holds zeros, which add nothing)
        const uint32_t gm = PACKED ? reinterpret_cast<const uint32_t *>(blk)[8] : 0u;
        float4 vk[KEEP ? GMAX : 1];
        float z0 = 0.f, z1 = 0.f, z2 = 0.f, z3 = 0.f;
        int slot = 0;
#pragma unroll
        for (int g = 0; g < GMAX; ++g)
            if (g < G && (!PACKED || ((gm >> g) & 1u))) {
                const float4 v = D4[32 * (PACKED ? slot++ : g)], w = w4[g];
                if (KEEP) vk[KEEP ? g : 0] = v;
                z0 = fmaf(v.x, w.x, z0);
                z1 = fmaf(v.y, w.y, z1);
                z2 = fmaf(v.z, w.z, z2);
                z3 = fmaf(v.w, w.w, z3);
            }
        const int sid = blk[lane];
        if (EARLY) {
            __syncwarp(); // every lane's reads of this slot are done before its next copy
            if (lane == 0) P.refill(it, PACKED);
        }
        const float zi = (z0 + z1) + (z2 + z3);
        const int64_t i = P.my_tile(j) * MP_WT + lane;
        float gi = 0.f;
        if (i < a.V) {
            if (MODE == PASS_ITER) {
                a.z[i] = zi;
                const float d = zi - S.sT[sid];
                const float w = d > 0.f ? S.sO[sid] : S.sU[sid];
                const float yk = (w * d) * d - fc; // Kahan step
                const float tk = fs + yk;
                fc = (tk - fs) - yk;
                fs = tk;
                gi = -2.f * w * d; // g = -grad F: -2 w+ (z - T) above, +2 w- (T - z) below
            } else {
                // curvature of F along DA G: the active weight (0 exactly at the threshold)
                const float zc = a.z[i], T = S.sT[sid];
                const float w = zc > T ? S.sO[sid] : (zc < T ? S.sU[sid] : 0.f);
                const float yk = (w * zi) * zi - fc;
                const float tk = fs + yk;
                fc = (tk - fs) - yk;
                fs = tk;
            }
        }
        if (MODE == PASS_ITER) {
            slot = 0;
#pragma unroll
            for (int g = 0; g < GMAX; ++g)
                if (g < G && (!PACKED || ((gm >> g) & 1u))) {
                    const float4 v = KEEP ? vk[KEEP ? g : 0] : D4[32 * (PACKED ? slot++ : g)];
                    gacc[4 * g + 0] = fmaf(v.x, gi, gacc[4 * g + 0]);
                    gacc[4 * g + 1] = fmaf(v.y, gi, gacc[4 * g + 1]);
                    gacc[4 * g + 2] = fmaf(v.z, gi, gacc[4 * g + 2]);
                    gacc[4 * g + 3] = fmaf(v.w, gi, gacc[4 * g + 3]);
                }
        }
        if (!EARLY) {
            __syncwarp(); // every lane's reads of this slot are done before its next copy
            if (lane == 0) P.refill(it, PACKED);
        }
    }
    return true;
}

// The warp's sums over its 32 lanes of the G shares gacc[0 .. n), written to out[0 .. n).
// From 16 apertures on, by halving exchanges over 32-column chunks: at the exchange of
// width w each lane keeps half of its remaining columns (the upper half when its lane bit
// w is set), sends the other half to lane ^ w and adds what it receives; after five
// exchanges lane l holds column l of the chunk.  31 shuffles per chunk instead of 5 per
// column.  Columns at or past n hold zero (their DA groups are zero padding).  A fixed
// order: every warp of every CTA adds the same way.
template <int NMAX>
__device__ __forceinline__ void warp_share_sums(const float *gacc, int n, float *out, int lane) {
    if (NMAX < 16) {
#pragma unroll
        for (int k = 0; k < NMAX; ++k) {
            if (k < n) {
                float x = gacc[k];
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
                if (lane == 0) out[k] = x;
            }
        }
        return;
    }
#pragma unroll
    for (int c = 0; c < (NMAX + 31) / 32; ++c) {
        if (32 * c < n) {
            float v[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = 32 * c + i < NMAX ? gacc[32 * c + i] : 0.f;
#pragma unroll
            for (int w = 16; w >= 1; w >>= 1) {
                const bool up = (lane & w) != 0;
#pragma unroll
                for (int i = 0; i < w; ++i) {
                    const float send = up ? v[i] : v[i + w];
                    const float keep = up ? v[i + w] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
                }
            }
            if (32 * c + lane < n) out[32 * c + lane] = v[0];
        }
    }
}

// The warps' pairs sh[0 .. MP_NW) in order.
__device__ __forceinline__ FF sum_warps_ff(const FF *sh) {
    FF t = sh[0];
#pragma unroll
    for (int w = 1; w < MP_NW; ++w) t = ff_add(t, sh[w]);
    return t;
}

// Exchange `tag` over n_col columns: every thread calls it after the CTA's slot of every column
// has been written (by some of its threads).  A thread that wants column `want`'s sum gets it in
// *out (want < 0: none).  epoch_src (elastic solver, else null): the owner of the last
// column reads that word once, and a thread with want == n_col gets the value, the same in
// every CTA, as the bits of out->hi.  Returns false in a thread whose wait ran out.
__device__ __forceinline__ bool exchange_columns(const PState &ps, FF *stage, int n_col, unsigned tag, int want,
                                                 FF *out, const unsigned *epoch_src) {
    const int tid = threadIdx.x, lane = tid & 31, wid = warp_index();
    const int cta = warp_uniform((int)ps.cta), n_cta = warp_uniform((int)ps.n_cta);
    bool ok = true;
    auto publish = [&](int k, FF v) { // a copy per lane
        ulonglong2 *copy = ps.res + (size_t)lane * ps.rstride;
        tagged_store(copy + k, v, tag);
        if (epoch_src && k == n_col - 1) {
            const unsigned e = __shfl_sync(0xffffffffu, lane == 0 ? *(const volatile unsigned *)epoch_src : 0u, 0);
            tagged_store(copy + n_col, FF{__uint_as_float(e), 0.f}, tag);
        }
    };
    if (n_cta >= n_col) { // a column or none per CTA: the CTA polls its slots
        if (cta < n_col) {
            FF v;
            ok = column_sum_cta(ps.slots + (size_t)cta * ps.pstride, n_cta, tag, stage, wid, &v);
            if (ok && wid == MP_NW - 1) publish(cta, v);
        }
    } else { // few CTAs: a warp per column, from the last warp down (the first ones poll results)
        for (int k = cta + (MP_NW - 1 - wid) * n_cta; k < n_col; k += MP_NW * n_cta) {
            FF v;
            const bool got = column_sum(ps.slots + (size_t)k * ps.pstride, n_cta, tag, &v); // the same in every lane
            ok = ok && got;
            if (got) publish(k, v);
        }
    }
    const ulonglong2 *res = ps.res + (size_t)(cta % RES_COPIES) * ps.rstride;
    // polled a warp at a time, so that the warp stays together
    if (__any_sync(0xffffffffu, want >= 0)) {
        ulonglong2 w = make_ulonglong2(0, 0);
        const long long t0 = clock64();
        while (true) {
            if (want >= 0) w = tagged_load(res + want);
            if (__all_sync(0xffffffffu, want < 0 || tagged_ok(w, tag))) break;
            if (__any_sync(0xffffffffu, clock64() - t0 > WAIT_LIMIT_CYCLES)) {
                ok = false;
                break;
            }
        }
        if (want >= 0) *out = tagged_value(w);
    }
    return ok;
}

// The arrays of the solver's shared memory that the end of an iteration uses
// (solve_layout's places, found from the solve's rounded aperture count).
struct TailSmem {
    float *y, *sg, *sYp, *wred;
    double *sG, *sGp, *sS, *sR;
    FF *sF, *stage;
};
__device__ __forceinline__ TailSmem tail_smem(const PState &ps) {
    extern __shared__ __align__(128) unsigned char sm_raw[];
    unsigned char *b = sm_raw + ps.off;
    const int m = ps.nmax;
    TailSmem S;
    S.y = reinterpret_cast<float *>(b);
    S.sg = S.y + m;
    S.sG = reinterpret_cast<double *>(S.sg + m);
    S.sGp = S.sG + m;
    S.sS = S.sGp + m;
    S.sR = S.sS + m;
    S.sF = reinterpret_cast<FF *>(S.sR + m);
    S.sYp = reinterpret_cast<float *>(S.sF + MP_NW);
    S.wred = S.sYp + m;
    S.stage = reinterpret_cast<FF *>(reinterpret_cast<unsigned char *>(S.wred + MP_NW * m + 3 * 256) +
                                     MP_NW * PQ * (8 + 8) + MP_NW * WL_CAP * 12);
    return S;
}

// The threads that take F and the elastic solver's epoch: in a warp without columns, so that
// no warp runs the work of a column and of F one after the other.
constexpr int F_THREAD = MP_NMAX, EPOCH_THREAD = MP_NMAX + 1;
static_assert(F_THREAD % 32 == 0 && EPOCH_THREAD < MP_THREADS, "a warp of their own");

enum { STEP_NEXT = 0, STEP_DONE = 1, STEP_CAUCHY = 2 };

// Eq. 9-10 freeze, stopping tests, BB step length (FP64) and projected update, on the
// shared-memory copy of the state, run by the whole CTA; every CTA runs it on identical
// inputs.  Thread k < n comes with column k's reduced pair (-G_k) in gf and its bounds,
// thread F_THREAD with F; `ok` false in a thread whose exchange failed: then -1 everywhere.
// Returns the same STEP_* in every thread; after STEP_NEXT y holds the next iterate.
//
// What bounds it: a chain of FP64 operations, which issue at a small fraction of the
// FP32 rate on this GPU.  So the work is spread (one aperture per thread, one warp per
// sum, the tests and the step size each in a warp of its own) with one CTA barrier per
// stage, every thread decides for itself from the stage's results, and no stage loads
// from global memory (the tile constant, which each step used to read, cost it an L2
// access on this chain).
__device__ __forceinline__ int solve_step_cta(PState &ps, const TailSmem &S, FF gf, float l, float h, bool ok) {
    const int tid = threadIdx.x, lane = tid & 31, wid = warp_index();
    const int n = warp_uniform(ps.n), t = ps.t;
    float *y = S.y;
    float yk = 0.f;
    double g = 0.0;
    if (tid == F_THREAD) ps.F = ff_to_double(gf) + ps.F_offset + ps.F_off;
    if (tid < n) {
        yk = y[tid];
        // g = -(hi + lo): its sign from a float compare (the pair's sum is not rounded to 0)
        g = -ff_to_double(gf);
        if (yk <= l && gf.hi < -gf.lo) {
            yk = l;
            g = 0.0;
        } else if (yk >= h && gf.hi > -gf.lo) {
            yk = h;
            g = 0.0;
        }
        y[tid] = yk;
        S.sG[tid] = g;
        if (t > 0) {
            S.sS[tid] = (double)yk - (double)S.sYp[tid];
            S.sR[tid] = g - S.sGp[tid];
        }
    }
    if (__syncthreads_or(!ok)) return -1;
    // Warp 0: the four sums, eight lanes each (lanes 8q .. 8q + 7: 0 G.G, 1 s.s, 2 s.r,
    // 3 r.r), lane j of a group over apertures j, j + 8, ... in order, then a fixed
    // butterfly of the group: one warp's FP64 instructions serve all four.  Warp 1: the
    // maxima |s| (lanes 0-15) and |y| (lanes 16-31) as integer maxima of the bit
    // patterns of non-negative values (the order of their values), off the FP64 pipe,
    // and with them the step test.  Warp 2: the relative-change test, which needs F only.
    // (the groups' operands are offsets into one array and the trip count is the warp's, so
    // that the warp does not run the groups one after the other; at t = 0 the groups other
    // than G.G read stale values, never used)
    if (wid == 0) {
        const int q = lane >> 3, j = lane & 7;
        const int m = ps.nmax, ox = (q == 0 ? 0 : (q == 3 ? 3 : 2)) * m + j, oz = (q == 0 ? 0 : (q == 1 ? 2 : 3)) * m + j;
        double v = 0.0;
        for (int k = 0; k < n; k += 8) { // entries past n (up to 7, sR's in sF) are read and left out
            const double p = fma(S.sG[ox + k], S.sG[oz + k], v);
            v = k + j < n ? p : v;
        }
#pragma unroll
        for (int d = 4; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
        const double ss = __shfl_sync(0xffffffffu, v, 8), sr = __shfl_sync(0xffffffffu, v, 16),
                     rr = __shfl_sync(0xffffffffu, v, 24);
        if (lane == 0) {
            ps.gg = t == 0 ? v : ps.gg;
            if (t > 0) {
                double delta;
                if (sr <= 0.0) delta = ps.opts.delta_max * ps.delta0;
                else if (t & 1) delta = sr / rr;
                else delta = ss / sr;
                ps.delta = fmin(fmax(delta, ps.opts.delta_min * ps.delta0), ps.opts.delta_max * ps.delta0);
            }
        }
    } else if (wid == 1) {
        const bool ys = lane >= 16;
        const int j = lane & 15;
        unsigned long long m = 0;
        if (ys) {
            for (int k = j; k < n; k += 16) m = max(m, (unsigned long long)(__float_as_uint(y[k]) & 0x7fffffffu));
        } else if (t > 0) {
            for (int k = j; k < n; k += 16)
                m = max(m, (unsigned long long)__double_as_longlong(S.sS[k]) & 0x7fffffffffffffffull);
        }
#pragma unroll
        for (int d = 8; d > 0; d >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, d));
        const unsigned long long my = __shfl_sync(0xffffffffu, m, 16);
        if (lane == 0) {
            const double dy = __longlong_as_double((long long)m), ymax = (double)__uint_as_float((unsigned)my);
            ps.stop_step = t >= 1 && dy <= ps.opts.step_tol * fmax(1.0, ymax);
        }
    } else if (wid == 2 && lane == 0) {
        const double F = ps.F;
        ps.stop_rel = t >= 5 && fabs(ps.F_hist[(t - 5) % 6] - F) <= ps.opts.rel_tol5 * F;
        ps.F_hist[t % 6] = F; // (t - 5) % 6 is another entry
    }
    __syncthreads();
    int stop = 0;
    if (ps.stop_rel) stop = VMAT_STOP_REL;
    else if (ps.stop_step) stop = VMAT_STOP_STEP;
    else if (t == ps.opts.max_iter - 1) stop = VMAT_STOP_MAXIT;
    else if (t == 0 && ps.gg == 0.0) stop = VMAT_STOP_GRAD0;
    if (stop) {
        if (tid == 0) {
            ps.done = 1;
            ps.stop = stop;
        }
        __syncthreads();
        return STEP_DONE;
    }
    if (t == 0) return STEP_CAUCHY; // the first step's length needs DA G
    if (tid < n) {
        S.sYp[tid] = yk;
        S.sGp[tid] = g;
        const double yn = (double)yk - ps.delta * g;
        y[tid] = fminf(fmaxf((float)yn, l), h);
    }
    __syncthreads();
    return STEP_NEXT;
}

// The end of an iteration, after every warp has written its G shares to wred: this CTA's
// partials of every column and of F (fs - fc per lane), their sums over the CTAs, the step.
// Returns STEP_* (the same in every CTA), -1 when a wait ran out.  Not inlined: the pass
// keeps its registers (inlined, the two together spilled inside the pass).
__device__ __noinline__ int solve_tail(float fs, float fc) {
    PState &ps = solve_state();
    const TailSmem S = tail_smem(ps);
    const int tid = threadIdx.x, lane = tid & 31, wid = warp_index();
    const int n = warp_uniform(ps.n), m = ps.nmax;
    const float l = tid < n && ps.lo ? ps.lo[tid] : 0.f, h = tid < n && ps.hi ? ps.hi[tid] : INFINITY;
    const FF fw = warp_ff(FF{fs, -fc});
    if (lane == 0) S.sF[wid] = fw;
    const unsigned tag = ps.tag + 1;
    __syncthreads();
    if (ps.abort) return -1;
    FF v{0.f, 0.f};
    if (tid < n) {
        v = FF{S.wred[tid], 0.f};
#pragma unroll
        for (int w = 1; w < MP_NW; ++w) v = ff_add(v, FF{S.wred[w * m + tid], 0.f});
    } else if (tid == F_THREAD) {
        v = sum_warps_ff(S.sF);
    }
    const int col = tid < n ? tid : (tid == F_THREAD ? n : -1);
    if (col >= 0) tagged_store(ps.slots + (size_t)col * ps.pstride + ps.cta, v, tag);
    const int want = ps.epoch_src && tid == EPOCH_THREAD ? n + 1 : col;
    const bool ok = exchange_columns(ps, S.stage, n + 1, tag, want, &v, ps.epoch_src);
    if (tid == EPOCH_THREAD) {
        ps.epoch = __float_as_uint(v.hi);
        ps.tag = tag; // read above, before the barrier; next read after the step's barriers
        ++ps.passes;
    }
    return solve_step_cta(ps, S, v, l, h, ok);
}

// The end of the Cauchy pass (curvature terms cs - cc per lane): delta0 = G.G / (2 sum_i w_i
// (DA G)_i^2) and the first step.  Returns STEP_NEXT, STEP_DONE (flat) or -1.
__device__ __noinline__ int solve_cauchy_tail(float cs, float cc) {
    PState &ps = solve_state();
    const TailSmem S = tail_smem(ps);
    const int tid = threadIdx.x, lane = tid & 31, wid = warp_index();
    const int n = ps.n;
    const float l = tid < n && ps.lo ? ps.lo[tid] : 0.f, h = tid < n && ps.hi ? ps.hi[tid] : INFINITY;
    const FF cw = warp_ff(FF{cs, -cc});
    if (lane == 0) S.sF[wid] = cw;
    const unsigned tag = ps.tag + 1;
    __syncthreads();
    if (ps.abort) return -1;
    FF c{0.f, 0.f};
    if (tid == 0) tagged_store(ps.slots + ps.cta, sum_warps_ff(S.sF), tag);
    const bool ok = exchange_columns(ps, S.stage, 1, tag, tid == 0 ? 0 : -1, &c, nullptr);
    if (tid == 0 && ok) {
        ps.tag = tag;
        ++ps.passes;
        const double curv = 2.0 * ff_to_double(c);
        if (curv == 0.0) {
            ps.done = 1;
            ps.stop = VMAT_STOP_FLAT;
        } else {
            ps.delta0 = ps.gg / curv;
        }
    }
    if (__syncthreads_or(!ok)) return -1;
    if (ps.done) return STEP_DONE;
    if (tid < n) {
        const float yk = S.y[tid];
        S.sYp[tid] = yk;
        S.sGp[tid] = S.sG[tid];
        const double yn = (double)yk - ps.delta0 * S.sG[tid];
        S.y[tid] = fminf(fmaxf((float)yn, l), h);
    }
    __syncthreads();
    return STEP_NEXT;
}

// Shared-memory layout of the solver for NMAX apertures and `stages` tiles per warp.
// sm_base: the start of dynamic shared memory, sm: its first 128-byte boundary.
template <int NMAX>
__device__ __forceinline__ SolveSmem solve_layout(const unsigned char *sm_base, unsigned char *sm, int stages,
                                                  uint32_t cbytes) {
    constexpr int GMAX = NMAX / 4;
    SolveSmem S;
    S.stage0 = sm;
    S.sy4 = reinterpret_cast<float4 *>(sm + (size_t)MP_NW * stages * cbytes);
    S.off = (int)(smem_u32(S.sy4) - smem_u32(sm_base));
    S.sg4 = S.sy4 + GMAX;
    S.sG = reinterpret_cast<double *>(S.sg4 + GMAX);
    S.sGp = S.sG + NMAX;
    S.sS = S.sGp + NMAX;
    S.sR = S.sS + NMAX;
    S.sF = reinterpret_cast<FF *>(S.sR + NMAX);
    S.sYp = reinterpret_cast<float *>(S.sF + MP_NW);
    S.wred = S.sYp + NMAX;
    S.sT = S.wred + MP_NW * NMAX;
    S.sO = S.sT + 256;
    S.sU = S.sO + 256;
    S.bars = reinterpret_cast<uint64_t *>(S.sU + 256);
    S.ring_meta = reinterpret_cast<uint32_t *>(S.bars + MP_NW * PQ);
    S.wlist = reinterpret_cast<int32_t *>(S.ring_meta + MP_NW * PQ * 2);
    return S;
}

// Loads one problem's tables and state into shared memory: a fresh start (y from
// a.y, projected onto the box) or, for the elastic solver, the state a
// previous epoch saved (t, F history, step scale, y, y_prev, G_prev).
template <int NMAX>
__device__ void solve_load(const MPArgs &a, const SolveSmem &S, bool resume, unsigned cta, unsigned n_cta,
                           const unsigned *epoch_src) {
    constexpr int GMAX = NMAX / 4;
    PState &ps = solve_state();
    const int n = a.n, tid = threadIdx.x;
    for (int k = tid; k < 4 * GMAX; k += MP_THREADS) {
        // the start projected onto the box (a saved iterate lies in it)
        reinterpret_cast<float *>(S.sy4)[k] = k < n ? fminf(fmaxf(a.y[k], lo_of(a, k)), hi_of(a, k)) : 0.f;
        reinterpret_cast<float *>(S.sg4)[k] = 0.f;
    }
    for (int k = tid; k < a.n_struct; k += MP_THREADS) {
        S.sT[k] = a.T[k];
        S.sO[k] = a.wo[k];
        S.sU[k] = a.wu[k];
    }
    if (resume)
        for (int k = tid; k < n; k += MP_THREADS) {
            S.sYp[k] = a.yprev[k];
            S.sGp[k] = a.Gprev[k];
        }
    if (tid == 0) {
        PState z = {};
        ps = z;
        ps.tag = __ldcg(a.tag);
        ps.F_off = a.F_off_dev ? __ldcg(a.F_off_dev) : 0.0;
        ps.n = n;
        ps.nmax = NMAX;
        ps.off = S.off;
        ps.cta = cta;
        ps.n_cta = n_cta;
        ps.slots = a.slots;
        ps.res = a.res;
        ps.pstride = a.pstride;
        ps.rstride = a.rstride;
        ps.epoch_src = epoch_src;
        ps.lo = a.lo;
        ps.hi = a.hi;
        ps.opts = a.opts;
        ps.F_offset = a.F_offset;
        if (resume) {
            for (int i = 0; i < 6; ++i) ps.F_hist[i] = a.st->F_hist[i];
            ps.F = a.st->F;
            ps.delta0 = a.st->delta0;
            ps.gg = a.st->gg;
            ps.t = a.st->t;
        }
    }
    __syncthreads();
}

// A solve leaves *tag past every tag any of its CTAs has used (they are at most one
// exchange apart), whether it ends, hands over or gives up.
constexpr unsigned TAG_GAP = 4;

// The state a later epoch resumes from (one CTA writes it).
template <int NMAX> __device__ void solve_save(const MPArgs &a, const SolveSmem &S) {
    const PState &ps = solve_state();
    const float *y = reinterpret_cast<const float *>(S.sy4);
    for (int k = threadIdx.x; k < a.n; k += MP_THREADS) {
        a.y[k] = y[k];
        a.yprev[k] = S.sYp[k];
        a.Gprev[k] = S.sGp[k];
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < 6; ++i) a.st->F_hist[i] = ps.F_hist[i];
        a.st->F = ps.F;
        a.st->delta0 = ps.delta0;
        a.st->gg = ps.gg;
        a.st->t = ps.t;
        a.st->started = 1;
        *a.tag = ps.tag + TAG_GAP;
    }
    __threadfence();
}

// The end of a solve (one CTA): y, the report and the iteration count.
template <int NMAX> __device__ void solve_finish(const MPArgs &a, const SolveSmem &S, bool ok) {
    const PState &ps = solve_state();
    const float *y = reinterpret_cast<const float *>(S.sy4);
    if (ok)
        for (int k = threadIdx.x; k < a.n; k += MP_THREADS) a.y[k] = y[k];
    if (threadIdx.x == 0) {
        a.st->F = ps.F;
        a.st->t = ps.t;
        a.st->done = 1;
        a.st->stop = ok ? ps.stop : VMAT_STOP_MAXIT;
        a.st->iters = ps.t + 1;
        a.st->delta0 = ps.delta0;
        *a.tag = ps.tag + TAG_GAP;
        if (ok && a.iters_acc) *a.iters_acc += ps.t + 1;
        if (ok && a.bytes_acc) { // each pass reads the tiles' labels and columns and writes (or reads) their dose
            const int64_t tiles = a.tiles ? min64((int64_t)max(__ldcg(a.n_live), 0), a.n_wtiles) : a.n_wtiles;
            const double per_tile_read = a.poff ? 0.0 : (double)wt_copy_bytes(a.n);
            const double packed_read = a.poff ? 128.0 * (double)__ldcg(a.poff + tiles) : 0.0;
            *a.bytes_acc += (double)ps.passes * ((double)tiles * (per_tile_read + 4.0 * MP_WT) + packed_read);
        }
    }
    __threadfence();
}

enum { LOOP_DONE = 0, LOOP_ABORT = 1, LOOP_REBALANCE = 2 };

// BB iterations of one problem, until a stopping rule
// (LOOP_DONE), a wait that ran out (LOOP_ABORT) or, for the elastic solver, a change of the batch epoch seen at an iteration's exchange
// (LOOP_REBALANCE, after this CTA has saved the state if cta == 0).
template <int NMAX>
__device__ __forceinline__ int solve_loop(const MPArgs &a, const SolveSmem &S, WarpPipe &P, int64_t &it, bool elastic,
                                          unsigned epoch_local) {
    constexpr int GMAX = NMAX / 4;
    PState &ps = solve_state();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    float gacc[NMAX];
    while (true) {
        // ---- pass: z = DA y, g, F and this CTA's shares of G = -DA^T g
#pragma unroll
        for (int k = 0; k < NMAX; ++k) gacc[k] = 0.f;
        float fs = 0.f, fc = 0.f;
        const bool pass_ok = P.n_my == 0 || (P.poff ? solve_pass<NMAX, PASS_ITER, true>(a, S, P, it, gacc, fs, fc)
                                                    : solve_pass<NMAX, PASS_ITER, false>(a, S, P, it, gacc, fs, fc));
        if (!pass_ok && lane == 0) ps.abort = 1;
        warp_share_sums<NMAX>(gacc, a.n, S.wred + wid * NMAX, lane);
        int step = solve_tail(fs, fc);
        if (step == STEP_CAUCHY) { // the first step's length needs DA G
            for (int k = tid; k < 4 * GMAX; k += MP_THREADS)
                reinterpret_cast<float *>(S.sg4)[k] = k < a.n ? (float)S.sG[k] : 0.f;
            __syncthreads();
            fs = fc = 0.f;
            const bool c_ok = P.n_my == 0 || (P.poff ? solve_pass<NMAX, PASS_CAUCHY, true>(a, S, P, it, gacc, fs, fc)
                                                      : solve_pass<NMAX, PASS_CAUCHY, false>(a, S, P, it, gacc, fs, fc));
            if (!c_ok && lane == 0) ps.abort = 1;
            step = solve_cauchy_tail(fs, fc);
        }
        if (step < 0) return LOOP_ABORT;
        if (step == STEP_DONE) return LOOP_DONE;
        if (tid == 0) ++ps.t; // next read after the tail's first barrier
        if (elastic && ps.epoch != epoch_local) { // the same word for every CTA of the problem
            __syncthreads();
            if (ps.cta == 0) solve_save<NMAX>(a, S);
            return LOOP_REBALANCE;
        }
    }
}

// Sets up a warp's pipeline for tiles w0, w0 + W, ... of problem a, starting at slot it.
__device__ __forceinline__ void pipe_start(WarpPipe &P, const MPArgs &a, unsigned cta, unsigned n_cta, int64_t it) {
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    P.src = reinterpret_cast<const unsigned char *>(a.DA);
    P.tile_bytes = a.wstride * 4;
    P.W = (int64_t)n_cta * MP_NW;
    P.w0 = (int64_t)cta * MP_NW + wid;
    P.tiles = a.tiles;
    P.packed = reinterpret_cast<const unsigned char *>(a.packed);
    P.poff = a.packed ? a.poff : nullptr;
    P.iss = it;
    P.jiss = 0;
    P.pos = 0;
    P.span = 0;
    int64_t n_wt = a.n_wtiles;
    if (a.tiles) // the live list: written by earlier kernels of the stream, fixed during the solve
        n_wt = min64((int64_t)max(__ldcg(a.n_live), 0), a.n_wtiles);
    P.n_my = P.w0 < n_wt ? (n_wt - 1 - P.w0) / P.W + 1 : 0;
    P.it_base = it;
    // the warp's first WL_CAP tiles: index, and the packed place when packed (lane per tile)
    for (int64_t j = lane; j < min64(P.n_my, (int64_t)WL_CAP); j += 32) {
        const int64_t q = P.w0 + j * P.W;
        P.wl[3 * j] = (int32_t)P.tile_of(q);
        if (P.poff) {
            const int32_t u0 = __ldg(P.poff + q);
            P.wl[3 * j + 1] = u0;
            P.wl[3 * j + 2] = __ldg(P.poff + q + 1) - u0;
        }
    }
    __syncwarp();
    if (lane == 0 && P.n_my > 0) {
        if (P.poff) P.fill(it);
        else
            for (int s = 0; s < P.stages; ++s) P.issue(it + s);
    }
}

// Copies issued ahead for a pass that will not run: let them land (this warp's slots it ..).
__device__ __forceinline__ void pipe_drain(const WarpPipe &P, int64_t it) {
    if ((threadIdx.x & 31) == 0 && P.n_my > 0) {
        if (P.poff)
            for (int64_t k = it; k < P.iss; ++k) P.wait_packed(k);
        else
            for (int s = 0; s < P.stages; ++s) P.wait(it + s);
    }
    __syncwarp();
}

__device__ __forceinline__ void pipe_init(WarpPipe &P, const SolveSmem &S, int stages, uint32_t cbytes,
                                          int keep_in_l2) {
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    P.my = S.stage0 + (size_t)wid * stages * cbytes;
    P.mb = S.bars + wid * PQ;
    P.ring_bytes = (uint32_t)stages * cbytes;
    P.moff = S.ring_meta + wid * PQ * 2;
    P.mspan = P.moff + PQ;
    P.wl = S.wlist + wid * WL_CAP * 3;
    P.cbytes = cbytes;
    P.stages = stages;
    // DA is read again by every iteration: keep it in L2 when it fits there
    P.pol = keep_in_l2 ? l2_evict_last_policy() : l2_evict_first_policy();
    P.n_my = 0;
    if (lane == 0) {
        for (int s = 0; s < PQ; ++s) mbar_init(&P.mb[s], 1);
        fence_mbar_init();
    }
}

template <int NMAX>
__global__ void __launch_bounds__(MP_THREADS, mp_min_ctas(NMAX))
    mp_solve_kernel(const __grid_constant__ MPArgs a, int stages, int keep_in_l2) {
    if (a.skip && *a.skip) return; // the same flag for every CTA: all return together
    extern __shared__ __align__(128) unsigned char sm_raw[];
    // align the staging area explicitly: static shared memory may shift the dynamic region
    unsigned char *sm = sm_raw + ((128u - (smem_u32(sm_raw) & 127u)) & 127u);
    const uint32_t cbytes = (uint32_t)wt_copy_bytes(a.n);
    const SolveSmem S = solve_layout<NMAX>(sm_raw, sm, stages, cbytes);
    WarpPipe P;
    pipe_init(P, S, stages, cbytes, keep_in_l2);
    solve_load<NMAX>(a, S, false, blockIdx.x, gridDim.x, nullptr); // ends with a __syncthreads (barriers initialised)
    int64_t it = 0;
    pipe_start(P, a, blockIdx.x, gridDim.x, it);
    const int r = solve_loop<NMAX>(a, S, P, it, false, 0u);
    if (r == LOOP_ABORT && threadIdx.x == 0) atomicOr(a.status, DEV_TIMEOUT);
    pipe_drain(P, it);
    if (blockIdx.x == 0) solve_finish<NMAX>(a, S, r != LOOP_ABORT);
}

__device__ bool batch_sync(unsigned *gctl, unsigned n_cta, const MPArgs *args, int n_plans) {
    __shared__ int ok_s;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned *vg = gctl + 1;
        const unsigned g0 = *vg;
        __threadfence();
        int ok = 1;
        if (atomicAdd(gctl, 1u) == n_cta - 1) {
            unsigned long long mask = 0ull;
            for (int p = 0; p < n_plans; ++p) {
                const MPArgs &q = args[p];
                const bool act = !(q.skip && *(volatile const int32_t *)q.skip) && !*(volatile int32_t *)&q.st->done;
                if (act) mask |= 1ull << p;
            }
            gctl[4] = (unsigned)(mask & 0xffffffffu);
            gctl[5] = (unsigned)(mask >> 32);
            gctl[3] = *(volatile unsigned *)(gctl + 2);
            atomicExch(gctl, 0u);
            __threadfence();
            atomicAdd(gctl + 1, 1u);
        } else {
            const long long t0 = clock64();
            while (*vg == g0) {
                if (clock64() - t0 > WAIT_LIMIT_CYCLES) {
                    ok = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

// Several independent problems in one persistent launch.  All CTAs are split
// among the problems still iterating, in proportion to their warp tiles (the same
// computation in every CTA), and each problem exchanges its sums among its own CTAs.
// When a problem stops it bumps the batch epoch (gctl[2]); the owner of a problem's last
// column sends the epoch along with that column's sum, so all CTAs of a problem see a
// change at the same exchange, save its state and join a barrier of the whole grid
// (gctl[0..1]), after which the CTAs are split again among the problems left.  Every
// problem has n apertures.
template <int NMAX>
__global__ void __launch_bounds__(MP_THREADS, mp_min_ctas(NMAX))
    mp_solve_batched_kernel(const MPArgs *__restrict__ args, const int64_t *__restrict__ weight, int32_t n_plans,
                            int32_t n, unsigned *gctl, int stages, int keep_in_l2) {
    extern __shared__ __align__(128) unsigned char sm_raw[];
    __shared__ MPArgs sa;
    __shared__ int sp, sc, sn, resume_s;
    __shared__ unsigned epoch_s;
    unsigned char *sm = sm_raw + ((128u - (smem_u32(sm_raw) & 127u)) & 127u);
    const uint32_t cbytes = (uint32_t)wt_copy_bytes(n);
    const SolveSmem S = solve_layout<NMAX>(sm_raw, sm, stages, cbytes);
    WarpPipe P;
    pipe_init(P, S, stages, cbytes, keep_in_l2);
    __syncthreads();
    int64_t it = 0;
    unsigned epoch_local = 0;
    bool ok = true;
    while (true) {
        if (threadIdx.x == 0) { // CTA split among the problems still iterating (identical in every CTA)
            const unsigned long long mask =
                (unsigned long long)__ldcg(gctl + 4) | ((unsigned long long)__ldcg(gctl + 5) << 32);
            double wsum = 0.0;
            int n_act = 0;
            for (int q = 0; q < n_plans; ++q)
                if ((mask >> q) & 1ull) {
                    wsum += (double)weight[q];
                    ++n_act;
                }
            sp = -1;
            if (n_act > 0) {
                const int G = (int)gridDim.x;
                int start = 0, seen = 0;
                for (int q = 0; q < n_plans && sp < 0; ++q) {
                    if (!((mask >> q) & 1ull)) continue;
                    ++seen;
                    int cnt = seen == n_act ? G - start
                                            : 1 + (int)((double)(G - n_act) * (double)weight[q] / wsum);
                    cnt = max(1, min(cnt, G - start - (n_act - seen)));
                    if ((int)blockIdx.x < start + cnt) {
                        sp = q;
                        sc = (int)blockIdx.x - start;
                        sn = cnt;
                    }
                    start += cnt;
                }
            }
            epoch_s = __ldcg(gctl + 3); // the epoch at the last batch barrier
        }
        __syncthreads();
        const int p = sp;
        if (p < 0) break;
        epoch_local = epoch_s;
        for (int i = threadIdx.x; i < (int)(sizeof(MPArgs) / 4); i += MP_THREADS)
            reinterpret_cast<int32_t *>(&sa)[i] = reinterpret_cast<const int32_t *>(args + p)[i];
        __syncthreads();
        if (threadIdx.x == 0) {
            sa.n = n;
            resume_s = *(volatile int32_t *)&args[p].st->started;
        }
        __syncthreads();
        const unsigned c = (unsigned)sc, nc = (unsigned)sn;
        solve_load<NMAX>(sa, S, resume_s != 0, c, nc, gctl + 2);
        pipe_start(P, sa, c, nc, it);
        const int r = solve_loop<NMAX>(sa, S, P, it, true, epoch_local);
        pipe_drain(P, it);
        if (P.n_my > 0) it += stages; // the drained slots were issued (a warp without tiles issued none)
        if (r == LOOP_ABORT) {
            ok = false;
            if (threadIdx.x == 0) atomicOr(sa.status, DEV_TIMEOUT);
            if (c == 0) solve_finish<NMAX>(sa, S, false);
            break;
        }
        if (r == LOOP_DONE && c == 0) {
            solve_finish<NMAX>(sa, S, true);
            if (threadIdx.x == 0) atomicAdd(gctl + 2, 1u);
        }
        if (!batch_sync(gctl, gridDim.x, args, n_plans)) {
            ok = false;
            if (threadIdx.x == 0) atomicOr(sa.status, DEV_TIMEOUT);
            break;
        }
    }
    (void)ok;
}

// Per-problem set-up of the batched solver (one block per problem).
// gctl words: [0] arrivals, [1] generation of the batch barrier, [2] the batch
// epoch (bumped when a problem stops), [3] the epoch seen at the last batch
// barrier, [4..5] the problems still iterating then (a 64-bit mask).
__global__ void mp_init_batched_kernel(const MPArgs *__restrict__ args, int32_t n_plans, int32_t n, unsigned *gctl) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        unsigned long long mask = 0ull;
        for (int p = 0; p < n_plans; ++p)
            if (!(args[p].skip && *args[p].skip)) mask |= 1ull << p;
        gctl[0] = gctl[1] = gctl[2] = gctl[3] = 0u;
        gctl[4] = (unsigned)(mask & 0xffffffffu);
        gctl[5] = (unsigned)(mask >> 32);
    }
    MPArgs a = args[blockIdx.x];
    a.n = n;
    if (a.skip && *a.skip) return;
    for (int k = threadIdx.x; k < n; k += blockDim.x) a.y[k] = fminf(fmaxf(a.y[k], lo_of(a, k)), hi_of(a, k));
    if (threadIdx.x == 0) {
        BBState st = {};
        *a.st = st;
    }
}

// The same iteration reading DA from global memory with per-tile reductions
// (more apertures than the register-resident shares hold).
__global__ void __launch_bounds__(MP_THREADS) mp_iter_ldg_kernel(MPArgs a) {
    if (a.st->done || a.st->need_cauchy) return;
    extern __shared__ __align__(16) unsigned char sm[];
    const int n = a.n;
    float *sy = reinterpret_cast<float *>(sm);                          // [n]
    double *accG = reinterpret_cast<double *>(sy + ((n + 3) & ~3));     // [n]
    float *gs = reinterpret_cast<float *>(accG + n);                    // [256]
    float *sT = gs + MP_THREADS, *sO = sT + 256, *sU = sO + 256;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int k = tid; k < n; k += MP_THREADS) {
        sy[k] = a.y[k];
        accG[k] = 0.0;
    }
    for (int k = tid; k < a.n_struct; k += MP_THREADS) {
        sT[k] = a.T[k];
        sO[k] = a.wo[k];
        sU[k] = a.wu[k];
    }
    __syncthreads();
    double facc = 0.0;
    for (int32_t tile = blockIdx.x; tile < a.n_tiles; tile += gridDim.x) {
        const int64_t i0 = (int64_t)tile * MP_THREADS, i = i0 + tid;
        float gi = 0.f;
        if (i < a.V) {
            float zi = 0.f;
            for (int k = 0; k < n; ++k) zi = fmaf(a.DA[da_at(a, i, k)], sy[k], zi);
            a.z[i] = zi;
            gi = voxel_terms(sT, sO, sU, a.sid[i], zi, facc);
        }
        gs[tid] = gi;
        __syncthreads();
        const int nvalid = (int)min64(MP_THREADS, a.V - i0);
        for (int k = wid; k < n; k += MP_NW) {
            float sum = 0.f;
#pragma unroll
            for (int m = lane; m < MP_THREADS; m += 32)
                if (m < nvalid) sum = fmaf(a.DA[da_at(a, i0 + m, k)], gs[m], sum);
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, d);
            if (lane == 0) accG[k] += (double)sum;
        }
        __syncthreads();
    }
    pass_epilogue(a, accG, facc, blockIdx.x, gridDim.x);
}

// Cauchy step, part 1: curvature 2 sum_i w_i (DA G)_i^2 with w the active penalty weight.
__global__ void __launch_bounds__(MP_THREADS) mp_cauchy_pass_kernel(MPArgs a) {
    if (a.st->done || !a.st->need_cauchy) return;
    extern __shared__ __align__(16) unsigned char sm[];
    float *sg = reinterpret_cast<float *>(sm); // [n]
    float *sT = sg + ((a.n + 3) & ~3), *sO = sT + 256, *sU = sO + 256;
    __shared__ double sh[MP_NW];
    const int tid = threadIdx.x;
    for (int k = tid; k < a.n; k += MP_THREADS) sg[k] = (float)a.G[k];
    for (int k = tid; k < a.n_struct; k += MP_THREADS) {
        sT[k] = a.T[k];
        sO[k] = a.wo[k];
        sU[k] = a.wu[k];
    }
    __syncthreads();
    double acc = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * MP_THREADS + tid; i < a.V; i += (int64_t)gridDim.x * MP_THREADS) {
        float q = 0.f;
        for (int k = 0; k < a.n; ++k) q = fmaf(a.DA[da_at(a, i, k)], sg[k], q);
        const int s = a.sid[i];
        const float zi = a.z[i], t = sT[s];
        const float w = zi > t ? sO[s] : (zi < t ? sU[s] : 0.f);
        acc += (double)w * (double)q * (double)q;
    }
    const double b = block_reduce_sum(acc, sh);
    if (tid == 0) a.cpart[blockIdx.x] = b;
}

// Cauchy step, part 2: delta0 = G.G / curvature, then the first projected step.
__global__ void __launch_bounds__(MP_THREADS) mp_cauchy_step_kernel(MPArgs a, int P) {
    BBState *st = a.st;
    if (st->done || !st->need_cauchy) return;
    __shared__ double curv_s;
    if (threadIdx.x == 0) {
        double c = 0.0;
        for (int b = 0; b < P; ++b) c += a.cpart[b];
        curv_s = 2.0 * c;
        st->need_cauchy = 0;
        if (curv_s == 0.0) finish(st, VMAT_STOP_FLAT, 0);
        else st->delta0 = st->gg / curv_s;
    }
    __syncthreads();
    if (curv_s == 0.0) return;
    take_step(a, st->delta0);
    if (threadIdx.x == 0) st->t = 1;
}


// Warp-tile layout from a column-major matrix (DA[k * ld + i]) and the labels; padding 0.
__global__ void to_warp_tiles(const float *src, int64_t ld, int32_t V, int32_t n, const uint8_t *sid,
                              int64_t wstride, int64_t n_wtiles, float *dst) {
    const int64_t total = n_wtiles * wstride;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < total;
         o += (int64_t)gridDim.x * blockDim.x) {
        const int64_t wt = o / wstride, r = o % wstride;
        if (r < MP_HEAD) { // labels of voxels 4r .. 4r + 3 of the tile (words 8 .. 31 stay 0)
            uint32_t packed = 0u;
            if (r < MP_WT / 4)
                for (int j = 0; j < 4; ++j) {
                    const int64_t i = wt * MP_WT + 4 * r + j;
                    if (i < V) packed |= (uint32_t)sid[i] << (8 * j);
                }
            reinterpret_cast<uint32_t *>(dst)[o] = packed;
        } else {
            const int64_t q = r - MP_HEAD;
            const int k = (int)((q >> 7) << 2) + (int)(q & 3);
            const int64_t i = wt * MP_WT + ((q & 127) >> 2);
            dst[o] = (k < n && i < V) ? src[(int64_t)k * ld + i] : 0.f;
        }
    }
}

// Label heads of every warp tile (the DA columns are written by the caller).
__global__ void write_label_heads(const uint8_t *sid, int32_t V, int64_t wstride, int64_t n_wtiles,
                                  uint32_t *dst) {
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < n_wtiles * (MP_WT / 4);
         o += (int64_t)gridDim.x * blockDim.x) {
        const int64_t wt = o / (MP_WT / 4), r = o % (MP_WT / 4);
        uint32_t packed = 0u;
        for (int j = 0; j < 4; ++j) {
            const int64_t i = wt * MP_WT + 4 * r + j;
            if (i < V) packed |= (uint32_t)sid[i] << (8 * j);
        }
        dst[wt * wstride + r] = packed;
    }
}

// ---------------------------------------------------------------------------
// Live tiles (MpLive): the 32-voxel tiles that some placed aperture reaches.
// ---------------------------------------------------------------------------

// Penalty at zero dose of each tile's voxels (a warp per tile, fixed butterfly).
__global__ void mp_tile_const_kernel(const uint8_t *sid, int32_t NA, const float *T, const float *wo,
                                     const float *wu, int64_t n_wtiles, double *c_tile) {
    const int64_t wt = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (wt >= n_wtiles) return; // warp-uniform
    const int lane = threadIdx.x & 31;
    const int64_t i = wt * MP_WT + lane;
    double f = 0.0;
    if (i < NA) {
        const int k = sid[i];
        const double d = -(double)T[k]; // z - T at z = 0
        const double w = d > 0.0 ? (double)wo[k] : (double)wu[k];
        f = w * d * d;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) f += __shfl_xor_sync(0xffffffffu, f, d);
    if (lane == 0) c_tile[wt] = f;
}

// Marks the tiles that column t of DA reaches (a warp per tile; the flag stays set).
__device__ __forceinline__ void live_mark(const MpLive &L, int32_t t, int64_t wt) {
    const int lane = threadIdx.x & 31;
    const float v = L.DA[wt * L.wstride + MP_HEAD + (int64_t)(t >> 2) * 128 + (lane << 2) + (t & 3)];
    if (__any_sync(0xffffffffu, v != 0.f) && lane == 0) {
        L.flag[wt] = 1;
        if (L.gmask) L.gmask[wt] |= 1u << (t >> 2); // one writer per tile and launch
    }
}

__global__ void mp_live_mark_kernel(MpLive L, int32_t t) {
    if (L.skip && *L.skip) return;
    const int64_t wt = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (wt < L.n_wtiles) live_mark(L, t, wt); // warp-uniform
}

__global__ void mp_live_mark_batched_kernel(const MpLive *plans, int32_t t) {
    const MpLive &L = plans[blockIdx.y];
    if (L.skip && *L.skip) return;
    const int64_t wt = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (wt < L.n_wtiles) live_mark(L, t, wt);
}

constexpr int LV_THREADS = MP_LIVE_BLOCK; // a thread per tile

// Block b of the list: the live count of tiles b * 1024 .. and the sum of the
// others' constants (a fixed tree).
__device__ void live_count(const MpLive &L) {
    __shared__ double sums[LV_THREADS];
    const int tid = threadIdx.x;
    const int64_t q = (int64_t)blockIdx.x * LV_THREADS + tid;
    const bool in = q < L.n_wtiles;
    const int f = in && L.flag[q];
    sums[tid] = in && !f ? L.c_tile[q] : 0.0;
    const int c = __syncthreads_count(f);
    for (int st = LV_THREADS / 2; st > 0; st >>= 1) {
        if (tid < st) sums[tid] += sums[tid + st];
        __syncthreads();
    }
    if (L.gmask) { // packed units of the block's live tiles: a head and 4 per marked group
        int32_t u = f ? 1 + 4 * __popc(L.gmask[q]) : 0;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) u += __shfl_xor_sync(0xffffffffu, u, d);
        __shared__ int32_t wu[LV_THREADS / 32];
        if ((tid & 31) == 0) wu[tid >> 5] = u;
        __syncthreads();
        if (tid == 0) {
            int32_t tot = 0;
            for (int w = 0; w < LV_THREADS / 32; ++w) tot += wu[w];
            L.bsize[blockIdx.x] = tot;
        }
    }
    if (tid == 0) {
        L.bcnt[blockIdx.x] = c;
        L.bpart[blockIdx.x] = sums[0];
    }
}

// Block b writes its live tiles after those of blocks 0 .. b-1 (ballot ranks within
// a warp, warp offsets by a scan of the 32 warp counts); block 0 also forms the
// count and F_off = F0 + the block sums in block order.
__device__ void live_write(const MpLive &L, int64_t n_blocks) {
    __shared__ int32_t woff[32];
    __shared__ int32_t base_s;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t q = (int64_t)blockIdx.x * LV_THREADS + tid;
    const bool f = q < L.n_wtiles && L.flag[q];
    const unsigned m = __ballot_sync(0xffffffffu, f);
    if (lane == 0) woff[wid] = __popc(m);
    if (tid == 0) {
        int32_t b = 0;
        for (int64_t k = 0; k < blockIdx.x; ++k) b += L.bcnt[k];
        base_s = b;
    }
    __syncthreads();
    if (wid == 0) { // exclusive scan of the warp counts
        const int32_t v = woff[lane];
        int32_t x = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        woff[lane] = x - v;
    }
    __syncthreads();
    const int32_t li = base_s + woff[wid] + __popc(m & ((1u << lane) - 1u)); // list index of a live tile
    if (f) L.tiles[li] = (int32_t)q;
    if (L.gmask) { // packed offsets in list order: earlier blocks' units, then a block scan
        __shared__ int32_t su[32];
        __shared__ int32_t ubase_s;
        const int32_t u = f ? 1 + 4 * __popc(L.gmask[q]) : 0;
        int32_t x = u;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        if (lane == 31) su[wid] = x;
        if (tid == 0) {
            int32_t b = 0;
            for (int64_t k = 0; k < blockIdx.x; ++k) b += L.bsize[k];
            ubase_s = b;
        }
        __syncthreads();
        if (wid == 0) {
            const int32_t v = su[lane];
            int32_t y = v;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int32_t o = __shfl_up_sync(0xffffffffu, y, d);
                if (lane >= d) y += o;
            }
            su[lane] = y - v;
        }
        __syncthreads();
        if (f) L.poff[li] = ubase_s + su[wid] + x - u;
    }
    if (blockIdx.x == 0 && tid == 0) {
        int32_t n = 0, units = 0;
        double acc = 0.0;
        for (int64_t k = 0; k < n_blocks; ++k) {
            n += L.bcnt[k];
            acc += L.bpart[k];
            if (L.gmask) units += L.bsize[k];
        }
        *L.n_live = n;
        *L.F_off = *L.F0 + acc;
        if (L.gmask) L.poff[n] = units;
    }
}

__global__ void __launch_bounds__(LV_THREADS) mp_live_count_kernel(MpLive L) {
    if (L.skip && *L.skip) return;
    if ((int64_t)blockIdx.x < mp_live_blocks(L.n_wtiles)) live_count(L);
}

__global__ void __launch_bounds__(LV_THREADS) mp_live_write_kernel(MpLive L) {
    if (L.skip && *L.skip) return;
    const int64_t nb = mp_live_blocks(L.n_wtiles);
    if ((int64_t)blockIdx.x < nb) live_write(L, nb);
}

__global__ void __launch_bounds__(LV_THREADS) mp_live_count_batched_kernel(const MpLive *plans) {
    const MpLive &L = plans[blockIdx.y];
    if (L.skip && *L.skip) return;
    if ((int64_t)blockIdx.x < mp_live_blocks(L.n_wtiles)) live_count(L);
}

__global__ void __launch_bounds__(LV_THREADS) mp_live_write_batched_kernel(const MpLive *plans) {
    const MpLive &L = plans[blockIdx.y];
    if (L.skip && *L.skip) return;
    const int64_t nb = mp_live_blocks(L.n_wtiles);
    if ((int64_t)blockIdx.x < nb) live_write(L, nb);
}

vmat_status mp_tile_consts(const uint8_t *sid_c, int32_t NA, const vmat_voxels *vox, int64_t n_wtiles, double *c_tile,
                           cudaStream_t s) {
    if (n_wtiles < 1) return VMAT_OK;
    const int64_t blocks = (n_wtiles * 32 + 255) / 256;
    mp_tile_const_kernel<<<(unsigned)blocks, 256, 0, s>>>(sid_c, NA, vox->T, vox->w_over, vox->w_under, n_wtiles,
                                                          c_tile);
    VMAT_LAUNCH_CHECK();
    return VMAT_OK;
}

// A warp per live list entry: the tile's labels and group mask, then its marked groups
// of the first G groups, ascending (float4 per lane; the group's 512 bytes per warp).
__global__ void mp_pack_kernel(MpLive L, int32_t G) {
    if (L.skip && *L.skip) return;
    const int lane = threadIdx.x & 31;
    const int64_t n_live = min64((int64_t)max(__ldcg(L.n_live), 0), L.n_wtiles);
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n_live;
         i += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t q = __ldcg(L.tiles + i);
        const float *src = L.DA + q * L.wstride;
        float *dst = L.packed + (int64_t)__ldcg(L.poff + i) * 32;
        const uint32_t mask = __ldcg(L.gmask + q);
        if (lane < 8) dst[lane] = src[lane]; // the 32 labels
        if (lane == 8) dst[8] = __uint_as_float(mask);
        int slot = 0;
        for (int g = 0; g < G; ++g) {
            if (!((mask >> g) & 1u)) continue; // warp-uniform
            const float4 v = reinterpret_cast<const float4 *>(src + MP_HEAD + g * 128)[lane];
            reinterpret_cast<float4 *>(dst + MP_HEAD + slot * 128)[lane] = v;
            ++slot;
        }
    }
}

vmat_status mp_pack(const MpLive &L, int32_t n, cudaStream_t s) {
    if (L.n_wtiles < 1 || !L.packed) return VMAT_OK;
    DeviceCtx *ctx;
    VMAT_TRY(device_ctx(&ctx));
    const int64_t want = (L.n_wtiles * 32 + 255) / 256;
    mp_pack_kernel<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)ctx->n_sm * 8)), 256, 0, s>>>(
        L, (n + 3) / 4);
    VMAT_LAUNCH_CHECK();
    return VMAT_OK;
}

vmat_status mp_live_mark(const MpLive &L, int32_t t, cudaStream_t s) {
    if (L.n_wtiles < 1) return VMAT_OK;
    mp_live_mark_kernel<<<(unsigned)((L.n_wtiles * 32 + 255) / 256), 256, 0, s>>>(L, t);
    VMAT_LAUNCH_CHECK();
    return VMAT_OK;
}

vmat_status mp_live_rebuild(const MpLive &L, cudaStream_t s) {
    if (L.n_wtiles < 1) return VMAT_OK;
    const unsigned nb = (unsigned)mp_live_blocks(L.n_wtiles);
    mp_live_count_kernel<<<nb, LV_THREADS, 0, s>>>(L);
    VMAT_LAUNCH_CHECK();
    mp_live_write_kernel<<<nb, LV_THREADS, 0, s>>>(L);
    VMAT_LAUNCH_CHECK();
    return VMAT_OK;
}

vmat_status mp_live_update(const MpLive &L, int32_t t, cudaStream_t s) {
    if (L.n_wtiles < 1) return VMAT_OK;
    mp_live_mark_kernel<<<(unsigned)((L.n_wtiles * 32 + 255) / 256), 256, 0, s>>>(L, t);
    VMAT_LAUNCH_CHECK();
    const unsigned nb = (unsigned)mp_live_blocks(L.n_wtiles);
    mp_live_count_kernel<<<nb, LV_THREADS, 0, s>>>(L);
    VMAT_LAUNCH_CHECK();
    mp_live_write_kernel<<<nb, LV_THREADS, 0, s>>>(L);
    VMAT_LAUNCH_CHECK();
    return VMAT_OK;
}

vmat_status mp_live_update_batched(const MpLive *plans, int32_t n_plans, int64_t max_wtiles, int32_t t,
                                   cudaStream_t s) {
    if (n_plans < 1 || max_wtiles < 1) return VMAT_OK;
    mp_live_mark_batched_kernel<<<dim3((unsigned)((max_wtiles * 32 + 255) / 256), n_plans), 256, 0, s>>>(plans, t);
    VMAT_LAUNCH_CHECK();
    const dim3 g((unsigned)mp_live_blocks(max_wtiles), (unsigned)n_plans);
    mp_live_count_batched_kernel<<<g, LV_THREADS, 0, s>>>(plans);
    VMAT_LAUNCH_CHECK();
    mp_live_write_batched_kernel<<<g, LV_THREADS, 0, s>>>(plans);
    VMAT_LAUNCH_CHECK();
    return VMAT_OK;
}

vmat_status mp_write_labels(const uint8_t *sid, int32_t V, int64_t wstride, float *DA, cudaStream_t s) {
    DeviceCtx *ctx;
    VMAT_TRY(device_ctx(&ctx));
    const int64_t n_wt = ((int64_t)V + MP_WT - 1) / MP_WT;
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>((n_wt * 8 + 255) / 256, (int64_t)ctx->n_sm * 8));
    write_label_heads<<<g, 256, 0, s>>>(sid, V, wstride, n_wt, reinterpret_cast<uint32_t *>(DA));
    VMAT_LAUNCH_CHECK();
    return VMAT_OK;
}

static int solve_nmax(int n) { return n <= 4 ? 4 : ((n + 7) / 8) * 8; }
static size_t solve_fixed(int n) {
    const int nmax = solve_nmax(n);
    return 128 /* alignment slack */ + 2 * (size_t)(nmax / 4) * 16 + 4 * (size_t)nmax * 8 + MP_NW * sizeof(FF) +
           (size_t)nmax * 4 + (size_t)MP_NW * nmax * 4 + 3 * 256 * 4 + (size_t)MP_NW * PQ * (8 + 8) +
           (size_t)MP_NW * WL_CAP * 12 + (size_t)mp_cta_cap(nmax) * sizeof(FF);
}
static size_t solve_smem(int n, int stages) { return solve_fixed(n) + (size_t)stages * MP_NW * wt_copy_bytes(n); }
// Tiles in flight per warp: as many as fit (up to 8) in ~110 KB, so that two CTAs
// share an SM (in 53 KB up to 4 apertures: four CTAs); where not even two fit there, up to
// the per-CTA limit (one CTA per SM).
static int solve_stages(int n) {
    const size_t per = MP_NW * wt_copy_bytes(n);
    const size_t small = (n <= 4 ? 53 : 110) * 1024;
    const size_t st = solve_fixed(n) + 2 * per <= small ? (small - solve_fixed(n)) / per
                                                        : (MP_SMEM_LIMIT - solve_fixed(n)) / per;
    return (int)std::min<size_t>(8, st);
}

using SolveFn = void (*)(MPArgs, int, int);
static SolveFn solve_kernel_for(int n) {
    switch ((n + 7) / 8) {
    case 1: return n <= 4 ? mp_solve_kernel<4> : mp_solve_kernel<8>;
    case 2: return mp_solve_kernel<16>;
    case 3: return mp_solve_kernel<24>;
    case 4: return mp_solve_kernel<32>;
    case 5: return mp_solve_kernel<40>;
    case 6: return mp_solve_kernel<48>;
    case 7: return mp_solve_kernel<56>;
    case 8: return mp_solve_kernel<64>;
    case 9: return mp_solve_kernel<72>;
    case 10: return mp_solve_kernel<80>;
    case 11: return mp_solve_kernel<88>;
    case 12: return mp_solve_kernel<96>;
    default: return nullptr;
    }
}
using SolveBatchFn = void (*)(const MPArgs *, const int64_t *, int32_t, int32_t, unsigned *, int, int);
static SolveBatchFn solve_batched_kernel_for(int n) {
    switch ((n + 7) / 8) {
    case 1: return n <= 4 ? mp_solve_batched_kernel<4> : mp_solve_batched_kernel<8>;
    case 2: return mp_solve_batched_kernel<16>;
    case 3: return mp_solve_batched_kernel<24>;
    case 4: return mp_solve_batched_kernel<32>;
    case 5: return mp_solve_batched_kernel<40>;
    case 6: return mp_solve_batched_kernel<48>;
    case 7: return mp_solve_batched_kernel<56>;
    case 8: return mp_solve_batched_kernel<64>;
    case 9: return mp_solve_batched_kernel<72>;
    case 10: return mp_solve_batched_kernel<80>;
    case 11: return mp_solve_batched_kernel<88>;
    case 12: return mp_solve_batched_kernel<96>;
    default: return nullptr;
    }
}
static size_t ldg_smem(int n) { return (size_t)((n + 3) & ~3) * 4 + (size_t)n * 8 + MP_THREADS * 4 + 3 * 256 * 4; }

int64_t mp_wtile_stride(int32_t n_cap) { return MP_HEAD + (int64_t)((n_cap + 3) / 4) * 128; }

// Launch configuration of one solve with n apertures over V voxels.
struct MPLaunch {
    bool persistent;
    SolveFn fn;
    int stages, keep_in_l2, P, Pc;
    size_t smem;
};

static vmat_status mp_set_attributes() {
    static bool attr = false;
    if (attr) return VMAT_OK;
    for (int n : {4, 8, 16, 24, 32, 40, 48, 56, 64, 72, 80, 88, 96}) { // every kernel
        VMAT_CUDA(cudaFuncSetAttribute(solve_kernel_for(n), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       MP_SMEM_LIMIT));
        VMAT_CUDA(cudaFuncSetAttribute(solve_batched_kernel_for(n), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       MP_SMEM_LIMIT));
    }
    VMAT_CUDA(cudaFuncSetAttribute(mp_iter_ldg_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MP_SMEM_LIMIT));
    VMAT_CUDA(cudaFuncSetAttribute(mp_cauchy_pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MP_SMEM_LIMIT));
    attr = true;
    return VMAT_OK;
}

// Persistent solver (one cooperative launch) up to MP_NMAX apertures, else one
// launch per iteration reading DA from global memory.
static vmat_status mp_configure(int32_t V, int32_t n_ap, const DeviceCtx *ctx, MPLaunch *L) {
    VMAT_TRY(mp_set_attributes());
    const int64_t n_wtiles = ((int64_t)V + MP_WT - 1) / MP_WT;
    const int32_t n_tiles = (int32_t)((V + MP_THREADS - 1) / MP_THREADS);
    L->stages = solve_stages(n_ap);
    L->persistent = n_ap <= MP_NMAX && L->stages >= 2 && solve_smem(n_ap, L->stages) <= MP_SMEM_LIMIT;
    L->fn = L->persistent ? solve_kernel_for(n_ap) : nullptr;
    L->smem = L->persistent ? solve_smem(n_ap, L->stages) : ldg_smem(n_ap);
    L->keep_in_l2 = (double)n_wtiles * (double)wt_copy_bytes(n_ap) <= 64.0 * 1024 * 1024 ? 1 : 0;
    int bps = 1;
    if (L->persistent) VMAT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, L->fn, MP_THREADS, L->smem));
    else VMAT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, mp_iter_ldg_kernel, MP_THREADS, L->smem));
    if (bps < 1) return set_error(VMAT_ECUDA, "mp_bb_solve: the solver kernel does not fit on an SM");
    // every CTA of the persistent grid must be resident at once (they wait for one another)
    L->P = (int)std::max<int64_t>(1, std::min<int64_t>(L->persistent ? (n_wtiles + MP_NW - 1) / MP_NW : n_tiles,
                                                        (int64_t)ctx->n_sm * bps));
    if (L->persistent) L->P = std::min(L->P, mp_cta_cap(solve_nmax(n_ap)));
    L->Pc = std::max(1, std::min<int>(n_tiles, ctx->n_sm * 4));
    return VMAT_OK;
}

// Upper bound on co-resident CTAs of MP_THREADS threads (2048 threads per SM).
static int mp_p_max(const DeviceCtx *ctx) { return ctx->n_sm * (2048 / MP_THREADS); }

// Slots and results of the persistent solvers' exchange; the fallback solver's [P][n + 1]
// partials take the slots' place.
static int32_t mp_rstride(int n_cap) { return (n_cap + 2 + 7) & ~7; } // whole 128-byte lines
static size_t mp_exchange_bytes(int n_cap, int p_max) {
    return ((size_t)p_max * (n_cap + 1) + (size_t)RES_COPIES * mp_rstride(n_cap)) * sizeof(ulonglong2);
}

static size_t mp_ws_bytes(int n_cap, int p_max) {
    return 256 + mp_exchange_bytes(n_cap, p_max) + (size_t)(n_cap + 1) * sizeof(double) +
           (size_t)n_cap * (sizeof(double) + sizeof(float)) + (size_t)p_max * sizeof(double) + 256;
}

// What has to be zero before the first solve on a workspace: the state word, the tag, the
// exchange's words.
static size_t mp_zero_bytes(int n_cap, int p_max) { return 256 + mp_exchange_bytes(n_cap, p_max); }

size_t mp_workspace_bytes(int32_t n_cap) {
    DeviceCtx *ctx;
    if (device_ctx(&ctx) != VMAT_OK) return 0;
    return mp_ws_bytes(n_cap, mp_p_max(ctx));
}

vmat_status mp_workspace_clear(void *ws, int32_t n_cap, cudaStream_t s) {
    DeviceCtx *ctx;
    VMAT_TRY(device_ctx(&ctx));
    VMAT_CUDA(cudaMemsetAsync(ws, 0, mp_zero_bytes(n_cap, mp_p_max(ctx)), s));
    return VMAT_OK;
}

static void mp_fill_args(MPArgs &a, void *ws, int n_cap, int p_max, const float *DA, int64_t wstride, int32_t V,
                         int32_t n_ap, const uint8_t *struct_id, const vmat_voxels *vox, const float *lo,
                         const float *hi, float *y, float *z, const vmat_bb_opts &opts, double F_offset,
                         const MPLaunch &L, const DeviceCtx *ctx) {
    char *p = static_cast<char *>(ws);
    a.st = reinterpret_cast<BBState *>(p);
    a.tag = reinterpret_cast<unsigned *>(p + 192);
    p += 256;
    a.slots = reinterpret_cast<ulonglong2 *>(p);
    a.res = a.slots + (size_t)p_max * (n_cap + 1);
    a.rstride = mp_rstride(n_cap);
    a.part = reinterpret_cast<double *>(p);
    a.G = reinterpret_cast<double *>(p + mp_exchange_bytes(n_cap, p_max)); // [n + 1]
    a.Gprev = a.G + n_cap + 1;
    a.cpart = a.Gprev + n_cap;
    a.yprev = reinterpret_cast<float *>(a.cpart + p_max);
    a.DA = DA;
    a.wstride = wstride;
    a.V = V;
    a.n = n_ap;
    a.sid = struct_id;
    a.T = vox->T;
    a.wo = vox->w_over;
    a.wu = vox->w_under;
    a.n_struct = vox->n_struct;
    a.y = y;
    a.z = z;
    a.lo = lo;
    a.hi = hi;
    a.pstride = p_max;
    a.n_tiles = (int32_t)((V + MP_THREADS - 1) / MP_THREADS);
    a.n_wtiles = ((int64_t)V + MP_WT - 1) / MP_WT;
    a.status = ctx->status;
    a.opts = opts;
    a.F_offset = F_offset;
    a.skip = nullptr;
    a.iters_acc = nullptr;
    a.bytes_acc = nullptr;
    a.tiles = nullptr;
    a.n_live = nullptr;
    a.F_off_dev = nullptr;
    a.packed = nullptr;
    a.poff = nullptr;
}

static vmat_status mp_launch_persistent(MPArgs &a, const MPLaunch &L, cudaStream_t s) {
    int st_arg = L.stages, l2_arg = L.keep_in_l2;
    void *args[] = {&a, &st_arg, &l2_arg};
    VMAT_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(L.fn), dim3(L.P), dim3(MP_THREADS), args,
                                          L.smem, s));
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return VMAT_OK;
}

vmat_status mp_bb_enqueue(const float *DA, int32_t V, int32_t n_ap, int32_t n_cap, int64_t wstride,
                          const uint8_t *struct_id, const vmat_voxels *vox, const float *lo, const float *hi, float *y,
                          float *z, const vmat_bb_opts *opts_in, double F_offset, void *ws, const int32_t *skip,
                          int32_t *iters_acc, cudaStream_t s, const MpLive *live, double *bytes_acc) {
    DeviceCtx *ctx;
    VMAT_TRY(device_ctx(&ctx));
    vmat_bb_opts opts = {500, 1e-6, 1e-9, 1e-12, 1e12};
    if (opts_in) opts = *opts_in;
    if (opts.max_iter < 1) return set_error(VMAT_EINVAL, "mp_bb_solve: max_iter must be >= 1");
    if (n_ap > n_cap) return set_error(VMAT_EINVAL, "mp_bb_enqueue: n_ap > n_cap");
    MPLaunch L;
    VMAT_TRY(mp_configure(V, n_ap, ctx, &L));
    if (!L.persistent)
        return set_error(VMAT_EUNSUPPORTED, "mp_bb_enqueue: %d apertures need the host-driven solver", n_ap);
    MPArgs a;
    mp_fill_args(a, ws, n_cap, mp_p_max(ctx), DA, wstride, V, n_ap, struct_id, vox, lo, hi, y, z, opts, F_offset, L,
                 ctx);
    a.skip = skip;
    a.iters_acc = iters_acc;
    a.bytes_acc = bytes_acc;
    if (live) {
        a.tiles = live->tiles;
        a.n_live = live->n_live;
        a.F_off_dev = live->F_off;
        a.packed = live->packed;
        a.poff = live->poff;
    }
    return mp_launch_persistent(a, L, s);
}

size_t mp_args_bytes() { return sizeof(MPArgs); }

vmat_status mp_fill_plan_args(void *out, void *ws, int32_t n_cap, const float *DA, int64_t wstride, int32_t V,
                              const uint8_t *struct_id, const vmat_voxels *vox, const float *lo, const float *hi,
                              float *y, float *z, const vmat_bb_opts *opts_in, double F_offset, const int32_t *skip,
                              int32_t *iters_acc, const MpLive *live) {
    DeviceCtx *ctx;
    VMAT_TRY(device_ctx(&ctx));
    vmat_bb_opts opts = {500, 1e-6, 1e-9, 1e-12, 1e12};
    if (opts_in) opts = *opts_in;
    if (opts.max_iter < 1) return set_error(VMAT_EINVAL, "mp_bb_solve: max_iter must be >= 1");
    MPLaunch L = {};
    L.P = 1;
    MPArgs a;
    mp_fill_args(a, ws, n_cap, mp_p_max(ctx), DA, wstride, V, n_cap, struct_id, vox, lo, hi, y, z, opts, F_offset, L,
                 ctx);
    a.skip = skip;
    a.iters_acc = iters_acc;
    if (live) {
        a.tiles = live->tiles;
        a.n_live = live->n_live;
        a.F_off_dev = live->F_off;
    }
    memcpy(out, &a, sizeof(MPArgs));
    return VMAT_OK;
}

vmat_status mp_batched_grid(int32_t n, int32_t n_plans, int32_t *grid, int32_t *stages, size_t *smem) {
    DeviceCtx *ctx;
    VMAT_TRY(device_ctx(&ctx));
    VMAT_TRY(mp_set_attributes());
    if (n < 1 || n > MP_NMAX) return set_error(VMAT_EUNSUPPORTED, "batched master problem: %d apertures (max %d)", n, MP_NMAX);
    const int st = solve_stages(n);
    const size_t sm = solve_smem(n, st);
    if (st < 2 || sm > MP_SMEM_LIMIT) return set_error(VMAT_EUNSUPPORTED, "batched master problem: no fit for %d", n);
    int bps = 0;
    VMAT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, solve_batched_kernel_for(n), MP_THREADS, sm));
    if (bps < 1) return set_error(VMAT_ECUDA, "batched master problem: kernel does not fit on an SM");
    // every CTA resident at once (they wait for one another)
    const int64_t P = std::min<int64_t>((int64_t)ctx->n_sm * bps, mp_cta_cap(solve_nmax(n)));
    if (P < n_plans) return set_error(VMAT_EUNSUPPORTED, "batched master problem: more plans than resident CTAs");
    *grid = (int32_t)P;
    *stages = st;
    *smem = sm;
    return VMAT_OK;
}

vmat_status mp_bb_enqueue_batched(const void *args, const int64_t *weight, unsigned *gctl, int32_t n_plans, int32_t n,
                                  int32_t grid, int32_t stages, size_t smem, int keep_in_l2, cudaStream_t s) {
    mp_init_batched_kernel<<<n_plans, 128, 0, s>>>(static_cast<const MPArgs *>(args), n_plans, n, gctl);
    VMAT_LAUNCH_CHECK();
    SolveBatchFn fn = solve_batched_kernel_for(n);
    if (!fn) return set_error(VMAT_EUNSUPPORTED, "batched master problem: %d apertures", n);
    const MPArgs *a = static_cast<const MPArgs *>(args);
    int32_t np = n_plans, nn = n;
    int st = stages, l2 = keep_in_l2;
    void *kargs[] = {&a, &weight, &np, &nn, &gctl, &st, &l2};
    VMAT_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(fn), dim3(grid), dim3(MP_THREADS), kargs, smem,
                                          s));
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return VMAT_OK;
}

vmat_status mp_bb_impl(const float *DA, int32_t V, int32_t n_ap, int64_t ld, const uint8_t *struct_id,
                       int64_t wstride, const vmat_voxels *vox, const float *lo, const float *hi, float *y,
                       float *z, const vmat_bb_opts *opts_in, double F_offset, vmat_bb_report *rep, cudaStream_t s) {
    DeviceCtx *ctx;
    VMAT_TRY(device_ctx(&ctx));
    vmat_bb_opts opts = {500, 1e-6, 1e-9, 1e-12, 1e12};
    if (opts_in) opts = *opts_in;
    if (opts.max_iter < 1) return set_error(VMAT_EINVAL, "mp_bb_solve: max_iter must be >= 1");
    if (ldg_smem(n_ap) > MP_SMEM_LIMIT) return set_error(VMAT_EUNSUPPORTED, "mp_bb_solve: too many apertures (%d)", n_ap);
    const int64_t n_wtiles = ((int64_t)V + MP_WT - 1) / MP_WT;

    MPLaunch L;
    VMAT_TRY(mp_configure(V, n_ap, ctx, &L));
    const int p_max = std::max(mp_p_max(ctx), std::max(L.P, L.Pc));
    const size_t conv_bytes =
        wstride == 0 ? (((size_t)n_wtiles * mp_wtile_stride(n_ap) * sizeof(float) + 255) & ~(size_t)255) : 0;
    const size_t bytes = conv_bytes + mp_ws_bytes(n_ap, p_max);
    // (from the default pool the 70 MB of a 422K-voxel, 40-aperture problem were mapped anew in every
    // call: 3.8 ms for a new state's first pass instead of 2.7)
    Scratch own;
    VMAT_TRY(own.alloc_kept(bytes, s));
    void *const mem = own.ptr;
    void *const ws = static_cast<char *>(mem) + conv_bytes;
    // a column-major input is copied once into the warp-tile layout (with the labels)
    if (wstride == 0) {
        wstride = mp_wtile_stride(n_ap);
        const int64_t total = n_wtiles * wstride;
        const int g = (int)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, (int64_t)ctx->n_sm * 16));
        to_warp_tiles<<<g, 256, 0, s>>>(DA, ld, V, n_ap, struct_id, wstride, n_wtiles, static_cast<float *>(mem));
        VMAT_LAUNCH_CHECK();
        DA = static_cast<const float *>(mem);
    }
    MPArgs a;
    mp_fill_args(a, ws, n_ap, p_max, DA, wstride, V, n_ap, struct_id, vox, lo, hi, y, z, opts, F_offset, L, ctx);
    const size_t smem_cauchy = (size_t)((n_ap + 3) & ~3) * 4 + 3 * 256 * 4;

    static thread_local BBState *host_st = nullptr;
    if (!host_st) VMAT_CUDA(cudaMallocHost(&host_st, sizeof(BBState)));

    if (L.persistent) {
        VMAT_CUDA(cudaMemsetAsync(ws, 0, mp_zero_bytes(n_ap, p_max), s));
        VMAT_TRY(mp_launch_persistent(a, L, s));
        VMAT_CUDA(cudaMemcpyAsync(host_st, a.st, sizeof(BBState), cudaMemcpyDeviceToHost, s));
        VMAT_CUDA(cudaStreamSynchronize(s));
    } else {
        mp_init_kernel<<<1, MP_THREADS, 0, s>>>(a);
        VMAT_LAUNCH_CHECK();
        int launched = 0;
        while (launched < opts.max_iter) {
            const int chunk = launched == 0 ? 1 : std::min(MP_CHUNK, opts.max_iter - launched);
            for (int c = 0; c < chunk; ++c) {
                mp_iter_ldg_kernel<<<L.P, MP_THREADS, L.smem, s>>>(a);
                g_launches.fetch_add(1, std::memory_order_relaxed);
                if (launched + c == 0) {
                    mp_cauchy_pass_kernel<<<L.Pc, MP_THREADS, smem_cauchy, s>>>(a);
                    mp_cauchy_step_kernel<<<1, MP_THREADS, 0, s>>>(a, L.Pc);
                    g_launches.fetch_add(2, std::memory_order_relaxed);
                }
            }
            VMAT_CUDA(cudaGetLastError());
            launched += chunk;
            VMAT_CUDA(cudaMemcpyAsync(host_st, a.st, sizeof(BBState), cudaMemcpyDeviceToHost, s));
            VMAT_CUDA(cudaStreamSynchronize(s));
            if (host_st->done) break;
        }
    }
    if (!host_st->done) return set_error(VMAT_ECUDA, "mp_bb_solve: solver did not reach a stopping rule");
    int32_t dev_status = 0;
    VMAT_CUDA(cudaMemcpy(&dev_status, ctx->status, 4, cudaMemcpyDeviceToHost));
    if (dev_status & DEV_TIMEOUT) return set_error(VMAT_ETIMEOUT, "mp_bb_solve: a device-side wait ran out");
    if (rep) {
        rep->iters = host_st->iters;
        rep->stop_reason = host_st->stop;
        rep->F = host_st->F;
    }
    return VMAT_OK;
}

} // namespace vmat

using namespace vmat;

extern "C" vmat_status mp_bb_solve(const float *DA, int32_t V, int32_t n_ap, int64_t ld, const vmat_voxels *vox,
                                   const float *lo, const float *hi, float *y, float *z, const vmat_bb_opts *opts,
                                   vmat_bb_report *rep, void *stream) {
    clear_error();
    VMAT_TRY(validate_voxels(vox));
    if (V <= 0 || n_ap <= 0 || ld < V || !DA || !y || !z)
        return set_error(VMAT_EINVAL, "mp_bb_solve: need V > 0, n_ap > 0, ld >= V and non-NULL DA, y, z");
    return mp_bb_impl(DA, V, n_ap, ld, vox->struct_id, 0, vox, lo, hi, y, z, opts, 0.0, rep, as_stream(stream));
}
