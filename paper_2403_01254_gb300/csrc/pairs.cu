// Candidate search and pair kernel of the hot path.
//
// For every edge (a, b) of the pose graph the points y_j of frame b are the
// queries: each is moved into frame a (y' = T_ab y, T_ab = T_a^-1 T_b; the
// pair distance of Eq. inner_product_actual_ba written in frame a, since
// |T_a x - T_b y| = |x - T_ab y|) and keyed by the frame-a grid cell holding
// it.  A stable radix sort groups the queries by home cell (order inside a
// cell = frame-b order, so results do not depend on thread timing), and the
// groups are cut into units of <= 32 queries.  A warp takes one unit, or one part
// of a unit with a long stream, holds its queries in registers and streams the candidates
// of the 27 surrounding cells, 32 at a time, through a box test against the unit's
// queries.  For every candidate x query pair inside r_c the weight
//     w = <l_i, l_j> * k_c(c_i, c_j) * exp(-|d|^2 / (2 ell^2))      Eq. (irls_weight)
// enters the sums that fix the 28 edge moments (layout in common.cuh), and
// through them the loss, the gradient of Eq. (inner_product_reformat) and the
// Gauss-Newton blocks of Eq. (irls_final).  Two unit bodies do this:
//   * the dense tile unit (no colour, no pruning): every element of the
//     32-candidate x unit tile in MMA fragment layout, label products and
//     per-query moment sums on the tensor cores (see "dense tile path");
//   * the lane unit (colour, semantic pruning, no labels): lanes over the
//     queries, all in FP32 (see "lane path").
// The moments of a unit (of each of its parts) are summed over the warp in a fixed order and
// rounded to 64-bit fixed point, so edge totals are exact integer sums, independent of which
// warp ran which unit and of the other edges.
//
// No FP64 arithmetic runs per query: the frame-a position of a frame-b cell
// centre comes from a per-edge affine map held as double-float pairs, evaluated
// with error-free transformations (Dekker product, Knuth sum) on the FP32 pipe.
#include "per_device.h"
#include "radix.cuh"

#include <type_traits>

namespace rk {

namespace {
constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t NO_KEY = 0xffffffffu;

// ---------------------------------------------------------- double-float --
struct df { float hi, lo; };

__device__ __forceinline__ df two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    const float e = (a - (s - bb)) + (b - bb);
    return {s, e};
}
__device__ __forceinline__ df fast_two_sum(float a, float b) {
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ df df_add(df a, df b) {
    const df s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, s.lo + a.lo + b.lo);
}
// (hi + lo) * c for a float c holding a small integer or half-integer
__device__ __forceinline__ df df_mul_f(float hi, float lo, float c) {
    const float p = hi * c;
    const float e = fmaf(hi, c, -p);
    return fast_two_sum(p, fmaf(lo, c, e));
}

// One edge's transform and its map of cell centres, by one warp: nine lanes an
// entry of R_ab each, three an entry of t_ab.
__device__ __forceinline__ void edge_transform(const double* __restrict__ poses, const EdgeDev& Ed, const FrameDev& Fb,
                                               double h, EdgeXf& X, int lane) {
    const double* Ta = poses + 16 * Ed.a;
    const double* Tb = poses + 16 * Ed.b;
    // R_ab = R_a^T R_b (lane 3 r + c: entry (r, c)),  t_ab = R_a^T (t_b - t_a) (lanes 9..11)
    const int r = lane < 9 ? lane / 3 : lane - 9, c = lane % 3;
    double v = 0.0, prod = 0.0;
    if (lane < 9) {
        for (int k = 0; k < 3; ++k) v += Ta[4 * k + r] * Tb[4 * k + c];
        X.R[lane] = v;
        X.Rf[lane] = (float)v;
        // P(l) = h R l + [R (lo_b + 1/2) h + t]
        const double A = h * v;
        X.Ahi[lane] = (float)A;
        X.Alo[lane] = (float)(A - (double)(float)A);
        prod = v * ((double)Fb.lo[c] + 0.5) * h;
    } else if (lane < 12) {
        v = Ta[r] * (Tb[3] - Ta[3]) + Ta[4 + r] * (Tb[7] - Ta[7]) + Ta[8 + r] * (Tb[11] - Ta[11]);
        X.t[r] = v;
    }
    const int src = lane >= 9 && lane < 12 ? 3 * r : 0;
    const double p0 = __shfl_sync(FULL, prod, src), p1 = __shfl_sync(FULL, prod, src + 1),
                 p2 = __shfl_sync(FULL, prod, src + 2);
    if (lane >= 9 && lane < 12) {
        const double B = v + p0 + p1 + p2;
        X.Bhi[r] = (float)B;
        X.Blo[r] = (float)(B - (double)(float)B);
    }
}

// Start of an evaluation: the edges' transforms, one warp per edge (nine lanes
// an entry of R_ab each: FP64 chains of a few operations instead of the ~100 of
// one thread per edge, 8.4 us at 28 edges), and everything cleared that the
// evaluation counts or adds into: the sort's digit counts and tile counters,
// the unit counters and the edges' accumulators.
__global__ void __launch_bounds__(128) k_eval_setup(const double* __restrict__ poses, const EdgeDev* __restrict__ edges,
                                                    int E, const FrameDev* __restrict__ frames, double h,
                                                    EdgeXf* __restrict__ xf, long long* __restrict__ ws, int n_ws,
                                                    int* __restrict__ ucount, long long* __restrict__ acc,
                                                    const int* done) {
    chain_enter();
    if (done && *done) return;
    const int gt = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    for (int i = gt; i < n_ws; i += nt) ws[i] = 0;
    for (long long i = gt; i < (long long)E * ACC_N; i += nt) acc[i] = 0;
    if (gt < 4) ucount[gt] = 0;
    const int lane = threadIdx.x & 31;
    for (int e = gt >> 5; e < E; e += nt >> 5) {
        edge_transform(poses, edges[e], frames[edges[e].b], h, xf[e], lane);
    }
}

__device__ __forceinline__ int find_edge_q(const EdgeDev* __restrict__ edges, int E, long long q) {
    int lo = 0, hi = E - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (edges[mid].q_off <= q) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int find_edge_bin(const EdgeDev* __restrict__ edges, int E, long long bin) {
    int lo = 0, hi = E - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (edges[mid].bin_off <= bin) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Home cell of one query among frame a's cells (NO_KEY: outside the grid) and
// its record, the FP32 offset from that cell's centre.  p: the point, relative to
// the centre of its own cell l of frame b; s: its index.
__device__ __forceinline__ uint32_t query_key(const FrameDev& Fa, const FrameDev& Fb, const EdgeXf& X, int l,
                                              const float4 p, int s, const GridParams& gp, float4& rec) {
    const float lf[3] = {(float)(l % Fb.dim[0]), (float)((l / Fb.dim[0]) % Fb.dim[1]),
                         (float)(l / (Fb.dim[0] * Fb.dim[1]))};
    float K[3], F[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        df P = {X.Bhi[r], X.Blo[r]};
#pragma unroll
        for (int c = 0; c < 3; ++c) P = df_add(P, df_mul_f(X.Ahi[3 * r + c], X.Alo[3 * r + c], lf[c]));
        float k = floorf(P.hi * gp.hf_inv);
        k = fminf(fmaxf(k, -4194304.f), 4194304.f);
        df C = df_mul_f(gp.hf, gp.hf_lo, k + 0.5f);
        df Rm = df_add(P, {-C.hi, -C.lo});
        float f = Rm.hi + Rm.lo;
        if (f < -0.5f * gp.hf) { k -= 1.f; C = df_mul_f(gp.hf, gp.hf_lo, k + 0.5f);
                                 Rm = df_add(P, {-C.hi, -C.lo}); f = Rm.hi + Rm.lo; }
        else if (f >= 0.5f * gp.hf) { k += 1.f; C = df_mul_f(gp.hf, gp.hf_lo, k + 0.5f);
                                      Rm = df_add(P, {-C.hi, -C.lo}); f = Rm.hi + Rm.lo; }
        K[r] = k;
        F[r] = f;
    }
    const float* R = X.Rf;
    const float vx = fmaf(R[2], p.z, fmaf(R[1], p.y, fmaf(R[0], p.x, F[0])));
    const float vy = fmaf(R[5], p.z, fmaf(R[4], p.y, fmaf(R[3], p.x, F[1])));
    const float vz = fmaf(R[8], p.z, fmaf(R[7], p.y, fmaf(R[6], p.x, F[2])));
    const float mx = floorf(fmaf(vx, gp.hf_inv, 0.5f));
    const float my = floorf(fmaf(vy, gp.hf_inv, 0.5f));
    const float mz = floorf(fmaf(vz, gp.hf_inv, 0.5f));
    const int hx = (int)(K[0] + mx) - Fa.lo[0];
    const int hy = (int)(K[1] + my) - Fa.lo[1];
    const int hz = (int)(K[2] + mz) - Fa.lo[2];
    const float ox = fmaf(-mx, gp.hf, vx), oy = fmaf(-my, gp.hf, vy), oz = fmaf(-mz, gp.hf, vz);
    rec = make_float4(ox, oy, oz, __int_as_float(s));
    if (hx < 0 || hy < 0 || hz < 0 || hx >= Fa.dim[0] || hy >= Fa.dim[1] || hz >= Fa.dim[2]) return NO_KEY;
    const uint32_t cell = (uint32_t)(((long long)hz * Fa.dim[1] + hy) * Fa.dim[0] + hx);
    // with key_sub = 3 the low bits hold the query's octant of its home
    // cell, so a cell's queries sort by octant and a unit's are close
    return gp.key_sub ? (cell << 3) | (ox >= 0.f ? 1u : 0u) | (oy >= 0.f ? 2u : 0u) | (oz >= 0.f ? 4u : 0u) : cell;
}

// One thread per query: frame-a home cell key and the query's FP32 offset
// from that cell's centre.  The block also counts its keys' digits and clears
// its share of the sort's tile records (radix.cuh).
__global__ void __launch_bounds__(RAD_T) k_query_keys(const EdgeDev* __restrict__ edges, int E,
                                                      const FrameDev* __restrict__ frames,
                                                      const EdgeXf* __restrict__ xf, const uint32_t* __restrict__ pt_cell,
                                                      const float4* __restrict__ pts4, GridParams gp, long long Q,
                                                      uint32_t* __restrict__ qkey, float4* __restrict__ qrec,
                                                      RadixWs ws, int rounds, const int* done) {
    chain_enter();
    if (done && *done) return;
    __shared__ int hist[RAD_PASSES][256];
#pragma unroll
    for (int p = 0; p < RAD_PASSES; ++p) hist[p][threadIdx.x] = 0;
    __syncthreads();
    for (int round = 0; round < rounds; ++round) {
        const long long q = ((long long)blockIdx.x * rounds + round) * RAD_T + threadIdx.x;
        uint32_t key = NO_KEY;
        if (q < Q) {
        const int e = find_edge_q(edges, E, q);
        const EdgeDev& Ed = edges[e];
        const FrameDev& Fa = frames[Ed.a];
        const FrameDev& Fb = frames[Ed.b];
        const int s = (int)(Fb.pt_off + (q - Ed.q_off));
        const uint32_t local = query_key(Fa, Fb, xf[e], (int)((long long)pt_cell[s] - Fb.cell_off), pts4[s], s, gp, qrec[q]);
        if (local != NO_KEY) key = (uint32_t)(Ed.bin_off << gp.key_sub) + local;
        qkey[q] = key;
        }
        radix_count(key, q < Q, ws.npass, hist);
    }
    __syncthreads();
    radix_finish(ws, hist);
}

// log2 of the parts that a unit of n queries of home cell `cell` comes in (see common.cuh): edge
// and unit decide, nothing else.  n_b: queries of the edge.
__device__ __forceinline__ int cut_shift(int cut_edge, const FrameDev& Fa, int n_b,
                                         const int* __restrict__ cell_start, int cell, int n) {
    if (n_b > cut_edge) return 0;
    const int least = max(min(max(n_b >> 3, CUT_SMALL), CUT_POINTS), n_b >> 6);
    // Runs of cells by their places in the flat grid (at its very edge, where a row would leave
    // it, other cells are counted, which make as good a rule).  First, for each of the three planes, all
    // cells from the first to the last of its nine: a bound that takes six reads; the eighteen of the
    // nine rows for every unit of a sparse cloud took a ten-iteration solve of 2 x 2000 points from
    // 746 to 785 us.
    const int dx = Fa.dim[0], plane = dx * Fa.dim[1], cells = plane * Fa.dim[2];
    const int* c = cell_start + Fa.cell_off;
    auto points = [&](int from, int to) { return __ldg(c + min(max(to + 1, 0), cells)) - __ldg(c + min(max(from, 0), cells)); };
    long long most = 0;
#pragma unroll
    for (int z = -1; z <= 1; ++z) most += points(cell + z * plane - dx - 1, cell + z * plane + dx + 1);
    if (most < 2 * least) return 0;
    int in_row[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int at = cell + (k % 3 - 1) * dx + (k / 3 - 1) * plane;
        in_row[k] = points(at - 1, at + 1);
    }
    long long all = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) all += in_row[k];
    int s = 0;
    while (s < 3 && (1 << s) <= n && (all >> (s + 1)) >= least) ++s;
    return s;
}

// Place of a lane's records among the warp's (2^s each where `start` holds), and their number.
__device__ __forceinline__ int unit_places(bool start, int s, int lane, int& total) {
    const unsigned m = __ballot_sync(FULL, start);
    int at = __popc(m & ((1u << lane) - 1u));
    total = __popc(m);
    if (__any_sync(FULL, s > 0)) {
        int more = (1 << s) - 1, inc = more;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += u;
        }
        at += inc - more;
        total += __shfl_sync(FULL, inc, 31);
    }
    return at;
}

// Sorted query records and the unit list, in one pass over the sorted keys: a
// unit starts at the first query of a home cell and every uq queries after.
// A block takes 256 sorted queries; where its first one continues a cell of
// an earlier block, the block looks for that cell's first query.  One atomic per block reserves its slots in the
// unit list; a record holds edge and queries, so that no warp of the pair
// kernels searches for either.
__global__ void __launch_bounds__(256) k_units(const uint32_t* __restrict__ key, const int* __restrict__ val,
                                               const float4* __restrict__ qrec, long long Q, int uq, int sub,
                                               int cut_edge,
                                               const EdgeDev* __restrict__ edges, int E,
                                               const FrameDev* __restrict__ frames,
                                               const int* __restrict__ cell_start,
                                               float4* __restrict__ slots, int2* __restrict__ units,
                                               int* __restrict__ n_units, const int* done) {
    chain_enter();
    if (done && *done) return;
    __shared__ int s_cnt[8], s_first[8];
    __shared__ int s_base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long base = (long long)blockIdx.x * blockDim.x; base < Q; base += (long long)gridDim.x * blockDim.x) {
        const long long k = base + threadIdx.x;
        uint32_t kk = NO_KEY, prev = NO_KEY;
        if (k < Q) {
            slots[k] = qrec[val[k]];
            kk = key[k];
            if (k > 0) prev = key[k - 1];
        }
        const bool valid = kk != NO_KEY;
        const bool head = valid && (k == 0 || (prev >> sub) != (kk >> sub));   // first query of its cell
        // last cell head at or before this query inside the block
        const unsigned hm = __ballot_sync(FULL, head) & (0xffffffffu >> (31 - lane));
        int start = hm ? warp * 32 + 31 - __clz(hm) : -1;
        if (lane == 31) s_first[warp] = start;
        __syncthreads();
        if (start < 0)
            for (int w = warp - 1; w >= 0 && start < 0; --w) start = s_first[w];
        // where the cell starts that the block's first query continues: among the 256
        // queries before it or, for a cell longer than that, found by a 256-ary search (the keys are
        // sorted; three reads for any cell, where a walk back over them took one per 256
        // queries: an evaluation with 400 000 queries in one cell 0.60 -> 0.13 ms)
        const uint32_t c0 = key[base] >> sub;
        long long from = base;
        if (key[base] != NO_KEY && base > 0 && (key[base - 1] >> sub) == c0) {
            from = base - __syncthreads_count(base > threadIdx.x && (key[base - 1 - threadIdx.x] >> sub) == c0);
            if (from == base - 256) {
                long long lo = 0;                    // the first query lies in [lo, from]
                while (lo < from) {
                    const long long step = (from - lo + 255) / 256, p = lo + threadIdx.x * step;
                    const int n = (int)((from - lo + step - 1) / step);
                    const int before = n - __syncthreads_count(p < from && (key[p] >> sub) == c0);
                    const long long last = lo + (before - 1) * step;      // the last probe of an earlier cell
                    if (before < n) from = lo + before * step;
                    if (before > 0) lo = last + 1;
                    else lo = from;
                }
            }
        }
        const long long run = start >= 0 ? base + start : from;
        const bool st = valid && ((k - run) % uq) == 0;
        int e = 0, n = 0, s = 0;
        if (st) {
            // queries of the cell from here on, uq at most (gallop, then bisect)
            int m = 1;
            while (m < uq && k + m < Q && (key[k + m] >> sub) == (kk >> sub)) m *= 2;
            int lo = m / 2 + 1, hi = m < uq ? m : uq;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (k + mid < Q && (key[k + mid] >> sub) == (kk >> sub)) lo = mid + 1; else hi = mid;
            }
            n = lo;
            e = find_edge_bin(edges, E, kk >> sub);
            s = cut_shift(cut_edge, frames[edges[e].a], frames[edges[e].b].n_pts, cell_start,
                          (int)((kk >> sub) - edges[e].bin_off), n);
        }
        int total;
        const int at = unit_places(st, s, lane, total);
        if (lane == 0) s_cnt[warp] = total;
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int w = 0; w < 8; ++w) { const int c = s_cnt[w]; s_cnt[w] = tot; tot += c; }
            s_base = tot ? atomicAdd(n_units, tot) : 0;
        }
        __syncthreads();
        if (st)
            for (int part = 0; part < 1 << s; ++part)
                units[s_base + s_cnt[warp] + at + part] = unit_record((int)k, e, n, s, part);
        __syncthreads();
    }
}

// ------------------------------------------------ binning by one block ----
// Problems whose edges have few queries (<= BIN_MAX each) are binned by one block per
// edge in one launch: transform, keys, the sort (in shared memory; edges' keys
// are apart, so sorting every edge by itself sorts them all, but for the queries
// of no home cell, which end their edge instead of the list), sorted records and
// units.  The chain of setup, keys, a kernel per 8-bit digit and the unit pass is
// bound by its 6 or 7 launches and the look-back between tiles: 2 x 2000 points, one
// evaluation 138 -> 119 us and one LM iteration 89 -> 84 us (this kernel 18 us, bound by the
// latency of its barriers and digit ranking), 60-rotation search of 2 x 4000 1283 ->
// 1250 us.  At 5003 queries per edge it takes as long as the chain (28 us: one SM's
// issue rate), at 8000 longer (39 us), so edges end at BIN_MAX.
constexpr int BIN_T = 1024;
constexpr int BIN_W = BIN_T / 32;

template <int IPT>
struct BinSmem {
    static constexpr int CAP = BIN_T * IPT;
    static constexpr size_t KEY = 0;                                     // [CAP] uint32
    static constexpr size_t VAL = KEY + 4 * CAP;                         // [CAP] uint16
    static constexpr size_t CNT = VAL + 2 * CAP;                         // [BIN_W][256] uint16
    static constexpr size_t BYTES = CNT + 2 * BIN_W * 256;
};

template <int IPT>
__global__ void __launch_bounds__(BIN_T) k_bin_edges(const double* __restrict__ poses, const EdgeDev* __restrict__ edges,
                                                     const FrameDev* __restrict__ frames,
                                                     const uint32_t* __restrict__ pt_cell,
                                                     const float4* __restrict__ pts4,
                                                     const int* __restrict__ cell_start, GridParams gp, int uq, int cut_edge,
                                                     EdgeXf* __restrict__ xf, uint32_t* qkey, float4* qrec,
                                                     float4* slots, int2* units, int* n_units,
                                                     long long* __restrict__ acc, const int* done) {
    chain_enter();
    if (done && *done) return;
    using L = BinSmem<IPT>;
    extern __shared__ float4 smem4[];
    unsigned char* sm = reinterpret_cast<unsigned char*>(smem4);
    uint32_t* s_key = reinterpret_cast<uint32_t*>(sm + L::KEY);
    uint16_t* s_val = reinterpret_cast<uint16_t*>(sm + L::VAL);
    uint16_t(*cnt)[256] = reinterpret_cast<uint16_t(*)[256]>(sm + L::CNT);
    __shared__ EdgeXf X;
    __shared__ int s_part[4][256], s_off[4][256], s_sum[BIN_W], s_first[BIN_W], s_base;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int e = blockIdx.x;
    const EdgeDev& Ed = edges[e];
    const FrameDev& Fa = frames[Ed.a];
    const FrameDev& Fb = frames[Ed.b];
    const int n = Fb.n_pts;
    if (warp == 0) edge_transform(poses, Ed, Fb, gp.h, X, lane);
    else if (warp == 1) acc[(long long)e * ACC_N + lane] = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) reinterpret_cast<uint32_t*>(cnt[warp])[lane + 32 * j] = 0u;
    __syncthreads();
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(&X);
        uint32_t* dst = reinterpret_cast<uint32_t*>(xf + e);
        for (int i = tid; i < (int)(sizeof(EdgeXf) / 4); i += BIN_T) dst[i] = src[i];
    }
    // a warp's queries are one run of the edge's
    const int at0 = warp * (32 * IPT) + lane;
    uint32_t key[IPT];
    int val[IPT];
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const int i = at0 + 32 * r;
        key[r] = NO_KEY;
        val[r] = i;
        if (i < n) {
            const int s = (int)Fb.pt_off + i;
            key[r] = query_key(Fa, Fb, X, (int)((long long)pt_cell[s] - Fb.cell_off), pts4[s], s, gp,
                               qrec[Ed.q_off + i]);
        }
    }
    // stable sort by 8-bit digits; bits such that NO_KEY's lie above every cell's
    const long long top = ((long long)Fa.dim[0] * Fa.dim[1] * Fa.dim[2]) << gp.key_sub;
    int bits = 1;
    while ((1LL << bits) <= top) ++bits;
    for (int shift = 0; shift < bits; shift += 8) {
        int rank[IPT];
#pragma unroll
        for (int r = 0; r < IPT; ++r) {
            const bool valid = at0 + 32 * r < n;
            const int d = valid ? (int)((key[r] >> shift) & 255u) : 256;
            const unsigned peers = __match_any_sync(FULL, d);
            const int leader = __ffs(peers) - 1;
            int old = 0;
            if (valid && lane == leader) {
                old = cnt[warp][d];
                cnt[warp][d] = (uint16_t)(old + __popc(peers));
            }
            rank[r] = __shfl_sync(FULL, old, leader) + __popc(peers & lt);
            __syncwarp();
        }
        __syncthreads();
        // exclusive sums over the warps, a quarter of them per group of 256 threads, then over the digits
        {
            const int d = tid & 255, q = tid >> 8;
            int sum = 0;
#pragma unroll
            for (int w = 0; w < BIN_W / 4; ++w) {
                const int c = cnt[q * (BIN_W / 4) + w][d];
                cnt[q * (BIN_W / 4) + w][d] = (uint16_t)sum;
                sum += c;
            }
            s_part[q][d] = sum;
        }
        __syncthreads();
        int tot = 0, inc = 0;
        if (tid < 256) {
            tot = s_part[0][tid] + s_part[1][tid] + s_part[2][tid] + s_part[3][tid];
            inc = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(FULL, inc, o);
                if (lane >= o) inc += u;
            }
            if (lane == 31) s_sum[warp] = inc;
        }
        __syncthreads();
        if (tid < 256) {
            int base = inc - tot;
            for (int w = 0; w < warp; ++w) base += s_sum[w];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                s_off[q][tid] = base;
                base += s_part[q][tid];
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < IPT; ++r) {
            if (at0 + 32 * r < n) {
                const int d = (int)((key[r] >> shift) & 255u);
                const int at = s_off[warp / (BIN_W / 4)][d] + cnt[warp][d] + rank[r];
                s_key[at] = key[r];
                s_val[at] = (uint16_t)val[r];
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < IPT; ++r) {
            const int i = at0 + 32 * r;
            if (i < n) {
                key[r] = s_key[i];
                val[r] = s_val[i];
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) reinterpret_cast<uint32_t*>(cnt[warp])[lane + 32 * j] = 0u;
        __syncwarp();
    }
    // sorted keys and records, and the last cell head at or before each query
    const uint32_t bin0 = (uint32_t)(Ed.bin_off << gp.key_sub);
    int start[IPT], carry = -1;
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const int i = at0 + 32 * r;
        bool head = false;
        if (i < n) {
            const long long q = Ed.q_off + i;
            slots[q] = qrec[Ed.q_off + val[r]];
            qkey[q] = key[r] == NO_KEY ? NO_KEY : bin0 + key[r];
            head = i == 0 || (s_key[i - 1] >> gp.key_sub) != (key[r] >> gp.key_sub);
        }
        const unsigned all = __ballot_sync(FULL, head);
        const unsigned hm = all & (lt | (1u << lane));
        start[r] = hm ? at0 - lane + 32 * r + 31 - __clz(hm) : carry;
        if (all) carry = at0 - lane + 32 * r + 31 - __clz(all);
    }
    if (lane == 0) s_first[warp] = carry;
    __syncthreads();
    for (int w = warp - 1, open = 1; w >= 0 && open; --w) {
        const int f = s_first[w];
        if (f >= 0) {
#pragma unroll
            for (int r = 0; r < IPT; ++r)
                if (start[r] < 0) start[r] = f;
            open = 0;
        }
    }
    // units: every uq queries of a cell
    int at[IPT], n_s[IPT], count = 0;            // place in the warp's records; queries << 2 | log2 of the parts
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const int i = at0 + 32 * r;
        const bool st = i < n && key[r] != NO_KEY && ((unsigned)(i - start[r]) % (unsigned)uq) == 0u;
        int s = 0;
        n_s[r] = 0;
        if (st) {
            const uint32_t c = key[r] >> gp.key_sub;
            auto same = [&](int k) { return k < n && (s_key[k] >> gp.key_sub) == c; };
            int m = 1;                               // queries of the cell from here on, uq at most
            while (m < uq && same(i + m)) m *= 2;
            int lo = m / 2 + 1, hi = m < uq ? m : uq;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (same(i + mid)) lo = mid + 1; else hi = mid;
            }
            s = cut_shift(cut_edge, Fa, n, cell_start, (int)c, lo);
            n_s[r] = lo << 2 | s;
        }
        int total;
        at[r] = count + unit_places(st, s, lane, total);
        count += total;
    }
    if (lane == 0) s_sum[warp] = count;
    __syncthreads();
    if (warp == 0) {
        const int c = s_sum[lane];
        int inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += u;
        }
        s_sum[lane] = inc - c;
        if (lane == 31) s_base = inc ? atomicAdd(n_units, inc) : 0;
    }
    __syncthreads();
    const int to = s_base + s_sum[warp];
#pragma unroll
    for (int r = 0; r < IPT; ++r)
        if (n_s[r])
            for (int part = 0; part < 1 << (n_s[r] & 3); ++part)
                units[to + at[r] + part] = unit_record((int)(Ed.q_off + at0 + 32 * r), e, n_s[r] >> 2, n_s[r] & 3, part);
}

// round(v * scale) to the nearest integer (ties to even) as int64, for
// |v * scale| < 2^62, with FP32 adds and integer operations only.  Below 2^22
// adding 2^23 leaves the rounded magnitude in the mantissa bits; from 2^22 up
// the value is m * 2^(e - 150) with a 24-bit mantissa m.
__device__ __forceinline__ long long to_fixed(float v, float scale) {
    const float x = v * scale;
    const int b = __float_as_int(x);
    const int ex = (b >> 23) & 0xff;
    long long mag;
    if (ex < 149) {
        const float t = fabsf(x) + 8388608.0f;
        mag = __float_as_int(t) & 0x7fffff;
    } else {
        const long long m = (b & 0x7fffff) | 0x800000;
        mag = (ex == 149) ? ((m >> 1) + (m & (m >> 1) & 1)) : (m << (ex - 150));
    }
    return b < 0 ? -mag : mag;
}

// ---------------------------------------------------- paired FP32 ops ----
// Two FP32 lanes in one 64-bit register: fma/mul/add .f32x2 issue one
// instruction for two IEEE FP32 operations (each rounded as its scalar form).
typedef unsigned long long u64;
__device__ __forceinline__ u64 f2(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 f2_split(u64 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ u64 ffma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 fmul2(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 fadd2(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

template <int DP, bool BF16>
struct Sem;

template <int DP>
struct Sem<DP, false> {   // FP32 label row of DP floats, as DP/2 pairs
    u64 q2[DP > 0 ? DP / 2 : 1];
    __device__ __forceinline__ void load(const void* base, int s, bool valid) {
        const ulonglong2* row = reinterpret_cast<const ulonglong2*>(base) + (size_t)s * (DP / 4);
#pragma unroll
        for (int k = 0; k < DP / 4; ++k) {
            const ulonglong2 v = valid ? __ldg(row + k) : make_ulonglong2(0ull, 0ull);
            q2[2 * k] = v.x;
            q2[2 * k + 1] = v.y;
        }
    }
};

__device__ __forceinline__ float bf_lo(unsigned u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(unsigned u) { return __uint_as_float(u & 0xffff0000u); }
__device__ __forceinline__ u64 bf_pair(unsigned u) { return f2(bf_lo(u), bf_hi(u)); }

template <int DP>
struct Sem<DP, true> {    // BF16 label row of DP values (DP % 8 == 0), widened to FP32 pairs
    u64 q2[DP / 2];
    __device__ __forceinline__ void load(const void* base, int s, bool valid) {
        const uint4* row = reinterpret_cast<const uint4*>(base) + (size_t)s * (DP / 8);
#pragma unroll
        for (int k = 0; k < DP / 8; ++k) {
            const uint4 v = valid ? __ldg(row + k) : make_uint4(0u, 0u, 0u, 0u);
            q2[4 * k + 0] = bf_pair(v.x);
            q2[4 * k + 1] = bf_pair(v.y);
            q2[4 * k + 2] = bf_pair(v.z);
            q2[4 * k + 3] = bf_pair(v.w);
        }
    }
};

// Label rows staged in shared memory (FP32 or BF16 rows) and their dot
// product with a row held in registers: even and odd terms summed in the
// two halves of a pair, then added.
template <int DP, bool BF16>
struct SemRow;
template <int DP>
struct SemRow<DP, false> {
    static constexpr int WORDS = DP;          // 32-bit words per row
    __device__ __forceinline__ static void stage(float* dst, const void* base, int i) {
        const float4* src = reinterpret_cast<const float4*>(base) + (size_t)i * (DP / 4);
        float4* d = reinterpret_cast<float4*>(dst);
#pragma unroll
        for (int k = 0; k < DP / 4; ++k) d[k] = __ldg(src + k);
    }
    __device__ __forceinline__ static float dot(const Sem<DP, false>& q, const float* row) {
        const ulonglong2* r = reinterpret_cast<const ulonglong2*>(row);
        u64 acc = 0ull;
#pragma unroll
        for (int k = 0; k < DP / 4; ++k) {
            const ulonglong2 v = r[k];
            acc = ffma2(q.q2[2 * k], v.x, acc);
            acc = ffma2(q.q2[2 * k + 1], v.y, acc);
        }
        const float2 s = f2_split(acc);
        return s.x + s.y;
    }
};
template <int DP>
struct SemRow<DP, true> {
    static constexpr int WORDS = DP / 2;
    __device__ __forceinline__ static void stage(float* dst, const void* base, int i) {
        const uint4* src = reinterpret_cast<const uint4*>(base) + (size_t)i * (DP / 8);
        uint4* d = reinterpret_cast<uint4*>(dst);
#pragma unroll
        for (int k = 0; k < DP / 8; ++k) d[k] = __ldg(src + k);
    }
    __device__ __forceinline__ static float dot(const Sem<DP, true>& q, const float* row) {
        const uint4* r = reinterpret_cast<const uint4*>(row);
        u64 acc = 0ull;
#pragma unroll
        for (int k = 0; k < DP / 8; ++k) {
            const uint4 v = r[k];
            acc = ffma2(q.q2[4 * k + 0], bf_pair(v.x), acc);
            acc = ffma2(q.q2[4 * k + 1], bf_pair(v.y), acc);
            acc = ffma2(q.q2[4 * k + 2], bf_pair(v.z), acc);
            acc = ffma2(q.q2[4 * k + 3], bf_pair(v.w), acc);
        }
        const float2 s = f2_split(acc);
        return s.x + s.y;
    }
};
template <>
struct SemRow<0, false> {
    static constexpr int WORDS = 0;
    __device__ __forceinline__ static void stage(float*, const void*, int) {}
    __device__ __forceinline__ static float dot(const Sem<0, false>&, const float*) { return 1.f; }
};


constexpr int PAIR_T = 256;
constexpr int UQ = UNIT_Q;
static_assert(UQ == 32, "a lane for every query of a unit");

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

constexpr int ROWS_WORDS = 9 * 4 + 9 * 2 + 2;   // segment list of the candidate stream (Rows)
constexpr int CQ_N = 64;            // ring of candidates that survived the unit's box test

// The candidate stream of a unit: the points of the 3x3x3 cells around its
// home cell are nine contiguous ranges (rows of three x-adjacent cells).  Cells
// farther than the cutoff from the bounding box of the unit's queries are left
// out, and rows without points skipped; what is left is a list of segments.
struct Rows {
    int4* seg;     // [<= 9] first and end point, first point of the home-x cell, of the x+1 cell
    float2* off;   // [<= 9] y and z offset of the row's cells from the home cell
};

// Fills the segment list (lanes 0..8 take a row each); returns the number of
// points on it and, in n_seg, of segments.  thr: squared cutoff with a margin,
// so that no cell holding a candidate that passes the box test is left out.
__device__ __forceinline__ int build_rows(const Rows& R, const int* __restrict__ cell_start, const FrameDev& F,
                                          int hx, int hy, int hz, float blo0, float blo1, float blo2, float bhi0,
                                          float bhi1, float bhi2, float hf, float thr, int lane, int& n_seg) {
    int len = 0;
    int4 sg = make_int4(0, 0, 0, 0);
    const int dy = (lane % 3) - 1, dz = (lane / 3) - 1;
    const float oy = (float)dy * hf, oz = (float)dz * hf;
    if (lane < 9) {
        const int ny = hy + dy, nz = hz + dz;
        const float hw = 0.50001f * hf;      // half a cell, with a margin for the rounding of the offsets
        const float ey = fmaxf(fmaxf(blo1 - (oy + hw), (oy - hw) - bhi1), 0.f);
        const float ez = fmaxf(fmaxf(blo2 - (oz + hw), (oz - hw) - bhi2), 0.f);
        const float left = 1.0001f * thr - fmaf(ey, ey, ez * ez);     // what the x distance may use
        if (ny >= 0 && ny < F.dim[1] && nz >= 0 && nz < F.dim[2] && left > 0.f) {
            const float el = fmaxf(blo0 + hf - hw, 0.f), er = fmaxf(hf - hw - bhi0, 0.f);
            const int xlo = max(hx - (el * el < left ? 1 : 0), 0), xhi = min(hx + (er * er < left ? 1 : 0), F.dim[0] - 1);
            const int* c = cell_start + F.cell_off + ((long long)nz * F.dim[1] + ny) * F.dim[0];
            sg.x = c[xlo];
            sg.y = c[xhi + 1];
            sg.z = c[hx];
            sg.w = c[hx + 1];
            len = sg.y - sg.x;
        }
    }
    const unsigned m = __ballot_sync(FULL, len > 0);
    if (len > 0) {
        const int at = __popc(m & ((1u << lane) - 1u));
        R.seg[at] = sg;
        R.off[at] = make_float2(oy, oz);
    }
    n_seg = __popc(m);
    const int total = __reduce_add_sync(FULL, len);
    __syncwarp();
    return total;
}

// A lane's place in the stream: it starts at a point of the list and steps 32 points at a time, crossing into the next segment when it must.
struct Cursor {
    int i, end, r, b1, b2;
    float oy, oz;
    __device__ __forceinline__ void enter(const Rows& R, int seg, int skip) {
        const int4 sg = R.seg[seg];
        const float2 o = R.off[seg];
        r = seg;
        i = sg.x + skip;
        end = sg.y;
        b1 = sg.z;
        b2 = sg.w;
        oy = o.x;
        oz = o.y;
    }
    __device__ __forceinline__ void settle(const Rows& R, int n_seg) {
        while (i >= end && r + 1 < n_seg) enter(R, r + 1, i - end);
    }
    __device__ __forceinline__ void start(const Rows& R, int n_seg, int at) {
        enter(R, 0, at);
        settle(R, n_seg);
    }
    __device__ __forceinline__ void next(const Rows& R, int n_seg) {
        i += 32;
        settle(R, n_seg);
    }
    __device__ __forceinline__ bool valid() const { return i < end; }
    // point i relative to the home cell's centre, with its index
    __device__ __forceinline__ float4 point(const float4* __restrict__ pts4, float hf) const {
        const float4 p = __ldg(pts4 + i);
        return make_float4(p.x + (i >= b2 ? hf : (i >= b1 ? 0.f : -hf)), p.y + oy, p.z + oz, __int_as_float(i));
    }
};

// Chunks [c0, c1) of 32 stream points that part `part` of 2^shift takes: an
// even share, but four at least (short streams stay whole, and their other
// parts are empty).
__device__ __forceinline__ void part_range(int C, int part, int shift, int& c0, int& c1) {
    const int n = (int)(((long long)C + 31) >> 5);
    const int per = max((n + (1 << shift) - 1) >> shift, 4);
    c0 = min(part * per, n);
    c1 = min(c0 + per, n);
}

// a + b with its rounding error (Knuth), two at a time: s = fl(a + b), s + e = a + b.
// Differences are multiplications by -1 (exact), which need no negated copies.
__device__ __forceinline__ u64 two_sum2(u64 a, u64 b, u64& e) {
    const u64 M1 = f2(-1.f, -1.f);
    const u64 s = fadd2(a, b);
    const u64 bb = ffma2(a, M1, s);
    e = fadd2(ffma2(ffma2(bb, M1, s), M1, a), ffma2(bb, M1, b));
    return s;
}

// One step of the moment reduce-scatter over pairs of moments hi + lo: lanes whose
// bit 2 N is clear keep the lower N pairs, the others the upper N, and each adds the half
// its partner sends.  FIRST: lo is zero on entry.
template <int N, bool FIRST>
__device__ __forceinline__ void reduce_half(u64 (&hi)[16], u64 (&lo)[16], int lane) {
    const bool up = (lane & (2 * N)) != 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const u64 keep = up ? hi[k + N] : hi[k], send = up ? hi[k] : hi[k + N];
        u64 e;
        hi[k] = two_sum2(keep, __shfl_xor_sync(FULL, send, 2 * N), e);
        if constexpr (FIRST) {
            lo[k] = e;
        } else {
            const u64 keep_l = up ? lo[k + N] : lo[k], send_l = up ? lo[k] : lo[k + N];
            lo[k] = fadd2(fadd2(keep_l, __shfl_xor_sync(FULL, send_l, 2 * N)), e);
        }
    }
}

// Unit end, shared by the pair kernels: the lanes' moments about the home cell
// centre are reduce-scattered over the warp (lane k ends with moment k), move to
// frame-a coordinates (y' += o), are rounded to 64-bit fixed point and added to the
// edge's accumulators with one integer atomic per moment.  The sums over lanes keep every
// addition's rounding error, and what a moment is made of is rounded to fixed point
// part by part, so nothing the lanes hold is lost to FP32 on the way (the lanes'
// moments cancel near convergence).  What enters the accumulators depends on the unit
// alone, and their sums are exact.
// Against plain FP32 sums (31 additions a lane and one rounded shift) this takes 6 us
// more of a 195 us evaluation of 5 x 20k RGB-D points (units of 5 queries), nothing that shows on
// LiDAR scans; two frames near convergence, 1500 points without labels: gradient off by
// 8.0e-7 with plain sums, 5.4e-7 with these (1500 points, eight neighbours: 2.8e-7, 2.4e-7).
// Rounding every lane's moments to 64 bits before the reduction takes ~1000 instructions a
// unit, four times as many.
__device__ __forceinline__ void store_moments(float W, const float (&Dv)[3], const float (&Sy)[3], const float (&Myy)[6],
                                              const float (&Mdy)[9], const float* Qm, int cnt, const FrameDev& Fa,
                                              int hx, int hy, int hz, const GridParams& gp,
                                              const float* __restrict__ scl, long long* __restrict__ acc_e,
                                              int lane) {
    u64 hi[16], lo[16];
    auto at = [&](int k) {
        return k == 0 ? W : k < 4 ? Dv[k - 1] : k < 7 ? Sy[k - 4] : k < 13 ? Myy[k - 7] : k < 22 ? Mdy[k - 13]
             : k < 28 ? Qm[k - 22] : 0.f;
    };
#pragma unroll
    for (int k = 0; k < 16; ++k) hi[k] = f2(at(2 * k), at(2 * k + 1));
    reduce_half<8, true>(hi, lo, lane);
    reduce_half<4, false>(hi, lo, lane);
    reduce_half<2, false>(hi, lo, lane);
    reduce_half<1, false>(hi, lo, lane);
    // a pair per two lanes is left: the even lane keeps its first, the odd one its second
    float x, xl;
    {
        const float2 h = f2_split(hi[0]), l = f2_split(lo[0]);
        const bool odd = lane & 1;
        const float keep = odd ? h.y : h.x, got = __shfl_xor_sync(FULL, odd ? h.x : h.y, 1);
        const float got_l = __shfl_xor_sync(FULL, odd ? l.x : l.y, 1);
        x = keep + got;
        const float bb = x - keep;
        xl = (odd ? l.y : l.x) + got_l + ((keep - (x - bb)) + (got - bb));
    }
    cnt = __reduce_add_sync(FULL, cnt);
    // rows m and columns l of the lane's moment: Sy (m), Myy and Mdy (m, l)
    const bool in_sy = lane >= 4 && lane < 7, in_yy = lane >= 7 && lane < 13, in_dy = lane >= 13 && lane < 22;
    const int q = lane - 13;
    const int m = in_sy ? lane - 4 : in_yy ? (lane < 10 ? 0 : (lane < 12 ? 1 : 2)) : in_dy ? q / 3 : 0;
    const int l = in_yy ? (lane < 10 ? lane - 7 : (lane < 12 ? lane - 9 : 2)) : in_dy ? q - 3 * m : 0;
    const float o0 = ((float)(hx + Fa.lo[0]) + 0.5f) * gp.hf, o1 = ((float)(hy + Fa.lo[1]) + 0.5f) * gp.hf,
                o2 = ((float)(hz + Fa.lo[2]) + 0.5f) * gp.hf;
    const float om = m == 0 ? o0 : (m == 1 ? o1 : o2), ol = l == 0 ? o0 : (l == 1 ? o1 : o2);
    // sum w y' += W o;  sum w y'y'^T += Sy o^T + o Sy^T + W o o^T;  sum w d y'^T += D o^T:
    // terms p1 + p2 + p3 of factors that are sums over the warp, and what their products round off
    const int src1 = in_sy ? 0 : in_yy ? 4 + m : 1 + m;
    const float w = __shfl_sync(FULL, x, 0), wl = __shfl_sync(FULL, xl, 0);
    float f1 = __shfl_sync(FULL, x, src1), f1l = __shfl_sync(FULL, xl, src1);
    float f2_ = __shfl_sync(FULL, x, 4 + l), f2l = __shfl_sync(FULL, xl, 4 + l);
    const float g1 = in_sy ? om : ol;
    if (!(in_sy || in_yy || in_dy)) f1 = f1l = 0.f;
    if (!in_yy) f2_ = f2l = 0.f;
    const float w3 = in_yy ? w : 0.f, oo = om * ol, ool = fmaf(om, ol, -oo);
    const float p1 = f1 * g1, p2 = f2_ * om, p3 = w3 * oo;
    const float rest = xl + (fmaf(f1, g1, -p1) + fmaf(f1l, g1, fmaf(f2_, om, -p2) + fmaf(f2l, om, fmaf(w3, oo, -p3)))) +
                       (in_yy ? fmaf(w3, ool, wl * oo) : 0.f);
    long long f = (long long)cnt;
    if (lane < N_MOM - 1) {
        const float sc = __ldg(scl + moment_class(lane));
        f = to_fixed(x, sc) + to_fixed(rest, sc);
        if (lane >= 4 && lane < 22) f += to_fixed(p1, sc) + to_fixed(p2, sc) + to_fixed(p3, sc);
    }
    if (lane < N_MOM && f != 0) atomicAdd(reinterpret_cast<unsigned long long*>(acc_e + lane), (unsigned long long)f);
}

// ------------------------------------------------------ dense tile path ----
// Labels without colour or pruning.  On the LiDAR workloads half to two
// thirds of a batch's candidate x query tests pass the cutoff after the box
// cull, so instead of taking pairs one by one the warp evaluates the
// whole tile in MMA fragment layout and moves the moment sums onto the tensor
// cores:
//   1. S = L_q L_c^T, the tile's label products (rows are the unit's queries
//      in m tiles of 16, columns the batch's 32 candidates): BF16 labels as
//      stored; FP32 labels scaled by a power of two and split into FP16
//      hi + lo parts, S = hi*hi + hi*lo + lo*hi;
//   2. per element: the exact cutoff test of the lane kernel (same FP32
//      formula, so the same pair set), w = s 2^(kg |d|^2) (one ex2), and 0
//      outside r_c; |d|^2 = |y|^2 - 2 x.y + |x|^2;
//   3. the weights, now an A operand in registers (the accumulator layout of
//      step 1 is the A-fragment layout of the next MMA), split into FP16
//      hi + lo, times the candidate features f(x) = (1, x, x x^T), also
//      split: per query q the sums k_q = sum_c w, X1_q = sum_c w x_c and
//      X2_q = sum_c w x_c x_c^T accumulate over the unit's batches
//      (hi*hi + hi*lo + lo*hi: products of 22-bit operands, FP32 sums,
//      added into FP32 running sums once per batch);
//   4. at the unit's end each lane takes one query and forms, with y = y_q,
//      W = k, D = X1 - k y, sum w y = k y, sum w y y^T = k y y^T,
//      sum w d y^T = D y^T and Q = X2 - X1 y^T - y X1^T + k y y^T, which
//      enter the same reduction as those of the lane kernel.
// Scaling: w is carried as w 2^KW with 2^KW |l|max^2 <= 2^14 and the
// features as x 2^-EX with 2^EX >= h, so every FP16 operand stays inside
// its range; both are powers of two and undone exactly at the unit's end.

// ldmatrix: four / two / one 8x8 b16 matrices from shared memory; lanes
// 8m..8m+7 give the row addresses of matrix m.
__device__ __forceinline__ void ldsm_x4(unsigned (&r)[4], const void* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldsm_x4_t(unsigned (&r)[4], const void* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldsm_x2_t(unsigned (&r)[2], const void* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}
__device__ __forceinline__ void ldsm_x2(unsigned& r0, unsigned& r1, const void* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(a));
}
__device__ __forceinline__ void ldsm_x1(unsigned& r0, const void* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x1.shared.b16 {%0}, [%1];" : "=r"(r0) : "r"(a));
}

__device__ __forceinline__ void mma_bf16_1688(float (&d)[4], unsigned a0, unsigned a1, unsigned b0) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ void mma_bf16_16816_r(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                                 unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16_16816(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// The first MMA of a sum: d = A B with the addend a zero operand of its own,
// so no accumulator registers are cleared beforehand.
__device__ __forceinline__ void mma_f16_16816_first(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// (lo, hi) rounded to FP16 (nearest even), lo in the low half
__device__ __forceinline__ unsigned f16x2_rn(float lo, float hi) {
    unsigned r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// v0 ~ hi.lo + lo.lo, v1 ~ hi.hi + lo.hi: two FP16 pieces per value (22 bits).
// The remainders v - hi are one mixed FP16 x FP16 + FP32 FMA each (exact: hi
// holds the leading bits of v), without widening hi first.
__device__ __forceinline__ void split_f16x2(float v0, float v1, unsigned& hi, unsigned& lo) {
    hi = f16x2_rn(v0, v1);
    float r0, r1;
    asm("{\n\t.reg .f16 l, h, m;\n\tmov.b32 {l, h}, %2;\n\tmov.b16 m, 0xBC00;\n\t"
        "fma.rn.f32.f16 %0, l, m, %3;\n\tfma.rn.f32.f16 %1, h, m, %4;\n\t}"
        : "=f"(r0), "=f"(r1) : "r"(hi), "f"(v0), "f"(v1));
    lo = f16x2_rn(r0, r1);
}

// w when t < thr (the pair is inside r_c), counted in cnt; else 0.  Selected, not
// multiplied by a mask of 0 and 1: outside r_c the label product may be infinite
// or NaN (labels beyond FP16's or BF16's range, on points that pair with nothing).  The
// mask's product took longer, too (64 x 100k mapping evaluation 64.1 against 62.4 ms).
__device__ __forceinline__ float inside_count(float t, float thr, float w, int& cnt) {
    float r;
    asm("{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %2, %3;\n\tselp.f32 %0, %4, 0f00000000, p;\n\t@p add.s32 %1, %1, 1;\n\t}"
        : "=f"(r), "+r"(cnt) : "f"(t), "f"(thr), "f"(w));
    return r;
}

// Per-warp shared memory of the dense path, in 32-bit words: the batch's
// candidates only (the unit's queries live in registers).  Label rows: BF16
// rows as stored (DP values); FP32 rows (SPLIT) as an FP16 hi part and an FP16
// lo part of DPH values each (DP rounded up to 8), scaled by a power of two.
template <int DP, bool SPLIT>
struct DenseSmem {
    static constexpr int DPH = SPLIT ? ((DP + 7) / 8) * 8 : DP;    // values per part
    static constexpr int PW = DPH / 2;                            // words per part
    static constexpr int RW = SPLIT ? 2 * PW : PW;                // words per staged row
    static constexpr int LW = (RW % 8 == 0) ? RW + 4 : RW;        // row stride: 4 x odd, conflict-free ldmatrix
    static constexpr int CL = 0;                                  // [32][LW] candidate label rows (first the
                                                                  //   unit's query rows, on their way to registers)
    static constexpr int CG = CL + 32 * LW;                       // [16][12] candidate pairs (2p, 2p+1):
                                                                  //   x0 x0' x1 x1' | x2 x2' thr thr' | xk xk' - -
    static constexpr int CF = CG + 16 * 12;                       // [32][12] features in FP16: hi of features 0..7,
                                                                  //   tile 1 (hi 8, hi 9, lo 8, lo 9, zeros), lo of
                                                                  //   features 0..7 (a 48-byte row: conflict-free
                                                                  //   ldmatrix)
    static constexpr int RING = CF + 32 * 12;                     // [CQ_N] float4 candidate ring
    static constexpr int ROWS = RING + 4 * CQ_N;                  // the stream's segments
    static constexpr int OLD = ROWS + ROWS_WORDS;                 // [4][32] float4: the lanes' sums over earlier pieces
    static constexpr int WORDS = OLD + 4 * 32 * 4;
};

// Power-of-two scales of the dense path's FP16 operands, from the frames'
// label-norm bounds and the cell size (see "Scaling" above): the weights carry
// 2^kw, the features 2^-ex, FP32 labels 2^-el.
struct DenseScales {
    int kw, ex, el;
};
__device__ __forceinline__ DenseScales dense_scales(float norm_a, float norm_b, float hf, bool split) {
    DenseScales d;
    int ew;
    frexpf(norm_a * norm_b, &ew);
    frexpf(hf, &d.ex);
    d.kw = min(max(14 - ew, -100), 100);
    d.el = 0;
    if (split) {
        frexpf(fmaxf(norm_a, norm_b), &d.el);
        d.el = min(max(d.el, -60), 60);
    }
    return d;
}

// Stage one label row into shared memory: BF16 rows copied; FP32 rows scaled
// by ls and split into FP16 hi and lo parts (zeros beyond DP); a zero row when
// !valid.
template <int DP, bool SPLIT>
__device__ __forceinline__ void stage_label_row(unsigned* row, const void* base, int i, float ls, bool valid) {
    using L = DenseSmem<DP, SPLIT>;
    uint4* dst = reinterpret_cast<uint4*>(row);
    if constexpr (!SPLIT) {
        const uint4* src = reinterpret_cast<const uint4*>(base) + (size_t)i * (L::PW / 4);
#pragma unroll
        for (int k = 0; k < L::PW / 4; ++k) dst[k] = valid ? __ldg(src + k) : make_uint4(0u, 0u, 0u, 0u);
    } else {
        float v[L::DPH];
        const float4* src = reinterpret_cast<const float4*>(base) + (size_t)i * (DP / 4);
#pragma unroll
        for (int k = 0; k < DP / 4; ++k) {
            const float4 t = valid ? __ldg(src + k) : make_float4(0.f, 0.f, 0.f, 0.f);
            v[4 * k] = t.x * ls;
            v[4 * k + 1] = t.y * ls;
            v[4 * k + 2] = t.z * ls;
            v[4 * k + 3] = t.w * ls;
        }
#pragma unroll
        for (int k = DP; k < L::DPH; ++k) v[k] = 0.f;
        unsigned hw[L::PW], lw[L::PW];
#pragma unroll
        for (int j = 0; j < L::PW; ++j) split_f16x2(v[2 * j], v[2 * j + 1], hw[j], lw[j]);
#pragma unroll
        for (int k = 0; k < L::PW / 4; ++k) {
            dst[k] = make_uint4(hw[4 * k], hw[4 * k + 1], hw[4 * k + 2], hw[4 * k + 3]);
            dst[L::PW / 4 + k] = make_uint4(lw[4 * k], lw[4 * k + 1], lw[4 * k + 2], lw[4 * k + 3]);
        }
    }
}

// The 8-wide chunks [0, NKC) of one part of the staged rows as MMA fragments:
// query side (A, rows 16 mt .. + 15; two registers per chunk) and candidate
// side (B, candidates 8 nt .. + 7; one register per chunk).
template <int NKC>
__device__ __forceinline__ void load_a_chunks(unsigned (&qa)[2 * NKC], const unsigned* rowp) {
    // rowp: this lane's row (16 mt + (lane & 7) + 8 ((lane >> 3) & 1)) at the part's first word
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int kc = 0; kc + 1 < NKC; kc += 2) {
        unsigned r[4];
        ldsm_x4(r, rowp + 4 * (kc + (lane >> 4)));
        qa[2 * kc] = r[0];
        qa[2 * kc + 1] = r[1];
        qa[2 * kc + 2] = r[2];
        qa[2 * kc + 3] = r[3];
    }
    if constexpr (NKC & 1) ldsm_x2(qa[2 * (NKC - 1)], qa[2 * (NKC - 1) + 1], rowp + 4 * (NKC - 1));
}
template <int NKC>
__device__ __forceinline__ void load_b_chunks(unsigned (&cb)[NKC], const unsigned* rowp) {
    // rowp: row of candidate 8 nt + (lane & 7) at the part's first word
    const int lane = threadIdx.x & 31;
    if constexpr (NKC == 4) {
        unsigned r[4];
        ldsm_x4(r, rowp + 4 * (lane >> 3));
#pragma unroll
        for (int k = 0; k < 4; ++k) cb[k] = r[k];
    } else if constexpr (NKC == 3) {
        ldsm_x2(cb[0], cb[1], rowp + 4 * ((lane >> 3) & 1));
        ldsm_x1(cb[2], rowp + 8);
    } else if constexpr (NKC == 2) {
        ldsm_x2(cb[0], cb[1], rowp + 4 * ((lane >> 3) & 1));
    } else {
        ldsm_x1(cb[0], rowp);
    }
}

__device__ __forceinline__ void mma_f16_1688(float (&d)[4], unsigned a0, unsigned a1, unsigned b0) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ void mma_f16_16816_r(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                                unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_bf16_16816_first(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                                     unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// s += A B over NKC chunks: BF16 (F16 false) or FP16 operands; FIRST: s = A B.
template <int NKC, bool F16, bool FIRST>
__device__ __forceinline__ void gram_chunks(float (&s)[4], const unsigned (&qa)[2 * NKC], const unsigned (&cb)[NKC]) {
    if constexpr (FIRST && NKC == 1) s[0] = s[1] = s[2] = s[3] = 0.f;
#pragma unroll
    for (int kc = 0; kc + 1 < NKC; kc += 2) {
        if (FIRST && kc == 0) {
            const unsigned a[4] = {qa[0], qa[1], qa[2], qa[3]};
            if constexpr (F16) mma_f16_16816_first(s, a, cb[0], cb[1]);
            else mma_bf16_16816_first(s, a[0], a[1], a[2], a[3], cb[0], cb[1]);
        } else if constexpr (F16) mma_f16_16816_r(s, qa[2 * kc], qa[2 * kc + 1], qa[2 * kc + 2], qa[2 * kc + 3], cb[kc], cb[kc + 1]);
        else mma_bf16_16816_r(s, qa[2 * kc], qa[2 * kc + 1], qa[2 * kc + 2], qa[2 * kc + 3], cb[kc], cb[kc + 1]);
    }
    if constexpr (NKC & 1) {
        if constexpr (F16) mma_f16_1688(s, qa[2 * (NKC - 1)], qa[2 * (NKC - 1) + 1], cb[NKC - 1]);
        else mma_bf16_1688(s, qa[2 * (NKC - 1)], qa[2 * (NKC - 1) + 1], cb[NKC - 1]);
    }
}

// One unit of the dense path: <= 32 queries of one frame-a home cell, MT m
// tiles of 16.  The queries live in registers for the whole unit (geometry as
// FP32 pairs, label rows as A fragments, running sums as accumulators), so
// that a batch reads each candidate's geometry, label row and features from
// shared memory once for all its queries: at one 16-query tile per read the
// shared-memory pipe was the kernel's bound (82% busy on the mapping workload,
// 98 wavefronts per 16 x 32 tile; 32 here).
template <int DP, bool SPLIT, bool PARTS>
__device__ __forceinline__ void pair_unit_dense(const PairArgs& A, int2 unit, float* wb, int lane) {
    using L = DenseSmem<DP, SPLIT>;
    constexpr int LW = L::LW, PW = L::PW;
    constexpr int NKC = L::DPH / 8;             // 8-wide chunks of a label row part (1..4)
    const GridParams& gp = A.gp;
    unsigned* cl = reinterpret_cast<unsigned*>(wb + L::CL);
    float* cg = wb + L::CG;
    unsigned* cf = reinterpret_cast<unsigned*>(wb + L::CF);
    float4* cq = reinterpret_cast<float4*>(wb + L::RING);
    const Rows R{reinterpret_cast<int4*>(wb + L::ROWS), reinterpret_cast<float2*>(wb + L::ROWS + 36)};
    const int g = lane >> 2, t4 = lane & 3;
    const float INF = __int_as_float(0x7f800000);

    const int k0 = unit.x, qcount = unit_queries(unit), e = unit_edge(unit);
    const uint32_t key0 = A.qkey[k0] >> gp.key_sub;
    const FrameDev& Fa = A.frames[A.edges[e].a];
    const FrameDev& Fb = A.frames[A.edges[e].b];
    const int cell = (int)(key0 - A.edges[e].bin_off);
    const int hx = cell % Fa.dim[0], hy = (cell / Fa.dim[0]) % Fa.dim[1], hz = cell / (Fa.dim[0] * Fa.dim[1]);
    const DenseScales sc = dense_scales(Fa.sem_norm_max, Fb.sem_norm_max, gp.hf, SPLIT);
    // FP32 labels enter the FP16 parts scaled by ls = 2^-el (|l| ls < 1), so
    // the products carry 2^-2el, which the exponent offset undoes
    const float ls = ldexpf(1.f, -sc.el);
    const float kwf = (float)(sc.kw + 2 * sc.el);
    const float xs = ldexpf(1.f, -sc.ex);
    // this lane's queries, rows g + 8 i: -2 y and |y|^2 doubled into pairs
    // (absent ones: |y|^2 = inf fails every test), and the unit's bounding box
    u64 qm[4][4];
    float blo0 = INF, blo1 = INF, blo2 = INF, bhi0 = -INF, bhi1 = -INF, bhi2 = -INF;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float mx = 0.f, my = 0.f, mz = 0.f, yy = INF;
        if (g + 8 * i < qcount) {
            const float4 r = A.slots[(long long)k0 + g + 8 * i];
            blo0 = fminf(blo0, r.x);
            bhi0 = fmaxf(bhi0, r.x);
            blo1 = fminf(blo1, r.y);
            bhi1 = fmaxf(bhi1, r.y);
            blo2 = fminf(blo2, r.z);
            bhi2 = fmaxf(bhi2, r.z);
            mx = -2.f * r.x;
            my = -2.f * r.y;
            mz = -2.f * r.z;
            yy = fmaf(r.x, r.x, fmaf(r.y, r.y, r.z * r.z));
        }
        qm[i][0] = f2(mx, mx);
        qm[i][1] = f2(my, my);
        qm[i][2] = f2(mz, mz);
        qm[i][3] = f2(yy, yy);
    }
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) {
        blo0 = fminf(blo0, __shfl_xor_sync(FULL, blo0, o));
        blo1 = fminf(blo1, __shfl_xor_sync(FULL, blo1, o));
        blo2 = fminf(blo2, __shfl_xor_sync(FULL, blo2, o));
        bhi0 = fmaxf(bhi0, __shfl_xor_sync(FULL, bhi0, o));
        bhi1 = fmaxf(bhi1, __shfl_xor_sync(FULL, bhi1, o));
        bhi2 = fmaxf(bhi2, __shfl_xor_sync(FULL, bhi2, o));
    }
    __syncwarp();
    const float box_thr = gp.rc2 * 1.0001f;
    int n_seg;
    const int C = build_rows(R, A.cell_start, Fa, hx, hy, hz, blo0, blo1, blo2, bhi0, bhi1, bhi2, gp.hf, box_thr, lane,
                             n_seg);
    int c_lo = 0, c_hi = (int)(((long long)C + 31) >> 5);    // chunks of the stream
    if constexpr (PARTS) part_range(C, unit_part(unit), unit_shift(unit), c_lo, c_hi);
    // query label rows (zero rows for absent queries) as A fragments, through
    // the candidates' rows
    {
        const bool qv = lane < qcount;
        const int s = qv ? __float_as_int(A.slots[(long long)k0 + lane].w) : 0;
        stage_label_row<DP, SPLIT>(cl + lane * LW, A.sem_sorted, s, ls, qv);
    }
    __syncwarp();
    unsigned qa[2][2 * NKC], qal[SPLIT ? 2 : 1][SPLIT ? 2 * NKC : 1];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
        const unsigned* qrowp = cl + (16 * mt + (lane & 7) + 8 * ((lane >> 3) & 1)) * LW;
        load_a_chunks<NKC>(qa[mt], qrowp);
        if constexpr (SPLIT) load_a_chunks<NKC>(qal[mt], qrowp + PW);
    }
    __syncwarp();
    const u64 KG2 = f2(gp.kg, gp.kg);
    // running sums of the moment MMAs, in the accumulator layout: feature tile
    // 0, and tile 1 (features 8 and 9: hi parts in the lanes with t4 = 0, lo
    // parts in those with t4 = 1, zeros elsewhere)
    float run[2][2][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int n2 = 0; n2 < 2; ++n2)
#pragma unroll
            for (int k = 0; k < 4; ++k) run[mt][n2][k] = 0.f;
    int cnt = 0;
    // the batches, compiled for one and for two m tiles
    auto batches = [&](auto mtc, int c_s, int c_hi) {
        constexpr int MT = decltype(mtc)::value;
        int qhead = 0, qlen = 0;
        Cursor cur;
        cur.start(R, n_seg, 32 * c_s + lane);
        while (c_s < c_hi || qlen > 0) {
            while (qlen < 32 && c_s < c_hi) {
                bool keep = false;
                float4 ent = make_float4(0.f, 0.f, 0.f, 0.f);
                if (cur.valid()) {
                    ent = cur.point(A.pts4, gp.hf);
                    const float e0 = fmaxf(fmaxf(blo0 - ent.x, ent.x - bhi0), 0.f);
                    const float e1 = fmaxf(fmaxf(blo1 - ent.y, ent.y - bhi1), 0.f);
                    const float e2 = fmaxf(fmaxf(blo2 - ent.z, ent.z - bhi2), 0.f);
                    keep = fmaf(e0, e0, fmaf(e1, e1, e2 * e2)) < box_thr;
                }
                const unsigned bal = __ballot_sync(FULL, keep);
                if (keep) cq[(qhead + qlen + __popc(bal & ((1u << lane) - 1u))) & (CQ_N - 1)] = ent;
                qlen += __popc(bal);
                ++c_s;
                cur.next(R, n_seg);
            }
            __syncwarp();
            const int nb = qlen < 32 ? qlen : 32;
            if (nb == 0) break;
            // lane c stages candidate c of the batch (absent ones: zero rows,
            // zero features, thr = -inf)
            {
                const bool has = lane < nb;
                const float4 ent = has ? cq[(qhead + lane) & (CQ_N - 1)] : make_float4(0.f, 0.f, 0.f, 0.f);
                const int i = __float_as_int(ent.w);
                stage_label_row<DP, SPLIT>(cl + lane * LW, A.sem_sorted, i, ls, has);
                const float x0 = ent.x, x1 = ent.y, x2 = ent.z;
                const float xx = fmaf(x0, x0, fmaf(x1, x1, x2 * x2));
                float* cgp = cg + 12 * (lane >> 1) + (lane & 1);
                cgp[0] = x0;
                cgp[2] = x1;
                cgp[4] = x2;
                cgp[6] = has ? gp.rc2 - xx : -INF;
                cgp[8] = fmaf(xx, gp.kg, kwf);
                const float u0 = x0 * xs, u1 = x1 * xs, u2 = x2 * xs;
                unsigned h0, h1, h2, h3, h4, l0, l1, l2, l3, l4;
                split_f16x2(has ? 1.f : 0.f, u0, h0, l0);
                split_f16x2(u1, u2, h1, l1);
                split_f16x2(u0 * u0, u0 * u1, h2, l2);
                split_f16x2(u0 * u2, u1 * u1, h3, l3);
                split_f16x2(u1 * u2, u2 * u2, h4, l4);
                uint4* frow = reinterpret_cast<uint4*>(cf + 12 * lane);
                frow[0] = make_uint4(h0, h1, h2, h3);
                frow[1] = make_uint4(h4, l4, 0u, 0u);
                frow[2] = make_uint4(l0, l1, l2, l3);
            }
            qhead = (qhead + nb) & (CQ_N - 1);
            qlen -= nb;
            __syncwarp();
            // 16 candidates at a time (one k step of the moment MMAs), not
            // unrolled: the smaller loop body fetches faster
#pragma unroll 1
            for (int ks = 0; ks < 2; ++ks) {
                if (16 * ks >= nb) break;
                // label products, then the weights of this lane's rows and of
                // columns 8 nt + 2 t4, + 1, split into the FP16 A operands of
                // the moment MMAs
                unsigned ah[MT][4], al[MT][4];
#pragma unroll
                for (int n1 = 0; n1 < 2; ++n1) {
                    const int nt = 2 * ks + n1;
                    const unsigned* crowp = cl + (8 * nt + (lane & 7)) * LW;
                    unsigned cb[NKC];
                    [[maybe_unused]] unsigned cbl[NKC];
                    load_b_chunks<NKC>(cb, crowp);
                    if constexpr (SPLIT) load_b_chunks<NKC>(cbl, crowp + PW);
                    const int p = 4 * nt + t4;
                    const ulonglong2 c01 = *reinterpret_cast<const ulonglong2*>(cg + 12 * p);
                    const ulonglong2 c2t = *reinterpret_cast<const ulonglong2*>(cg + 12 * p + 4);
                    const u64 XK = *reinterpret_cast<const u64*>(cg + 12 * p + 8);
                    const float2 thr = f2_split(c2t.y);
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        float s[4];
                        if constexpr (SPLIT) {
                            // FP32 labels: hi*hi + hi*lo + lo*hi of the FP16 parts
                            gram_chunks<NKC, true, true>(s, qa[mt], cb);
                            gram_chunks<NKC, true, false>(s, qa[mt], cbl);
                            gram_chunks<NKC, true, false>(s, qal[mt], cb);
                        } else {
                            gram_chunks<NKC, false, true>(s, qa[mt], cb);
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const u64(&m)[4] = qm[2 * mt + i];
                            const u64 T = ffma2(c01.x, m[0], ffma2(c01.y, m[1], ffma2(c2t.x, m[2], m[3])));
                            const float2 t = f2_split(T);
                            const float2 a = f2_split(ffma2(T, KG2, XK));
                            const float2 w = f2_split(fmul2(f2(s[2 * i], s[2 * i + 1]), f2(ex2_approx(a.x), ex2_approx(a.y))));
                            split_f16x2(inside_count(t.x, thr.x, w.x, cnt), inside_count(t.y, thr.y, w.y, cnt),
                                        ah[mt][2 * n1 + i], al[mt][2 * n1 + i]);
                        }
                    }
                }
                // per query: sum over the 16 candidates of w (1, x, x x^T);
                // feature B fragments, FP16 hi and lo
                unsigned fh[4], fl[2];
                const unsigned* rowp = cf + 12 * (16 * ks + (lane & 7) + 8 * ((lane >> 3) & 1));
                ldsm_x4_t(fh, rowp + 4 * (lane >> 4));
                ldsm_x2_t(fl, rowp + 8);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    float t[2][4];
                    mma_f16_16816_first(t[0], ah[mt], fh[0], fh[1]);
                    mma_f16_16816_first(t[1], ah[mt], fh[2], fh[3]);
                    mma_f16_16816(t[1], al[mt], fh[2], fh[3]);
                    mma_f16_16816(t[0], ah[mt], fl[0], fl[1]);
                    mma_f16_16816(t[0], al[mt], fh[0], fh[1]);
#pragma unroll
                    for (int n2 = 0; n2 < 2; ++n2)
#pragma unroll
                        for (int k = 0; k < 4; k += 2) {
                            const float2 r = f2_split(fadd2(f2(run[mt][n2][k], run[mt][n2][k + 1]),
                                                            f2(t[n2][k], t[n2][k + 1])));
                            run[mt][n2][k] = r.x;
                            run[mt][n2][k + 1] = r.y;
                        }
                }
            }
        }
    };
    // Streams of more than PIECE chunks are taken in pieces of that length, whose sums are added up
    // in shared memory: no chain of FP32 additions is longer than 2 PIECE (and one per
    // piece).  Every piece ends with a batch that is not full (a batch in sixty), and the inner loop
    // stays as it was: sums folded inside it, every 8 or 32 batches, cost 3% of every case.
    constexpr int PIECE = 64;
    float4* older = reinterpret_cast<float4*>(wb + L::OLD) + lane;
    auto pieces = [&](auto mtc) {
        constexpr int MT = decltype(mtc)::value;
#pragma unroll 1
        for (int c0 = c_lo; c0 < c_hi; c0 += PIECE) {
            batches(mtc, c0, min(c0 + PIECE, c_hi));
            if (c_hi - c_lo <= PIECE) break;
            const bool first = c0 == c_lo, last = c0 + PIECE >= c_hi;
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int n2 = 0; n2 < 2; ++n2) {
                    float(&r)[4] = run[mt][n2];
                    float4& o = older[32 * (2 * mt + n2)];
                    float4 v = make_float4(r[0], r[1], r[2], r[3]);
                    if (!first) v = make_float4(o.x + v.x, o.y + v.y, o.z + v.z, o.w + v.w);
                    if (!last) {
                        o = v;
                        v = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    r[0] = v.x;
                    r[1] = v.y;
                    r[2] = v.z;
                    r[3] = v.w;
                }
        }
    };
    if (qcount > 16) pieces(std::integral_constant<int, 2>{});
    else pieces(std::integral_constant<int, 1>{});
    if (!__any_sync(FULL, cnt != 0)) return;     // no pair: every sum is zero
    // unit end: the per-query sums through shared memory (the features' place)
    // to one lane per query, formed into the lane's moments
    float* sq = reinterpret_cast<float*>(cf);    // [32][12] (features 0..9 used)
    __syncwarp();
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
        float (&r1)[4] = run[mt][1];
#pragma unroll
        for (int k = 0; k < 4; ++k) r1[k] += __shfl_xor_sync(FULL, r1[k], 1);    // hi and lo parts of features 8, 9
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float* row = sq + 12 * (16 * mt + 8 * i + g);
            *reinterpret_cast<float2*>(row + 2 * t4) = make_float2(run[mt][0][2 * i], run[mt][0][2 * i + 1]);
            if (t4 == 0) *reinterpret_cast<float2*>(row + 8) = make_float2(r1[2 * i], r1[2 * i + 1]);
        }
    }
    __syncwarp();
    const float4 r0 = *reinterpret_cast<const float4*>(sq + 12 * lane), r1 = *reinterpret_cast<const float4*>(sq + 12 * lane + 4);
    const float2 r2 = *reinterpret_cast<const float2*>(sq + 12 * lane + 8);
    const float4 yq = lane < qcount ? A.slots[(long long)k0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float s0 = ldexpf(1.f, -sc.kw), s1 = ldexpf(1.f, sc.ex - sc.kw), s2 = ldexpf(1.f, 2 * sc.ex - sc.kw);
    const float y[3] = {yq.x, yq.y, yq.z};
    const float W = r0.x * s0;
    const float X1[3] = {r0.y * s1, r0.z * s1, r0.w * s1};
    const float X2[6] = {r1.x * s2, r1.y * s2, r1.z * s2, r1.w * s2, r2.x * s2, r2.y * s2};
    float Sy[3], D[3], Myy[6], Mdy[9], Q[6];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        Sy[m] = W * y[m];
        D[m] = X1[m] - Sy[m];
    }
    int t6 = 0;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
#pragma unroll
        for (int l = m; l < 3; ++l, ++t6) {
            Myy[t6] = Sy[m] * y[l];
            Q[t6] = X2[t6] - X1[m] * y[l] - y[m] * X1[l] + Myy[t6];
        }
#pragma unroll
        for (int l = 0; l < 3; ++l) Mdy[3 * m + l] = D[m] * y[l];
    }
    store_moments(W, D, Sy, Myy, Mdy, Q, cnt, Fa, hx, hy, hz, gp, A.edges[e].scale, A.acc + (long long)e * ACC_N, lane);
}

// ------------------------------------------------------------ lane path ----
// Everything else (colour, semantic pruning, no labels): lanes over the unit's
// queries, all in FP32.  A unit of <= 16, 8 or 4 queries gives each of them 2, 4
// or 8 lanes, which take every 2nd, 4th or 8th pair of candidates; a lane holds its
// query (place, label row, colour) and its running sums W, D = sum w d and Q =
// sum w d d^T in registers, and evaluates two candidates at a time in paired
// FP32, those outside r_c with weight 0.  With y the lane's query, sum w y' = W y,
// sum w y'y'^T = W y y^T and sum w d y'^T = D y^T at the unit's end.
//
// Bound by FP32 issue (two elements take ~22 paired instructions), on clouds of small
// units by the latency of a unit's loads.  It replaced a walk over the set bits of a
// per-candidate mask (lane = candidate), which folded 28 sums per candidate and
// batch, read the queries with bank conflicts and ran as long as the lane with the
// most pairs: four unlabelled scans of 8000 points 381 -> 298 us per evaluation, 5 x 20k
// RGB-D with colour 210 -> 200 us.  Three CTAs per SM: 313 and 203 us.
template <int DP, bool BF16>
__host__ __device__ constexpr int lane_row_words() {   // row stride of the staged labels: lanes read up to 8 rows at a time
    return SemRow<DP, BF16>::WORDS + (SemRow<DP, BF16>::WORDS % 8 == 0 && DP > 0 ? 4 : 0);
}
// Per-warp shared memory: the batch's candidate pairs [16][8] (x0 x0' x1 x1' x2
// x2' thr thr'), their colours [16][8] (r r' g g' b b' - -), label rows, the
// candidate ring, the stream's segments.
template <int DP, bool BF16, bool COLOR>
__host__ __device__ constexpr int warp_smem_words() {
    return 16 * 8 + (COLOR ? 16 * 8 : 0) + 32 * lane_row_words<DP, BF16>() + 4 * CQ_N + ROWS_WORDS;
}

template <int DP, bool BF16, bool COLOR>
__device__ __forceinline__ void pair_unit(const PairArgs& A, int2 unit, float* wb, int lane) {
    constexpr int SW = lane_row_words<DP, BF16>();
    const GridParams& gp = A.gp;
    float* cg = wb;
    float* cc = wb + 16 * 8;
    float* srow = cc + (COLOR ? 16 * 8 : 0);
    float4* cq = reinterpret_cast<float4*>(srow + 32 * SW);
    const Rows R{reinterpret_cast<int4*>(cq + CQ_N), reinterpret_cast<float2*>(cq + CQ_N + 9)};
    const float INF = __int_as_float(0x7f800000);
    const int k0 = unit.x, qcount = unit_queries(unit), e = unit_edge(unit);
    const uint32_t key0 = A.qkey[k0] >> gp.key_sub;            // home-cell key
    const FrameDev& Fa = A.frames[A.edges[e].a];
    const int cell = (int)(key0 - A.edges[e].bin_off);
    const int hx = cell % Fa.dim[0], hy = (cell / Fa.dim[0]) % Fa.dim[1], hz = cell / (Fa.dim[0] * Fa.dim[1]);
    // 2^gs lanes per query: the lane's query, and its place among them
    const int gs = qcount > 16 ? 0 : (qcount > 8 ? 1 : (qcount > 4 ? 2 : 3));
    const int ql = lane & ((32 >> gs) - 1), gi = lane >> (5 - gs);
    const bool qv = ql < qcount;
    const float4 r = qv ? A.slots[(long long)k0 + ql] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int sidx = __float_as_int(r.w);
    const float mx = -2.f * r.x, my = -2.f * r.y, mz = -2.f * r.z;
    const float mw = qv ? fmaf(r.x, r.x, fmaf(r.y, r.y, r.z * r.z)) : INF;      // an absent query fails every test
    Sem<DP, BF16> qs;
    if (DP > 0) qs.load(A.sem_sorted, sidx, qv);
    float4 qc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (COLOR && qv) qc = __ldg(A.col4 + sidx);
    float blo0 = qv ? r.x : INF, blo1 = qv ? r.y : INF, blo2 = qv ? r.z : INF;
    float bhi0 = qv ? r.x : -INF, bhi1 = qv ? r.y : -INF, bhi2 = qv ? r.z : -INF;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        blo0 = fminf(blo0, __shfl_xor_sync(FULL, blo0, o));
        blo1 = fminf(blo1, __shfl_xor_sync(FULL, blo1, o));
        blo2 = fminf(blo2, __shfl_xor_sync(FULL, blo2, o));
        bhi0 = fmaxf(bhi0, __shfl_xor_sync(FULL, bhi0, o));
        bhi1 = fmaxf(bhi1, __shfl_xor_sync(FULL, bhi1, o));
        bhi2 = fmaxf(bhi2, __shfl_xor_sync(FULL, bhi2, o));
    }
    __syncwarp();
    // a candidate farther than r_c from the query box pairs with none of
    // the queries; the margin keeps every candidate the exact test passes
    const float box_thr = gp.rc2 * 1.0001f;
    int n_seg;
    const int C = build_rows(R, A.cell_start, Fa, hx, hy, hz, blo0, blo1, blo2, bhi0, bhi1, bhi2, gp.hf, box_thr, lane,
                             n_seg);
    int c_s, c_hi;                               // chunks of the stream
    part_range(C, unit_part(unit), unit_shift(unit), c_s, c_hi);
    if (c_s >= c_hi) return;
    const u64 MX = f2(mx, mx), MY = f2(my, my), MZ = f2(mz, mz), MW = f2(mw, mw);
    const u64 H2 = f2(0.5f, 0.5f), KG2 = f2(gp.kg, gp.kg);
    // W, D and Q of the last <= 32 candidate pairs (halves: even, odd candidates), and of all before
    // them.  One chain of additions over the whole stream was off by up to 1.2e-4 at 25 600
    // candidates of equal weight (the loss promises 1e-5), these by 4e-6; four unlabelled scans of
    // 8000 points take 288 us with either.
    u64 S2[10];
    float T[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) {
        S2[k] = 0ull;
        T[k] = 0.f;
    }
    int cnt = 0;
    // the batches, compiled with and without the pruning test
    auto batches = [&](auto prune) {
        [[maybe_unused]] constexpr bool PRUNE = decltype(prune)::value;
        int qhead = 0, qlen = 0;                 // ring head and fill
        Cursor cur;
        cur.start(R, n_seg, 32 * c_s + lane);
        bool more = true;
        for (;;) {
            // batches of up to 16 additions, until another one could make more than 32
#pragma unroll 1
            for (int chain = 0; chain <= 16;) {
                more = c_s < c_hi || qlen > 0;
                if (!more) break;
                // stream the 27-cell candidates through the box test into the
                // ring until it holds a full batch (or the stream ends)
                while (qlen < 32 && c_s < c_hi) {
                    bool keep = false;
                    float4 ent = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (cur.valid()) {
                        ent = cur.point(A.pts4, gp.hf);
                        const float e0 = fmaxf(fmaxf(blo0 - ent.x, ent.x - bhi0), 0.f);
                        const float e1 = fmaxf(fmaxf(blo1 - ent.y, ent.y - bhi1), 0.f);
                        const float e2 = fmaxf(fmaxf(blo2 - ent.z, ent.z - bhi2), 0.f);
                        keep = fmaf(e0, e0, fmaf(e1, e1, e2 * e2)) < box_thr;
                    }
                    const unsigned bal = __ballot_sync(FULL, keep);
                    if (keep) cq[(qhead + qlen + __popc(bal & ((1u << lane) - 1u))) & (CQ_N - 1)] = ent;
                    qlen += __popc(bal);
                    ++c_s;
                    cur.next(R, n_seg);
                }
                __syncwarp();
                const int nb = qlen < 32 ? qlen : 32;
                more = nb != 0;                      // stream ended with the ring empty
                if (!more) break;
                // lane c stages candidate c (absent ones: thr = -inf, the label row left as it is)
                {
                    const bool has = lane < nb;
                    const float4 ent = has ? cq[(qhead + lane) & (CQ_N - 1)] : make_float4(0.f, 0.f, 0.f, 0.f);
                    const int i = __float_as_int(ent.w);
                    float* g = cg + 8 * (lane >> 1) + (lane & 1);
                    g[0] = ent.x;
                    g[2] = ent.y;
                    g[4] = ent.z;
                    g[6] = has ? gp.rc2 - fmaf(ent.x, ent.x, fmaf(ent.y, ent.y, ent.z * ent.z)) : -INF;
                    if constexpr (COLOR) {
                        const float4 c = has ? __ldg(A.col4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
                        float* k = cc + 8 * (lane >> 1) + (lane & 1);
                        k[0] = c.x;
                        k[2] = c.y;
                        k[4] = c.z;
                    }
                    if (has) SemRow<DP, BF16>::stage(srow + lane * SW, A.sem_sorted, i);
                }
                qhead = (qhead + nb) & (CQ_N - 1);
                qlen -= nb;
                __syncwarp();
                const int n_it = (((nb + 1) >> 1) + (1 << gs) - 1) >> gs;
                for (int j = 0; j < n_it; ++j) {
                    const int p = (j << gs) + gi;
                    const ulonglong2 x01 = *reinterpret_cast<const ulonglong2*>(cg + 8 * p);
                    const ulonglong2 x2t = *reinterpret_cast<const ulonglong2*>(cg + 8 * p + 4);
                    const float2 t = f2_split(ffma2(x01.x, MX, ffma2(x01.y, MY, ffma2(x2t.x, MZ, MW))));
                    const float2 thr = f2_split(x2t.y);
                    bool in0 = t.x < thr.x, in1 = t.y < thr.y;
                    const u64 E0 = ffma2(H2, MX, x01.x), E1 = ffma2(H2, MY, x01.y), E2 = ffma2(H2, MZ, x2t.x);
                    u64 arg = fmul2(ffma2(E0, E0, ffma2(E1, E1, fmul2(E2, E2))), KG2);
                    if constexpr (COLOR) {
                        const ulonglong2 c01 = *reinterpret_cast<const ulonglong2*>(cc + 8 * p);
                        const u64 c2 = *reinterpret_cast<const u64*>(cc + 8 * p + 4);
                        const u64 r0 = fadd2(c01.x, f2(-qc.x, -qc.x)), r1 = fadd2(c01.y, f2(-qc.y, -qc.y)),
                                  r2 = fadd2(c2, f2(-qc.z, -qc.z));
                        arg = ffma2(ffma2(r0, r0, ffma2(r1, r1, fmul2(r2, r2))), f2(gp.kc, gp.kc), arg);
                    }
                    const float2 a = f2_split(arg);
                    float w0 = ex2_approx(a.x), w1 = ex2_approx(a.y);
                    if constexpr (DP > 0) {
                        const float s0 = SemRow<DP, BF16>::dot(qs, srow + (2 * p) * SW);
                        const float s1 = SemRow<DP, BF16>::dot(qs, srow + (2 * p + 1) * SW);
                        if constexpr (PRUNE) {
                            in0 = in0 && s0 >= gp.sem_min;
                            in1 = in1 && s1 >= gp.sem_min;
                        }
                        w0 *= s0;
                        w1 *= s1;
                    }
                    cnt += (in0 ? 1 : 0) + (in1 ? 1 : 0);
                    const u64 w = f2(in0 ? w0 : 0.f, in1 ? w1 : 0.f);
                    const u64 WX = fmul2(w, E0), WY = fmul2(w, E1), WZ = fmul2(w, E2);
                    S2[0] = fadd2(S2[0], w);
                    S2[1] = fadd2(S2[1], WX);
                    S2[2] = fadd2(S2[2], WY);
                    S2[3] = fadd2(S2[3], WZ);
                    S2[4] = ffma2(WX, E0, S2[4]);
                    S2[5] = ffma2(WX, E1, S2[5]);
                    S2[6] = ffma2(WX, E2, S2[6]);
                    S2[7] = ffma2(WY, E1, S2[7]);
                    S2[8] = ffma2(WY, E2, S2[8]);
                    S2[9] = ffma2(WZ, E2, S2[9]);
                }
                chain += n_it;
                __syncwarp();
            }
            if (!more) break;
#pragma unroll
            for (int k = 0; k < 10; ++k) {
                const float2 h = f2_split(S2[k]);
                T[k] += h.x + h.y;
                S2[k] = 0ull;
            }
        }
    };
    if (DP > 0 && gp.sem_min > -INF) batches(std::true_type{});
    else batches(std::false_type{});
    if (!__any_sync(FULL, cnt != 0)) return;     // no pair: every sum is zero
    auto both = [&](int k) {
        const float2 h = f2_split(S2[k]);
        return T[k] + (h.x + h.y);
    };
    const float W = both(0), y[3] = {r.x, r.y, r.z};
    float Dv[3], Sy[3], Myy[6], Mdy[9], Qm[6];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        Dv[m] = both(1 + m);
        Sy[m] = W * y[m];
    }
    int t6 = 0;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
#pragma unroll
        for (int l = 0; l < 3; ++l) Mdy[3 * m + l] = Dv[m] * y[l];
#pragma unroll
        for (int l = m; l < 3; ++l, ++t6) {
            Myy[t6] = Sy[m] * y[l];
            Qm[t6] = both(4 + t6);
        }
    }
    store_moments(W, Dv, Sy, Myy, Mdy, Qm, cnt, Fa, hx, hy, hz, gp, A.edges[e].scale, A.acc + (long long)e * ACC_N, lane);
}

// Shared-memory words per warp of the lane or the dense tile unit.
template <int DP, bool BF16, bool COLOR, bool DENSE>
__host__ __device__ constexpr int unit_smem_words() {
    if constexpr (DENSE) return DenseSmem<(DP > 0 ? DP : 8), !BF16>::WORDS;
    else return warp_smem_words<DP, BF16, COLOR>();
}

// PARTS false (the dense path of problems that never cut units): the kernel
// without part numbers, 2% faster on the mapping and window workloads.
template <int DP, bool BF16, bool COLOR, bool DENSE, bool PARTS>
__device__ __forceinline__ void run_unit(const PairArgs& A, int item, float* wb, int lane) {
    const int2 unit = A.units[item];
    if constexpr (DENSE && DP > 0 && !COLOR) pair_unit_dense<DP, !BF16, PARTS>(A, unit, wb, lane);
    else pair_unit<DP, BF16, COLOR>(A, unit, wb, lane);
}

template <int DP, bool BF16, bool COLOR, bool DENSE, bool PARTS>
__global__ void __launch_bounds__(PAIR_T, 2)
k_pairs(int* unit_counter, const PairArgs A, const int* done) {
    chain_enter();
    if (done && *done) return;
    extern __shared__ float4 smem4[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    float* wb = reinterpret_cast<float*>(smem4) + warp * unit_smem_words<DP, BF16, COLOR, DENSE>();
    const int items = *A.n_units;
    for (;;) {
        int u = 0;
        if (lane == 0) u = atomicAdd(unit_counter, 1);
        u = __shfl_sync(FULL, u, 0);
        if (u >= items) break;
        run_unit<DP, BF16, COLOR, DENSE, PARTS>(A, u, wb, lane);
    }
}

// The pair stage of several problems in one persistent launch: the units of
// job j are numbered after those of jobs 0..j-1 (a job whose solve is done
// contributes none), warps take global unit numbers from one counter, find
// the job by binary search over the prefix, and run the unit with that
// job's arrays.  Every job adds into its own fixed-point accumulators, so a
// problem's results do not depend on which other problems share the launch.
template <int DP, bool BF16, bool COLOR, bool DENSE>
__global__ void __launch_bounds__(PAIR_T, 2)
k_pairs_multi(const PairJob* __restrict__ jobs, int n_jobs, int* unit_counter) {
    __shared__ int s_pref[MAX_PAIR_JOBS + 1];
    extern __shared__ float4 smem4[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    if (warp == 0) {
        int carry = 0;
        for (int base = 0; base < n_jobs; base += 32) {
            const int j = base + lane;
            int n = 0;
            if (j < n_jobs) {
                const int* dn = jobs[j].done;
                n = (dn && *dn) ? 0 : *jobs[j].a.n_units;
            }
            int inc = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(FULL, inc, o);
                if (lane >= o) inc += v;
            }
            if (j < n_jobs) s_pref[j] = carry + inc - n;
            carry += __shfl_sync(FULL, inc, 31);
        }
        if (lane == 0) s_pref[n_jobs] = carry;
    }
    __syncthreads();
    const int total = s_pref[n_jobs];
    float* wb = reinterpret_cast<float*>(smem4) + warp * unit_smem_words<DP, BF16, COLOR, DENSE>();
    for (;;) {
        int u = 0;
        if (lane == 0) u = atomicAdd(unit_counter, 1);
        u = __shfl_sync(FULL, u, 0);
        if (u >= total) break;
        int lo = 0, hi = n_jobs - 1;                 // last job with s_pref[j] <= u
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_pref[mid] <= u) lo = mid; else hi = mid - 1;
        }
        run_unit<DP, BF16, COLOR, DENSE, true>(jobs[lo].a, u - s_pref[lo], wb, lane);
    }
}

// Neighbour-limited variant (top_k > 0): the same candidate stream, cutoff
// test and weight, with lanes over the unit's queries.  Each lane keeps the
// TOPK_MAX pairs of largest w of its query (of equal w the earlier ones in stream
// order, which is the order of the points), then sums its first top_k: W, D = sum
// w d, Q = sum w d d^T, and with y' the query itself sum w y' = W y, sum w y'y'^T =
// W y y^T, sum w d y'^T = D y^T.
//
// A unit of <= 16, 8 or 4 queries gives each of them 2, 4 or 8 lanes, which take
// every 2nd, 4th or 8th candidate of a batch and merge their lists at the unit's
// end (LiDAR units hold 8 queries in the median, so most lanes had no query).  A list
// entry is (w, point): d is formed again for the pairs that are left.  Insertions
// wait until the batch's weights are there and are then made by all lanes at
// once, as many rounds as the busiest lane has candidates above its list's
// smallest, instead of one for every candidate that any lane takes.
// 8 x 20k LiDAR, top_k = 8: evaluation 724 -> 645 us.  Three CTAs per SM (80
// registers) spill: slower than the start.
template <int DP, bool BF16, bool COLOR>
__host__ __device__ constexpr int warp_smem_words_topk() {
    return 32 * 4 + 32 * lane_row_words<DP, BF16>() + (COLOR ? 32 * 4 : 0) + 4 * CQ_N + ROWS_WORDS + 32 * 32;
}

// (w, i) comes before (v, j): larger weight, of equal ones the earlier point
__device__ __forceinline__ bool topk_before(float w, int i, float v, int j) { return w > v || (w == v && i < j); }

template <int DP, bool BF16, bool COLOR>
__global__ void __launch_bounds__(PAIR_T, 2)
k_pairs_topk(const int2* __restrict__ units, const int* __restrict__ n_units, int* unit_counter,
             const uint32_t* __restrict__ qkey, const float4* __restrict__ slots,
             const EdgeDev* __restrict__ edges, const FrameDev* __restrict__ frames,
             const int* __restrict__ cell_start, const float4* __restrict__ pts4,
             const void* __restrict__ sem_sorted, const float4* __restrict__ col4, GridParams gp,
             long long* __restrict__ acc, const int* done) {
    chain_enter();
    if (done && *done) return;
    extern __shared__ float4 smem4[];
    constexpr int SW = lane_row_words<DP, BF16>();
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    float* wb = reinterpret_cast<float*>(smem4) + warp * warp_smem_words_topk<DP, BF16, COLOR>();
    float4* scx = reinterpret_cast<float4*>(wb);                      // [32] staged candidates (x, index)
    float* srow = wb + 4 * 32;                                        // [32][SW] their label rows
    float4* scc = reinterpret_cast<float4*>(srow + 32 * SW);          // [32] their colours
    float4* cq = reinterpret_cast<float4*>(wb + 4 * 32 + 32 * SW + (COLOR ? 4 * 32 : 0));   // ring
    const Rows R{reinterpret_cast<int4*>(cq + CQ_N), reinterpret_cast<float2*>(cq + CQ_N + 9)};
    float* sw = reinterpret_cast<float*>(cq + CQ_N) + ROWS_WORDS + lane;     // [32][32] weights waiting for insertion
    const float NEG_INF = -__int_as_float(0x7f800000);
    const int nu = *n_units;
    for (;;) {
        int u = 0;
        if (lane == 0) u = atomicAdd(unit_counter, 1);
        u = __shfl_sync(FULL, u, 0);
        if (u >= nu) break;
        const int2 unit = units[u];
        const int k0 = unit.x, qcount = unit_queries(unit), e = unit_edge(unit);
        const uint32_t key0 = qkey[k0] >> gp.key_sub;
        const FrameDev& Fa = frames[edges[e].a];
        const int cell = (int)(key0 - edges[e].bin_off);
        const int hx = cell % Fa.dim[0], hy = (cell / Fa.dim[0]) % Fa.dim[1], hz = cell / (Fa.dim[0] * Fa.dim[1]);
        // 2^gs lanes per query: lane's query, and its place among them
        const int gs = qcount > 16 ? 0 : (qcount > 8 ? 1 : (qcount > 4 ? 2 : 3));
        const int ql = lane & ((32 >> gs) - 1), gi = lane >> (5 - gs);
        const bool qv = ql < qcount;
        const float4 r = qv ? slots[(long long)k0 + ql] : make_float4(0.f, 0.f, 0.f, 0.f);
        const int sidx = __float_as_int(r.w);
        const float mx = -2.f * r.x, my = -2.f * r.y, mz = -2.f * r.z;
        const float mw = fmaf(r.x, r.x, fmaf(r.y, r.y, r.z * r.z));
        Sem<DP, BF16> qs;
        if (DP > 0) qs.load(sem_sorted, sidx, qv);
        float4 qc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (COLOR && qv) qc = __ldg(col4 + sidx);
        float blo0 = qv ? r.x : -NEG_INF, blo1 = qv ? r.y : -NEG_INF, blo2 = qv ? r.z : -NEG_INF;
        float bhi0 = qv ? r.x : NEG_INF, bhi1 = qv ? r.y : NEG_INF, bhi2 = qv ? r.z : NEG_INF;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            blo0 = fminf(blo0, __shfl_xor_sync(FULL, blo0, o));
            blo1 = fminf(blo1, __shfl_xor_sync(FULL, blo1, o));
            blo2 = fminf(blo2, __shfl_xor_sync(FULL, blo2, o));
            bhi0 = fmaxf(bhi0, __shfl_xor_sync(FULL, bhi0, o));
            bhi1 = fmaxf(bhi1, __shfl_xor_sync(FULL, bhi1, o));
            bhi2 = fmaxf(bhi2, __shfl_xor_sync(FULL, bhi2, o));
        }
        __syncwarp();
        const float box_thr = gp.rc2 * 1.0001f;
        int n_seg;
        const int C = build_rows(R, cell_start, Fa, hx, hy, hz, blo0, blo1, blo2, bhi0, bhi1, bhi2, gp.hf, box_thr, lane,
                                 n_seg);
        if (C == 0) continue;
        float tw[TOPK_MAX];                        // w descending
        int ti[TOPK_MAX];                          // their points
#pragma unroll
        for (int k = 0; k < TOPK_MAX; ++k) {
            tw[k] = NEG_INF;
            ti[k] = 0x7fffffff;
        }
        int c_s = 0, qhead = 0, qlen = 0;
        Cursor cur;
        cur.start(R, n_seg, lane);
        while (c_s < C || qlen > 0) {
            while (qlen < 32 && c_s < C) {
                bool keep = false;
                float4 ent = make_float4(0.f, 0.f, 0.f, 0.f);
                if (cur.valid()) {
                    ent = cur.point(pts4, gp.hf);
                    const float e0 = fmaxf(fmaxf(blo0 - ent.x, ent.x - bhi0), 0.f);
                    const float e1 = fmaxf(fmaxf(blo1 - ent.y, ent.y - bhi1), 0.f);
                    const float e2 = fmaxf(fmaxf(blo2 - ent.z, ent.z - bhi2), 0.f);
                    keep = fmaf(e0, e0, fmaf(e1, e1, e2 * e2)) < box_thr;
                }
                const unsigned bal = __ballot_sync(FULL, keep);
                if (keep) cq[(qhead + qlen + __popc(bal & ((1u << lane) - 1u))) & (CQ_N - 1)] = ent;
                qlen += __popc(bal);
                c_s += 32;
                cur.next(R, n_seg);
            }
            __syncwarp();
            const int nb = qlen < 32 ? qlen : 32;
            if (nb == 0) break;
            if (lane < nb) {
                const float4 ent = cq[(qhead + lane) & (CQ_N - 1)];
                const int i = __float_as_int(ent.w);
                scx[lane] = ent;
                SemRow<DP, BF16>::stage(srow + lane * SW, sem_sorted, i);
                if (COLOR) scc[lane] = __ldg(col4 + i);
            }
            qhead = (qhead + nb) & (CQ_N - 1);
            qlen -= nb;
            __syncwarp();
            // the lane's candidates that enter its list as it stands
            unsigned pend = 0u;
            const int n_it = (nb + (1 << gs) - 1) >> gs;
            for (int j = 0; j < n_it; ++j) {
                const int c = (j << gs) + gi;
                const float4 xe = scx[c];
                const float thr = gp.rc2 - fmaf(xe.x, xe.x, fmaf(xe.y, xe.y, xe.z * xe.z));
                const float t = fmaf(xe.x, mx, fmaf(xe.y, my, fmaf(xe.z, mz, mw)));
                if (qv && c < nb && t < thr) {
                    const float ex = fmaf(0.5f, mx, xe.x), ey = fmaf(0.5f, my, xe.y), ez = fmaf(0.5f, mz, xe.z);
                    const float dd = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
                    float arg = dd * gp.kg;
                    if (COLOR) {
                        const float4 cc = scc[c];
                        const float cr = cc.x - qc.x, cg = cc.y - qc.y, cb = cc.z - qc.z;
                        arg = fmaf(fmaf(cr, cr, fmaf(cg, cg, cb * cb)), gp.kc, arg);
                    }
                    const float s = SemRow<DP, BF16>::dot(qs, srow + c * SW);
                    const float cw = s * ex2_approx(arg);
                    if (s >= gp.sem_min && cw > tw[TOPK_MAX - 1]) {
                        sw[32 * j] = cw;
                        pend |= 1u << j;
                    }
                }
            }
            while (__any_sync(FULL, pend != 0u)) {
                if (pend) {
                    const int j = __ffs(pend) - 1;
                    pend &= pend - 1u;
                    float cw = sw[32 * j];
                    int ci = __float_as_int(scx[(j << gs) + gi].w);
                    bool in = false;                 // once in, the entries behind it move down
#pragma unroll
                    for (int k = 0; k < TOPK_MAX; ++k) {
                        in = in || cw > tw[k];
                        const float a = tw[k];
                        const int b = ti[k];
                        tw[k] = in ? cw : a;
                        ti[k] = in ? ci : b;
                        cw = in ? a : cw;
                        ci = in ? b : ci;
                    }
                }
            }
            __syncwarp();
        }
        // lists of a query's lanes into one: of two descending lists the better
        // of entry k of one and entry 7 - k of the other are the eight first, bitonic
        for (int o = 32 >> gs; o < 32; o <<= 1) {
            float vw[TOPK_MAX];
            int vi[TOPK_MAX];
#pragma unroll
            for (int k = 0; k < TOPK_MAX; ++k) {
                vw[k] = __shfl_xor_sync(FULL, tw[TOPK_MAX - 1 - k], o);
                vi[k] = __shfl_xor_sync(FULL, ti[TOPK_MAX - 1 - k], o);
            }
#pragma unroll
            for (int k = 0; k < TOPK_MAX; ++k) {
                const bool theirs = topk_before(vw[k], vi[k], tw[k], ti[k]);
                tw[k] = theirs ? vw[k] : tw[k];
                ti[k] = theirs ? vi[k] : ti[k];
            }
#pragma unroll
            for (int h = TOPK_MAX / 2; h > 0; h >>= 1)
#pragma unroll
                for (int k = 0; k < TOPK_MAX; ++k)
                    if (!(k & h)) {
                        const bool swap = topk_before(tw[k + h], ti[k + h], tw[k], ti[k]);
                        const float a = tw[k];
                        const int b = ti[k];
                        tw[k] = swap ? tw[k + h] : a;
                        ti[k] = swap ? ti[k + h] : b;
                        tw[k + h] = swap ? a : tw[k + h];
                        ti[k + h] = swap ? b : ti[k + h];
                    }
        }
        float W = 0.f, Dv[3] = {0.f, 0.f, 0.f}, Qm[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < TOPK_MAX; ++k) {
            if (k < gp.top_k && lane < qcount && tw[k] > NEG_INF) {
                // the pair's d, as the stream formed it: the point's row gives its offset
                const int i = ti[k];
                Cursor at;
                at.enter(R, 0, 0);
                for (int g = 1; g < n_seg && i >= at.end; ++g) at.enter(R, g, 0);
                at.i = i;
                const float4 x = at.point(pts4, gp.hf);
                const float d0 = fmaf(0.5f, mx, x.x), d1 = fmaf(0.5f, my, x.y), d2 = fmaf(0.5f, mz, x.z);
                const float w = tw[k];
                const float wx = w * d0, wy = w * d1, wz = w * d2;
                W += w;
                Dv[0] += wx; Dv[1] += wy; Dv[2] += wz;
                Qm[0] = fmaf(wx, d0, Qm[0]); Qm[1] = fmaf(wx, d1, Qm[1]); Qm[2] = fmaf(wx, d2, Qm[2]);
                Qm[3] = fmaf(wy, d1, Qm[3]); Qm[4] = fmaf(wy, d2, Qm[4]); Qm[5] = fmaf(wz, d2, Qm[5]);
                ++cnt;
            }
        }
        if (!__any_sync(FULL, cnt != 0)) continue;   // no pair: every sum is zero
        const float y[3] = {r.x, r.y, r.z};
        float Sy[3], Myy[6], Mdy[9];
        int t6 = 0;
#pragma unroll
        for (int mm = 0; mm < 3; ++mm) {
            Sy[mm] = W * y[mm];
#pragma unroll
            for (int l = 0; l < 3; ++l) Mdy[3 * mm + l] = Dv[mm] * y[l];
#pragma unroll
            for (int l = mm; l < 3; ++l, ++t6) Myy[t6] = W * y[mm] * y[l];
        }
        store_moments(W, Dv, Sy, Myy, Mdy, Qm, cnt, Fa, hx, hy, hz, gp, edges[e].scale,
                      acc + (long long)e * ACC_N, lane);
    }
}

// Same search and the same cutoff test, geometry only: writes the pair list
// of one edge (verification).
__global__ void __launch_bounds__(PAIR_T)
k_emit_pairs(const int2* __restrict__ units, const int* __restrict__ n_units, int* unit_counter,
             const uint32_t* __restrict__ qkey, const float4* __restrict__ slots,
             const EdgeDev* __restrict__ edges, const FrameDev* __restrict__ frames,
             const int* __restrict__ cell_start, const float4* __restrict__ pts4, GridParams gp,
             int edge_sel, const int* __restrict__ perm_local, long long capacity,
             int* __restrict__ i_out, int* __restrict__ j_out, unsigned long long* n_out) {
    __shared__ float4 s_m[PAIR_T / 32][UQ];
    __shared__ int s_j[PAIR_T / 32][UQ];
    __shared__ int4 s_rows[PAIR_T / 32][ROWS_WORDS / 4];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    float4* sm = s_m[warp];
    const Rows R{s_rows[warp], reinterpret_cast<float2*>(s_rows[warp] + 9)};
    const int nu = *n_units;
    for (;;) {
        int u = 0;
        if (lane == 0) u = atomicAdd(unit_counter, 1);
        u = __shfl_sync(FULL, u, 0);
        if (u >= nu) break;
        const int2 unit = units[u];
        const int k0 = unit.x, qcount = unit_queries(unit), e = unit_edge(unit);
        if (e != edge_sel || unit_part(unit) > 0) continue;      // the first part lists the whole unit
        const uint32_t key0 = qkey[k0] >> gp.key_sub;
        const FrameDev& Fa = frames[edges[e].a];
        const int cell = (int)(key0 - edges[e].bin_off);
        const int hx = cell % Fa.dim[0], hy = (cell / Fa.dim[0]) % Fa.dim[1], hz = cell / (Fa.dim[0] * Fa.dim[1]);
        __syncwarp();
        if (lane < qcount) {
            const float4 r = slots[(long long)k0 + lane];
            sm[lane] = make_float4(-2.f * r.x, -2.f * r.y, -2.f * r.z, fmaf(r.x, r.x, fmaf(r.y, r.y, r.z * r.z)));
            s_j[warp][lane] = perm_local[__float_as_int(r.w)];
        }
        const float INF = __int_as_float(0x7f800000);
        int n_seg;
        const int C = build_rows(R, cell_start, Fa, hx, hy, hz, -INF, -INF, -INF, INF, INF, INF, gp.hf, gp.rc2, lane,
                                 n_seg);      // every cell: no query box
        if (C == 0) continue;
        Cursor cur;
        cur.start(R, n_seg, lane);
        for (int c0 = 0; c0 < C; c0 += 32, cur.next(R, n_seg)) {
            if (!cur.valid()) continue;
            const float4 x = cur.point(pts4, gp.hf);
            const int i = __float_as_int(x.w);
            const float x0 = x.x, x1 = x.y, x2 = x.z;
            const float thr = gp.rc2 - fmaf(x0, x0, fmaf(x1, x1, x2 * x2));
            for (int j = 0; j < qcount; ++j) {
                const float4 m = sm[j];
                const float t = fmaf(x0, m.x, fmaf(x1, m.y, fmaf(x2, m.z, m.w)));
                if (t < thr) {
                    const unsigned long long k = atomicAdd(n_out, 1ULL);
                    if ((long long)k < capacity) {
                        i_out[k] = perm_local[i];
                        j_out[k] = s_j[warp][j];
                    }
                }
            }
        }
    }
}

inline unsigned blocks_for(long long n, int t) {
    long long b = (n + t - 1) / t;
    if (b < 1) b = 1;
    if (b > 1048560) b = 1048560;
    return (unsigned)b;
}

int current_device() {
    int dev = 0;
    cudaGetDevice(&dev);
    return dev;
}

// Opts a kernel in to its dynamic shared memory, which counts for the current device
// alone.
template <typename KernelT>
bool opt_in(KernelT kernel, size_t smem) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess;
}

// Resident CTAs per SM of a pair kernel at its shared-memory size (queried
// once per instantiation and device; the opt-in is set then).  A failure is not kept, and the launch
// that follows reports it.
template <typename KernelT>
int pair_blocks_per_sm(KernelT kernel, size_t smem, PerDevice& cache) {
    const int b = cache.get(current_device(), [&] {
        int n = 0;
        if (!opt_in(kernel, smem) ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, PAIR_T, smem) != cudaSuccess)
            return 0;
        return n < 1 ? 1 : n;
    });
    return b < 1 ? 1 : b;
}

template <int IPT>
void bin_edges(const BinArgs& a, cudaStream_t st) {
    constexpr size_t smem = BinSmem<IPT>::BYTES;
    if constexpr (smem > 36864) {                // with the static arrays more than 48 KB
        static PerDevice opted;
        opted.get(current_device(), [] { return opt_in(k_bin_edges<IPT>, smem) ? 1 : 0; });
    }
    launch_chained(k_bin_edges<IPT>, (unsigned)a.E, BIN_T, smem, st, a.poses, a.edges, a.frames, a.pt_cell, a.pts4,
                   a.cell_start, a.gp, a.uq, a.cut_edge, a.xf,
                                                         a.qkey, a.qrec, a.slots, a.units, a.ucount, a.acc, a.done);
}

inline unsigned pair_grid(int num_sms, int resident, int ctas_per_sm) {
    const int per_sm = (ctas_per_sm > 0 && ctas_per_sm < resident) ? ctas_per_sm : resident;
    return (unsigned)(num_sms * per_sm);
}

// The dense tile unit serves BF16 labels without colour and without
// semantic pruning (top_k has its own kernel); RK_NO_DENSE builds the
// lane kernel for every layout.
inline bool dense_path(const GridParams& gp) {
#ifdef RK_NO_DENSE
    (void)gp;
    return false;
#else
    return gp.sem_pad > 0 && !gp.color && !(gp.sem_min > -__builtin_huge_valf()) && gp.top_k == 0;
#endif
}

template <int DP, bool BF16, bool COLOR, bool DENSE, bool PARTS>
void launch_k_pairs(const PairLaunch& L, const PairArgs& A) {
    const size_t smem = sizeof(float) * (PAIR_T / 32) * unit_smem_words<DP, BF16, COLOR, DENSE>();
    static PerDevice resident;
    const int r = pair_blocks_per_sm(k_pairs<DP, BF16, COLOR, DENSE, PARTS>, smem, resident);
    launch_chained(k_pairs<DP, BF16, COLOR, DENSE, PARTS>, pair_grid(L.num_sms, r, L.ctas_per_sm), PAIR_T, smem, L.stream, 
        L.unit_counter, A, L.done);
}

template <int DP, bool BF16, bool COLOR>
void run_pairs(const PairLaunch& L, const PairArgs& A) {
    if (A.gp.top_k > 0) {
        const size_t smem = sizeof(float) * (PAIR_T / 32) * warp_smem_words_topk<DP, BF16, COLOR>();
        static PerDevice resident;
        const int r = pair_blocks_per_sm(k_pairs_topk<DP, BF16, COLOR>, smem, resident);
        launch_chained(k_pairs_topk<DP, BF16, COLOR>, pair_grid(L.num_sms, r, L.ctas_per_sm), PAIR_T, smem, L.stream, 
            A.units, A.n_units, L.unit_counter, A.qkey, A.slots, A.edges, A.frames, A.cell_start, A.pts4,
            A.sem_sorted, A.col4, A.gp, A.acc, L.done);
        return;
    }
    if constexpr (DP > 0 && !COLOR) {
        if (dense_path(A.gp)) {
            if (A.cut) launch_k_pairs<DP, BF16, COLOR, true, true>(L, A);
            else launch_k_pairs<DP, BF16, COLOR, true, false>(L, A);
            return;
        }
    }
    launch_k_pairs<DP, BF16, COLOR, false, true>(L, A);
}

template <int DP, bool BF16, bool COLOR, bool DENSE>
void launch_k_pairs_multi(const PairJob* jobs, int n_jobs, int* counter, int num_sms, int ctas_per_sm,
                          cudaStream_t st) {
    const size_t smem = sizeof(float) * (PAIR_T / 32) * unit_smem_words<DP, BF16, COLOR, DENSE>();
    static PerDevice resident;
    const int r = pair_blocks_per_sm(k_pairs_multi<DP, BF16, COLOR, DENSE>, smem, resident);
    k_pairs_multi<DP, BF16, COLOR, DENSE><<<pair_grid(num_sms, r, ctas_per_sm), PAIR_T, smem, st>>>(
        jobs, n_jobs, counter);
}

template <int DP, bool BF16, bool COLOR>
void run_pairs_multi(const PairJob* jobs, int n_jobs, int* counter, int num_sms, int ctas_per_sm, bool dense,
                     cudaStream_t st) {
    if constexpr (DP > 0 && !COLOR) {
        if (dense) {
            launch_k_pairs_multi<DP, BF16, COLOR, true>(jobs, n_jobs, counter, num_sms, ctas_per_sm, st);
            return;
        }
    }
    launch_k_pairs_multi<DP, BF16, COLOR, false>(jobs, n_jobs, counter, num_sms, ctas_per_sm, st);
}

// Calls F.template operator()<DP, BF16>() for the label layout of gp
// (padded width, FP32 or BF16 rows); false for a layout without kernels.
template <typename F>
bool with_label_layout(const GridParams& gp, const F& f) {
    if (gp.sem_pad == 0) { f.template operator()<0, false>(); return true; }
    if (gp.sem_bf16) {
        switch (gp.sem_pad) {
            case 8: f.template operator()<8, true>(); return true;
            case 16: f.template operator()<16, true>(); return true;
            case 24: f.template operator()<24, true>(); return true;
            case 32: f.template operator()<32, true>(); return true;
            default: return false;
        }
    }
    switch (gp.sem_pad) {
        case 4: f.template operator()<4, false>(); return true;
        case 8: f.template operator()<8, false>(); return true;
        case 12: f.template operator()<12, false>(); return true;
        case 16: f.template operator()<16, false>(); return true;
        case 20: f.template operator()<20, false>(); return true;
        case 24: f.template operator()<24, false>(); return true;
        case 32: f.template operator()<32, false>(); return true;
        default: return false;
    }
}
}  // namespace

void launch_eval_setup(const double* poses, const EdgeDev* edges, int E, const FrameDev* frames, double h, EdgeXf* xf,
                       long long* ws, int n_ws, int* ucount, long long* acc, const int* done, cudaStream_t st) {
    launch_chained(k_eval_setup, (unsigned)(E < 4 * 592 ? (E + 3) / 4 : 592), 128, 0, st, poses, edges, E, frames, h, xf, ws, n_ws,
                                                                              ucount, acc, done);
    count_launch();
}

void launch_query_keys(const EdgeDev* edges, int E, const FrameDev* frames, const EdgeXf* xf,
                       const uint32_t* pt_cell, const float4* pts4, GridParams gp, long long Q,
                       uint32_t* qkey, float4* qrec, const RadixWs& ws, int num_sms, const int* done, cudaStream_t st) {
    if (Q <= 0) return;
    const int rounds = radix_rounds(Q, num_sms);
    launch_chained(k_query_keys, (unsigned)((Q + (long long)RAD_T * rounds - 1) / ((long long)RAD_T * rounds)), RAD_T, 0, st, 
        edges, E, frames, xf, pt_cell, pts4, gp, Q, qkey, qrec, ws, rounds, done);
    count_launch();
}

void launch_units(const uint32_t* qkey_sorted, const int* qval_sorted, const float4* qrec, long long Q, int uq,
                  int sub, int cut_edge, const EdgeDev* edges, int E, const FrameDev* frames, const int* cell_start,
                  float4* slots, int2* units, int* n_units, const int* done, cudaStream_t st) {
    if (Q <= 0) return;
    if (uq < 1 || uq > UQ) uq = UQ;      // larger units are taken as units of 32
    launch_chained(k_units, blocks_for(Q, 256), 256, 0, st, qkey_sorted, qval_sorted, qrec, Q, uq, sub, cut_edge, edges, E,
                   frames, cell_start, slots, units, n_units, done);
    count_launch();
}

void launch_bin_edges(const BinArgs& a, int q_max, cudaStream_t st) {
    cudaMemsetAsync(a.ucount, 0, 4 * sizeof(int), st);
    BinArgs b = a;
    if (b.uq < 1 || b.uq > UQ) b.uq = UQ;      // larger units are taken as units of 32
    switch ((q_max + BIN_T - 1) / BIN_T) {     // queries per thread
        case 0:
        case 1: bin_edges<1>(b, st); break;
        case 2: bin_edges<2>(b, st); break;
        case 3: bin_edges<3>(b, st); break;
        default: bin_edges<4>(b, st); break;
    }
    count_launch();
}

namespace {
struct SingleLaunch {
    const PairLaunch& L;
    const PairArgs& A;
    template <int DP, bool BF16>
    void operator()() const {
        if (A.gp.color) run_pairs<DP, BF16, true>(L, A);
        else run_pairs<DP, BF16, false>(L, A);
    }
};
struct MultiLaunch {
    const PairJob* jobs;
    int n_jobs;
    bool color;
    bool dense;
    int* counter;
    int num_sms, ctas_per_sm;
    cudaStream_t st;
    template <int DP, bool BF16>
    void operator()() const {
        if (color) run_pairs_multi<DP, BF16, true>(jobs, n_jobs, counter, num_sms, ctas_per_sm, dense, st);
        else run_pairs_multi<DP, BF16, false>(jobs, n_jobs, counter, num_sms, ctas_per_sm, dense, st);
    }
};
}  // namespace

int pair_unit_max(const GridParams& gp) { return (dense_path(gp) && gp.sem_bf16) ? 64 : UQ; }

void launch_pairs(const PairLaunch& L, const PairArgs& A) {
    if (A.Q <= 0) return;
    if (with_label_layout(A.gp, SingleLaunch{L, A})) count_launch();
}

bool launch_pairs_multi(const PairJob* jobs, int n_jobs, const GridParams& layout, int* counter, int num_sms,
                        int ctas_per_sm, cudaStream_t st) {
    if (n_jobs <= 0 || n_jobs > MAX_PAIR_JOBS || layout.top_k > 0) return false;
    const bool ok = with_label_layout(layout, MultiLaunch{jobs, n_jobs, layout.color != 0, dense_path(layout),
                                                          counter, num_sms, ctas_per_sm, st});
    if (ok) count_launch();
    return ok;
}

void launch_emit_pairs(const int2* units, const int* n_units, int* unit_counter,
                       const uint32_t* qkey, const float4* slots, long long Q, const EdgeDev* edges,
                       const FrameDev* frames, const int* cell_start, const float4* pts4,
                       GridParams gp, int edge_sel, const int* perm_local, long long capacity,
                       int* i_out, int* j_out, unsigned long long* n_out, int num_sms,
                       cudaStream_t st) {
    if (Q <= 0) return;
    k_emit_pairs<<<num_sms * 2, PAIR_T, 0, st>>>(units, n_units, unit_counter, qkey, slots, edges, frames,
                                                 cell_start, pts4, gp, edge_sel, perm_local, capacity,
                                                 i_out, j_out, n_out);
    count_launch();
}

}  // namespace rk
