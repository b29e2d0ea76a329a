// Stable LSD radix sort of uint32 keys with an int32 payload (the key's first
// position): the plumbing of the grid build (points by cell) and of the
// per-evaluation query binning (queries by home cell).  The pair sum needs a
// spatial index (the paper names GPU voxel hashing as future work); this one is
// rebuilt by sorting.
//
// The kernels that make the keys also histogram their 8-bit digits (radix.cuh);
// each pass is then a single kernel ("one sweep"): a block takes the next tile
// of keys (tiles are handed out in order by an atomic counter), ranks its keys
// stably (each warp its own run of keys by match.any and a digit counter of its
// own; one exclusive sum over the warps), publishes its per-digit counts, obtains
// the counts of all earlier tiles by looking back over their published records
// (decoupled look-back, eight records read at a time), and writes the tile in
// digit order from shared memory.  A record holds a flag (aggregate of the tile
// / inclusive prefix up to the tile) and a count in one 64-bit word.  Every wait
// is bounded; a wait that gives up sets an error word and the kernel finishes
// with what it has.
//
// Ranking by warps costs two block barriers per tile where rounds of 256 keys in
// input order cost three each (24 per tile of 2048).
#include "radix.cuh"

#include <utility>
#include <vector>

namespace rk {

namespace {
constexpr int RAD_WARPS = RAD_T / 32;
constexpr unsigned long long ST_AGG = 1ull << 62;      // count = this tile's
constexpr unsigned long long ST_PRE = 2ull << 62;      // count = tiles 0..t inclusive
constexpr unsigned long long ST_CNT = (1ull << 62) - 1ull;
constexpr int SPIN_LIMIT = 1 << 22;         // polls of one look-back wait before it gives up
constexpr int LOOK = 8;                     // records a look-back reads at a time

// exclusive scan of one value per thread over a 256-thread block
template <typename T>
__device__ __forceinline__ T block_excl_scan256(T v, T* s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    T before = 0;
#pragma unroll
    for (int w = 0; w < RAD_WARPS; ++w) before += w < warp ? s_warp[w] : T(0);
    __syncthreads();
    return before + inc - v;
}

// FIRST: the payload is the key's position, not read.
template <int IPT, bool FIRST>
__global__ void __launch_bounds__(RAD_T) k_onesweep(const uint32_t* __restrict__ kin,
                                                    const int* __restrict__ vin,
                                                    uint32_t* __restrict__ kout, int* __restrict__ vout,
                                                    long long n, int shift,
                                                    const unsigned long long* __restrict__ counts,
                                                    unsigned long long* status, int* tile_ctr, int* err,
                                                    int spin_limit, const int* done) {
    chain_enter();
    if (done && *done) return;
    constexpr int TILE = RAD_T * IPT;
    __shared__ int s_tile;
    __shared__ int wcnt[RAD_WARPS][256];
    __shared__ int s_loc[256];            // first place of a digit inside the tile
    __shared__ long long s_out[256];      // what to add to a place inside the tile for its place in the output
    __shared__ long long s_warp[RAD_WARPS];
    __shared__ int s_warpi[RAD_WARPS];
    __shared__ uint32_t s_key[TILE];
    __shared__ int s_val[TILE];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_tile = atomicAdd(tile_ctr, 1);
#pragma unroll
    for (int w = 0; w < RAD_WARPS; ++w) wcnt[w][tid] = 0;
    __syncthreads();
    const int t = s_tile;
    const long long base = (long long)t * TILE;
    const unsigned lt = (1u << lane) - 1u;
    const int off = warp * (32 * IPT) + lane;       // a warp's keys are one run of the input
    uint32_t key[IPT];
    int val[IPT], rank[IPT];
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const long long i = base + off + 32 * r;
        key[r] = i < n ? kin[i] : 0u;
        val[r] = FIRST ? (int)i : (i < n ? vin[i] : 0);
    }
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const bool valid = base + off + 32 * r < n;
        const int d = valid ? (int)((key[r] >> shift) & 255u) : 256;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int leader = __ffs(peers) - 1;
        int old = 0;
        if (valid && lane == leader) {
            old = wcnt[warp][d];
            wcnt[warp][d] = old + __popc(peers);
        }
        rank[r] = __shfl_sync(0xffffffffu, old, leader) + __popc(peers & lt);
        __syncwarp();
    }
    __syncthreads();
    // digit tid: exclusive sum over the warps, this tile's count
    const int d = tid;
    int cnt = 0;
#pragma unroll
    for (int w = 0; w < RAD_WARPS; ++w) {
        const int c = wcnt[w][d];
        wcnt[w][d] = cnt;
        cnt += c;
    }
    // publish it, then look back for the prefix
    volatile unsigned long long* st = status + (long long)t * 256 + d;
    *st = (t == 0 ? ST_PRE : ST_AGG) | (unsigned long long)cnt;
    const int loc = block_excl_scan256<int>(cnt, s_warpi);
    const long long first = block_excl_scan256<long long>((long long)counts[d], s_warp);
    s_loc[d] = loc;
    __syncthreads();
    // the tile in digit order (places below the tile's key count)
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        if (base + off + 32 * r < n) {
            const int dd = (int)((key[r] >> shift) & 255u);
            const int at = s_loc[dd] + wcnt[warp][dd] + rank[r];
            s_key[at] = key[r];
            s_val[at] = val[r];
        }
    }
    long long excl = 0;
    if (t > 0) {
        bool open = true;                           // no inclusive prefix met yet
        for (int p = t - 1; p >= 0 && open; p -= LOOK) {
            unsigned long long v[LOOK];
#pragma unroll
            for (int j = 0; j < LOOK; ++j)
                v[j] = p - j >= 0 ? *(volatile unsigned long long*)(status + (long long)(p - j) * 256 + d) : 0ull;
#pragma unroll
            for (int j = 0; j < LOOK; ++j) {
                if (open && p - j >= 0) {
                    volatile unsigned long long* sp = status + (long long)(p - j) * 256 + d;
                    int spins = 0;
                    while ((v[j] >> 62) == 0ull) {
                        if (++spins > spin_limit) {   // give up: the prefix stays short, writes stay in bounds
                            atomicOr(err, 1);
                            open = false;
                            break;
                        }
                        __nanosleep(20);
                        v[j] = *sp;
                    }
                    excl += (long long)(v[j] & ST_CNT);
                    if ((v[j] >> 62) == 2ull) open = false;
                }
            }
        }
        *st = ST_PRE | (unsigned long long)(excl + cnt);
    }
    s_out[d] = first + excl - loc;
    __syncthreads();
    const int m = n - base < TILE ? (int)(n - base) : TILE;
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const int j = tid + RAD_T * r;
        if (j < m) {
            const uint32_t k = s_key[j];
            const long long o = s_out[(k >> shift) & 255u] + j;
            kout[o] = k;
            vout[o] = s_val[j];
        }
    }
}

template <int IPT>
void sort_passes(uint32_t* keys, int* vals, uint32_t* keys_alt, int* vals_alt, long long n, const RadixWs& ws,
                 int* err, const int* done, cudaStream_t st) {
    const long long nb = (n + RAD_T * IPT - 1) / (RAD_T * IPT);
    uint32_t* ki = keys;
    int* vi = vals;
    uint32_t* ko = keys_alt;
    int* vo = vals_alt;
    for (int p = 0; p < ws.npass; ++p) {
        auto kernel = p == 0 ? k_onesweep<IPT, true> : k_onesweep<IPT, false>;
        launch_chained(kernel, (unsigned)nb, RAD_T, 0, st, ki, vi, ko, vo, n, 8 * p, ws.counts + 256 * p,
                                               ws.status + (size_t)256 * nb * p, ws.ctr + p, err, SPIN_LIMIT, done);
        count_launch();
        std::swap(ki, ko);
        std::swap(vi, vo);
    }
}
// Tiles of 4096 keys once there are enough of them for every SM several times
// over (half the records per key), else of 2048.
constexpr long long BIG_SORT = 4096LL * 152 * 8;
}  // namespace

size_t scan_ws_elems(long long) { return (size_t)(RAD_PASSES * 256 + 2 * RAD_PASSES); }

size_t radix_hist_elems(long long n) {
    const long long nb = (n + RAD_TILE_MIN - 1) / RAD_TILE_MIN;
    return (size_t)(RAD_PASSES * 256 * (nb > 0 ? nb : 1));
}

RadixWs radix_ws(long long n, int nbits, long long* hist, long long* ws) {
    RadixWs r{};
    r.counts = reinterpret_cast<unsigned long long*>(ws);
    r.ctr = reinterpret_cast<int*>(ws + RAD_PASSES * 256);
    r.status = reinterpret_cast<unsigned long long*>(hist);
    r.npass = (nbits + 7) / 8;
    const long long tile = n >= BIG_SORT ? 4096 : 2048;
    r.n_status = 256 * ((n + tile - 1) / tile) * r.npass;
    return r;
}

bool radix_sort_u32(uint32_t* keys, int* vals, uint32_t* keys_alt, int* vals_alt, long long n, const RadixWs& ws,
                    int* err, const int* done, cudaStream_t st) {
    if (n <= 0 || ws.npass <= 0) return false;
    if (n >= BIG_SORT) sort_passes<16>(keys, vals, keys_alt, vals_alt, n, ws, err, done, st);
    else sort_passes<8>(keys, vals, keys_alt, vals_alt, n, ws, err, done, st);
    return (ws.npass & 1) != 0;
}

}  // namespace rk

// Failure-detection self-test of the look-back's bounded wait (declared in
// include/rkhsba.h).  Two tiles of keys; tile_ctr starts at 1, so the single
// launched block takes tile 1 while the record of tile 0 is never published.
// Every thread of the block then polls a record that stays zero, gives up
// after spin_limit polls, raises the error word and finishes with a short
// prefix (zero): each output index is the digit's base from the global counts
// plus the key's rank inside tile 1, below n, so all writes land inside the
// output arrays.  Guard words on both sides of the outputs are checked.
extern "C" rkhsba_status rkhsba_selftest_lookback_timeout(int32_t spin_limit, int32_t* writes_in_bounds) {
    using namespace rk;
    if (writes_in_bounds) *writes_in_bounds = 0;
    if (spin_limit < 1 || spin_limit > (1 << 20)) {
        set_thread_error("rkhsba_selftest_lookback_timeout: spin_limit must be in [1, 2^20]");
        return RKHSBA_EINVAL;
    }
    const long long n = 2LL * RAD_TILE_MIN;
    const long long G = 256;                        // guard words on each side of the outputs
    uint32_t* kin = nullptr;
    uint32_t* kout = nullptr;
    int* vin = nullptr;
    int* vout = nullptr;
    unsigned long long* status = nullptr;
    unsigned long long* counts = nullptr;
    int* ctl = nullptr;                              // [0] tile counter, [1] error word
    auto release = [&] {
        cudaFree(kin); cudaFree(kout); cudaFree(vin); cudaFree(vout);
        cudaFree(status); cudaFree(counts); cudaFree(ctl);
    };
    auto cuda_fail = [&](cudaError_t e) {
        release();
        cudaGetLastError();
        set_thread_error(cudaGetErrorString(e));
        return RKHSBA_ECUDA;
    };
    cudaError_t e = cudaSuccess;
    if ((e = cudaMalloc(&kin, sizeof(uint32_t) * n)) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMalloc(&vin, sizeof(int) * n)) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMalloc(&kout, sizeof(uint32_t) * (n + 2 * G))) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMalloc(&vout, sizeof(int) * (n + 2 * G))) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMalloc(&status, sizeof(unsigned long long) * 2 * 256)) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMalloc(&counts, sizeof(unsigned long long) * 256)) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMalloc(&ctl, sizeof(int) * 2)) != cudaSuccess) return cuda_fail(e);
    std::vector<uint32_t> hk(n);
    std::vector<int> hv(n);
    for (long long i = 0; i < n; ++i) {
        hk[i] = (uint32_t)((unsigned long long)(i + 1) * 2654435761ull);
        hv[i] = (int)i;
    }
    const int ctl0[2] = {1, 0};
    if ((e = cudaMemcpy(kin, hk.data(), sizeof(uint32_t) * n, cudaMemcpyHostToDevice)) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMemcpy(vin, hv.data(), sizeof(int) * n, cudaMemcpyHostToDevice)) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMemset(kout, 0xAB, sizeof(uint32_t) * (n + 2 * G))) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMemset(vout, 0xAB, sizeof(int) * (n + 2 * G))) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMemset(status, 0, sizeof(unsigned long long) * 2 * 256)) != cudaSuccess) return cuda_fail(e);
    std::vector<unsigned long long> hc(256, 0ull);
    for (long long i = 0; i < n; ++i) ++hc[hk[i] & 255u];
    if ((e = cudaMemcpy(counts, hc.data(), sizeof(unsigned long long) * 256, cudaMemcpyHostToDevice)) != cudaSuccess)
        return cuda_fail(e);
    if ((e = cudaMemcpy(ctl, ctl0, sizeof(ctl0), cudaMemcpyHostToDevice)) != cudaSuccess) return cuda_fail(e);
    k_onesweep<RAD_TILE_MIN / RAD_T, false><<<1, RAD_T>>>(kin, vin, kout + G, vout + G, n, 0, counts, status, ctl, ctl + 1, spin_limit, nullptr);
    count_launch();
    if ((e = cudaDeviceSynchronize()) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e);
    int ctl1[2] = {0, 0};
    std::vector<uint32_t> gk(n + 2 * G);
    std::vector<int> gv(n + 2 * G);
    if ((e = cudaMemcpy(ctl1, ctl, sizeof(ctl1), cudaMemcpyDeviceToHost)) != cudaSuccess) return cuda_fail(e);
    if ((e = cudaMemcpy(gk.data(), kout, sizeof(uint32_t) * (n + 2 * G), cudaMemcpyDeviceToHost)) != cudaSuccess)
        return cuda_fail(e);
    if ((e = cudaMemcpy(gv.data(), vout, sizeof(int) * (n + 2 * G), cudaMemcpyDeviceToHost)) != cudaSuccess)
        return cuda_fail(e);
    release();
    bool guards = true;
    for (long long i = 0; i < G; ++i) {
        guards = guards && gk[i] == 0xABABABABu && gk[n + G + i] == 0xABABABABu;
        guards = guards && gv[i] == (int)0xABABABABu && gv[n + G + i] == (int)0xABABABABu;
    }
    if (writes_in_bounds) *writes_in_bounds = guards ? 1 : 0;
    if (ctl1[1]) {
        set_thread_error("a bounded wait of the radix sort's look-back gave up (self-test)");
        return RKHSBA_ETIMEOUT;
    }
    set_thread_error("");
    return RKHSBA_OK;
}
