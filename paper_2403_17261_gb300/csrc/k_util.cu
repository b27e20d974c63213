// k_util.cu -- scan, stable grouping by key, and fills used by the step.
#include "common.cuh"

#include <atomic>

namespace ovl {

namespace {
std::atomic<long long> g_launches{0};
}
void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
void note_launches(long long k) { g_launches.fetch_add(k, std::memory_order_relaxed); }
long long launch_count() { return g_launches.load(std::memory_order_relaxed); }

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

__device__ __forceinline__ int warp_incl_scan(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// exclusive scan of one value per thread across the block (blockDim a
// multiple of 32); returns the block total through *total
__device__ int block_excl_scan(int v, int *total) {
    __shared__ int warp_sums[32];
    __shared__ int block_total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    int inc = warp_incl_scan(v);
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int w = lane < nwarps ? warp_sums[lane] : 0;
        int wi = warp_incl_scan(w);
        warp_sums[lane] = wi - w;
        if (lane == 31) block_total = wi;
    }
    __syncthreads();
    int res = inc - v + warp_sums[warp];
    *total = block_total;
    __syncthreads();
    return res;
}

// Exclusive scan in one launch: every tile publishes its sum, then its prefix
// once it has added up its predecessors' (decoupled look-back, Merrill and
// Garland 2016).  A step scans a dozen arrays, most of a few thousand words,
// so launches count: three kernels per scan (tile sums, their scan, tile
// scan) took 8-10 us each time, this one 2.5.  Tiles are taken by ticket, so
// a tile's predecessors are always running.  The state words carry an epoch,
// so nothing is cleared between scans: ctl = (next ticket, tiles done, epoch),
// advanced by the tile that finishes last.  A wait that reaches its limit adds
// up the missing inputs itself.
constexpr unsigned long long kAggregate = 1, kPrefix = 2;
constexpr int kScanPolls = 1 << 16;

__global__ void __launch_bounds__(SCAN_THREADS)
k_scan(const int *__restrict__ in, int n, int *__restrict__ out, int nb, unsigned *ctl, unsigned long long *state,
       int *host_total) {
    __shared__ int sh_tile, sh_prefix;
    const int tid = threadIdx.x, lane = tid & 31;
    unsigned long long epoch = 0;
    if (nb > 1) {
        epoch = *reinterpret_cast<volatile unsigned *>(ctl + 2) & 0x3fffffffu;
        if (tid == 0) sh_tile = (int)atomicAdd(ctl, 1u);
        __syncthreads();
    } else if (tid == 0) {
        sh_tile = 0;
    }
    if (nb == 1) __syncthreads();
    const int tile = sh_tile, base = tile * SCAN_TILE + tid * SCAN_ITEMS;
    int v[SCAN_ITEMS], sum = 0;
    const bool whole = base + SCAN_ITEMS <= n && (reinterpret_cast<uintptr_t>(in) & 15) == 0;
    if (whole) {
        const int4 a = *reinterpret_cast<const int4 *>(in + base), b = *reinterpret_cast<const int4 *>(in + base + 4);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k) v[k] = base + k < n ? in[base + k] : 0;
    }
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) sum += v[k];
    int total;
    const int ex = block_excl_scan(sum, &total);
    int prefix = 0;
    if (nb > 1) {
        auto word = [&](unsigned long long flag, int x) {
            return (epoch << 2 | flag) << 32 | (unsigned long long)(unsigned)x;
        };
        volatile unsigned long long *st = state;
        if (tid == 0) st[tile] = word(tile == 0 ? kPrefix : kAggregate, total);
        if (tid < 32) {
            int run = 0;
            for (int j = tile - 1; j >= 0; j -= 32) {
                const int k = j - lane;
                unsigned long long w = 0;
                bool ready = false;
                for (int it = 0; it < kScanPolls; ++it) {
                    w = k >= 0 ? st[k] : word(kPrefix, 0);
                    ready = (w >> 34) == epoch && (w >> 32 & 3) != 0;
                    if (__all_sync(0xffffffffu, ready)) break;
                }
                int add;
                if (!__all_sync(0xffffffffu, ready)) {
                    add = 0;
                    for (long long i = lane; i < (long long)(j + 1) * SCAN_TILE; i += 32) add += in[i];
                    for (int o = 16; o > 0; o >>= 1) add += __shfl_xor_sync(0xffffffffu, add, o);
                    run += add;
                    break;
                }
                const unsigned full = __ballot_sync(0xffffffffu, (w >> 32 & 3) == kPrefix);
                add = !full || lane <= __ffs(full) - 1 ? (int)(unsigned)w : 0;
                for (int o = 16; o > 0; o >>= 1) add += __shfl_xor_sync(0xffffffffu, add, o);
                run += add;
                if (full) break;
            }
            if (lane == 0) {
                if (tile > 0) st[tile] = word(kPrefix, run + total);
                sh_prefix = run;
            }
        }
        __syncthreads();
        prefix = sh_prefix;
    }
    int e = prefix + ex;
    if (whole && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
        int o[SCAN_ITEMS];
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k) { o[k] = e; e += v[k]; }
        *reinterpret_cast<int4 *>(out + base) = make_int4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<int4 *>(out + base + 4) = make_int4(o[4], o[5], o[6], o[7]);
    } else {
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k) {
            if (base + k < n) out[base + k] = e;
            e += v[k];
        }
    }
    if (tid == 0) {
        if (tile == nb - 1) {
            out[n] = prefix + total;
            if (host_total) *host_total = prefix + total;
        }
        if (nb > 1 && atomicAdd(ctl + 1, 1u) == (unsigned)nb - 1) {
            ctl[0] = 0;
            ctl[1] = 0;
            ctl[2] = (unsigned)epoch + 1;
        }
    }
}

}  // namespace

void scan_i32(const int *in, int *out, int n, DBuf<int> &tmp, cudaStream_t s, int *host_total) {
    const int nb = n > 0 ? (n + SCAN_TILE - 1) / SCAN_TILE : 1;
    const size_t need = 4 + 2 * (size_t)nb;   // ctl, then a state word per tile
    if (need > tmp.cap || !tmp.p) {
        tmp.ensure(need);
        CK(cudaMemsetAsync(tmp.p, 0, sizeof(int) * tmp.cap, s));
    }
    k_scan<<<nb, SCAN_THREADS, 0, s>>>(in, n, out, nb, reinterpret_cast<unsigned *>(tmp.p),
                                       reinterpret_cast<unsigned long long *>(tmp.p + 4), host_total);
    note_launch();
    CK(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// stable LSD radix sort, 8-bit digits
// ---------------------------------------------------------------------------
namespace {

constexpr int RS_THREADS = 256;
constexpr int RS_ROUNDS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ROUNDS;
constexpr int RS_WARPS = RS_THREADS / 32;

__global__ void k_rs_hist(const uint32_t *keys, int n, int shift, int nblocks, int *hist) {
    __shared__ int h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    int base = blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ROUNDS; ++r) {
        int i = base + r * RS_THREADS + threadIdx.x;
        if (i < n) atomicAdd(&h[(keys[i] >> shift) & 255u], 1);
    }
    __syncthreads();
    hist[threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

__global__ void k_rs_scatter(const uint32_t *keys, const uint32_t *vals, int n, int shift,
                             int nblocks, const int *offs, uint32_t *keys_out, uint32_t *vals_out) {
    __shared__ int running[256];
    __shared__ int wcnt[RS_WARPS][256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    running[tid] = 0;
    for (int w = 0; w < RS_WARPS; ++w) wcnt[w][tid] = 0;
    __syncthreads();
    const int base = blockIdx.x * RS_TILE;
    const unsigned lt = (1u << lane) - 1u;
    for (int r = 0; r < RS_ROUNDS; ++r) {
        int i = base + r * RS_THREADS + tid;
        bool valid = i < n;
        uint32_t k = valid ? keys[i] : 0u;
        int d = valid ? (int)((k >> shift) & 255u) : 256;
        unsigned peers = __match_any_sync(0xffffffffu, d);
        int lrank = __popc(peers & lt);
        if (valid && lrank == 0) wcnt[warp][d] = __popc(peers);
        __syncthreads();
        int pos = 0;
        if (valid) {
            int pre = 0;
            for (int w = 0; w < warp; ++w) pre += wcnt[w][d];
            pos = offs[d * nblocks + blockIdx.x] + running[d] + pre + lrank;
        }
        __syncthreads();
        {
            int add = 0;
            for (int w = 0; w < RS_WARPS; ++w) {
                add += wcnt[w][tid];
                wcnt[w][tid] = 0;
            }
            running[tid] += add;
        }
        if (valid) {
            keys_out[pos] = k;
            vals_out[pos] = vals ? vals[i] : (uint32_t)i;
        }
        __syncthreads();
    }
}

}  // namespace

const uint32_t *group_by_key(const uint32_t *key, int n, int nbits, uint32_t *out, GroupBuf &b, DBuf<int> &tmp,
                             cudaStream_t s) {
    b.k0.ensure((size_t)n + 1);
    if (n == 0) return b.k0.p;
    const int nblocks = (n + RS_TILE - 1) / RS_TILE, passes = nbits > 8 ? (nbits + 7) / 8 : 1;
    b.hist.ensure((size_t)256 * nblocks + 1);
    b.offs.ensure((size_t)256 * nblocks + 1);
    if (passes > 1) { b.k1.ensure((size_t)n + 1); b.v0.ensure((size_t)n + 1); b.v1.ensure((size_t)n + 1); }
    const uint32_t *ki = key, *vi = nullptr;
    for (int p = 0; p < passes; ++p) {
        uint32_t *ko = p & 1 ? b.k1.p : b.k0.p, *vo = p + 1 == passes ? out : (p & 1 ? b.v1.p : b.v0.p);
        k_rs_hist<<<nblocks, RS_THREADS, 0, s>>>(ki, n, 8 * p, nblocks, b.hist.p);
        note_launch();
        scan_i32(b.hist.p, b.offs.p, 256 * nblocks, tmp, s);
        k_rs_scatter<<<nblocks, RS_THREADS, 0, s>>>(ki, vi, n, 8 * p, nblocks, b.offs.p, ko, vo);
        note_launch();
        CK(cudaGetLastError());
        ki = ko;
        vi = vo;
    }
    return ki;
}

namespace {
__global__ void k_fill_u8(uint8_t *p, uint8_t v, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        p[i] = v;
}
// start[p] = first index of a sorted key >= p, for p <= P, here and on the
// host: every change between neighbouring keys sets the starts it passes (a
// binary search per p took 12 us, twenty dependent loads)
__global__ void k_key_starts(const uint32_t *keys, int n, int P, int *start, int *host_start) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x) {
        const int lo = i > 0 ? (int)keys[i - 1] + 1 : 0, hi = i < n ? (int)keys[i] : P;
        for (int p = lo; p <= hi; ++p) {
            start[p] = i;
            host_start[p] = i;
        }
    }
}
int grid_for(size_t n, int threads) {
    size_t g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 152 * 16) g = 152 * 16;
    return (int)g;
}
}  // namespace

void fill_u8(uint8_t *p, uint8_t v, size_t n, cudaStream_t s) {
    if (!n) return;
    k_fill_u8<<<grid_for(n, 256), 256, 0, s>>>(p, v, n);
    note_launch();
    CK(cudaGetLastError());
}
void key_starts(const uint32_t *keys, int n, int P, int *start, int *host_start, cudaStream_t s) {
    k_key_starts<<<grid_for((size_t)n + 1, 256), 256, 0, s>>>(keys, n, P, start, host_start);
    note_launch();
    CK(cudaGetLastError());
}

}  // namespace ovl
