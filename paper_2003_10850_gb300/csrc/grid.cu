// grid.cu -- quantisation, Morton keys, LSD radix sort, and the implicit
// bounding-volume hierarchy over Morton-sorted particles.
//
// The paper's modules each walk a tree to find the neighbours of active
// particles (Sec. 1, Sec. 2.4); its tree is built on the CPU, which it names
// as a coming bottleneck (Sec. 4). Here the whole neighbour structure is built
// on the GPU: integer positions -> 63-bit Morton keys -> stable radix sort ->
// fixed fan-out hierarchy whose level-k node t covers sorted particles
// [t*8^(k+1), (t+1)*8^(k+1)) of its box, with integer bounding boxes.
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "internal.cuh"

namespace sph {

// ---------------------------------------------------------------------------
// a1: quantise + key
// ---------------------------------------------------------------------------

// Spread the low 21 bits of v so that bit b lands at bit 3b (bit tricks of
// the usual "part1by2" form on 64-bit words).
__device__ __forceinline__ unsigned long long spread3(unsigned v) {
    unsigned long long x = v & 0x1fffffu;
    x = (x | (x << 32)) & 0x1f00000000ffffull;
    x = (x | (x << 16)) & 0x1f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

// x / L is a product when L is a power of two: x * (S 2^-32) with S = 2^32 / L
// exact, so the value is the division's (FP64 division is a long sequence on
// the narrow FP64 pipe).
__device__ __forceinline__ unsigned quantize1(double x, const BoxDesc& B, bool& bad) {
    if (!isfinite(x)) { bad = true; return 0u; }
    double t = B.pow2 ? x * (B.S * 2.3283064365386962890625e-10) : x / B.L;
    t = t - floor(t);
    double v = rint(t * 4294967296.0);
    if (v >= 4294967296.0) v -= 4294967296.0;
    return (unsigned)(unsigned long long)v;
}

// FP32 positions inside [0, L) of a power-of-two box take an FP32 path with
// the same result: t = x / L is in [0, 1), so frac(t) = t, and t 2^32 = x Hs
// (Hs = 2^32 / L, a power of two) is exact in FP32; rint of that float is the
// FP64 rint of the same value. Everything else takes the FP64 definition.
__device__ __forceinline__ unsigned quantize_p(float x, const BoxDesc& B, bool& bad) {
    if (B.pow2 && x >= 0.f && x < B.Lf && (double)B.Lf == B.L) {
        const float v = rintf(x * B.Hs);
        return v >= 4294967296.0f ? 0u : (unsigned)(unsigned long long)v;
    }
    return quantize1((double)x, B, bad);
}
__device__ __forceinline__ unsigned quantize_p(double x, const BoxDesc& B, bool& bad) {
    return quantize1(x, B, bad);
}

template <typename P>
__global__ void k_quantize(const P* __restrict__ pos, const float* __restrict__ mass, int n,
                           const long long* __restrict__ box_off, const BoxDesc* __restrict__ boxes,
                           int nb, int bb, uint4* __restrict__ xq, unsigned long long* __restrict__ keys,
                           Counters* ctr) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo = 0, hi = nb - 1;  // largest b with box_off[b] <= i
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (box_off[mid] <= i) lo = mid; else hi = mid - 1;
    }
    const BoxDesc& B = boxes[lo];
    bool bad = false;
    unsigned X = quantize_p(pos[3 * (size_t)i], B, bad);
    unsigned Y = quantize_p(pos[3 * (size_t)i + 1], B, bad);
    unsigned Z = quantize_p(pos[3 * (size_t)i + 2], B, bad);
    float m = mass[i];
    if (!(m > 0.f) || !isfinite(m)) bad = true;
    if (bad) atomicOr(&ctr->status, ST_INVALID);
    unsigned long long key = (spread3(X >> 11) << 2) | (spread3(Y >> 11) << 1) | spread3(Z >> 11);
    if (bb) key = ((unsigned long long)lo << (63 - bb)) | (key >> bb);
    xq[i] = make_uint4(X, Y, Z, __float_as_uint(m));
    keys[i] = key;
}

// ---------------------------------------------------------------------------
// a2: stable LSD radix sort of (64-bit key, 32-bit index), 9-bit digits
// ---------------------------------------------------------------------------
//
// One kernel counts every pass's digits, then one kernel per pass ranks and
// moves the items: a tile of 4096 items finds where its digit runs start from
// the digit totals and from the tiles before it, whose counts it reads as they
// appear (each tile publishes its own counts first, then its running totals).
// Tiles are numbered by a ticket, so a tile only ever waits for tiles that
// already run; a wait is bounded, and a tile whose wait runs out counts the items
// before it by itself, so that the result never depends on the wait. 63-bit keys
// take 7 passes of 9 bits: 9 launches in all.
//
// What bounds it: at 10M keys the 24 bytes per item and pass (HBM); below a
// few hundred thousand the chain of passes, a few microseconds each. A
// separate count, scan (three launches) and scatter per 8-bit pass, ranking
// with four block barriers per 256 items, took 40 launches.

constexpr int kRsT = 512, kRsIPT = 8, kRsWarps = kRsT / 32;
constexpr int kRsDig = 1 << kRsBits;
static_assert(kRsTile == kRsT * kRsIPT && kRsDig == kRsT, "one digit per thread");
#ifndef SPH_WAIT_POLLS
#define SPH_WAIT_POLLS (1 << 22)
#endif
constexpr int kRsSpin = SPH_WAIT_POLLS;   // polls of a predecessor's word before counting its tile's items
constexpr int kRsBack = 8;         // predecessors read at a time

struct RsSmem {
    unsigned long long key[kRsTile];
    unsigned val[kRsTile];
    unsigned short wcnt[kRsWarps][kRsDig];   // per warp: items of each digit so far; then the warps before
    unsigned start[kRsDig];                  // first place of each digit's run in the tile
    unsigned gbase[kRsDig];                  // global place of the run's first item - start
    unsigned long long wsum[kRsWarps];
    unsigned tile;
};

// The digit counts of every pass at once (keys are only permuted between passes).
__global__ void __launch_bounds__(kRsT) k_rs_hist(const unsigned long long* __restrict__ keys, int n, int passes,
                                                  unsigned* __restrict__ hist) {
    __shared__ unsigned h[kRsMaxPass][kRsDig];
    for (int p = 0; p < passes; ++p) h[p][threadIdx.x] = 0u;
    __syncthreads();
    for (long long base = (long long)blockIdx.x * kRsTile; base < n; base += (long long)gridDim.x * kRsTile) {
        unsigned long long key[kRsIPT];
#pragma unroll
        for (int r = 0; r < kRsIPT; ++r) {
            const long long k = base + r * kRsT + threadIdx.x;
            key[r] = k < n ? keys[k] : 0ull;
        }
#pragma unroll
        for (int r = 0; r < kRsIPT; ++r) {
            if (base + r * kRsT + threadIdx.x < n)
                for (int p = 0; p < passes; ++p)
                    atomicAdd(&h[p][(unsigned)(key[r] >> (p * kRsBits)) & (kRsDig - 1u)], 1u);
        }
    }
    __syncthreads();
    for (int p = 0; p < passes; ++p) {
        const unsigned c = h[p][threadIdx.x];
        if (c) atomicAdd(&hist[p * kRsDig + threadIdx.x], c);
    }
}

// A word of the tiles' published counts: count, flag and the pass it belongs
// to in one 64-bit word, so that no fence is needed and words of earlier
// passes read as "not yet".
__device__ __forceinline__ void rs_put(unsigned long long* p, unsigned tag, unsigned v) {
    const unsigned long long w = ((unsigned long long)tag << 32) | v;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ unsigned long long rs_get(const unsigned long long* p) {
    unsigned long long w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    return w;
}

// One pass. A warp ranks its 256 consecutive items in rounds of 32 (equal
// digits in lane order, then round order: stable), the block adds the warps
// before, and the items leave through shared memory in digit order, so that
// consecutive threads write consecutive places of a digit's run. vin NULL: the
// items' own indices.
__global__ void __launch_bounds__(kRsT, 2) k_rs_pass(const unsigned long long* __restrict__ kin,
                                                     const unsigned* __restrict__ vin,
                                                     unsigned long long* __restrict__ kout,
                                                     unsigned* __restrict__ vout, int n, int pass,
                                                     const unsigned* __restrict__ hist, unsigned* ticket,
                                                     unsigned long long* status) {
    extern __shared__ __align__(16) unsigned char raw[];
    RsSmem& sm = *reinterpret_cast<RsSmem*>(raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int shift = pass * kRsBits;
    const unsigned agg = (unsigned)(pass + 1) * 2u, incl = agg + 1u;   // word tags: tile count, running total
    if (tid == 0) sm.tile = atomicAdd(ticket, 1u);
    {
        unsigned* w = reinterpret_cast<unsigned*>(sm.wcnt[warp]);
#pragma unroll
        for (int k = 0; k < kRsDig / 64; ++k) w[k * 32 + lane] = 0u;
    }
    const unsigned total = hist[tid];
    __syncthreads();
    const int tile = (int)sm.tile;
    const long long base = (long long)tile * kRsTile;
    const int tn = (int)min((long long)kRsTile, n - base);
    // places past n carry the last digit and the largest indices: they rank behind every item
    unsigned long long key[kRsIPT];
    unsigned val[kRsIPT], rank[kRsIPT];
#pragma unroll
    for (int r = 0; r < kRsIPT; ++r) {
        const int i = warp * (32 * kRsIPT) + r * 32 + lane;
        key[r] = i < tn ? kin[base + i] : ~0ull;
        val[r] = i < tn ? (vin ? vin[base + i] : (unsigned)(base + i)) : 0u;
    }
    // the lanes of each round with the same digit, bit by bit (independent of one
    // another, unlike the running counts that follow)
    unsigned peers[kRsIPT];
#pragma unroll
    for (int r = 0; r < kRsIPT; ++r) {
        const int i = warp * (32 * kRsIPT) + r * 32 + lane;
        const unsigned d = i < tn ? (unsigned)(key[r] >> shift) & (kRsDig - 1u) : kRsDig - 1u;
        unsigned m = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < kRsBits; ++b) {
            const bool one = (d >> b) & 1u;
            const unsigned v = __ballot_sync(0xffffffffu, one);
            m &= one ? v : ~v;
        }
        peers[r] = m;
        rank[r] = d;
    }
#pragma unroll
    for (int r = 0; r < kRsIPT; ++r) {
        const unsigned d = rank[r], b = sm.wcnt[warp][d];
        const unsigned before = __popc(peers[r] & ((1u << lane) - 1u));
        __syncwarp();   // every lane has read its digit's count
        if (before == 0u) sm.wcnt[warp][d] = (unsigned short)(b + __popc(peers[r]));
        rank[r] = b + before;
        __syncwarp();
    }
    __syncthreads();
    // thread tid serves digit tid from here on
    unsigned cnt = 0u;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) {
        const unsigned c = sm.wcnt[w][tid];
        sm.wcnt[w][tid] = (unsigned short)cnt;
        cnt += c;
    }
    unsigned long long* mine = status + (size_t)tile * kRsDig + tid;
    rs_put(mine, tile == 0 ? incl : agg, cnt);
    // exclusive scans over the digits of the tile's counts (low word) and the totals (high word)
    unsigned long long x = ((unsigned long long)total << 32) | cnt;
    const unsigned long long own = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sm.wsum[warp] = x;
    __syncthreads();
    unsigned long long before = 0ull;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) before += w < warp ? sm.wsum[w] : 0ull;
    x += before - own;
    sm.start[tid] = (unsigned)x;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRsIPT; ++r) {
        const int i = warp * (32 * kRsIPT) + r * 32 + lane;
        const unsigned d = i < tn ? (unsigned)(key[r] >> shift) & (kRsDig - 1u) : kRsDig - 1u;
        const unsigned p = sm.start[d] + sm.wcnt[warp][d] + rank[r];
        sm.key[p] = key[r];
        sm.val[p] = val[r];
    }
    // the items of this digit in the tiles before: add their counts back to the
    // nearest running total, several words in flight at a time
    unsigned prefix = 0u;
    int t = tile - 1, spins = 0;
    while (t >= 0) {
        unsigned long long w[kRsBack];
#pragma unroll
        for (int k = 0; k < kRsBack; ++k) w[k] = t - k >= 0 ? rs_get(status + (size_t)(t - k) * kRsDig + tid) : 0ull;
        bool more = true;
#pragma unroll
        for (int k = 0; k < kRsBack; ++k) {
            if (!more) continue;
            const unsigned tag = (unsigned)(w[k] >> 32);
            if (t < 0 || (tag != agg && tag != incl)) {
                more = false;   // not published yet: read again from here
            } else {
                prefix += (unsigned)w[k];
                t = tag == incl ? -1 : t - 1;
                if (tag == incl) more = false;
            }
        }
        if (t >= 0 && !more && ++spins > kRsSpin) break;
    }
    if (__syncthreads_or(t >= 0)) {   // a wait ran out: count the items before the tile (nobody writes kin)
        sm.gbase[tid] = 0u;
        __syncthreads();
        for (long long i = tid; i < base; i += kRsT)
            atomicAdd(&sm.gbase[(unsigned)(kin[i] >> shift) & (kRsDig - 1u)], 1u);
        __syncthreads();
        prefix = sm.gbase[tid];
    }
    if (tile > 0) rs_put(mine, incl, prefix + cnt);
    sm.gbase[tid] = (unsigned)(x >> 32) + prefix - sm.start[tid];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRsIPT; ++r) {
        const int p = r * kRsT + tid;
        if (p < tn) {
            const unsigned long long k = sm.key[p];
            const unsigned g = sm.gbase[(unsigned)(k >> shift) & (kRsDig - 1u)] + (unsigned)p;
            if (g < (unsigned)n) {   // (always, unless the caller's keys change under the sort)
                kout[g] = k;
                vout[g] = sm.val[p];
            }
        }
    }
}

// The whole sort in one block, for up to kRsSmall items: the passes follow one
// another in shared memory, ranked and placed as k_rs_pass does. A set this small
// is one or two tiles of the passes above, and pays their launches and round trips
// through global memory (about 8 us each) for a microsecond or two of work:
// 4,096 keys 63 -> 34 us.
constexpr int kRsSmallT = 1024, kRsSmallWarps = kRsSmallT / 32;
static_assert(kRsSmall == kRsSmallT * kRsIPT, "items of the block");
struct RsSmallSmem {
    unsigned long long key[kRsSmall];
    unsigned val[kRsSmall];
    unsigned short wcnt[kRsSmallWarps][kRsDig];
    unsigned start[kRsDig];
    unsigned wsum[kRsDig / 32];
};
__global__ void __launch_bounds__(kRsSmallT) k_rs_small(const unsigned long long* __restrict__ kin,
                                                        unsigned long long* __restrict__ kout,
                                                        unsigned* __restrict__ vout, int n, int passes) {
    extern __shared__ __align__(16) unsigned char raw[];
    RsSmallSmem& sm = *reinterpret_cast<RsSmallSmem*>(raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int first = warp * (32 * kRsIPT) + lane;   // this lane's items: first + 32 r
    const bool any = warp * (32 * kRsIPT) < n;       // the warp has items
    unsigned long long key[kRsIPT];
    unsigned val[kRsIPT], rank[kRsIPT];
#pragma unroll
    for (int r = 0; r < kRsIPT; ++r) {
        val[r] = (unsigned)(first + 32 * r);
        key[r] = first + 32 * r < n ? kin[first + 32 * r] : 0ull;
    }
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = pass * kRsBits;
        {
            unsigned* w = reinterpret_cast<unsigned*>(sm.wcnt[warp]);
#pragma unroll
            for (int k = 0; k < kRsDig / 64; ++k) w[k * 32 + lane] = 0u;
        }
        __syncwarp();
        // places past n carry the last digit: behind every item in every pass
        auto digit = [&](int r) {
            return first + 32 * r < n ? (unsigned)(key[r] >> shift) & (kRsDig - 1u) : kRsDig - 1u;
        };
        if (any) {
            unsigned peers[kRsIPT];
#pragma unroll
            for (int r = 0; r < kRsIPT; ++r) {
                const unsigned d = digit(r);
                unsigned m = 0xffffffffu;
#pragma unroll
                for (int b = 0; b < kRsBits; ++b) {
                    const bool one = (d >> b) & 1u;
                    const unsigned v = __ballot_sync(0xffffffffu, one);
                    m &= one ? v : ~v;
                }
                peers[r] = m;
            }
#pragma unroll
            for (int r = 0; r < kRsIPT; ++r) {
                const unsigned d = digit(r), b = sm.wcnt[warp][d];
                const unsigned before = __popc(peers[r] & ((1u << lane) - 1u));
                __syncwarp();   // every lane has read its digit's count
                if (before == 0u) sm.wcnt[warp][d] = (unsigned short)(b + __popc(peers[r]));
                rank[r] = b + before;
                __syncwarp();
            }
        }
        __syncthreads();
        unsigned cnt = 0u, x = 0u;
        if (tid < kRsDig) {
#pragma unroll
            for (int w = 0; w < kRsSmallWarps; ++w) {
                const unsigned c = sm.wcnt[w][tid];
                sm.wcnt[w][tid] = (unsigned short)cnt;
                cnt += c;
            }
            x = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) sm.wsum[warp] = x;
        }
        __syncthreads();
        if (tid < kRsDig) {
            unsigned before = 0u;
#pragma unroll
            for (int w = 0; w < kRsDig / 32; ++w) before += w < warp ? sm.wsum[w] : 0u;
            sm.start[tid] = before + x - cnt;
        }
        __syncthreads();
        if (any) {
#pragma unroll
            for (int r = 0; r < kRsIPT; ++r) {
                const unsigned d = digit(r), q = sm.start[d] + sm.wcnt[warp][d] + rank[r];
                sm.key[q] = key[r];
                sm.val[q] = val[r];
            }
        }
        __syncthreads();
        if (any) {
#pragma unroll
            for (int r = 0; r < kRsIPT; ++r) {
                key[r] = sm.key[first + 32 * r];
                val[r] = sm.val[first + 32 * r];
            }
        }
    }
#pragma unroll
    for (int r = 0; r < kRsIPT; ++r) {
        if (first + 32 * r < n) {
            kout[first + 32 * r] = key[r];
            vout[first + 32 * r] = val[r];
        }
    }
}

// Sorts keys of key_bits bits with their indices. kin is read by the first
// pass only (and not written); the passes write (ka, va), (kb, vb), (ka, va),
// ... in turn, so an odd number of passes ends in (ka, va). With an odd number
// kin may be kb, with an even number kin may not be ka. (Up to kRsSmall items go
// straight to where the last pass would end.)
cudaError_t rs_sort(const unsigned long long* kin, unsigned long long* ka, unsigned* va, unsigned long long* kb,
                    unsigned* vb, int n, int key_bits, unsigned char* work, int sm_count, cudaStream_t s,
                    unsigned* launches) {
    const int passes = (key_bits + kRsBits - 1) / kRsBits;
    const int tiles = (n + kRsTile - 1) / kRsTile;
    if (n <= kRsSmall) {
        cudaError_t e = cudaFuncSetAttribute(k_rs_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(RsSmallSmem));
        if (e) return e;
        k_rs_small<<<1, kRsSmallT, sizeof(RsSmallSmem), s>>>(kin, passes & 1 ? ka : kb, passes & 1 ? va : vb, n, passes);
        ++*launches;
        return cudaGetLastError();
    }
    unsigned* hist = reinterpret_cast<unsigned*>(work);
    unsigned* ticket = hist + kRsMaxPass * kRsDig;
    unsigned long long* status = reinterpret_cast<unsigned long long*>(work + kRsHead);
    cudaError_t e = cudaFuncSetAttribute(k_rs_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RsSmem));
    if (e) return e;
    if ((e = cudaMemsetAsync(work, 0, rs_work_bytes(n), s))) return e;
    k_rs_hist<<<std::min(tiles, 2 * sm_count), kRsT, 0, s>>>(kin, n, passes, hist);
    if ((e = cudaGetLastError())) return e;
    for (int p = 0; p < passes; ++p) {
        k_rs_pass<<<tiles, kRsT, sizeof(RsSmem), s>>>(p == 0 ? kin : p & 1 ? ka : kb,
                                                      p == 0 ? nullptr : p & 1 ? va : vb, p & 1 ? kb : ka,
                                                      p & 1 ? vb : va, n, p, hist + p * kRsDig, ticket + p, status);
        if ((e = cudaGetLastError())) return e;
    }
    *launches += 1 + passes;
    return cudaSuccess;
}

// ---------------------------------------------------------------------------
// a3: gather into sorted order, hierarchy bounding boxes, h_max
// ---------------------------------------------------------------------------

__global__ void k_gather(const uint4* __restrict__ xq, int n, uint4* __restrict__ posm, const int32_t* __restrict__ perm,
                         int32_t* __restrict__ rank) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    int i = perm[k];
    posm[k] = xq[i];
    rank[i] = k;
}

// Node centre (integer) and half extents (box units, padded by two integer
// units) -- the form the thread-per-particle walk tests against.
__device__ __forceinline__ void node_geom(uint4 a, uint4 b, double s, uint4& c, float4& e) {
    c = make_uint4(a.x + ((b.x - a.x) >> 1), a.y + ((b.y - a.y) >> 1), a.z + ((b.z - a.z) >> 1), 0u);
    e = make_float4((float)((double)(((b.x - a.x) >> 1) + 2u) * s), (float)((double)(((b.y - a.y) >> 1) + 2u) * s),
                    (float)((double)(((b.z - a.z) >> 1) + 2u) * s), 0.f);
}

// The hierarchy is built in two launches: blocks of kTreeT leaves form levels
// 0 to 3 of their part (a level's results pass through shared memory), then one
// block per box forms the few nodes of the levels above, one level after another.
// (One launch per level, most of them a handful of threads, took five to seven.)

// Bounds and geometry of node nd.
__device__ __forceinline__ void put_bbox(int nd, uint4 a, uint4 b, double s, uint4* __restrict__ lo,
                                         uint4* __restrict__ hi, uint4* __restrict__ nc, float4* __restrict__ ne,
                                         uint4& c) {
    float4 e;
    node_geom(a, b, s, c, e);
    lo[nd] = a;
    hi[nd] = b;
    nc[nd] = c;
    ne[nd] = e;
}
__device__ __forceinline__ void join_bbox(uint4& a, uint4& b, uint4 x, uint4 y) {
    a.x = min(a.x, x.x); a.y = min(a.y, x.y); a.z = min(a.z, x.z);
    b.x = max(b.x, y.x); b.y = max(b.y, y.y); b.z = max(b.z, y.z);
}

__global__ void __launch_bounds__(kTreeT) k_tree_low(const uint4* __restrict__ posm, const BoxDesc* __restrict__ boxes,
                                                     uint4* __restrict__ lo, uint4* __restrict__ hi,
                                                     uint4* __restrict__ nc, float4* __restrict__ ne,
                                                     float4* __restrict__ posf) {
    __shared__ uint4 sa[kTreeT], sb[kTreeT];
    const BoxDesc& B = boxes[blockIdx.y];
    const int tid = threadIdx.x, t = blockIdx.x * kTreeT + tid;
    if (blockIdx.x * kTreeT >= B.lvl_n[0]) return;
    const double s = ldexp(B.L, -32);
    const uint4 a0 = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0), b0 = make_uint4(0, 0, 0, 0);
    uint4 a = a0, b = b0, c;
    if (t < B.lvl_n[0]) {
        const long long p0 = B.off + (long long)t * kLeaf;
        const int np = (int)min((long long)kLeaf, B.off + B.n - p0);
        uint4 x[kLeaf];   // all loads in flight together
#pragma unroll
        for (int k = 0; k < kLeaf; ++k)
            if (k < np) x[k] = posm[p0 + k];
#pragma unroll
        for (int k = 0; k < kLeaf; ++k)
            if (k < np) join_bbox(a, b, x[k], x[k]);
        put_bbox(B.lvl_off[0] + t, a, b, s, lo, hi, nc, ne, c);
        // leaf-relative FP32 coordinates (box units) and mass of the leaf's particles
        const float sf = (float)s;
#pragma unroll
        for (int k = 0; k < kLeaf; ++k)
            if (k < np)
                posf[p0 + k] = make_float4((float)(int)(x[k].x - c.x) * sf, (float)(int)(x[k].y - c.y) * sf,
                                           (float)(int)(x[k].z - c.z) * sf, __uint_as_float(x[k].w));
    }
    sa[tid] = a;
    sb[tid] = b;
    int w = kTreeT;
#pragma unroll
    for (int lev = 1; lev < kTreeLow; ++lev) {
        w /= kFan;
        __syncthreads();
        const int tt = blockIdx.x * w + tid;
        a = a0;
        b = b0;
        if (tid < w)   // (children past the level's end hold the neutral bounds)
            for (int k = 0; k < kFan; ++k) join_bbox(a, b, sa[tid * kFan + k], sb[tid * kFan + k]);
        __syncthreads();
        if (tid < w) {
            sa[tid] = a;
            sb[tid] = b;
            if (lev < B.nlev && tt < B.lvl_n[lev]) put_bbox(B.lvl_off[lev] + tt, a, b, s, lo, hi, nc, ne, c);
        }
    }
}

__global__ void __launch_bounds__(kTreeTopT) k_tree_top(const BoxDesc* __restrict__ boxes, uint4* lo, uint4* hi,
                                                        uint4* __restrict__ nc, float4* __restrict__ ne) {
    const BoxDesc& B = boxes[blockIdx.x];
    const double s = ldexp(B.L, -32);
    for (int lev = kTreeLow; lev < B.nlev; ++lev) {
        for (int t = threadIdx.x; t < B.lvl_n[lev]; t += kTreeTopT) {
            const int c0 = t * kFan, c1 = min(c0 + kFan, B.lvl_n[lev - 1]);
            uint4 a = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0), b = make_uint4(0, 0, 0, 0), c;
            for (int k = c0; k < c1; ++k) join_bbox(a, b, lo[B.lvl_off[lev - 1] + k], hi[B.lvl_off[lev - 1] + k]);
            put_bbox(B.lvl_off[lev] + t, a, b, s, lo, hi, nc, ne, c);
        }
        __syncthreads();
    }
}

// h_max of every node, as the bounds.
__global__ void __launch_bounds__(kTreeT) k_hmax_low(const int32_t* __restrict__ perm, const float* __restrict__ h,
                                                     const BoxDesc* __restrict__ boxes, float* __restrict__ hmax,
                                                     float4* __restrict__ ne) {
    __shared__ float sm[kTreeT];
    const BoxDesc& B = boxes[blockIdx.y];
    const int tid = threadIdx.x, t = blockIdx.x * kTreeT + tid;
    if (blockIdx.x * kTreeT >= B.lvl_n[0]) return;
    float m = 0.f;
    if (t < B.lvl_n[0]) {
        const long long p0 = B.off + (long long)t * kLeaf;
        const int np = (int)min((long long)kLeaf, B.off + B.n - p0);
        float x[kLeaf];   // all gathers in flight together
#pragma unroll
        for (int k = 0; k < kLeaf; ++k) x[k] = k < np ? h[perm[p0 + k]] : 0.f;
#pragma unroll
        for (int k = 0; k < kLeaf; ++k) m = fmaxf(m, x[k]);
        hmax[B.lvl_off[0] + t] = m;
        ne[B.lvl_off[0] + t].w = m;
    }
    sm[tid] = m;
    int w = kTreeT;
#pragma unroll
    for (int lev = 1; lev < kTreeLow; ++lev) {
        w /= kFan;
        __syncthreads();
        const int tt = blockIdx.x * w + tid;
        m = 0.f;
        if (tid < w)
            for (int k = 0; k < kFan; ++k) m = fmaxf(m, sm[tid * kFan + k]);
        __syncthreads();
        if (tid < w) {
            sm[tid] = m;
            if (lev < B.nlev && tt < B.lvl_n[lev]) {
                hmax[B.lvl_off[lev] + tt] = m;
                ne[B.lvl_off[lev] + tt].w = m;
            }
        }
    }
}

__global__ void __launch_bounds__(kTreeTopT) k_hmax_top(const BoxDesc* __restrict__ boxes, float* hmax,
                                                        float4* __restrict__ ne) {
    const BoxDesc& B = boxes[blockIdx.x];
    for (int lev = kTreeLow; lev < B.nlev; ++lev) {
        for (int t = threadIdx.x; t < B.lvl_n[lev]; t += kTreeTopT) {
            const int c0 = t * kFan, c1 = min(c0 + kFan, B.lvl_n[lev - 1]);
            float m = 0.f;
            for (int c = c0; c < c1; ++c) m = fmaxf(m, hmax[B.lvl_off[lev - 1] + c]);
            hmax[B.lvl_off[lev] + t] = m;
            ne[B.lvl_off[lev] + t].w = m;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// a6: active list
// ---------------------------------------------------------------------------

// What a call clears before its kernels, in the launch that makes its active list
// (each a memset or a launch of its own otherwise).
__device__ __forceinline__ void call_begin(const CallBegin& b, int k) {
    if (k < kQueues && ((b.queue_mask >> k) & 1u)) b.queue[k] = 0u;
    if (b.list_zero && k < 2) b.list_zero[k] = 0u;
    if (b.list_new) {   // a density call that records lists: clear the status words, one more generation
        if (k < kListGen) b.list_new[k] = 0u;
        else if (k == kListGen) b.list_new[kListGen] += 1u;
    }
}

// all particles active: the identity list, and its length
__global__ void k_iota_count(int32_t* a, int n, uint32_t* count, CallBegin b) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) {
        a[k] = k;
        if (b.ext_n) b.ext_n[k] = 0u;
    }
    if (k == 0) *count = (uint32_t)n;
    if (blockIdx.x == 0) call_begin(b, k);
}

__global__ void k_mark(const int32_t* __restrict__ active, int na, const int32_t* __restrict__ rank,
                       uint8_t* __restrict__ flag, int n, Counters* ctr) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= na) return;
    int i = active[k];
    if (i < 0) return;   // a padding entry (a list of fixed capacity whose count lives on the device)
    if (i >= n) { atomicOr(&ctr->status, ST_INVALID); return; }
    flag[rank[i]] = 1;
}

// The indices whose flag is set, ascending, and their number, in one pass:
// a tile of 4096 flags counts its own, publishes the count, and adds the counts
// of the tiles before it (32 of them at a time), or counts their flags itself when
// a wait runs out (as k_rs_pass). flag: a byte per index, or (max_bin >= 0) its time
// bin, set if the bin ends a step at `tick`. work: a ticket and a word per tile,
// cleared. One launch in place of a three-launch scan and a placing pass over every
// flag and its scan.
constexpr int kCpT = 256, kCpPer = 16;
static_assert(kCpTile == kCpT * kCpPer, "flags per block");
__global__ void __launch_bounds__(kCpT) k_flag_list(const uint8_t* __restrict__ flag, int n, long long tick, int max_bin,
                                                    unsigned long long* work, int32_t* __restrict__ list,
                                                    uint32_t* __restrict__ count, CallBegin b) {
    __shared__ unsigned s_tile, s_before, s_late, s_warp[kCpT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (blockIdx.x == 0) call_begin(b, tid);
    if (tid == 0) s_tile = atomicAdd(reinterpret_cast<unsigned*>(work), 1u);
    __syncthreads();
    const int tile = (int)s_tile;
    unsigned long long* status = work + 1;
    const long long i0 = (long long)tile * kCpTile + tid * kCpPer;
    unsigned set = 0u;   // bit k: flag i0 + k
    auto is_set = [&](unsigned v) {
        return max_bin >= 0 ? (tick & ((1ll << (max_bin - min((int)v, max_bin))) - 1)) == 0 : v != 0u;
    };
    auto take = [&](int k, unsigned v) { set |= is_set(v) ? 1u << k : 0u; };
    if (i0 + kCpPer <= n && (reinterpret_cast<uintptr_t>(flag) & 15) == 0) {
        const uint4 v = *reinterpret_cast<const uint4*>(flag + i0);
        const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < kCpPer; ++k) take(k, (w[k >> 2] >> (8 * (k & 3))) & 255u);
    } else {
        for (int k = 0; k < kCpPer; ++k)
            if (i0 + k < n) take(k, flag[i0 + k]);
    }
    const unsigned c = __popc(set);
    unsigned x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    unsigned before = x - c, total = 0u;
#pragma unroll
    for (int w = 0; w < kCpT / 32; ++w) {
        before += w < warp ? s_warp[w] : 0u;
        total += s_warp[w];
    }
    constexpr unsigned kAgg = 1u, kIncl = 2u;
    auto publish = [&](unsigned prefix) {
        if (tile > 0) rs_put(status + tile, kIncl, prefix + total);
        if ((long long)(tile + 1) * kCpTile >= n) *count = min(prefix + total, (unsigned)n);
    };
    if (warp == 0) {
        if (lane == 0) rs_put(status + tile, tile == 0 ? kIncl : kAgg, total);
        unsigned prefix = 0u;
        int t = tile - 1;
        for (int spins = 0; t >= 0;) {
            const unsigned long long w = t >= lane ? rs_get(status + (t - lane)) : (unsigned long long)kIncl << 32;
            const unsigned tag = (unsigned)(w >> 32);
            const unsigned incl = __ballot_sync(0xffffffffu, tag == kIncl);
            const unsigned wait = __ballot_sync(0xffffffffu, tag != kIncl && tag != kAgg);
            const int fi = incl ? __ffs(incl) - 1 : 32, fw = wait ? __ffs(wait) - 1 : 32;
            const int use = fi < fw ? fi + 1 : fw;   // words that count: up to the first running total
            prefix += warp_sum(lane < use ? (unsigned)w : 0u);
            t = fi < fw ? -1 : t - fw;
            if (fw < fi && ++spins > kRsSpin) break;
        }
        if (lane == 0) {
            s_late = t >= 0 ? 1u : 0u;
            s_before = t >= 0 ? 0u : prefix;
            if (t < 0) publish(prefix);
        }
    }
    __syncthreads();
    if (s_late) {   // a wait ran out: count the flags before the tile
        unsigned k = 0u;
        for (long long i = tid; i < (long long)tile * kCpTile; i += kCpT) k += is_set(flag[i]) ? 1u : 0u;
        k = warp_sum(k);
        if (lane == 0) atomicAdd(&s_before, k);
        __syncthreads();
        if (tid == 0) publish(s_before);
    }
    unsigned pos = s_before + before;
    while (set) {
        const int k = __ffs(set) - 1;
        set &= set - 1u;
        if (pos < (unsigned)n) list[pos] = (int32_t)(i0 + k);
        ++pos;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

#define GRID_CHECK(call)                                                                  \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) {                                                          \
            ctx->err = std::string("CUDA error in grid build: ") + cudaGetErrorString(e_); \
            grid_free(g);                                                                 \
            return e_ == cudaErrorMemoryAllocation ? SPH_ERR_OOM : SPH_ERR_CUDA;          \
        }                                                                                 \
    } while (0)

void grid_free(sph_grid* g) {
    if (!g) return;
    for (void* p : {g->arena, g->list_arena, g->bw_arena})
        if (p) cudaFree(p);
    delete g;
}

cudaError_t carve(void** base, const Part* parts, int n) {
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    size_t total = 0;
    for (int k = 0; k < n; ++k) total += up(parts[k].bytes);
    *base = nullptr;
    const cudaError_t e = cudaMalloc(base, total);
    if (e) return e;
    char* p = static_cast<char*>(*base);
    for (int k = 0; k < n; ++k) {
        *parts[k].ptr = p;
        p += up(parts[k].bytes);
    }
    return cudaSuccess;
}

static cudaError_t grid_fill(sph_grid* g, const void* pos, int f64, const float* mass, cudaStream_t s) {
    sph_ctx* ctx = g->ctx;
    const int n = (int)g->n, nb = g->n_boxes;
    const int blocks = (n + 255) / 256;
    // 7 passes: the sort starts from k2 and ends in (keys, perm)
    unsigned long long* keys = (unsigned long long*)g->keys;
    if (f64)
        k_quantize<double><<<blocks, 256, 0, s>>>((const double*)pos, mass, n, g->d_off, g->boxes, nb, g->box_bits,
                                                  g->xq, g->k2, ctx->counters);
    else
        k_quantize<float><<<blocks, 256, 0, s>>>((const float*)pos, mass, n, g->d_off, g->boxes, nb, g->box_bits,
                                                 g->xq, g->k2, ctx->counters);
    ++ctx->launches;
    static_assert(((63 + kRsBits - 1) / kRsBits) % 2 == 1, "an odd number of passes ends in (keys, perm)");
    const cudaError_t e =
        rs_sort(g->k2, keys, (unsigned*)g->perm, g->k2, g->v2, n, 63, g->rs_work, ctx->sm_count, s, &ctx->launches);
    if (e) return e;
    k_gather<<<blocks, 256, 0, s>>>(g->xq, n, g->posm, g->perm, g->rank);
    k_tree_low<<<dim3((g->max_leaves + kTreeT - 1) / kTreeT, nb), kTreeT, 0, s>>>(
        g->posm, g->boxes, g->node_lo, g->node_hi, g->node_c, g->node_e, g->posf);
    ctx->launches += 2;
    if (g->max_lev > kTreeLow) {
        k_tree_top<<<nb, kTreeTopT, 0, s>>>(g->boxes, g->node_lo, g->node_hi, g->node_c, g->node_e);
        ++ctx->launches;
    }
    return cudaGetLastError();
}

sph_status grid_build(sph_ctx* ctx, const void* pos, int f64, const float* mass, bool lists, const int64_t* offs,
                      const double* Ls, int nb, cudaStream_t s, sph_grid** out) {
    sph_grid* g = new sph_grid();
    g->ctx = ctx;
    g->device = ctx->device;
    const int n = (int)offs[nb];
    g->n = n;
    g->n_boxes = nb;
    int bb = 0;
    while ((1 << bb) < nb) ++bb;
    g->box_bits = bb;
    // implicit hierarchy layout, box-major, level-minor
    g->boxes_h.resize(nb);
    int node = 0, maxleaf = 0, maxlev = 0;
    for (int b = 0; b < nb; ++b) {
        BoxDesc& B = g->boxes_h[b];
        B = BoxDesc();
        B.off = offs[b];
        B.n = offs[b + 1] - offs[b];
        B.L = Ls[b];
        int cnt = (int)((B.n + kLeaf - 1) / kLeaf), lev = 0;
        while (true) {
            if (lev >= kMaxLev) { ctx->err = "box too large for the hierarchy"; delete g; return SPH_ERR_INVALID; }
            B.lvl_off[lev] = node;
            B.lvl_n[lev] = cnt;
            node += cnt;
            ++lev;
            if (cnt == 1) break;
            cnt = (cnt + kFan - 1) / kFan;
        }
        B.nlev = lev;
        B.sf = (float)std::ldexp(B.L, -32);
        B.S = 4294967296.0 / B.L;
        B.Hs = (float)B.S;
        int ex = 0;
        B.pow2 = std::frexp(B.L, &ex) == 0.5 ? 1 : 0;
        B.Lf = (float)B.L;
        B.wideL = 0.45f * B.Lf;
        const double cap = 0.5 * B.L * (1.0 - 1e-9);
        B.capu = (float)cap;
        if ((double)B.capu < cap) B.capu = std::nextafter(B.capu, INFINITY);
        maxlev = std::max(maxlev, lev);
        maxleaf = std::max(maxleaf, B.lvl_n[0]);
    }
    g->n_nodes = node;
    g->max_leaves = maxleaf;
    g->max_lev = maxlev;

    // One allocation for everything the grid holds, a second for the neighbour lists
    // (46 separate ones, and as many frees, took 3 ms of a 262k differentiable step).
    {
        const size_t N = (size_t)n, M = (size_t)node, mpw = (size_t)ctx->sm_count * kMpWarpsPerSm * kMpMembers;
        const Part parts[] = {
            {&g->boxes, sizeof(BoxDesc) * nb}, {&g->d_off, sizeof(long long) * (nb + 1)}, {&g->d_L, sizeof(double) * nb},
            // (padded: the gravity kernel reads whole leaves, the last one past its end)
            {&g->posm, sizeof(uint4) * (N + kLeaf)},
            {&g->xq, sizeof(uint4) * N}, {&g->perm, sizeof(int32_t) * N}, {&g->rank, sizeof(int32_t) * N},
            {&g->keys, sizeof(uint64_t) * N},
            {&g->node_lo, sizeof(uint4) * M}, {&g->node_hi, sizeof(uint4) * M}, {&g->node_hmax, sizeof(float) * M},
            {&g->node_c, sizeof(uint4) * M}, {&g->node_e, sizeof(float4) * M},
            {&g->posf, sizeof(float4) * N}, {&g->fvel, sizeof(float4) * N}, {&g->fthermo, sizeof(float4) * N},
            {&g->fposh, sizeof(float4) * N}, {&g->fvm, sizeof(float4) * N}, {&g->fbal, sizeof(float) * N},
            {&g->fcond, sizeof(float2) * N}, {&g->fvisc, sizeof(float2) * N},
            {&g->node_m, sizeof(float4) * M}, {&g->grav_box, (size_t)kGravBoxBytes * nb},
            // the near-list indices of the density pass's member-parallel path, one
            // block of kMpMembers x kMpCap per persistent warp
            {&g->mp_j, sizeof(int32_t) * mpw * kMpCap}, {&g->den_left, sizeof(int32_t) * N},
            {&g->act, sizeof(int32_t) * N}, {&g->flag, flag_bytes(n) + flag_work_bytes(n)}, {&g->act_n, sizeof(uint32_t)},
            {&g->list_a, sizeof(int32_t) * N}, {&g->list_b, sizeof(int32_t) * N},
            {&g->st_lo, sizeof(float) * N}, {&g->st_hi, sizeof(float) * N}, {&g->list_n, sizeof(int) * 2},
            {&g->k2, sizeof(unsigned long long) * N}, {&g->v2, sizeof(unsigned) * N}, {&g->rs_work, rs_work_bytes(n)}};
        GRID_CHECK(carve(&g->arena, parts));
        if (lists) {
            // Neighbour-list pools (int32 offsets: at most 2^31 - 2^12 entries each).
            // Lists are an optimisation: if they cannot be allocated the grid is
            // built without them and the force pass walks.
            const long long lim = (1ll << 31) - (1ll << 12);
            g->list_pool = (int64_t)std::min<long long>((long long)n * kListPool, lim);
            const Part lp[] = {
                {&g->nbr, sizeof(int32_t) * (size_t)g->list_pool}, {&g->nbr_off, sizeof(int32_t) * N},
                {&g->nbr_n, sizeof(int32_t) * N}, {&g->ext_n, sizeof(uint32_t) * N},
                {&g->ext, sizeof(int32_t) * N * kExtCap}, {&g->list_xh, sizeof(uint4) * N},
                {&g->list_st, sizeof(unsigned) * kListSt}, {&g->fb_list, sizeof(int32_t) * N},
                {&g->list_ep, sizeof(uint32_t) * N}, {&g->mp_x, sizeof(int32_t) * mpw * kMpFar}};
            if (carve(&g->list_arena, lp) == cudaSuccess) {
                GRID_CHECK(cudaMemsetAsync(g->list_st, 0, sizeof(unsigned) * kListSt, s));
                GRID_CHECK(cudaMemsetAsync(g->list_ep, 0, sizeof(uint32_t) * N, s));
            } else {
                (void)cudaGetLastError();
            }
        }
        GRID_CHECK(cudaMemsetAsync(g->node_e, 0, sizeof(float4) * M, s));
        GRID_CHECK(cudaMemsetAsync(g->act, 0, sizeof(int32_t) * N, s));
    }
    // (the host staging outlives the copies: the build ends with a synchronisation)
    std::vector<long long> offh(offs, offs + nb + 1);
    std::vector<double> Lh(Ls, Ls + nb);
    GRID_CHECK(cudaMemcpyAsync(g->boxes, g->boxes_h.data(), sizeof(BoxDesc) * nb, cudaMemcpyHostToDevice, s));
    GRID_CHECK(cudaMemcpyAsync(g->d_off, offh.data(), sizeof(long long) * (nb + 1), cudaMemcpyHostToDevice, s));
    GRID_CHECK(cudaMemcpyAsync(g->d_L, Lh.data(), sizeof(double) * nb, cudaMemcpyHostToDevice, s));
    GRID_CHECK(grid_fill(g, pos, f64, mass, s));
    GRID_CHECK(cudaStreamSynchronize(s));
    *out = g;
    return SPH_OK;
}

sph_status grid_update(sph_grid* g, const void* pos, int f64, const float* mass, cudaStream_t s) {
    g->lists_rec = false;   // the particles may have moved: recorded neighbour lists are stale
    const cudaError_t e = grid_fill(g, pos, f64, mass, s);
    if (e) {
        g->ctx->err = std::string("CUDA error in grid update: ") + cudaGetErrorString(e);
        return SPH_ERR_CUDA;
    }
    return SPH_OK;
}

void grid_refresh_hmax(sph_grid* g, const float* h, cudaStream_t s) {
    int nb = g->n_boxes;
    k_hmax_low<<<dim3((g->max_leaves + kTreeT - 1) / kTreeT, nb), kTreeT, 0, s>>>(g->perm, h, g->boxes, g->node_hmax,
                                                                              g->node_e);
    ++g->ctx->launches;
    if (g->max_lev > kTreeLow) {
        k_hmax_top<<<nb, kTreeTopT, 0, s>>>(g->boxes, g->node_hmax, g->node_e);
        ++g->ctx->launches;
    }
}

void flag_list(sph_grid* g, const uint8_t* flag, long long tick, int max_bin, int32_t* list, uint32_t* count,
               cudaStream_t s, const CallBegin& b) {
    const int n = (int)g->n;
    k_flag_list<<<(n + kCpTile - 1) / kCpTile, kCpT, 0, s>>>(flag, n, tick, max_bin,
                                                             (unsigned long long*)(g->flag + flag_bytes(n)), list, count,
                                                             b);
    ++g->ctx->launches;
}

void grid_active(sph_grid* g, const int32_t* active, int64_t n_active, cudaStream_t s, const CallBegin& b) {
    int n = (int)g->n;
    unsigned& nl = g->ctx->launches;
    if (!active) {
        k_iota_count<<<(n + 255) / 256, 256, 0, s>>>(g->act, n, g->act_n, b);
        ++nl;
    } else {
        cudaMemsetAsync(g->flag, 0, flag_bytes(n) + flag_work_bytes(n), s);   // flags and flag_list's words
        if (n_active > 0) {
            k_mark<<<(int)((n_active + 255) / 256), 256, 0, s>>>(active, (int)n_active, g->rank, g->flag, n,
                                                                  g->ctx->counters);
            ++nl;
        }
        if (b.ext_n) cudaMemsetAsync(b.ext_n, 0, sizeof(uint32_t) * n, s);
        flag_list(g, g->flag, 0, -1, g->act, g->act_n, s, b);
    }
}

}  // namespace sph
