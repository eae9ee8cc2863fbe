// Selection of the k seeds of lowest RSS (Sec. 2.1; top-k as in Sec. 3.1's ten best seeds per side).
//
// Order: ascending RSS, equal RSS by ascending seed index, NaN after every number.  With the index
// as tie-break every key is unique, so round r of a selection is simply "the smallest key greater
// than the key chosen in round r-1".
//
// Pass 1: each block selects the k smallest keys of a contiguous chunk of the RSS array into the
// scratch buffer.  Pass 2: one block selects among all blocks' candidates.  For the smallest k (select_how)
// that is k rounds of a block argmin (per-thread minimum, warp-shuffle reduction, then a shared-memory
// reduction over the warps), bound by the barriers' latency.  For larger k every warp keeps the 64 smallest
// keys it has seen as a sorted list, two per lane: 64 keys at a time are sorted by a bitonic network of
// shuffles and merged in, or skipped by one vote when none of them precedes the list's k-th; the warps'
// lists are then merged pairwise through shared memory: 13 us for any k up to 64 and 59,535 FP32 seeds,
// where 16 rounds take 52.  Deterministic: no atomics, fixed networks.
#include <float.h>
#include <stdint.h>

#include <mutex>

#include "device.cuh"
#include "internal.h"

namespace comet {

namespace {

constexpr int kSelThreads = 256;
constexpr int kChunk = 2048;
constexpr int64_t kNone = INT64_MAX;

template <typename T>
struct Key {
    T v;
    int64_t i;
};

// a < b in (NaN last, value, index) order; the "none" key (index kNone) is greater than all others.
template <typename T>
__device__ __forceinline__ bool key_less(const Key<T> &a, const Key<T> &b)
{
    if (a.i == kNone || b.i == kNone) return a.i < b.i;
    const bool an = isnan(a.v), bn = isnan(b.v);
    if (an != bn) return bn;
    if (!an && a.v != b.v) return a.v < b.v;
    return a.i < b.i;
}

template <typename T>
__device__ __forceinline__ Key<T> warp_min(Key<T> k)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        Key<T> o;
        o.v = __shfl_xor_sync(0xffffffffu, k.v, off);
        o.i = __shfl_xor_sync(0xffffffffu, k.i, off);
        if (key_less(o, k)) k = o;
    }
    return k;
}

// k rounds of block argmin over the keys produced by get(j) for j in [0, n), each the smallest key after the
// last round's (ONE: k = 1).  Thread 0 writes round r's key to out_v[r], out_i[r].
template <typename T, bool ONE, class Get>
__device__ void block_rounds(int64_t n, int k, Get get, T *out_v, int64_t *out_i)
{
    __shared__ Key<T> red[kSelThreads / 32];
    __shared__ Key<T> last;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int r = 0; r < (ONE ? 1 : k); ++r) {
        [[maybe_unused]] Key<T> lk{T(0), -1};   // below every key
        if constexpr (!ONE)
            if (r > 0) lk = last;
        Key<T> best{T(0), kNone};
        for (int64_t j = tid; j < n; j += kSelThreads) {
            const Key<T> c = get(j);
            const bool later = ONE || lk.i < 0 || key_less(lk, c);
            if (later && key_less(c, best)) best = c;
        }
        best = warp_min(best);
        if (lane == 0) red[wid] = best;
        __syncthreads();
        if (wid == 0) {
            Key<T> b = lane < kSelThreads / 32 ? red[lane] : Key<T>{T(0), kNone};
            b = warp_min(b);
            if (lane == 0) {
                out_v[r] = b.v;
                out_i[r] = b.i;
                if constexpr (!ONE) last = b;
            }
        }
        if constexpr (!ONE) __syncthreads();
    }
}

// Sort keys of the top-k path: an unsigned image of the value (ascending like the value, -0 as +0, NaN
// after every number) and the position of the candidate, which orders equal values.  Candidates stand in
// ascending seed order among equal values (chunk by chunk, and inside a chunk as pass 1 left them), so
// the position decides ties as the seed index does.  No candidate: all ones, after everything.
struct Key32 {
    unsigned long long k;   // image << 32 | position
};
struct Key64 {
    unsigned long long u;   // image
    uint32_t p;             // position
};
template <typename T>
struct SortKey;
template <>
struct SortKey<float> {
    using type = Key32;
};
template <>
struct SortKey<double> {
    using type = Key64;
};

__device__ __forceinline__ Key32 sort_key(float v, uint32_t pos)
{
    const uint32_t b = __float_as_uint(v == 0.f ? 0.f : v);
    const uint32_t u = v != v ? 0xffffffffu : ((b & 0x80000000u) ? ~b : (b | 0x80000000u));
    return Key32{((unsigned long long)u << 32) | pos};
}
__device__ __forceinline__ Key64 sort_key(double v, uint32_t pos)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v == 0.0 ? 0.0 : v);
    const unsigned long long u = v != v ? ~0ull : ((b >> 63) ? ~b : (b | (1ull << 63)));
    return Key64{u, pos};
}
__device__ __forceinline__ void set_none(Key32 &k) { k.k = ~0ull; }
__device__ __forceinline__ void set_none(Key64 &k)
{
    k.u = ~0ull;
    k.p = 0xffffffffu;
}
__device__ __forceinline__ bool less(Key32 a, Key32 b) { return a.k < b.k; }
__device__ __forceinline__ bool less(Key64 a, Key64 b) { return a.u != b.u ? a.u < b.u : a.p < b.p; }
__device__ __forceinline__ uint32_t position(Key32 k) { return (uint32_t)k.k; }
__device__ __forceinline__ uint32_t position(Key64 k) { return k.p; }
__device__ __forceinline__ Key32 shfl_xor(Key32 k, int m) { return Key32{__shfl_xor_sync(0xffffffffu, k.k, m)}; }
__device__ __forceinline__ Key64 shfl_xor(Key64 k, int m)
{
    return Key64{__shfl_xor_sync(0xffffffffu, k.u, m), __shfl_xor_sync(0xffffffffu, k.p, m)};
}
__device__ __forceinline__ Key32 shfl(Key32 k, int l) { return Key32{__shfl_sync(0xffffffffu, k.k, l)}; }
__device__ __forceinline__ Key64 shfl(Key64 k, int l)
{
    return Key64{__shfl_sync(0xffffffffu, k.u, l), __shfl_sync(0xffffffffu, k.p, l)};
}

// A list of 64 keys over a warp: element l in lane l's a, element 32 + l in its b.
template <typename K>
struct List64 {
    K a, b;
};

// One stage of a bitonic network over 64 keys: elements e and e ^ stride, ascending where up(e).
template <typename K, class Up>
__device__ __forceinline__ void bitonic_stage(List64<K> &x, int lane, int stride, Up up)
{
    if (stride == 32) {
        if (less(x.b, x.a) == up(lane)) {
            const K t = x.a;
            x.a = x.b;
            x.b = t;
        }
        return;
    }
    const K oa = shfl_xor(x.a, stride), ob = shfl_xor(x.b, stride);
    const bool low = (lane & stride) == 0;
    // the lower element of an ascending pair (the upper of a descending one) keeps the smaller key
    if (less(oa, x.a) == (low == up(lane))) x.a = oa;
    if (less(ob, x.b) == (low == up(lane + 32))) x.b = ob;
}

// Sorts 64 keys in descending order.
template <typename K>
__device__ __forceinline__ void sort_descending(List64<K> &x, int lane)
{
#pragma unroll
    for (int size = 2; size <= 64; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1)
            bitonic_stage(x, lane, stride, [&](int e) { return (e & size) != 0; });
}

// best <- the 64 smallest of best (ascending) and d (descending), ascending: the element-wise minimum of
// the two is bitonic.
template <typename K>
__device__ __forceinline__ void merge_smallest(List64<K> &best, const List64<K> &d, int lane)
{
    if (less(d.a, best.a)) best.a = d.a;
    if (less(d.b, best.b)) best.b = d.b;
#pragma unroll
    for (int stride = 32; stride > 0; stride >>= 1) bitonic_stage(best, lane, stride, [](int) { return true; });
}

// The k <= 64 smallest of n candidates val(j), j in [0, n): warp 0 returns them sorted (element r in
// lane r & 31's a or b), n < 2^32.  NW warps.
template <typename T, int NW, class Val>
__device__ List64<typename SortKey<T>::type> block_smallest(int64_t n, int k, Val val)
{
    using K = typename SortKey<T>::type;
    __shared__ K lists[NW / 2 > 0 ? NW / 2 : 1][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    List64<K> best;
    set_none(best.a);
    set_none(best.b);
    for (int64_t j0 = (int64_t)warp * 64; j0 < n; j0 += NW * 64) {
        List64<K> x;
        set_none(x.a);
        set_none(x.b);
        const int64_t ja = j0 + lane, jb = ja + 32;
        if (ja < n) x.a = sort_key(val(ja), (uint32_t)ja);
        if (jb < n) x.b = sort_key(val(jb), (uint32_t)jb);
        const K kth = shfl(k > 32 ? best.b : best.a, (k - 1) & 31);
        if (!__any_sync(0xffffffffu, less(x.a, kth) || less(x.b, kth))) continue;
        sort_descending(x, lane);
        merge_smallest(best, x, lane);
    }
#pragma unroll
    for (int half = NW / 2; half > 0; half >>= 1) {
        __syncthreads();
        if (warp >= half && warp < 2 * half) {
            lists[warp - half][lane] = best.a;
            lists[warp - half][lane + 32] = best.b;
        }
        __syncthreads();
        if (warp < half) {
            const List64<K> o{lists[warp][63 - lane], lists[warp][31 - lane]};
            merge_smallest(best, o, lane);
        }
    }
    return best;
}

enum Select { kOne, kRounds, kLists };   // k = 1; a few rounds of block argmin; sorted lists

constexpr int kMaxRounds = 3;
constexpr int kSel2Threads = 1024;   // pass 2 over lists: one block, as many warps as it can have

// Rounds are faster than the lists' sorting networks for the smallest k (rounds and lists, both passes,
// 59,535 seeds: FP32 k = 2 8.2 and 13.1 us, 3 11.2 and 12.8, 4 13.8 and 12.0; FP64 k = 2 20.5 and 20.0,
// but 256 seeds 11.0 and 12.7, 2^18 23.0 and 20.7).
template <typename T>
static Select select_how(int k, int n_blocks)
{
    if (k == 1) return kOne;
    if (sizeof(T) == 4) return k <= kMaxRounds ? kRounds : kLists;
    return k == 2 && n_blocks == 1 ? kRounds : kLists;
}

template <typename T, Select HOW>
__global__ void __launch_bounds__(kSelThreads) select_pass1(const T *__restrict__ rss, int64_t S,
                                                            int k, T *pv, int64_t *pi)
{
    const int64_t b0 = (int64_t)blockIdx.x * kChunk;
    const int64_t n = min((int64_t)kChunk, S - b0);
    pv += (int64_t)blockIdx.x * k;
    pi += (int64_t)blockIdx.x * k;
    if constexpr (HOW != kLists) {
        block_rounds<T, HOW == kOne>(n, k, [&](int64_t j) { return Key<T>{rss[b0 + j], b0 + j}; }, pv, pi);
    } else {
        const auto best = block_smallest<T, kSelThreads / 32>(n, k, [&](int64_t j) { return rss[b0 + j]; });
        const int lane = threadIdx.x;
        if (lane >= 32) return;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = lane + 32 * h;
            const uint32_t j = position(h ? best.b : best.a);
            if (r < k) {
                pv[r] = j < n ? rss[b0 + j] : T(0);
                pi[r] = j < n ? b0 + j : kNone;
            }
        }
    }
}

template <typename T, Select HOW>
__global__ void __launch_bounds__(HOW == kLists ? kSel2Threads : kSelThreads)
    select_pass2(const T *__restrict__ pv, const int64_t *__restrict__ pi, int64_t n, int k, int64_t *idx_out,
                 T *rss_out)
{
    if constexpr (HOW != kLists) {
        __shared__ T ov[kMaxRounds];
        __shared__ int64_t oi[kMaxRounds];
        block_rounds<T, HOW == kOne>(n, k, [&](int64_t j) { return Key<T>{pv[j], pi[j]}; }, ov, oi);
        if (threadIdx.x == 0)   // which wrote them
            for (int r = 0; r < (HOW == kOne ? 1 : k); ++r) {
                idx_out[r] = oi[r];
                if (rss_out) rss_out[r] = ov[r];
            }
    } else {
        // places that pass 1 left empty (the last chunk shorter than k) stand after every candidate and
        // are never among the k <= S smallest; as NaN they sort after every number, and after every
        // NaN by their position
        const auto best = block_smallest<T, kSel2Threads / 32>(n, k, [&](int64_t j) {
            return pi[j] == kNone ? (T)NAN : pv[j];
        });
        const int lane = threadIdx.x;
        if (lane >= 32) return;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = lane + 32 * h;
            const uint32_t j = position(h ? best.b : best.a);
            if (r < k) {
                idx_out[r] = pi[j];
                if (rss_out) rss_out[r] = pv[j];
            }
        }
    }
}

// A batch (k = 1): pass 1 block b serves the chunk batch_find gives inside its event; pass 2 block e
// serves event e.  Each event's partial results live at its SelArgs.scratch (ids first, then values).
template <typename T>
__global__ void __launch_bounds__(kSelThreads) select_pass1_batch(BatchLaunch L)
{
    int e;
    int64_t lb;
    if (!batch_find(L.sel_start, L.B, blockIdx.x, e, lb)) return;
    const SelArgs a = L.ev[e].sel;
    int64_t *pi = (int64_t *)a.scratch;
    T *pv = (T *)(pi + a.n_blocks);
    const T *__restrict__ rss = (const T *)a.rss;
    const int64_t b0 = lb * kChunk;
    const int64_t n = min((int64_t)kChunk, a.S - b0);
    block_rounds<T, true>(n, 1, [&](int64_t j) { return Key<T>{rss[b0 + j], b0 + j}; }, pv + lb, pi + lb);
}

template <typename T>
__global__ void __launch_bounds__(kSelThreads) select_pass2_batch(BatchLaunch L)
{
    if ((int)blockIdx.x >= L.B) return;
    const SelArgs a = L.ev[blockIdx.x].sel;
    if (a.S <= 0) return;
    const int64_t *pi = (const int64_t *)a.scratch;
    const T *pv = (const T *)(pi + a.n_blocks);
    __shared__ T ov;
    __shared__ int64_t oi;
    block_rounds<T, true>(a.n_blocks, 1, [&](int64_t j) { return Key<T>{pv[j], pi[j]}; }, &ov, &oi);
    if (threadIdx.x == 0) {
        *a.idx_out = oi;
        if (a.rss_out) *(T *)a.rss_out = ov;
    }
}

} // namespace

cudaError_t launch_select_batch(comet_dtype dt, const BatchLaunch &L, cudaStream_t st)
{
    if (L.B == 0) return cudaSuccess;
    if (dt == COMET_F32) {
        if (L.sel_blocks) select_pass1_batch<float><<<L.sel_blocks, kSelThreads, 0, st>>>(L);
        select_pass2_batch<float><<<(unsigned)L.B, kSelThreads, 0, st>>>(L);
    } else {
        if (L.sel_blocks) select_pass1_batch<double><<<L.sel_blocks, kSelThreads, 0, st>>>(L);
        select_pass2_batch<double><<<(unsigned)L.B, kSelThreads, 0, st>>>(L);
    }
    return cudaGetLastError();
}

int select_chunk() { return kChunk; }

size_t select_scratch_bytes(comet_dtype dt, int64_t S, int k, int *n_blocks)
{
    const int64_t nb = (S + kChunk - 1) / kChunk;
    *n_blocks = (int)nb;
    const size_t es = dt == COMET_F32 ? sizeof(float) : sizeof(double);
    return (size_t)nb * k * (es + sizeof(int64_t)) + 64;
}

template <typename T, Select HOW>
static void sel_launch_how(const SelArgs &a, cudaStream_t st)
{
    const int nb = a.n_blocks;
    int64_t *pi = (int64_t *)a.scratch;
    T *pv = (T *)(pi + (int64_t)nb * a.k);
    select_pass1<T, HOW><<<nb, kSelThreads, 0, st>>>((const T *)a.rss, a.S, a.k, pv, pi);
    select_pass2<T, HOW><<<1, HOW == kLists ? kSel2Threads : kSelThreads, 0, st>>>(pv, pi, (int64_t)nb * a.k, a.k,
                                                                                  a.idx_out, (T *)a.rss_out);
}

template <typename T>
static void sel_launch(const SelArgs &a, cudaStream_t st)
{
    switch (select_how<T>(a.k, a.n_blocks)) {
    case kOne: sel_launch_how<T, kOne>(a, st); break;
    case kRounds: sel_launch_how<T, kRounds>(a, st); break;
    default: sel_launch_how<T, kLists>(a, st); break;
    }
}

// Scratch of comet_scan_select_noalloc: one file-scope device array per device that loads the
// library, held until the process exits.  In host code `g_select_scratch` is only a host-side
// stand-in for the symbol, never a device address: the device address is looked up once per device
// with cudaGetSymbolAddress, with that device current, and cached here.
static __device__ __align__(256) unsigned char g_select_scratch[kStaticSelectScratchBytes];

cudaError_t static_select_scratch(void **ptr)
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static void *addr[kMaxDevices] = {};
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_select_scratch);
        if (e != cudaSuccess) return e;
        addr[dev] = p;
    }
    *ptr = addr[dev];
    return cudaSuccess;
}

cudaError_t kernel_binary_version(int *version)
{
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, select_pass1<float, kOne>);
    if (e == cudaSuccess) *version = fa.binaryVersion;
    return e;
}

cudaError_t launch_select(comet_dtype dt, const SelArgs &a, cudaStream_t st)
{
    if (dt == COMET_F32)
        sel_launch<float>(a, st);
    else
        sel_launch<double>(a, st);
    return cudaGetLastError();
}

} // namespace comet
