// Many-to-many overlap seeding before the extension: the step that the
// paper's application (Sec. V) runs to find read pairs worth extending and
// a seed for each, and the adaptive threshold applied to the extension
// score.  The paper gives these steps in words only; the definitions here:
//   k-mer codes   base codes A0 C1 G2 T3; forward code of the k-mer at p =
//                 sum_t c[p+t] << 2t; reverse complement sum_t (3 - c[p+k-1-t])
//                 << 2t; canonical = the smaller, strand 1 when the reverse
//                 complement is strictly smaller (k <= 31)
//   reliable      min_freq <= occurrences of the canonical code <= max_freq
//   hits          two occurrences of a reliable k-mer in reads a < b:
//                 (a, b, strand_a ^ strand_b, pos_a, pos_b)
//   candidates    (a, b, o) with >= min_shared hits; the seed is the hit at
//                 index count / 2 in (pos_a, pos_b) order
//   threshold     keep when score * den >= ratio_num * L - delta * den, L the
//                 overlap the seed's diagonal implies
// Sorting runs on CUB radix sorts (library primitives; stable, so equal
// keys keep the order of their input); every other step is a kernel here.
#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>
#include <cub/device/device_select.cuh>

#include <algorithm>
#include <cstdint>
#include <utility>
#include <vector>

#include "ctx_ext.h"
#include "internal.h"

#include "../../include/logan.h"

namespace logan {

namespace {

constexpr int kThreads = 256;

inline unsigned blocks_for(uint64_t n, unsigned t = kThreads) {
    return unsigned(std::min<uint64_t>((n + t - 1) / t, 1u << 20));
}

inline int bit_width(uint64_t v) {
    int b = 0;
    while (v >> b) ++b;
    return b;
}

// 2k bits of codes starting at pool position P (code of P in the low bits)
__device__ __forceinline__ uint64_t codes_at(const uint32_t* __restrict__ w, uint64_t P, int k) {
    const uint64_t i0 = P >> 4;
    const uint32_t sh = uint32_t(P & 15) * 2u;
    const uint64_t lo = uint64_t(__ldg(w + i0)) | (uint64_t(__ldg(w + i0 + 1)) << 32);
    uint64_t v = lo >> sh;
    if (sh && sh + 2u * k > 64u) v |= uint64_t(__ldg(w + i0 + 2)) << (64u - sh);
    return k == 32 ? v : (v & ((1ull << (2 * k)) - 1ull));
}

__device__ __forceinline__ uint64_t revcomp_code(uint64_t f, int k) {
    uint64_t v = __brevll(~f);
    v = ((v >> 1) & 0x5555555555555555ull) | ((v & 0x5555555555555555ull) << 1);
    return v >> (64 - 2 * k);
}

// k-mer positions per read (0 when the read is shorter than k)
__global__ void k_kmer_counts(const uint32_t* __restrict__ len, uint32_t n, int k,
                              uint64_t* __restrict__ cnt) {
    for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x)
        cnt[r] = len[r] >= uint32_t(k) ? uint64_t(len[r] - k + 1) : 0ull;
}

// Occurrence i (in (read, pos) order) belongs to the last read r with
// first[r] <= i (reads without k-mers share their start with the next one).
// cell[c] is the read of occurrence c << shift, so the search covers the few
// reads that start inside a cell.
struct ReadIndex {
    const uint64_t* first;  // n_reads + 1 entries
    const uint32_t* cell;   // (n_occurrences >> shift) + 2 entries
    int shift;
    __device__ __forceinline__ uint32_t find(uint64_t i) const {
        uint32_t lo = __ldg(cell + (i >> shift)), hi = __ldg(cell + (i >> shift) + 1) + 1u;
        while (hi - lo > 1u) {  // first[lo] <= i < first[hi]
            const uint32_t mid = lo + ((hi - lo) >> 1);
            if (__ldg(first + mid) <= i) lo = mid;
            else hi = mid;
        }
        return lo;
    }
};

__global__ void k_read_cells(const uint64_t* __restrict__ first, uint32_t n_reads, uint64_t nk,
                             int shift, uint64_t n_cells, uint32_t* __restrict__ cell) {
    for (uint64_t c = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; c < n_cells;
         c += uint64_t(gridDim.x) * blockDim.x) {
        const uint64_t i = min(c << shift, nk - 1);
        uint32_t lo = 0, hi = n_reads;
        while (hi - lo > 1u) {
            const uint32_t mid = lo + ((hi - lo) >> 1);
            if (first[mid] <= i) lo = mid;
            else hi = mid;
        }
        cell[c] = lo;
    }
}

constexpr int kPerThread = 8;
constexpr int kTile = kThreads * kPerThread;
constexpr int kMaxClasses = 16;

struct KmerArgs {
    const uint32_t* w;
    const uint64_t* off;
    ReadIndex ix;
    uint64_t nk;
    int k;
};

// canonical code and strand of occurrence i
__device__ __forceinline__ uint64_t kmer_of(const KmerArgs& a, uint64_t i, uint32_t& strand) {
    const uint32_t r = a.ix.find(i);
    const uint64_t f = codes_at(a.w, __ldg(a.off + r) + (i - __ldg(a.ix.first + r)), a.k);
    const uint64_t rc = revcomp_code(f, a.k);
    strand = rc < f ? 1u : 0u;
    return rc < f ? rc : f;
}

// Occurrence of the tile that thread t's j-th turn takes: a warp's turns are
// consecutive, so a tile's order is (warp, turn, lane).
__device__ __forceinline__ uint64_t tile_item(uint64_t tile, int j) {
    return tile * kTile + uint64_t(threadIdx.x >> 5) * (32 * kPerThread) + 32 * j +
           (threadIdx.x & 31u);
}

// k-mers of each tile per class (the code's bits above the low 32)
__global__ void __launch_bounds__(kThreads)
    k_kmer_classes(KmerArgs a, int classes, uint64_t tiles, uint64_t* __restrict__ at) {
    __shared__ uint32_t cnt[kMaxClasses];
    if (threadIdx.x < kMaxClasses) cnt[threadIdx.x] = 0u;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) {
        const uint64_t i = tile_item(blockIdx.x, j);
        uint32_t c = 0xffffffffu, strand;
        if (i < a.nk) c = uint32_t(kmer_of(a, i, strand) >> 32);
        const uint32_t m = __match_any_sync(0xffffffffu, c);
        if (c < uint32_t(classes) && int(threadIdx.x & 31u) == __ffs(m) - 1)
            atomicAdd(&cnt[c], uint32_t(__popc(m)));
    }
    __syncthreads();
    if (threadIdx.x < uint32_t(classes)) at[threadIdx.x * tiles + blockIdx.x] = cnt[threadIdx.x];
}

// (key, occurrence << 1 | strand) of every k-mer, class by class, each class in
// occurrence order (a stable partition).  Sorting 32-bit keys class by class
// moves 16 bytes per k-mer and pass where 64-bit keys with read and position
// moved 32, in one pass less; read and position are looked up again only
// for the occurrences that make hits.
template <typename K, typename V>
__global__ void __launch_bounds__(kThreads)
    k_kmer_emit(KmerArgs a, int classes, uint64_t tiles, const uint64_t* __restrict__ at,
                K* __restrict__ keys, V* __restrict__ vals) {
    __shared__ uint32_t cnt[kThreads / 32][kMaxClasses];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane < kMaxClasses) cnt[w][lane] = 0u;
    __syncwarp();
    K key[kPerThread];
    uint32_t cls[kPerThread], rank[kPerThread], strand[kPerThread];
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) {
        const uint64_t i = tile_item(blockIdx.x, j);
        uint64_t code = 0ull;
        strand[j] = 0u;
        if (i < a.nk) code = kmer_of(a, i, strand[j]);
        key[j] = K(code);
        cls[j] = sizeof(K) == 4 ? uint32_t(code >> 32) : 0u;
        if (classes > 1) {
            if (i >= a.nk) cls[j] = kMaxClasses;
            const uint32_t m = __match_any_sync(0xffffffffu, cls[j]);
            const uint32_t below = uint32_t(__popc(m & ((1u << lane) - 1u)));
            const uint32_t base = cls[j] < kMaxClasses ? cnt[w][cls[j]] : 0u;
            rank[j] = base + below;
            __syncwarp();
            if (below == 0u && cls[j] < kMaxClasses) cnt[w][cls[j]] = base + uint32_t(__popc(m));
            __syncwarp();
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) {
        const uint64_t i = tile_item(blockIdx.x, j);
        if (i >= a.nk) continue;
        uint64_t o = i;
        if (classes > 1) {
            o = at[cls[j] * tiles + blockIdx.x] + rank[j];
            for (int t = 0; t < w; ++t) o += cnt[t][cls[j]];
        }
        keys[o] = key[j];
        vals[o] = V((i << 1) | strand[j]);
    }
}

// Length of the run of equal keys that starts at i, 0 when i is not a run's
// start or the code is not reliable.  Most codes of reads with errors occur
// once, so a thread mostly reads its key and the two beside it (of lines
// that its neighbours read too) and is done; no run is walked past fmax + 1.
template <typename K>
__device__ __forceinline__ uint32_t reliable_run(const K* __restrict__ keys, uint64_t n, uint64_t i,
                                                 uint32_t fmin, uint32_t fmax) {
    const K key = keys[i];
    if (i > 0 && keys[i - 1] == key) return 0u;
    uint32_t f = 1;
    while (f <= fmax && i + f < n && keys[i + f] == key) ++f;
    return f >= fmin && f <= fmax ? f : 0u;
}

// exclusive prefix of v over the block, and its total
__device__ __forceinline__ uint64_t block_prefix(uint64_t v, uint64_t* warp_sum, uint64_t& all) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint64_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) warp_sum[w] = incl;
    __syncthreads();
    uint64_t before = 0ull;
    all = 0ull;
#pragma unroll
    for (int t = 0; t < kThreads / 32; ++t) {
        if (t < w) before += warp_sum[t];
        all += warp_sum[t];
    }
    return before + incl - v;
}

// The reliable runs among the sorted keys [0, n) of one class, as (place << 11 |
// length), places counted from `base`, appended to runs in no particular
// order.  One pass over the keys (flags, scan, scatter, run lengths and a
// scan over all run starts moved ten times as much).
template <typename K>
__global__ void __launch_bounds__(kThreads)
    k_find_runs(const K* __restrict__ keys, uint64_t n, uint64_t base, uint32_t fmin, uint32_t fmax,
                unsigned long long* __restrict__ n_runs, uint64_t* __restrict__ runs) {
    __shared__ uint64_t warp_sum[kThreads / 32];
    __shared__ unsigned long long at;
    uint32_t run[kPerThread];
    uint32_t mine = 0u;
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) {
        const uint64_t i = uint64_t(blockIdx.x) * kTile + uint64_t(j) * kThreads + threadIdx.x;
        run[j] = i < n ? reliable_run(keys, n, i, fmin, fmax) : 0u;
        mine += run[j] ? 1u : 0u;
    }
    uint64_t all;
    const uint64_t before = block_prefix(mine, warp_sum, all);
    if (threadIdx.x == 0 && all) at = atomicAdd(n_runs, all);
    __syncthreads();
    if (!mine) return;
    uint64_t o = at + before;
#pragma unroll
    for (int j = 0; j < kPerThread; ++j)
        if (run[j]) {
            const uint64_t i = uint64_t(blockIdx.x) * kTile + uint64_t(j) * kThreads + threadIdx.x;
            runs[o++] = ((base + i) << 11) | run[j];
        }
}

// Hits of the reliable runs, a thread per run: pairs of occurrences in different
// reads (a run is in (read, pos) order, so read_i <= read_j).  EMIT = false:
// the block's number of hits; EMIT = true: the hits from the block's place on.
// COMPOSITE: hit key (read a, read b, o, pos_a) and 32-bit value pos_b; else
// key (read a, read b, o), value (pos_a, pos_b).
template <typename V, typename H, bool EMIT, bool COMPOSITE>
__global__ void __launch_bounds__(kThreads)
    k_run_hits(const uint64_t* __restrict__ runs, uint64_t n_runs, const V* __restrict__ vals,
               ReadIndex ix, int rb, int pb, uint64_t* __restrict__ block_hits,
               uint64_t* __restrict__ hk, H* __restrict__ hv) {
    __shared__ uint64_t warp_sum[kThreads / 32];
    const uint64_t t = uint64_t(blockIdx.x) * kThreads + threadIdx.x;
    const uint64_t run = t < n_runs ? runs[t] : 0ull;
    const uint32_t f = uint32_t(run & 2047u);
    const V* v = vals + (run >> 11);
    uint64_t mine = 0ull;
    for (uint32_t a = 0; a + 1 < f; ++a) {
        // occurrences are in order: those of other reads follow the end of a's read
        const uint64_t end = __ldg(ix.first + ix.find(uint64_t(v[a]) >> 1) + 1);
        for (uint32_t b = a + 1; b < f; ++b) mine += (uint64_t(v[b]) >> 1) >= end ? 1 : 0;
    }
    uint64_t all;
    const uint64_t before = block_prefix(mine, warp_sum, all);
    if constexpr (!EMIT) {
        if (threadIdx.x == 0) block_hits[blockIdx.x] = all;
    } else {
        uint64_t o = block_hits[blockIdx.x] + before;
        for (uint32_t a = 0; mine && a + 1 < f; ++a) {
            const uint64_t va = v[a], ia = va >> 1;
            const uint64_t ra = ix.find(ia);
            const uint64_t fa = __ldg(ix.first + ra), end = __ldg(ix.first + ra + 1);
            for (uint32_t b = a + 1; b < f; ++b) {
                const uint64_t vb = v[b], ib = vb >> 1;
                if (ib < end) continue;
                const uint64_t rb_ = ix.find(ib);
                const uint64_t pair = (ra << (rb + 1)) | (rb_ << 1) | ((va ^ vb) & 1ull);
                const uint64_t pa = ia - fa, pbv = ib - __ldg(ix.first + rb_);
                hk[o] = COMPOSITE ? (pair << pb) | pa : pair;
                hv[o] = COMPOSITE ? H(pbv) : H((pa << pb) | pbv);
                ++o;
            }
        }
    }
}

// 1 where a run of equal keys (above their low `shift` bits) starts (flag[n] =
// 0 pads the scan)
__global__ void k_head_flags(const uint64_t* __restrict__ keys, uint64_t n, int shift,
                             uint64_t* __restrict__ flag) {
    for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i <= n;
         i += uint64_t(gridDim.x) * blockDim.x)
        flag[i] = (i < n && (i == 0 || (keys[i] >> shift) != (keys[i - 1] >> shift))) ? 1ull : 0ull;
}

// starts[rank[i]] = i for every run head i
__global__ void k_head_scatter(const uint64_t* __restrict__ flag, const uint64_t* __restrict__ rank,
                               uint64_t n, uint64_t* __restrict__ starts) {
    for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < n;
         i += uint64_t(gridDim.x) * blockDim.x)
        if (flag[i]) starts[rank[i]] = i;
}

// Per (a, b, o) segment of the sorted hits: its middle hit in (pos_a, pos_b)
// order, kept when the segment has at least min_shared hits.  COMPOSITE: the
// hits are ordered by pos_a only; those that share the middle one's pos_a (the
// occurrences of one code in read b, at most max_freq) are ranked by pos_b
// here.
template <typename H, bool COMPOSITE>
__global__ void k_segment_pick(const uint64_t* __restrict__ starts, uint64_t n_seg, uint64_t n,
                               const uint64_t* __restrict__ hk, const H* __restrict__ hv, int rb,
                               int pb, uint32_t min_shared, logan_candidate_t* __restrict__ cand,
                               uint8_t* __restrict__ keep) {
    for (uint64_t j = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; j < n_seg;
         j += uint64_t(gridDim.x) * blockDim.x) {
        const uint64_t s = starts[j], e = j + 1 < n_seg ? starts[j + 1] : n;
        const uint64_t cnt = e - s, m = s + cnt / 2;
        const uint64_t key = COMPOSITE ? hk[m] >> pb : hk[m];
        const uint64_t low = (1ull << pb) - 1ull;
        logan_candidate_t c;
        c.a = uint32_t(key >> (rb + 1));
        c.b = uint32_t((key >> 1) & ((1ull << rb) - 1ull));
        c.o = uint32_t(key & 1ull);
        if constexpr (COMPOSITE) {
            uint64_t l = m, r = m + 1;
            while (l > s && hk[l - 1] == hk[m]) --l;
            while (r < e && hk[r] == hk[m]) ++r;
            H pick = hv[m];
            for (uint64_t x = l; r - l > 1 && x < r; ++x) {  // the (m - l)-th smallest of [l, r)
                uint64_t less = 0, same = 0;
                for (uint64_t y = l; y < r; ++y) {
                    less += hv[y] < hv[x] ? 1 : 0;
                    same += hv[y] == hv[x] ? 1 : 0;
                }
                if (less <= m - l && m - l < less + same) pick = hv[x];
            }
            c.pos_a = uint32_t(hk[m] & low);
            c.pos_b = uint32_t(pick);
        } else {
            c.pos_a = uint32_t(hv[m] >> pb);
            c.pos_b = uint32_t(hv[m] & low);
        }
        c.count = uint32_t(cnt);
        cand[j] = c;
        keep[j] = cnt >= min_shared ? 1 : 0;
    }
}

// the reverse complement of every read, 16-base aligned after the forward
// pool's words: thread per output word
__global__ void k_revcomp_pool(const uint32_t* __restrict__ w, const uint64_t* __restrict__ off,
                               const uint32_t* __restrict__ len, uint32_t n,
                               const uint64_t* __restrict__ word_first, uint64_t fwd_words,
                               uint32_t* __restrict__ out, uint64_t* __restrict__ out_off) {
    for (uint32_t r = blockIdx.y; r < n; r += gridDim.y) {
        const uint64_t nw = (uint64_t(len[r]) + 15) / 16;
        if (blockIdx.x == 0 && threadIdx.x == 0) out_off[r] = (fwd_words + word_first[r]) * 16;
        for (uint64_t q = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; q < nw;
             q += uint64_t(gridDim.x) * blockDim.x) {
            uint32_t word = 0u;
            for (uint32_t t = 0; t < 16; ++t) {
                const uint64_t i = q * 16 + t;  // base i of the reverse complement
                if (i < len[r]) {
                    const uint32_t c = code_at(w, off[r] + len[r] - 1 - i);
                    word |= (3u - c) << (2 * t);
                }
            }
            out[fwd_words + word_first[r] + q] = word;
        }
    }
}

__global__ void k_overlap_seeds(const logan_candidate_t* __restrict__ c, uint64_t n,
                                const uint32_t* __restrict__ len, uint32_t n_reads, int k,
                                logan_seed_t* __restrict__ seeds) {
    for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < n;
         i += uint64_t(gridDim.x) * blockDim.x) {
        const logan_candidate_t x = c[i];
        logan_seed_t s;
        s.idxA = x.a;
        s.idxB = x.o ? n_reads + x.b : x.b;
        s.posA = x.pos_a;
        s.posB = x.o ? len[x.b] - x.pos_b - uint32_t(k) : x.pos_b;
        s.len = uint32_t(k);
        seeds[i] = s;
    }
}

__global__ void k_overlap_keep(const logan_result_t* __restrict__ res,
                               const logan_seed_t* __restrict__ seeds, uint64_t n,
                               const uint32_t* __restrict__ lenA, const uint32_t* __restrict__ lenB,
                               int64_t ratio_num, int64_t den, int64_t delta,
                               uint8_t* __restrict__ keep) {
    for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < n;
         i += uint64_t(gridDim.x) * blockDim.x) {
        const logan_seed_t s = seeds[i];
        const int64_t la = lenA[s.idxA], lb = lenB[s.idxB];
        const int64_t pa = s.posA, pbv = s.posB, k = s.len;
        const int64_t L = min(pa, pbv) + k + min(la - pa - k, lb - pbv - k);
        keep[i] = (res[i].status == 0 && int64_t(res[i].score) * den >= ratio_num * L - delta * den)
                      ? 1
                      : 0;
    }
}

// stream-ordered scratch that frees itself
struct Scratch {
    cudaStream_t s;
    cudaMemPool_t pool;  // the context's scratch pool (null: the default one)
    std::vector<void*> ptrs;
    bool ok = true;
    Scratch(cudaStream_t st, cudaMemPool_t p) : s(st), pool(p) {}
    template <typename T>
    T* get(size_t n) {
        void* p = nullptr;
        const size_t bytes = std::max<size_t>(n, 1) * sizeof(T);
        if (!ok || (pool ? cudaMallocFromPoolAsync(&p, bytes, pool, s)
                         : cudaMallocAsync(&p, bytes, s)) != cudaSuccess) {
            ok = false;
            return nullptr;
        }
        ptrs.push_back(p);
        return static_cast<T*>(p);
    }
    ~Scratch() {
        for (void* p : ptrs) cudaFreeAsync(p, s);
    }
};

// Start index of every run of equal keys (above their low `shift` bits) in
// keys[0, n) (sorted); returns
// the number of runs (synchronises the stream), or -1 on failure.
int64_t run_heads(Scratch& sc, const uint64_t* keys, uint64_t n, int shift, uint64_t*& starts) {
    cudaStream_t s = sc.s;
    uint64_t* flag = sc.get<uint64_t>(n + 1);
    uint64_t* rank = sc.get<uint64_t>(n + 1);
    starts = sc.get<uint64_t>(n);
    size_t tb = 0;
    cub::DeviceScan::ExclusiveSum(nullptr, tb, flag, rank, n + 1, s);
    void* tmp = sc.get<char>(tb);
    if (!sc.ok) return -1;
    k_head_flags<<<blocks_for(n + 1), kThreads, 0, s>>>(keys, n, shift, flag);
    cub::DeviceScan::ExclusiveSum(tmp, tb, flag, rank, n + 1, s);
    k_head_scatter<<<blocks_for(n), kThreads, 0, s>>>(flag, rank, n, starts);
    uint64_t nr = 0;
    if (cudaMemcpyAsync(&nr, rank + n, sizeof(uint64_t), cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return -1;
    return int64_t(nr);
}

// exclusive prefix of v[0, n) (v[n] is set to 0), *total = its sum when asked
bool prefix(Scratch& sc, uint64_t* v, uint64_t n, uint64_t*& out, uint64_t* total) {
    out = sc.get<uint64_t>(n + 1);
    size_t tb = 0;
    cub::DeviceScan::ExclusiveSum(nullptr, tb, v, out, n + 1, sc.s);
    void* tmp = sc.get<char>(tb);
    if (!sc.ok) return false;
    cudaMemsetAsync(v + n, 0, sizeof(uint64_t), sc.s);
    cub::DeviceScan::ExclusiveSum(tmp, tb, v, out, n + 1, sc.s);
    return !total || cudaMemcpyAsync(total, out + n, sizeof(uint64_t), cudaMemcpyDeviceToHost,
                                     sc.s) == cudaSuccess;
}

// The hits of the runs, sorted by (a, b, o), then position; their (a, b, o)
// segments' middle hits, compacted: candidates `kept`, `nkept` of them.
template <typename V, typename H, bool COMPOSITE>
int candidates_of(Scratch& sc, const uint64_t* runs, uint64_t n_runs, const V* vals, ReadIndex ix,
                  int rb, int pb, uint32_t min_shared, logan_candidate_t*& kept, uint64_t& nkept) {
    cudaStream_t s = sc.s;
    const uint64_t blocks = (n_runs + kThreads - 1) / kThreads;
    uint64_t* block_hits = sc.get<uint64_t>(blocks + 1);
    uint64_t* block_at = nullptr;
    if (!sc.ok) return LOGAN_ENOMEM;
    k_run_hits<V, H, false, COMPOSITE><<<unsigned(blocks), kThreads, 0, s>>>(
        runs, n_runs, vals, ix, rb, pb, block_hits, nullptr, nullptr);
    uint64_t nh = 0;
    if (!prefix(sc, block_hits, blocks, block_at, &nh)) return sc.ok ? LOGAN_ECUDA : LOGAN_ENOMEM;
    if (cudaStreamSynchronize(s) != cudaSuccess) return LOGAN_ECUDA;
    if (nh == 0) return LOGAN_OK;
    uint64_t* hk = sc.get<uint64_t>(nh);
    uint64_t* hk2 = sc.get<uint64_t>(nh);
    H* hv = sc.get<H>(nh);
    H* hv2 = sc.get<H>(nh);
    if (!sc.ok) return LOGAN_ENOMEM;
    k_run_hits<V, H, true, COMPOSITE><<<unsigned(blocks), kThreads, 0, s>>>(
        runs, n_runs, vals, ix, rb, pb, block_at, hk, hv);
    const int key_bits = COMPOSITE ? 2 * rb + 1 + pb : 2 * rb + 1;
    size_t t0 = 0, t1 = 0;
    if constexpr (COMPOSITE) {
        cub::DeviceRadixSort::SortPairs(nullptr, t0, hk, hk2, hv, hv2, nh, 0, key_bits, s);
        void* tmp = sc.get<char>(t0);
        if (!sc.ok) return LOGAN_ENOMEM;
        cub::DeviceRadixSort::SortPairs(tmp, t0, hk, hk2, hv, hv2, nh, 0, key_bits, s);
        std::swap(hk, hk2);
        std::swap(hv, hv2);
    } else {  // by position, then stably by pair
        cub::DeviceRadixSort::SortPairs(nullptr, t0, hv, hv2, hk, hk2, nh, 0, 2 * pb, s);
        cub::DeviceRadixSort::SortPairs(nullptr, t1, hk2, hk, hv2, hv, nh, 0, key_bits, s);
        void* tmp = sc.get<char>(std::max(t0, t1));
        if (!sc.ok) return LOGAN_ENOMEM;
        cub::DeviceRadixSort::SortPairs(tmp, t0, hv, hv2, hk, hk2, nh, 0, 2 * pb, s);
        cub::DeviceRadixSort::SortPairs(tmp, t1, hk2, hk, hv2, hv, nh, 0, key_bits, s);
    }
    uint64_t* sstart = nullptr;
    const int64_t nseg_i = run_heads(sc, hk, nh, COMPOSITE ? pb : 0, sstart);
    if (nseg_i < 0) return sc.ok ? LOGAN_ECUDA : LOGAN_ENOMEM;
    const uint64_t nseg = uint64_t(nseg_i);
    logan_candidate_t* all = sc.get<logan_candidate_t>(nseg);
    uint8_t* keep = sc.get<uint8_t>(nseg);
    kept = sc.get<logan_candidate_t>(nseg);
    uint64_t* nkept_d = sc.get<uint64_t>(1);
    if (!sc.ok) return LOGAN_ENOMEM;
    k_segment_pick<H, COMPOSITE><<<blocks_for(nseg), kThreads, 0, s>>>(sstart, nseg, nh, hk, hv, rb,
                                                                      pb, min_shared, all, keep);
    size_t t8 = 0;
    cub::DeviceSelect::Flagged(nullptr, t8, all, keep, kept, nkept_d, nseg, s);
    void* tmp8 = sc.get<char>(t8);
    if (!sc.ok) return LOGAN_ENOMEM;
    cub::DeviceSelect::Flagged(tmp8, t8, all, keep, kept, nkept_d, nseg, s);
    return cudaMemcpyAsync(&nkept, nkept_d, sizeof(uint64_t), cudaMemcpyDeviceToHost, s) ==
                       cudaSuccess &&
                   cudaStreamSynchronize(s) == cudaSuccess
               ? LOGAN_OK
               : LOGAN_ECUDA;
}

// Every step after the occurrences are counted (first): keys of type K --
// 32-bit with the code's upper bits as up to 16 classes, else 64-bit -- and
// occurrence numbers of type V.
template <typename K, typename V>
int find_candidates(Scratch& sc, const logan_seqs_t* reads, int k, const uint64_t* first, uint64_t nk,
                    uint32_t min_freq, uint32_t max_freq, uint32_t min_shared,
                    logan_candidate_t*& kept, uint64_t& nkept) {
    cudaStream_t s = sc.s;
    const uint32_t R = reads->count;
    // about four cells per read
    int shift = 0;
    while ((nk >> shift) > 4ull * R && shift < 30) ++shift;
    const uint64_t n_cells = (nk >> shift) + 2;
    uint32_t* cell = sc.get<uint32_t>(n_cells);
    if (!sc.ok) return LOGAN_ENOMEM;
    k_read_cells<<<blocks_for(n_cells), kThreads, 0, s>>>(first, R, nk, shift, n_cells, cell);
    const KmerArgs ka = {static_cast<const uint32_t*>(reads->bases), reads->offsets,
                         ReadIndex{first, cell, shift}, nk, k};
    const int classes = sizeof(K) == 4 && 2 * k > 32 ? 1 << (2 * k - 32) : 1;
    const uint64_t tiles = (nk + kTile - 1) / kTile;
    if (tiles > 0x7fffffffull) return LOGAN_EINVAL;
    uint64_t* at = nullptr;
    uint64_t start[kMaxClasses + 1] = {};
    if (classes > 1) {
        uint64_t* cnt = sc.get<uint64_t>(classes * tiles + 1);
        if (!sc.ok) return LOGAN_ENOMEM;
        k_kmer_classes<<<unsigned(tiles), kThreads, 0, s>>>(ka, classes, tiles, cnt);
        if (!prefix(sc, cnt, classes * tiles, at, nullptr)) return LOGAN_ENOMEM;
        for (int c = 1; c < classes; ++c)
            if (cudaMemcpyAsync(&start[c], at + c * tiles, sizeof(uint64_t), cudaMemcpyDeviceToHost,
                                s) != cudaSuccess)
                return LOGAN_ECUDA;
    }
    K* keys = sc.get<K>(nk);
    V* vals = sc.get<V>(nk);
    K* keys2 = sc.get<K>(nk);
    V* vals2 = sc.get<V>(nk);
    uint64_t* runs = sc.get<uint64_t>(nk / 2 + 1);
    unsigned long long* n_runs_d = sc.get<unsigned long long>(1);
    if (!sc.ok) return LOGAN_ENOMEM;
    k_kmer_emit<K, V><<<unsigned(tiles), kThreads, 0, s>>>(ka, classes, tiles, at, keys, vals);
    std::vector<uint32_t> hl(R);
    if (cudaMemsetAsync(n_runs_d, 0, sizeof(*n_runs_d), s) != cudaSuccess ||
        cudaMemcpyAsync(hl.data(), reads->lengths, sizeof(uint32_t) * R, cudaMemcpyDeviceToHost,
                        s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return LOGAN_ECUDA;
    start[classes] = nk;
    // sort each class by code (stable: equal codes stay in (read, pos) order)
    // and list its reliable runs
    uint64_t most = 0;
    for (int c = 0; c < classes; ++c) most = std::max(most, start[c + 1] - start[c]);
    const int bits = sizeof(K) == 4 ? std::min(2 * k, 32) : 2 * k;
    size_t tsort = 0;
    cub::DeviceRadixSort::SortPairs(nullptr, tsort, keys, keys2, vals, vals2, most, 0, bits, s);
    void* tmp = sc.get<char>(tsort);
    if (!sc.ok) return LOGAN_ENOMEM;
    for (int c = 0; c < classes; ++c) {
        const uint64_t b = start[c], n = start[c + 1] - b;
        if (n == 0) continue;
        size_t tb = tsort;
        if (cub::DeviceRadixSort::SortPairs(tmp, tb, keys + b, keys2 + b, vals + b, vals2 + b, n, 0,
                                            bits, s) != cudaSuccess)
            return LOGAN_ECUDA;
        k_find_runs<K><<<unsigned((n + kTile - 1) / kTile), kThreads, 0, s>>>(
            keys2 + b, n, b, min_freq, max_freq, n_runs_d, runs);
    }
    unsigned long long n_runs = 0;
    if (cudaMemcpyAsync(&n_runs, n_runs_d, sizeof(n_runs), cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return LOGAN_ECUDA;
    if (n_runs == 0) return LOGAN_OK;
    uint32_t maxlen = 0;
    for (uint32_t v : hl) maxlen = std::max(maxlen, v);
    const int rb = std::max(1, bit_width(R)), pb = std::max(1, bit_width(maxlen));
    if (2 * rb + 1 > 64 || 2 * pb > 64) return LOGAN_EINVAL;
    // one sort by (a, b, o, pos_a) when that fits 64 bits (50,000 reads up to
    // 64 kbp: 49), else two
    return 2 * rb + 1 + pb <= 64
               ? candidates_of<V, uint32_t, true>(sc, runs, n_runs, vals2, ka.ix, rb, pb, min_shared,
                                                  kept, nkept)
               : candidates_of<V, uint64_t, false>(sc, runs, n_runs, vals2, ka.ix, rb, pb,
                                                   min_shared, kept, nkept);
}

}  // namespace

}  // namespace logan

using namespace logan;

extern "C" int logan_overlap_candidates(logan_ctx_t* ctx, const logan_seqs_t* reads, int k,
                                        uint32_t min_freq, uint32_t max_freq,
                                        uint32_t min_shared, logan_candidate_t* out,
                                        uint64_t capacity, uint64_t* n_found, void* stream) {
    if (!ctx || !reads || !n_found || k < 1 || k > 31 || min_freq < 2 || max_freq < min_freq ||
        max_freq > 1024 || min_shared < 1)
        return LOGAN_EINVAL;
    if (!reads->packed2bit || (reads->count && (!reads->bases || !reads->offsets || !reads->lengths)))
        return LOGAN_EINVAL;
    if (capacity && !out) return LOGAN_EINVAL;
    *n_found = 0;
    const uint32_t R = reads->count;
    if (R < 2) return LOGAN_OK;
    int64_t dev = 0;
    logan_get_option(ctx, LOGAN_OPT_DEVICE, &dev);
    int prev = 0;
    cudaGetDevice(&prev);
    if (prev != int(dev) && cudaSetDevice(int(dev)) != cudaSuccess) return LOGAN_ECUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = LOGAN_OK;
    {
        Scratch sc(s, ctx_scratch_pool(ctx));
        // 1. k-mer occurrences, (read, pos) order: first[r] = k-mers of
        // reads below r, first[R] = all of them
        uint64_t* cnt = sc.get<uint64_t>(R + 1);
        uint64_t* first = sc.get<uint64_t>(R + 1);
        size_t tb = 0;
        cub::DeviceScan::ExclusiveSum(nullptr, tb, cnt, first, R + 1, s);
        void* tmp = sc.get<char>(tb);
        if (!sc.ok) return LOGAN_ENOMEM;
        k_kmer_counts<<<blocks_for(R), kThreads, 0, s>>>(reads->lengths, R, k, cnt);
        cudaMemsetAsync(cnt + R, 0, sizeof(uint64_t), s);
        cub::DeviceScan::ExclusiveSum(tmp, tb, cnt, first, R + 1, s);
        uint64_t* nk_d = first + R;
        uint64_t nk = 0;
        cudaMemcpyAsync(&nk, nk_d, sizeof(uint64_t), cudaMemcpyDeviceToHost, s);
        if (cudaStreamSynchronize(s) != cudaSuccess) return LOGAN_ECUDA;
        if (nk < 2) return LOGAN_OK;
        // 2. the candidates: 32-bit keys when the codes' upper bits make at most
        // 16 classes (k <= 18), 32-bit occurrence numbers below 2^31 of them
        logan_candidate_t* kept = nullptr;
        uint64_t nkept = 0;
        const bool k32 = 2 * k <= 36, v32 = nk < (1ull << 31);
        const int frc =
            k32 && v32 ? find_candidates<uint32_t, uint32_t>(sc, reads, k, first, nk, min_freq, max_freq,
                                                             min_shared, kept, nkept)
            : k32      ? find_candidates<uint32_t, uint64_t>(sc, reads, k, first, nk, min_freq, max_freq,
                                                             min_shared, kept, nkept)
            : v32      ? find_candidates<uint64_t, uint32_t>(sc, reads, k, first, nk, min_freq, max_freq,
                                                             min_shared, kept, nkept)
                       : find_candidates<uint64_t, uint64_t>(sc, reads, k, first, nk, min_freq, max_freq,
                                                             min_shared, kept, nkept);
        if (frc != LOGAN_OK) return frc;
        *n_found = nkept;
        const uint64_t ncopy = std::min(nkept, capacity);
        if (ncopy)
            cudaMemcpyAsync(out, kept, sizeof(logan_candidate_t) * ncopy, cudaMemcpyDeviceToDevice,
                            s);
        if (cudaStreamSynchronize(s) != cudaSuccess || cudaGetLastError() != cudaSuccess)
            rc = LOGAN_ECUDA;
    }
    if (prev != int(dev)) cudaSetDevice(prev);
    return rc;
}

extern "C" int logan_overlap_pool_words(logan_ctx_t* ctx, const logan_seqs_t* reads,
                                        uint64_t* words, void* stream) {
    if (!ctx || !reads || !words || !reads->packed2bit || (reads->count && !reads->lengths))
        return LOGAN_EINVAL;
    // the forward pool's words (with its spare word), then every reverse
    // complement 16-base aligned, then one spare word
    const uint32_t R = reads->count;
    std::vector<uint32_t> hl(R);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (R && (cudaMemcpyAsync(hl.data(), reads->lengths, sizeof(uint32_t) * R,
                              cudaMemcpyDeviceToHost, s) != cudaSuccess ||
              cudaStreamSynchronize(s) != cudaSuccess))
        return LOGAN_ECUDA;
    uint64_t tot = (reads->pool_bases + 15) / 16 + 1;
    for (uint32_t v : hl) tot += (uint64_t(v) + 15) / 16;
    *words = tot + 1;
    return LOGAN_OK;
}

extern "C" int logan_overlap_pool(logan_ctx_t* ctx, const logan_seqs_t* reads,
                                  uint32_t* words_out, uint64_t words_capacity,
                                  uint64_t* offsets_out, uint32_t* lengths_out,
                                  logan_seqs_t* pool_out, void* stream) {
    if (!ctx || !reads || !pool_out || !reads->packed2bit || !words_out || !offsets_out ||
        !lengths_out)
        return LOGAN_EINVAL;
    const uint32_t R = reads->count;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const uint64_t fwd = (reads->pool_bases + 15) / 16 + 1;
    std::vector<uint32_t> hl(R);
    if (R && (cudaMemcpyAsync(hl.data(), reads->lengths, sizeof(uint32_t) * R,
                              cudaMemcpyDeviceToHost, s) != cudaSuccess ||
              cudaStreamSynchronize(s) != cudaSuccess))
        return LOGAN_ECUDA;
    std::vector<uint64_t> wf(R);
    uint64_t tot = 0;
    for (uint32_t r = 0; r < R; ++r) {
        wf[r] = tot;
        tot += (uint64_t(hl[r]) + 15) / 16;
    }
    const uint64_t need = fwd + tot + 1;
    if (words_capacity < need) return LOGAN_ENOMEM;
    int rc = LOGAN_OK;
    {
        Scratch sc(s, ctx_scratch_pool(ctx));
        uint64_t* wfd = sc.get<uint64_t>(R);
        if (!sc.ok) return LOGAN_ENOMEM;
        if (R) cudaMemcpyAsync(wfd, wf.data(), sizeof(uint64_t) * R, cudaMemcpyHostToDevice, s);
        cudaMemcpyAsync(words_out, reads->bases, sizeof(uint32_t) * fwd, cudaMemcpyDeviceToDevice, s);
        cudaMemsetAsync(words_out + fwd + tot, 0, sizeof(uint32_t), s);
        if (R) {
            cudaMemcpyAsync(offsets_out, reads->offsets, sizeof(uint64_t) * R,
                            cudaMemcpyDeviceToDevice, s);
            cudaMemcpyAsync(lengths_out, reads->lengths, sizeof(uint32_t) * R,
                            cudaMemcpyDeviceToDevice, s);
            cudaMemcpyAsync(lengths_out + R, reads->lengths, sizeof(uint32_t) * R,
                            cudaMemcpyDeviceToDevice, s);
            dim3 grid(64, std::min<uint32_t>(R, 65535u));
            k_revcomp_pool<<<grid, 128, 0, s>>>(static_cast<const uint32_t*>(reads->bases),
                                                reads->offsets, reads->lengths, R, wfd, fwd,
                                                words_out, offsets_out + R);
        }
        // the host copies above read pageable host vectors: finish before they go
        if (cudaStreamSynchronize(s) != cudaSuccess || cudaGetLastError() != cudaSuccess)
            rc = LOGAN_ECUDA;
    }
    pool_out->bases = words_out;
    pool_out->offsets = offsets_out;
    pool_out->lengths = lengths_out;
    pool_out->count = 2 * R;
    pool_out->packed2bit = 1;
    pool_out->pool_bases = (need - 1) * 16;
    return rc;
}

extern "C" int logan_overlap_seeds(logan_ctx_t* ctx, const logan_candidate_t* cands, uint64_t n,
                                   const logan_seqs_t* reads, int k, logan_seed_t* seeds,
                                   void* stream) {
    if (!ctx || !reads || (n && (!cands || !seeds)) || k < 1 || k > 31) return LOGAN_EINVAL;
    if (!n) return LOGAN_OK;
    k_overlap_seeds<<<blocks_for(n), kThreads, 0, static_cast<cudaStream_t>(stream)>>>(
        cands, n, reads->lengths, reads->count, k, seeds);
    return cudaGetLastError() == cudaSuccess ? LOGAN_OK : LOGAN_ECUDA;
}

extern "C" int logan_overlap_keep(logan_ctx_t* ctx, const logan_result_t* results,
                                  const logan_seed_t* seeds, uint64_t n,
                                  const logan_seqs_t* seqsA, const logan_seqs_t* seqsB,
                                  int64_t ratio_num, int64_t den, int64_t delta, uint8_t* keep,
                                  void* stream) {
    if (!ctx || !seqsA || !seqsB || den <= 0 || (n && (!results || !seeds || !keep)))
        return LOGAN_EINVAL;
    if (!n) return LOGAN_OK;
    k_overlap_keep<<<blocks_for(n), kThreads, 0, static_cast<cudaStream_t>(stream)>>>(
        results, seeds, n, seqsA->lengths, seqsB->lengths, ratio_num, den, delta, keep);
    return cudaGetLastError() == cudaSuccess ? LOGAN_OK : LOGAN_ECUDA;
}
