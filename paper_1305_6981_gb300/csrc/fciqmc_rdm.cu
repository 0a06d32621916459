// Energy functional E(h, V; c) = c^T H c / c^T c over a fixed determinant list, and its gradient with
// respect to the one- and two-electron integrals (the 1- and 2-RDMs of c divided by c^T c).
//
// The pair structure. Every determinant I emits, for each pair {x < y} of its occupied spin orbitals, the key
// K = I - {x, y}. With v_K(xy) = +-c_I, the sign being that of a_y a_x |I>, the off-diagonal part of the
// energy is a sum over keys of small quadratic forms,
//   c^T H c - diagonal = sum_K sum_{xy != zw} v_K(xy) v_K(zw) <xy|T|zw>,
//   T = the antisymmetrised two-electron integral + (one-electron elements) / (N - 1),
// because two determinants that differ by a double excitation share one key and two that differ by a single
// share N - 1 of them, whose T elements add up to the whole Slater-Condon element (its spectator sum runs
// over the keys). So no pair needs to be decoded: a member of a key's group is (pair code, signed
// amplitude), T is a table over pair codes, and a pair of members costs one table read and one FMA. The
// two-body density matrix is the same sum with T's element replaced by its index.
// Only keys shared by two or more determinants matter; the diagonal comes from the occupation-pair sums
// O_pq = sum_I c_I^2 n_p n_q.
//
// Grouping is a radix partition by a 64-bit XOR hash of the key (one word per spin orbital, so a key's hash
// is the determinant's with two words taken out): keys are 8-byte records, scattered once into partitions
// that fit in shared memory, where one block groups them exactly (the hash only routes; determinants decide).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <new>

#include "fciqmc.h"
#include "fciqmc_device.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kPartMax = 1 << 15;     // most partitions (their counters fill 128 KB of shared memory)
constexpr int kBins = 1024;           // most bins of one scatter pass
constexpr int kFineBits = 7;          // bins of the second pass, where one pass is not enough
constexpr int kTileKeys = 4096;       // keys scattered at a time by one block (two blocks fit on an SM)
constexpr int kCursorStride = 16;     // first-pass cursors, one per 64 bytes: every tile of every block takes room there
constexpr int kHashThreads = 1024;    // threads of the passes over the keys
static_assert(kBins == kHashThreads, "the first scatter pass has one thread per bin");
constexpr int kGroupThreads = 512;
// Records grouped at a time by one block and slots of its table: 110 KB of shared memory, so two blocks fit on
// an SM. An average partition holds at most about 3,700 records up to 1.2e8 keys; longer ones are taken in
// several parts.
constexpr int kGroupCap = 4608;
constexpr int kGroupSlots = 8192;
constexpr int kBigLeaders = 16;       // distinct keys of one hash value that the oversized path tells apart
// Groups from this size on are large: walked as triangles, by warps of all blocks. The largest that a member's code can
// tell apart; E and gradient of 1e6 determinants of 16e/40o 1.27 and 1.40 ms with 62, 1.32 and 1.47 with 48, 1.52 and 1.48
// with 24; 3e5 of 24e/60o 0.51, 0.53 and 0.62 (E).
constexpr int kTriangle = 63;
constexpr int kTaskPartners = 128;    // partners of a row beyond which more warps share it
constexpr int kTaskShares = 16;       // most warps that do
constexpr int kMergeThreads = 128;

// A determinant in the group of a key: its signed amplitude, its pair code (bits 0..12 the index within the
// class, 13..14 the class: 0 alpha alpha, 1 beta beta, 2 mixed; bits 15..20 the group size, kLarge from kTriangle
// on), and the position of the group's first member in the partition.
constexpr unsigned kLarge = 63;
static_assert(kTriangle <= kLarge, "a small group's size is not kLarge");
struct alignas(16) Member {
    double v;
    unsigned code;
    unsigned first;
};

// A large group: its first member (of all) and size.
struct Head {
    unsigned first, m;
};

// A warp's share of a large group of m members from `first` on: rows row0 + lane, each with the members before it, of
// those the blocks of 64 numbered share, share + n_shares, ...
struct alignas(16) Task {
    unsigned first, m, row0;
    unsigned short share, n_shares;
};

struct RdmState {
    unsigned long long n_buckets;
    unsigned long long n_members;  // members of buckets with two or more entries
    unsigned long long n_pairs;    // candidate pairs
    unsigned long long n_shared;   // pairs of members that share one spin orbital (counted on request)
    unsigned long long n_apart;    // pairs that share none
    unsigned long long n_tasks;
    unsigned n_heads;
    unsigned pad0;
    double norm;
    int status;
    int pad;
};

struct RdmLayout {
    size_t dets, c, total_p, base_p, cursor_p, coarse_p, count_p, records, members, heads, state, gh, ge, share, table,
        occ_part, occ_pair, partial;
    size_t total;
};

size_t align256(size_t x) { return (x + 255) / 256 * 256; }
long long next_pow2(long long x) {
    long long p = 1;
    while (p < x) p <<= 1;
    return p;
}
int log2i(long long x) {
    int b = 0;
    while ((1LL << b) < x) ++b;
    return b;
}

constexpr int kSms = 152;                     // blocks of the passes that take one block per SM
constexpr int kPairGrid = kSms * 32;          // most blocks of the pair passes (several waves: partitions differ in cost)
constexpr int kPairThreads = 128;
constexpr int kDiagBlocks = 16;               // blocks of the energy's diagonal
constexpr int kLargeGrid = kSms * 16;         // most blocks of the pair passes for large groups
constexpr int kNormGrid = kSms;

struct Dims {
    int n_elec, n_orb, n_so, W, npairs;
    int n1, n2;          // pair codes of one spin (p < q) and of mixed spin (p, q)
    int parts, pbits;    // partitions of the key records
    int tbits;           // bits of a key's number
    int hash_blocks;     // blocks of the passes over the determinants
    long long n, n_keys, n_eri;
};

bool dims_of(int n_elec, int n_orb, long long n, Dims &d) {
    if (n_orb < 1 || n_orb > 64 || n_elec < 2 || n_elec > fq::MAXN || n_elec >= 2 * n_orb || n < 1 || n > (1LL << 30))
        return false;
    d.n_elec = n_elec;
    d.n_orb = n_orb;
    d.n_so = 2 * n_orb;
    d.W = (2 * n_orb + 63) / 64;
    d.npairs = n_elec * (n_elec - 1) / 2;
    d.n1 = n_orb * (n_orb - 1) / 2;
    d.n2 = n_orb * n_orb;
    d.n = n;
    d.n_keys = n * d.npairs;
    // about 4096 records a partition; small lists get up to 512 partitions of at least 256, to spread over the SMs
    d.parts = (int)std::min<long long>(
        kPartMax, next_pow2(std::max<long long>(d.n_keys / 4096, std::min<long long>(512, std::max<long long>(1, d.n_keys / 256)))));
    d.pbits = log2i(d.parts);
    d.tbits = std::max(1, log2i(d.n_keys));
    d.hash_blocks = (int)std::min<long long>(kSms, (n + 31) / 32);
    long long np = (long long)n_orb * (n_orb + 1) / 2;
    d.n_eri = np * (np + 1) / 2;
    return d.n_keys < (1LL << 31);
}

RdmLayout layout_of(const Dims &d) {
    RdmLayout L{};
    size_t off = 0;
    auto take = [&](size_t b) {
        size_t o = off;
        off = align256(off + b);
        return o;
    };
    L.dets = take(sizeof(unsigned long long) * d.W * d.n);
    L.c = take(sizeof(double) * d.n);
    L.total_p = take(sizeof(unsigned) * d.parts);
    L.base_p = take(sizeof(unsigned) * (d.parts + 1));
    L.cursor_p = take(sizeof(unsigned) * d.parts);
    L.coarse_p = take(sizeof(unsigned) * kBins * kCursorStride);
    L.count_p = take(sizeof(unsigned) * d.parts);
    L.records = take(sizeof(unsigned long long) * d.n_keys);
    L.members = take(sizeof(Member) * d.n_keys);
    L.heads = take(sizeof(Head) * (d.n_keys / kTriangle + 1));
    L.state = take(sizeof(RdmState));
    L.gh = take(sizeof(double) * d.n_orb * d.n_orb);
    L.ge = take(sizeof(double) * d.n_eri);
    L.share = take(sizeof(double) * d.n_orb * d.n_orb);
    L.table = take(sizeof(double) * ((size_t)d.n1 * d.n1 + (size_t)d.n2 * d.n2));
    L.occ_part = take(2 * sizeof(double) * kSms * ((size_t)d.n_so * (d.n_so + 1) / 2));
    L.occ_pair = take(sizeof(double) * ((size_t)d.n_so * (d.n_so + 1) / 2));
    L.partial = take(sizeof(double) * 2 * (kPairGrid + kLargeGrid + kDiagBlocks + kNormGrid));
    L.total = off;
    return L;
}

// ------------------------------------------------------------------------------------ device helpers
template <int W>
__device__ __forceinline__ void load_det(const unsigned long long *dets, long long i, unsigned long long (&d)[W]) {
    if (W == 2) {
        const ulonglong2 x = __ldg(reinterpret_cast<const ulonglong2 *>(dets) + i);
        d[0] = x.x;
        d[W - 1] = x.y;
    } else {
        d[0] = __ldg(dets + i);
    }
}

// A key's hash as it is used. -DFQ_RDM_HASH_BITS=b leaves 2^b different ones, so that a test can have keys that share
// all hash bits in every partition of a small list.
__device__ __forceinline__ unsigned long long used_hash(unsigned long long h) {
#ifdef FQ_RDM_HASH_BITS
    return fq::mix64(h & ((1ull << FQ_RDM_HASH_BITS) - 1ull));
#else
    return h;
#endif
}

// The hash word of a spin orbital.
__device__ __forceinline__ unsigned long long orbital_word(int k) { return fq::mix64(0x9E3779B97F4A7C15ull * (unsigned long long)(k + 1)); }

// Electron pairs in order k = y (y - 1) / 2 + x, x < y, packed x | y << 8.
__device__ __forceinline__ void triangle_of(int k, int &x, int &y) {  // k = y (y - 1) / 2 + x, x < y
    y = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)k)) * 0.5f);
    while (y > 1 && y * (y - 1) / 2 > k) --y;
    while ((y + 1) * y / 2 <= k) ++y;
    x = k - y * (y - 1) / 2;
}
__device__ __forceinline__ void fill_pairs(int n_elec, unsigned short *pairs) {
    for (int k = threadIdx.x; k < n_elec * (n_elec - 1) / 2; k += blockDim.x) {
        int x, y;
        triangle_of(k, x, y);
        pairs[k] = (unsigned short)(x | (y << 8));
    }
}

// A key record: the low tbits bits are the emitting (determinant, pair) t = I npairs + k, the others the hash bits after
// those that chose the partition (64 - tbits of them, at least 33; tbits = bits of the number of keys).
__device__ __forceinline__ unsigned rec_t(unsigned long long r, int tbits) { return (unsigned)r & ((1u << tbits) - 1u); }
__device__ __forceinline__ unsigned long long rec_hash(unsigned long long r, int tbits) { return r >> tbits; }
__device__ __forceinline__ unsigned long long make_rec(unsigned long long hash, int used, int tbits, unsigned t) {
    return (((hash << used) >> tbits) << tbits) | (unsigned long long)t;
}

// Key and removed spin orbitals of a record.
struct KeyOf {
    unsigned I;
    int k, ox, oy;
};
template <int W>
__device__ __forceinline__ KeyOf key_of(const unsigned long long *dets, const unsigned short *pairs, int npairs, unsigned t,
                                        unsigned long long (&key)[W]) {
    KeyOf q;
    q.I = t / (unsigned)npairs;
    q.k = (int)(t - q.I * (unsigned)npairs);
    const unsigned short pr = pairs[q.k];
    load_det<W>(dets, q.I, key);
    q.ox = fq::select_bit<W>(key, pr & 0xFF);
    q.oy = fq::select_bit<W>(key, pr >> 8);
    fq::flip<W>(key, q.ox);
    fq::flip<W>(key, q.oy);
    return q;
}

// Code of the pair ox < oy: class << 13 | index. Mixed pairs are indexed alpha first. kNoPair for orbitals outside the
// basis or out of order (a determinant that is none of the run's): such members carry no amplitude.
constexpr unsigned kNoPair = 0x7FFFu;
__device__ __forceinline__ unsigned pair_code(int ox, int oy, int n_orb) {
    if (ox >= oy || oy >= 2 * n_orb) return kNoPair;
    const int p = ox >> 1, q = oy >> 1, sx = ox & 1, sy = oy & 1;
    if (sx == sy) return ((unsigned)sx << 13) | (unsigned)(q * (q - 1) / 2 + p);
    return (2u << 13) | (unsigned)(sx == 0 ? p * n_orb + q : q * n_orb + p);
}

// ------------------------------------------------------------------------------------ construction kernels
// The keys of determinants [lo, hi), one determinant per warp at a time: the lanes decode it together (each set bit's
// rank is a population count) and then take its pairs. f(pair's key number t, its 64-bit hash).
struct HashShared {
    unsigned long long z[fq::MAXSO];
    unsigned long long zo[kHashThreads / 32][fq::MAXN];
    unsigned short pairs[fq::MAXPAIRS];
};
__device__ __forceinline__ void hash_setup(HashShared &s, int n_elec) {
    fill_pairs(n_elec, s.pairs);
    for (int k = threadIdx.x; k < fq::MAXSO; k += blockDim.x) s.z[k] = orbital_word(k);
}
template <int W, typename F>
__device__ __forceinline__ void for_keys(HashShared &s, const unsigned long long *dets, long long lo, long long hi, int n_elec, F f) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long *zo = s.zo[warp];
    const int npairs = n_elec * (n_elec - 1) / 2;
    for (long long I = lo + warp; I < hi; I += kHashThreads / 32) {
        unsigned long long d[W];
        load_det<W>(dets, I, d);
        unsigned long long z = 0;
        int base = 0;
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 2 * W; ++c) {
            const unsigned bits = (unsigned)(d[c >> 1] >> (32 * (c & 1)));
            if ((bits >> lane) & 1u) {
                const int r = base + __popc(bits & ((1u << lane) - 1u));
                const unsigned long long w = s.z[32 * c + lane];
                z ^= w;
                if (r < fq::MAXN) zo[r] = w;
            }
            base += __popc(bits);
        }
        for (int r = base + lane; r < n_elec; r += 32) zo[r] = 0ull;  // (a determinant short of electrons)
        const unsigned zl = __reduce_xor_sync(0xFFFFFFFFu, (unsigned)z), zh = __reduce_xor_sync(0xFFFFFFFFu, (unsigned)(z >> 32));
        const unsigned long long H = (unsigned long long)zl | ((unsigned long long)zh << 32);
        __syncwarp();
        const unsigned t0 = (unsigned)(I * npairs);
        for (int k = lane; k < npairs; k += 32) {
            const unsigned short pr = s.pairs[k];
            f(t0 + (unsigned)k, used_hash(H ^ zo[pr & 0xFF] ^ zo[pr >> 8]));
        }
    }
}

// Keys per partition, counted in shared memory.
template <int W>
__global__ void __launch_bounds__(kHashThreads) k_key_hist(const unsigned long long *dets, long long n, int n_elec, int parts,
                                                           int pbits, unsigned *total_p) {
    extern __shared__ unsigned s_count[];
    __shared__ HashShared s_h;
    hash_setup(s_h, n_elec);
    for (int p = threadIdx.x; p < parts; p += blockDim.x) s_count[p] = 0;
    __syncthreads();
    for_keys<W>(s_h, dets, n * blockIdx.x / gridDim.x, n * (blockIdx.x + 1) / gridDim.x, n_elec, [&](unsigned, unsigned long long h) {
        atomicAdd(&s_count[pbits ? (unsigned)(h >> (64 - pbits)) : 0u], 1u);
    });
    __syncthreads();
    for (int p = threadIdx.x; p < parts; p += blockDim.x) {
        const unsigned m = s_count[p];
        if (m) atomicAdd(&total_p[p], m);
    }
}

// First record of every partition and of every bin of the first scatter pass (one block).
__global__ void __launch_bounds__(1024) k_part_scan(const unsigned *total_p, int parts, int fine, unsigned *base_p, unsigned *cursor_p,
                                                    unsigned *coarse_p) {
    __shared__ unsigned s_w[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned carry = 0;
    for (int p0 = 0; p0 < parts; p0 += 4096) {  // four neighbouring partitions per thread, so loads are coalesced
        unsigned m[4], sum = 0;
        const int p = p0 + 4 * (int)threadIdx.x;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            m[k] = p + k < parts ? total_p[p + k] : 0u;
            sum += m[k];
        }
        unsigned x = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        __syncthreads();
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        unsigned off = carry + x - sum, all = 0;
#pragma unroll
        for (int w = 0; w < 32; ++w) {
            const unsigned y = s_w[w];
            off += w < warp ? y : 0u;
            all += y;
        }
        carry += all;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (p + k < parts) {
                base_p[p + k] = off;
                cursor_p[p + k] = off;
                if (((p + k) & ((1 << fine) - 1)) == 0) coarse_p[((p + k) >> fine) * kCursorStride] = off;
            }
            off += m[k];
        }
    }
    if (threadIdx.x == 0) base_p[parts] = carry;
}

// Scatter of the key records to their partitions, a tile of up to kTileKeys at a time: the block counts the tile's
// bins, takes room for each with one atomic, sorts the tile by bin in shared memory and writes it in that order, so
// that neighbouring lanes write neighbouring records. (One store per lane wherever its record belongs took 2.4 ms
// for 1.2e8 keys and 256 bins, every warp touching 32 pages; all 32,768 partitions at once took 4.5 ms.) Up to kBins
// partitions one pass does; beyond, this pass takes the leading bits and k_refine the rest.
// First pass: the records are made from the determinants. bits: of the bin number.
struct ScatterShared {
    HashShared h;
    unsigned long long hash[kTileKeys];
    unsigned long long rec[kTileKeys];
    unsigned short bin[kTileKeys];
    unsigned at[kBins];      // a bin's next place in the tile
    unsigned to[kBins];      // where the tile's first record would go if it belonged to the bin
    unsigned scan[kHashThreads / 32];
};
template <int W>
__global__ void __launch_bounds__(kHashThreads, 2) k_key_scatter(const unsigned long long *dets, long long n, int n_elec,
                                                                 int bits, int tbits, unsigned *cursor, unsigned long long *out) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    ScatterShared &s = *reinterpret_cast<ScatterShared *>(s_raw);
    hash_setup(s.h, n_elec);
    const int npairs = n_elec * (n_elec - 1) / 2, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = max(1, kTileKeys / npairs);  // determinants of a tile (npairs <= MAXPAIRS < kTileKeys)
    for (long long lo = (long long)blockIdx.x * per; lo < n; lo += (long long)gridDim.x * per) {
        const long long hi = min(lo + per, n);
        const int m = (int)((hi - lo) * npairs);
        s.at[threadIdx.x] = 0;  // kBins = kHashThreads
        __syncthreads();
        const unsigned t0 = (unsigned)(lo * npairs);
        for_keys<W>(s.h, dets, lo, hi, n_elec, [&](unsigned t, unsigned long long h) {
            s.hash[t - t0] = h;
            atomicAdd(&s.at[bits ? (unsigned)(h >> (64 - bits)) : 0u], 1u);
        });
        __syncthreads();
        const unsigned c = s.at[threadIdx.x];
        unsigned x = c;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s.scan[warp] = x;
        __syncthreads();
        unsigned off = x - c;
#pragma unroll
        for (int w = 0; w < kHashThreads / 32; ++w) off += w < warp ? s.scan[w] : 0u;
        s.at[threadIdx.x] = off;
        s.to[threadIdx.x] = c ? atomicAdd(&cursor[threadIdx.x * kCursorStride], c) - off : 0u;
        __syncthreads();
        for (int k = threadIdx.x; k < m; k += kHashThreads) {
            const unsigned long long h = s.hash[k];
            const unsigned b = bits ? (unsigned)(h >> (64 - bits)) : 0u, at = atomicAdd(&s.at[b], 1u);
            s.rec[at] = make_rec(h, bits, tbits, t0 + (unsigned)k);
            s.bin[at] = (unsigned short)b;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < m; k += kHashThreads) out[s.to[s.bin[k]] + (unsigned)k] = s.rec[k];
        __syncthreads();
    }
}

// Second pass: the records of coarse bin blockIdx.y to its 2^kFineBits partitions, by their hash's leading bits, which
// are shifted out (the last kFineBits of the hash become zero).
__global__ void __launch_bounds__(kHashThreads) k_refine(const unsigned long long *in, int tbits, const unsigned *base_p, unsigned *cursor_p,
                                                         unsigned long long *out) {
    constexpr int kFine = 1 << kFineBits;
    __shared__ unsigned long long s_rec[4096];
    __shared__ unsigned s_at[kFine];
    const unsigned lo = base_p[blockIdx.y << kFineBits], hi = base_p[(blockIdx.y + 1) << kFineBits];
    unsigned *cursor = cursor_p + (blockIdx.y << kFineBits);
    for (unsigned long long t = (unsigned long long)lo + blockIdx.x * 4096ull; t < hi; t += gridDim.x * 4096ull) {
        const int m = (int)min(4096ull, hi - t);
        if (threadIdx.x < kFine) s_at[threadIdx.x] = 0;
        __syncthreads();
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
            const unsigned long long r = in[t + k];
            s_rec[k] = r;
            atomicAdd(&s_at[(unsigned)(r >> (64 - kFineBits))], 1u);
        }
        __syncthreads();
        if (threadIdx.x < kFine) {
            const unsigned c = s_at[threadIdx.x];
            s_at[threadIdx.x] = c ? atomicAdd(&cursor[threadIdx.x], c) : 0u;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
            const unsigned long long r = s_rec[k];
            out[atomicAdd(&s_at[(unsigned)(r >> (64 - kFineBits))], 1u)] = make_rec(rec_hash(r, tbits) << tbits, kFineBits, tbits, rec_t(r, tbits));
        }
        __syncthreads();
    }
}

template <int W>
__device__ __forceinline__ bool same_key(const unsigned long long (&a)[W], const unsigned long long (&b)[W]) {
    bool e = true;
#pragma unroll
    for (int w = 0; w < W; ++w) e = e && a[w] == b[w];
    return e;
}

// Exclusive block scan of a 64-bit value (packed 16-bit fields); total in `sum`.
__device__ __forceinline__ unsigned long long block_scan64(unsigned long long v, unsigned long long *s_w, unsigned long long &sum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    unsigned long long off = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kGroupThreads / 32; ++w) {
        const unsigned long long y = s_w[w];
        off += w < warp ? y : 0ull;
        tot += y;
    }
    sum = tot;
    return x - v + off;
}

// Signed amplitude of a member: the parity of removing the x-th and y-th electron, and one more exchange when a
// mixed pair has its beta orbital first (pair codes put alpha first).
__device__ __forceinline__ double signed_c(const double *c, unsigned I, unsigned short pr, int ox, int oy) {
    const double v = __ldg(c + I);
    const int par = ((pr & 0xFF) + (pr >> 8) + (((ox ^ oy) & ox) & 1)) & 1;
    return par ? -v : v;
}

template <int W>
struct GroupShared {
    unsigned long long rec[kGroupCap];
    unsigned table[kGroupSlots];       // (leading record << 16) | count, later (start << 16) | members placed
    unsigned short slot[kGroupCap];    // a record's slot
    unsigned short order[kGroupCap];   // record at each place of the kept members
    unsigned short code[kGroupCap];    // of the member at a place: pair code, bit 15: negative sign
    unsigned short orb[kGroupCap];     // its spin orbitals, x | y << 8
    unsigned short pairs[fq::MAXPAIRS];
    unsigned long long scan[kGroupThreads / 32];
    unsigned long long lo, hi;         // smallest and largest hash of a selection
    unsigned long long leader[kBigLeaders][W];
    unsigned long long acc[3];
    unsigned n, min_t, kept;
};

// Records s.rec[0, s.n) grouped by key; groups of two and more go to members + base + s.kept, longer groups first (four size
// classes), members in the order of their codes, so that the lanes of the pair passes have rows of similar length
// and neighbouring table columns. Grouping goes by the hash bits; every member's key is then compared with its
// group's first, and where two keys share the hash, false is returned to the whole block and nothing is written:
// called again with `exact`, the keys themselves are compared on insertion. That happens to about
// 2850^2 / 2 / 2^30 = 0.4% of the partitions of 1.2e8 keys (2,850 distinct keys, 30 hash bits left in a
// partition), 120 of 32,768.
template <int W>
__device__ __forceinline__ bool group_shared(GroupShared<W> &s, const unsigned long long *dets, const double *c, int npairs,
                                             int n_orb, int tbits, Member *members, unsigned base, Head *heads, RdmState *st,
                                             bool exact) {
    Member *out = members + base;
    constexpr unsigned kFree = 0xFFFFFFFFu;
    const unsigned n = s.n;
    for (int h = threadIdx.x; h < kGroupSlots; h += kGroupThreads) s.table[h] = kFree;
    __syncthreads();
    for (unsigned i = threadIdx.x; i < n; i += kGroupThreads) {
        const unsigned long long r = s.rec[i];
        unsigned h = (unsigned)(rec_hash(r, tbits) >> kFineBits) & (kGroupSlots - 1);
        for (int probe = 0; probe < kGroupSlots; ++probe) {  // ends earlier: the table has more slots than records
            unsigned e = *(volatile unsigned *)&s.table[h];
            if (e == kFree) {
                e = atomicCAS(&s.table[h], kFree, (i << 16) | 1u);
                if (e == kFree) {
                    s.slot[i] = (unsigned short)h;
                    break;
                }
            }
            const unsigned long long q = s.rec[e >> 16];
            bool match = rec_hash(q, tbits) == rec_hash(r, tbits);
            if (exact && match) {
                unsigned long long key[W], other[W];
                key_of<W>(dets, s.pairs, npairs, rec_t(r, tbits), key);
                key_of<W>(dets, s.pairs, npairs, rec_t(q, tbits), other);
                match = same_key<W>(key, other);
            }
            if (match) {
                atomicAdd(&s.table[h], 1u);
                s.slot[i] = (unsigned short)h;
                break;
            }
            h = (h + 1) & (kGroupSlots - 1);
        }
    }
    __syncthreads();
    // member places by size class: 32 and more, 8.., 3.., 2 (16-bit fields of one scan)
    constexpr int kPer = kGroupSlots / kGroupThreads;
    unsigned long long mine = 0, buckets = 0, pairs = 0;
    for (int k = 0; k < kPer; ++k) {
        const unsigned e = s.table[k * kGroupThreads + threadIdx.x];
        if (e == kFree) continue;
        const unsigned m = e & 0xFFFFu;
        ++buckets;
        if (m < 2) continue;
        pairs += (unsigned long long)m * (m - 1) / 2;
        mine += (unsigned long long)m << (m >= 32 ? 0 : m >= 8 ? 16 : m >= 3 ? 32 : 48);
    }
    unsigned long long total = 0;
    unsigned long long off = block_scan64(mine, s.scan, total);
    const unsigned t0 = (unsigned)(total & 0xFFFF), t1 = (unsigned)((total >> 16) & 0xFFFF), t2 = (unsigned)((total >> 32) & 0xFFFF),
                   t3 = (unsigned)(total >> 48);
    const unsigned placed = t0 + t1 + t2 + t3;
    off += ((unsigned long long)t0 << 16) + ((unsigned long long)(t0 + t1) << 32) + ((unsigned long long)(t0 + t1 + t2) << 48);
    for (int k = 0; k < kPer; ++k) {
        const unsigned h = k * kGroupThreads + threadIdx.x, e = s.table[h];
        if (e == kFree) continue;
        const unsigned m = e & 0xFFFFu;
        if (m < 2) {
            s.table[h] = kFree;  // a key of one determinant: dropped
        } else {
            const int sh = m >= 32 ? 0 : m >= 8 ? 16 : m >= 3 ? 32 : 48;
            s.table[h] = (unsigned)((off >> sh) & 0xFFFF) << 16;
            off += (unsigned long long)m << sh;
        }
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < n; i += kGroupThreads) {
        const unsigned h = s.slot[i];
        if (s.table[h] == kFree) continue;
        const unsigned e = atomicAdd(&s.table[h], 1u);
        s.order[(e >> 16) + (e & 0xFFFFu)] = (unsigned short)i;
    }
    __syncthreads();
    for (unsigned at = threadIdx.x; at < placed; at += kGroupThreads) {
        unsigned long long key[W];
        const KeyOf q = key_of<W>(dets, s.pairs, npairs, rec_t(s.rec[s.order[at]], tbits), key);
        const unsigned short pr = s.pairs[q.k];
        const unsigned par = ((pr & 0xFF) + (pr >> 8) + (((q.ox ^ q.oy) & q.ox) & 1)) & 1;
        s.code[at] = (unsigned short)(pair_code(q.ox, q.oy, n_orb) | (par << 15));
        s.orb[at] = (unsigned short)(q.ox | (q.oy << 8));
    }
    __syncthreads();
    if (!exact) {
        // the same key: the determinants differ by the two pairs
        bool bad = false;
        for (unsigned at = threadIdx.x; at < placed; at += kGroupThreads) {
            const unsigned i = s.order[at], first = s.table[s.slot[i]] >> 16;
            if (first == at) continue;
            unsigned long long a[W], b[W];
            load_det<W>(dets, rec_t(s.rec[i], tbits) / (unsigned)npairs, a);
            load_det<W>(dets, rec_t(s.rec[s.order[first]], tbits) / (unsigned)npairs, b);
            const unsigned x = s.orb[at], y = s.orb[first];
            fq::flip<W>(a, x & 0xFF);
            fq::flip<W>(a, x >> 8);
            fq::flip<W>(b, y & 0xFF);
            fq::flip<W>(b, y >> 8);
            if (!same_key<W>(a, b)) bad = true;
        }
        // one verdict for the block, and the barrier after which the caller may fill the table again (a flag in shared
        // memory would be cleared by the next call while slower warps still read it)
        if (__syncthreads_or(bad)) return false;
    }
    const unsigned kept = s.kept;
    for (unsigned at = threadIdx.x; at < placed; at += kGroupThreads) {
        const unsigned i = s.order[at], e = s.table[s.slot[i]];
        const unsigned first = e >> 16, m = e & 0xFFFFu, ci = s.code[at], code = ci & 0x7FFFu;
        unsigned rank = 0;
        for (unsigned j = first; j < first + m; ++j) {
            const unsigned cj = s.code[j] & 0x7FFFu;
            rank += (cj < code || (cj == code && j < at)) ? 1u : 0u;
        }
        const double v = __ldg(c + rec_t(s.rec[i], tbits) / (unsigned)npairs);
        Member o;
        o.v = code == kNoPair ? 0.0 : (ci & 0x8000u) ? -v : v;
        o.code = (code == kNoPair ? 0u : code) | ((m >= kTriangle ? kLarge : m) << 15);
        o.first = kept + first;
        out[kept + first + rank] = o;
        if (at == first && m >= kTriangle) heads[atomicAdd(&st->n_heads, 1u)] = Head{base + kept + first, m};
    }
    for (int o = 16; o > 0; o >>= 1) {
        buckets += __shfl_down_sync(0xFFFFFFFFu, buckets, o);
        pairs += __shfl_down_sync(0xFFFFFFFFu, pairs, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&s.acc[0], buckets);
        atomicAdd(&s.acc[2], pairs);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        s.kept = kept + placed;
        s.acc[1] += placed;
    }
    __syncthreads();
    return true;
}

// More than kGroupCap records of one partition with the same hash bits (a key shared by thousands of
// determinants): the distinct keys are taken one after another (smallest record first), each in two passes
// over the partition; its members are written in the order the threads meet them.
template <int W>
__device__ void group_big(GroupShared<W> &s, const unsigned long long *rec, unsigned size, unsigned long long hash,
                          const unsigned long long *dets, const double *c, int npairs, int n_orb, int tbits, Member *members, unsigned base,
                          Head *heads, RdmState *st) {
    Member *out = members + base;
    for (int nl = 0;; ++nl) {
        if (threadIdx.x == 0) {
            s.min_t = 0xFFFFFFFFu;
            s.n = 0;
        }
        __syncthreads();
        for (unsigned i = threadIdx.x; i < size; i += kGroupThreads) {
            const unsigned long long r = rec[i];
            if (rec_hash(r, tbits) != hash) continue;
            unsigned long long key[W];
            key_of<W>(dets, s.pairs, npairs, rec_t(r, tbits), key);
            bool seen = false;
            for (int l = 0; l < nl; ++l) seen = seen || same_key<W>(key, s.leader[l]);
            if (!seen) atomicMin(&s.min_t, rec_t(r, tbits));
        }
        __syncthreads();
        const unsigned t = s.min_t;
        if (t == 0xFFFFFFFFu) return;
        if (nl >= kBigLeaders) {
            if (threadIdx.x == 0) atomicCAS(&st->status, 0, FCIQMC_ERR_CAPACITY);
            return;
        }
        unsigned long long lead[W];
        key_of<W>(dets, s.pairs, npairs, t, lead);
        if (threadIdx.x == 0)
            for (int w = 0; w < W; ++w) s.leader[nl][w] = lead[w];
        for (unsigned i = threadIdx.x; i < size; i += kGroupThreads) {
            const unsigned long long r = rec[i];
            if (rec_hash(r, tbits) != hash) continue;
            unsigned long long key[W];
            key_of<W>(dets, s.pairs, npairs, rec_t(r, tbits), key);
            if (same_key<W>(key, lead)) atomicAdd(&s.n, 1u);
        }
        __syncthreads();
        const unsigned m = s.n, kept = s.kept;
        __syncthreads();
        if (threadIdx.x == 0) {
            s.acc[0] += 1;
            s.n = 0;
            if (m >= 2) {
                s.acc[1] += m;
                s.acc[2] += (unsigned long long)m * (m - 1) / 2;
                s.kept = kept + m;
                if (m >= kTriangle) heads[atomicAdd(&st->n_heads, 1u)] = Head{base + kept, m};
            }
        }
        __syncthreads();
        if (m < 2) continue;
        for (unsigned i = threadIdx.x; i < size; i += kGroupThreads) {
            const unsigned long long r = rec[i];
            if (rec_hash(r, tbits) != hash) continue;
            unsigned long long key[W];
            const KeyOf q = key_of<W>(dets, s.pairs, npairs, rec_t(r, tbits), key);
            if (!same_key<W>(key, lead)) continue;
            Member o;
            const unsigned code = pair_code(q.ox, q.oy, n_orb);
            o.v = code == kNoPair ? 0.0 : signed_c(c, q.I, s.pairs[q.k], q.ox, q.oy);
            o.code = (code == kNoPair ? 0u : code) | ((m >= kTriangle ? kLarge : m) << 15);
            o.first = kept;
            out[kept + atomicAdd(&s.n, 1u)] = o;
        }
        __syncthreads();
    }
}

// One block per partition: its records in shared memory (in parts by further hash bits when there are more than
// fit), grouped by key, the groups of two and more written as members at the partition's place.
template <int W>
__global__ void __launch_bounds__(kGroupThreads, 2) k_group(const unsigned long long *dets, const double *c, int n_elec, int n_orb,
                                                            int tbits, const unsigned long long *records, const unsigned *base_p,
                                                            Member *members, unsigned *count_p, Head *heads, RdmState *st) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    GroupShared<W> &s = *reinterpret_cast<GroupShared<W> *>(s_raw);
    const int npairs = n_elec * (n_elec - 1) / 2;
    fill_pairs(n_elec, s.pairs);
    if (threadIdx.x < 3) s.acc[threadIdx.x] = 0;
    if (threadIdx.x == 0) s.kept = 0;
    const unsigned base = base_p[blockIdx.x], size = base_p[blockIdx.x + 1] - base;
    const unsigned long long *rec = records + base;
    if (size <= (unsigned)kGroupCap) {
        for (unsigned i = threadIdx.x; i < size; i += kGroupThreads) s.rec[i] = rec[i];
        if (threadIdx.x == 0) s.n = size;
        __syncthreads();
        if (size && !group_shared<W>(s, dets, c, npairs, n_orb, tbits, members, base, heads, st, false)) group_shared<W>(s, dets, c, npairs, n_orb, tbits, members, base, heads, st, true);
    } else {
        // sub-partitions by the leading `depth` bits of the hash, deeper where one is still too long
        int d0 = 1;
        while (((unsigned)kGroupCap / 2) << d0 < size && d0 < 20) ++d0;
        int depth = d0;
        unsigned long long sub = 0;
        while (sub < (1ull << depth)) {
            if (threadIdx.x == 0) {
                s.n = 0;
                s.lo = ~0ull;
                s.hi = 0;
            }
            __syncthreads();
            for (unsigned i = threadIdx.x; i < size; i += kGroupThreads) {
                const unsigned long long r = rec[i];
                if (rec_hash(r, tbits) >> (64 - tbits - depth) != sub) continue;
                const unsigned k = atomicAdd(&s.n, 1u);
                if (k < (unsigned)kGroupCap) s.rec[k] = r;
                atomicMin(&s.lo, rec_hash(r, tbits));
                atomicMax(&s.hi, rec_hash(r, tbits));
            }
            __syncthreads();
            const unsigned m = s.n;
            if (m > (unsigned)kGroupCap && s.lo != s.hi) {  // two hashes share these bits, so there are more
                ++depth;
                sub <<= 1;
                __syncthreads();
                continue;
            }
            const unsigned long long hash = s.lo;
            __syncthreads();
            if (m > (unsigned)kGroupCap) group_big<W>(s, rec, size, hash, dets, c, npairs, n_orb, tbits, members, base, heads, st);
            else if (m && !group_shared<W>(s, dets, c, npairs, n_orb, tbits, members, base, heads, st, false)) group_shared<W>(s, dets, c, npairs, n_orb, tbits, members, base, heads, st, true);
            __syncthreads();
            ++sub;
            while (depth > d0 && !(sub & 1ull)) {
                sub >>= 1;
                --depth;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        count_p[blockIdx.x] = s.kept;
        if (s.acc[0]) atomicAdd(&st->n_buckets, s.acc[0]);
        if (s.acc[1]) atomicAdd(&st->n_members, s.acc[1]);
        if (s.acc[2]) atomicAdd(&st->n_pairs, s.acc[2]);
    }
}

// The tasks of the large groups, a warp per group. They lie where the records were: at most m / 2 of 16 bytes for a
// group of m (one for 32 rows up to kTaskPartners, kTaskShares at most), and a record is 8 bytes.
__device__ __forceinline__ void make_tasks(const Head *heads, Task *tasks, RdmState *st, unsigned g, unsigned warps) {
    const int lane = threadIdx.x & 31;
    const unsigned n = st->n_heads;
    for (; g < n; g += warps) {
        const Head q = heads[g];
        for (unsigned t0 = 0; t0 * 32u < q.m; t0 += 32) {  // a tile of 32 rows per lane
            const unsigned row0 = 32u * (t0 + (unsigned)lane);
            const unsigned mine = row0 < q.m ? min((row0 + 32u + kTaskPartners - 1) / kTaskPartners, (unsigned)kTaskShares) : 0u;
            unsigned x = mine;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                if (lane >= o) x += y;
            }
            unsigned long long at = 0;
            if (lane == 31) at = atomicAdd(&st->n_tasks, (unsigned long long)x);
            at = __shfl_sync(0xFFFFFFFFu, at, 31) + (x - mine);
            for (unsigned k = 0; k < mine; ++k) tasks[at + k] = Task{q.first, q.m, row0, (unsigned short)k, (unsigned short)mine};
        }
    }
}

// ------------------------------------------------------------------------------------ compensated sums
// Sum and running error of a sequence of FP64 additions (Knuth's TwoSum per addition, Neumaier's
// compensated summation): the result is the rounded exact sum up to a few ulp whatever the number of
// additions, so finite differences of E are not swamped by accumulated rounding. A compensated addition costs
// seven plain ones, so terms are added plainly first, a bounded number at a time (k_pair_energy).
struct alignas(16) CSum {
    double s, c;
};
__device__ __forceinline__ void csum_add(CSum &a, double x) {
    const double t = __dadd_rn(a.s, x);
    const double bb = __dsub_rn(t, a.s);
    const double err = __dadd_rn(__dsub_rn(a.s, __dsub_rn(t, bb)), __dsub_rn(x, bb));
    a.s = t;
    a.c = __dadd_rn(a.c, err);
}
__device__ __forceinline__ void csum_merge(CSum &a, const CSum &b) {
    csum_add(a, b.s);
    a.c = __dadd_rn(a.c, b.c);
}

// Fixed-tree merges (the same order in every run): lanes pairwise by shuffles, then the warps' results.
__device__ __forceinline__ CSum warp_csum(CSum a) {
    for (int o = 16; o > 0; o >>= 1) {
        const CSum b{__shfl_down_sync(0xFFFFFFFFu, a.s, o), __shfl_down_sync(0xFFFFFFFFu, a.c, o)};
        csum_merge(a, b);
    }
    return a;  // lane 0 holds the warp's sum
}
// Block sum of every thread's acc, in thread 0; s: one slot per warp.
__device__ __forceinline__ CSum block_csum(CSum acc, CSum *s) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    acc = warp_csum(acc);
    if (lane == 0) s[warp] = acc;
    __syncthreads();
    CSum x{0.0, 0.0};
    if (warp == 0) {
        if (lane < (int)(blockDim.x >> 5)) x = s[lane];
        x = warp_csum(x);
    }
    __syncthreads();
    return x;
}

// ------------------------------------------------------------------------------------ diagonal
// Occupation-pair sums over spin orbitals p <= q, O_pq = sum_I c_I^2 n_p n_q at q (q + 1) / 2 + p (p == q: the
// occupations). One determinant per warp at a time: the lanes hold its occupied list and take its pairs, which are
// distinct, so each warp adds into a copy of its own in shared memory without atomics (shared FP64 atomics are
// compare-and-swap loops, and the core pairs, occupied in nearly every determinant, made all lanes retry on
// one word). A warp adds kOccPlain determinants plainly; then the block adds its copies, in warp order, to its compensated
// sums in occ_part[block] (all of a warp's determinants added plainly, the occupation of a core orbital came out 188 times
// 2^-53 off for 4e5 equal amplitudes in 64 orbitals, and E of 1e6 determinants of 16e/40o 1.7e-13; now 13 times and 5e-15).
// Bound by the FP64 pipe: construction for 1e6 determinants of 16e/40o and 3e5 of 24e/60o 5.48 and 4.12 ms without the
// compensated sums, 5.60 and 4.20 with 128 determinants between them, 5.70 and 4.29 with 64.
constexpr int kOccPlain = 64;
constexpr int kOccThreads = 256;
template <int W>
__global__ void __launch_bounds__(kOccThreads) k_occ_pairs(const unsigned long long *dets, const double *c, long long n, int n_elec,
                                                           int n_so, int nw, CSum *occ_part) {
    extern __shared__ double s_o[];
    __shared__ unsigned short s_pairs[fq::MAXPAIRS];
    fill_pairs(n_elec, s_pairs);
    const int nent = n_so * (n_so + 1) / 2, npairs = n_elec * (n_elec - 1) / 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < nent * nw; k += blockDim.x) s_o[k] = 0.0;
    __syncthreads();
    double *o = s_o + nent * warp;
    const long long step = (long long)gridDim.x * nw;
    long long I = warp < nw ? (long long)blockIdx.x * nw + warp : n;
    // the lane's occupied orbitals (ranks lane and lane + 32; ranks beyond the electrons are not used) and c^2, of the
    // next determinant while the current one's sums are in flight
    auto decode = [&](long long i, int &k0, int &k1, double &c2) {
        unsigned long long d[W];
        load_det<W>(dets, i, d);
        const double ci = __ldg(c + i);
        k0 = fq::select_bit<W>(d, lane);
        k1 = n_elec > 32 ? fq::select_bit<W>(d, lane + 32) : 0;
        c2 = __dmul_rn(ci, ci);
    };
    int k0 = 0, k1 = 0, nk0 = 0, nk1 = 0;
    double c2 = 0.0, nc2 = 0.0;
    if (I < n) decode(I, k0, k1, c2);
    CSum *sums = occ_part + (size_t)blockIdx.x * nent;
    for (long long i0 = (long long)blockIdx.x * nw; i0 < n; i0 += step * kOccPlain) {
        for (int left = kOccPlain; left > 0 && I < n; --left, I += step, k0 = nk0, k1 = nk1, c2 = nc2) {
            if (I + step < n) decode(I + step, nk0, nk1, nc2);
            // four pairs of a lane at a time: their words are distinct, so the loads need not wait for the stores
            for (int k0s = 0; k0s < npairs; k0s += 128) {
                double *e[4], x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = k0s + 32 * u + lane;
                    const unsigned short pr = k < npairs ? s_pairs[k] : 0;
                    const int rx = pr & 0xFF, ry = pr >> 8;
                    int p = __shfl_sync(0xFFFFFFFFu, k0, rx & 31), q = __shfl_sync(0xFFFFFFFFu, k0, ry & 31);
                    if (n_elec > 32) {
                        const int p1 = __shfl_sync(0xFFFFFFFFu, k1, rx & 31), q1 = __shfl_sync(0xFFFFFFFFu, k1, ry & 31);
                        if (rx >= 32) p = p1;
                        if (ry >= 32) q = q1;
                    }
                    e[u] = k < npairs && p <= q && q < n_so ? o + q * (q + 1) / 2 + p : nullptr;
                    x[u] = e[u] ? *e[u] : 0.0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (e[u]) *e[u] = __dadd_rn(x[u], c2);
            }
            if (lane < n_elec && k0 < n_so) {
                double *e = o + k0 * (k0 + 1) / 2 + k0;
                *e = __dadd_rn(*e, c2);
            }
            if (lane + 32 < n_elec && k1 < n_so) {
                double *e = o + k1 * (k1 + 1) / 2 + k1;
                *e = __dadd_rn(*e, c2);
            }
            __syncwarp();
        }
        __syncthreads();
        const bool first = i0 < step, last = i0 + step * kOccPlain >= n;
        for (int k0 = threadIdx.x; k0 < nent; k0 += 4 * kOccThreads) {  // four entries in flight
            CSum a[4];
            double t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + u * kOccThreads;
                a[u] = !first && k < nent ? sums[k] : CSum{0.0, 0.0};
                t[u] = k < nent ? s_o[k] : 0.0;
            }
            for (int w = 1; w < nw; ++w)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (k0 + u * kOccThreads < nent) t[u] = __dadd_rn(t[u], s_o[nent * w + k0 + u * kOccThreads]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + u * kOccThreads;
                if (k >= nent) continue;
                if (first) a[u].s = t[u];
                else csum_add(a[u], t[u]);
                sums[k] = a[u];
                if (!last)
                    for (int w = 0; w < nw; ++w) s_o[nent * w + k] = 0.0;
            }
        }
        __syncthreads();
    }
}

// Sums of the blocks' occupation pairs (compensated): a warp adds 8 entries, four lanes each taking every fourth block in
// order, merged in a fixed tree (the first n_merge blocks). The next block adds the partial sums of c^2, the others make
// the tasks of the large groups, which need k_group's heads only and here cost no launch and no time.
__global__ void __launch_bounds__(kMergeThreads) k_occ_merge(const CSum *occ_part, int nblocks, int nent, double *occ_pair, int n_merge,
                                                             const double *norm_part, int n_norm, const Head *heads, Task *tasks,
                                                             RdmState *st) {
    if ((int)blockIdx.x > n_merge) {
        constexpr unsigned kWarps = kMergeThreads / 32;
        make_tasks(heads, tasks, st, (blockIdx.x - n_merge - 1) * kWarps + (threadIdx.x >> 5), (gridDim.x - n_merge - 1) * kWarps);
        return;
    }
    if ((int)blockIdx.x == n_merge) {
        __shared__ CSum s[kMergeThreads / 32];
        CSum a{0.0, 0.0};
        for (int b = threadIdx.x; b < n_norm; b += kMergeThreads) csum_merge(a, CSum{norm_part[2 * b], norm_part[2 * b + 1]});
        a = block_csum(a, s);
        if (threadIdx.x == 0) st->norm = __dadd_rn(a.s, a.c);
        return;
    }
    const int lane = threadIdx.x & 31, part = lane >> 3;
    const int k = (blockIdx.x * (kMergeThreads / 32) + (threadIdx.x >> 5)) * 8 + (lane & 7);
    CSum a{0.0, 0.0};
    if (k < nent)
        for (int b0 = part; b0 < nblocks; b0 += 16) {  // four reads in flight
            CSum x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = b0 + 4 * u < nblocks ? occ_part[(size_t)(b0 + 4 * u) * nent + k] : CSum{0.0, 0.0};
#pragma unroll
            for (int u = 0; u < 4; ++u) csum_merge(a, x[u]);
        }
    for (int o = 16; o >= 8; o >>= 1) {
        const CSum b{__shfl_down_sync(0xFFFFFFFFu, a.s, o), __shfl_down_sync(0xFFFFFFFFu, a.c, o)};
        csum_merge(a, b);
    }
    if (k < nent && part == 0) occ_pair[k] = __dadd_rn(a.s, a.c);
}

__global__ void __launch_bounds__(kThreads) k_norm(const double *c, long long n, double *partial) {
    __shared__ CSum s[kThreads / 32];
    CSum v{0.0, 0.0};
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        csum_add(v, __dmul_rn(c[i], c[i]));
    v = block_csum(v, s);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = v.s;
        partial[2 * blockIdx.x + 1] = v.c;
    }
}

// ------------------------------------------------------------------------------------ pairs
// h / (N - 1), the share of one key in a one-electron element (divided for each entry that needs it, k_pair_table and k_fold
// took far longer; a product with the rounded inverse has two roundings, the same ones at all N - 1 keys).
__global__ void __launch_bounds__(kThreads) k_share(const double *h, int n, double keys, double *share) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) share[k] = __ddiv_rn(h[k], keys);
}

// T over pair codes: the same-spin block (n1 x n1, rows and columns p < q), then the mixed block (n2 x n2, alpha
// first); zero on the diagonals (the diagonal of H comes from the occupation-pair sums), and only columns from the
// diagonal on: T is symmetric and the pair passes read and add at (smaller code, larger code). The table grows with the
// basis and not with the list: E of 5,000 determinants of 8e/64o, 2.1e7 entries, took 228 us with whole rows, 163 so.
__global__ void __launch_bounds__(kThreads) k_pair_table(const double *share, const double *eri, int n_orb, int n1, int n2,
                                                         double *table) {
    const int row = blockIdx.y;
    if (row < n1) {
        int p, q;
        triangle_of(row, p, q);
        for (int col = row + blockIdx.x * blockDim.x + threadIdx.x; col < n1; col += gridDim.x * blockDim.x) {
            int r, s;
            triangle_of(col, r, s);
            double v = 0.0;
            if (col != row) {
                v = __dsub_rn(__ldg(eri + fq::eidx(p, r, q, s)), __ldg(eri + fq::eidx(p, s, q, r)));
                if (q == s) v = __dadd_rn(v, __ldg(share + p * n_orb + r));
                if (p == r) v = __dadd_rn(v, __ldg(share + q * n_orb + s));
                if (q == r) v = __dsub_rn(v, __ldg(share + p * n_orb + s));
                if (p == s) v = __dsub_rn(v, __ldg(share + q * n_orb + r));
            }
            table[(size_t)row * n1 + col] = v;
        }
    } else {
        const int row2 = row - n1, p = row2 / n_orb, q = row2 - p * n_orb;
        for (int col = row2 + blockIdx.x * blockDim.x + threadIdx.x; col < n2; col += gridDim.x * blockDim.x) {
            const int r = col / n_orb, s = col - r * n_orb;
            double v = 0.0;
            if (col != row2) {
                v = __ldg(eri + fq::eidx(p, r, q, s));
                if (q == s) v = __dadd_rn(v, __ldg(share + p * n_orb + r));
                if (p == r) v = __dadd_rn(v, __ldg(share + q * n_orb + s));
            }
            table[(size_t)n1 * n1 + (size_t)row2 * n2 + col] = v;
        }
    }
}

// The partners of member j of a group of m starting at `first`, so that every pair is met once: small groups
// cyclically (each member takes about half of the others, so the lanes of a warp, in groups of similar size,
// finish together). Large ones (m >= kTriangle) are not a partition's business: their rows are triangles, in which
// the lanes of a warp meet the same partner at the same time and read neighbouring columns of its table row, and
// they are dealt out to the warps of all blocks (Task). A list of few keys is a few large groups (two electrons: one), and
// in a vector around a reference they hold most pairs; as rows of the block that has the partition, the 3.3e7 pairs of
// 8,128 determinants of two electrons took E 68.6 ms and its gradient 24.1 (0.41 and 0.25 as tasks), those of 1e6
// determinants of 16e/40o 1.86 and 1.59 (1.33 and 1.40; shares of 512 partners instead of 128, in launches of their own:
// 1.47 and 1.62, and 12 us more for 3e3 determinants, whose longest share was the launch).
struct RowRange {
    int n;        // partners
    int at;       // first partner, counted from the group's start
    int wrap;     // group size
};
__device__ __forceinline__ RowRange row_range(unsigned packed, int local) {
    const int m = (int)(packed >> 15);
    if (m == (int)kLarge) return RowRange{0, 0, 0};
    const int half = (m - 1) >> 1, even = (m & 1) == 0 && local < (m >> 1) ? 1 : 0;
    return RowRange{half + even, local + 1 < m ? local + 1 : 0, m};
}

__device__ __forceinline__ double pair_entry(const double *t, int stride, unsigned a, unsigned b) {
    return __ldg(t + (size_t)min(a, b) * stride + max(a, b));
}

// The tasks of warp g of `warps`, a lane per row: f(its member, the group, k0, k1) for the task's blocks of 64 members
// before it.
template <typename F>
__device__ __forceinline__ void for_task_rows(const Member *members, const Task *tasks, unsigned long long n_tasks, unsigned g,
                                              unsigned warps, F f) {
    for (unsigned long long i = g; i < n_tasks; i += warps) {
        const Task t = tasks[i];
        const Member *grp = members + t.first;
        const unsigned row = t.row0 + (threadIdx.x & 31u);
        if (row >= t.m) continue;
        const Member u = grp[row];
        for (unsigned k0 = 64u * t.share; k0 < row; k0 += 64u * t.n_shares) f(u, grp, k0, min(k0 + 64u, row));
    }
}

// Thread t of n: half of its share of the diagonal, sum_p O_pp h_pp + sum_{p<q} O_pq ((pp|qq) - delta_spin (pq|qp)).
__device__ __forceinline__ CSum diagonal_energy(const double *occ_pair, const double *h, const double *eri, int n_orb, int t, int n) {
    CSum acc{0.0, 0.0};
    for (int k = t; k < n_orb * (2 * n_orb + 1); k += n) {
        int q = (int)((sqrtf(8.0f * (float)k + 1.0f) - 1.0f) * 0.5f);
        while (q * (q + 1) / 2 > k) --q;
        while ((q + 1) * (q + 2) / 2 <= k) ++q;
        const int p = k - q * (q + 1) / 2, P = p >> 1, Q = q >> 1;
        double x;
        if (p == q) {
            x = __ldg(h + P * n_orb + P);
        } else {
            x = __ldg(eri + fq::eidx(P, P, Q, Q));
            if ((p & 1) == (q & 1)) x = __dsub_rn(x, __ldg(eri + fq::eidx(P, Q, Q, P)));
        }
        csum_add(acc, 0.5 * __dmul_rn(occ_pair[k], x));
    }
    return acc;
}

// 2 c_I c_J H_IJ summed over the pairs of members, without the factor 2. The first `large` blocks take the tasks of the
// large groups, a warp each, the last kDiagBlocks half of the diagonal (in the one block that merges the sums it took 8 us in 40
// orbitals and 24 in 64), those between the partitions' small groups. A row is an FMA chain of eight partners at a time;
// per thread these parts are added plainly, at most eight of a large group's row or the four of kPlainRows rows of small
// ones, and then compensated, the blocks' sums in a fixed tree. So a pair is followed by at most 8 + 4 + kPlainRows plain
// additions whatever the length of the list (with one plain sum per row, thread and partition, 8.4e6 equal pairs of one
// key came out 48 times 2^-53 off).
// Bound by the FP64 pipe (one FMA per pair, charged per warp instruction) and the table reads from L2.
constexpr int kPlainRows = 16;
__global__ void __launch_bounds__(kPairThreads) k_pair_energy(const Member *members, const unsigned *base_p, const unsigned *count_p,
                                                          int parts, const Task *tasks, unsigned long long n_tasks, int large,
                                                          int n1, int n2, const double *table, const double *occ_pair,
                                                          const double *h, const double *eri, int n_orb, double *partial) {
    __shared__ CSum s_red[kPairThreads / 32];
    CSum acc{0.0, 0.0};
    const double *mixed = table + (size_t)n1 * n1;
    const int small = (int)gridDim.x - large - kDiagBlocks;
    if ((int)blockIdx.x < large) {
        constexpr unsigned kWarps = kPairThreads / 32;
        for_task_rows(members, tasks, n_tasks, blockIdx.x * kWarps + (threadIdx.x >> 5), (unsigned)large * kWarps,
                      [&](const Member &u, const Member *grp, unsigned k0, unsigned k1) {
            const unsigned cls = (u.code >> 13) & 3u, cu = u.code & 0x1FFFu;
            const double *t = cls == 2u ? mixed : table;
            const int stride = cls == 2u ? n2 : n1;
            double row = 0.0;
            for (; k0 < k1; k0 += 8) {
                double part = 0.0;
                const unsigned end = min(k0 + 8u, k1);
#pragma unroll 4
                for (unsigned k = k0; k < end; ++k) {
                    const Member w = grp[k];
                    if (((w.code >> 13) & 3u) == cls) part = __fma_rn(pair_entry(t, stride, cu, w.code & 0x1FFFu), w.v, part);
                }
                row = __dadd_rn(row, part);
            }
            csum_add(acc, __dmul_rn(u.v, row));
        });
    } else if ((int)blockIdx.x >= large + small) {
        acc = diagonal_energy(occ_pair, h, eri, n_orb, ((int)blockIdx.x - large - small) * kPairThreads + threadIdx.x, kDiagBlocks * kPairThreads);
    } else {
        for (int p = (int)blockIdx.x - large; p < parts; p += small) {
            const Member *mem = members + base_p[p];
            const int cnt = (int)count_p[p];
            if ((int)threadIdx.x >= cnt) continue;
            for (int j0 = threadIdx.x; j0 < cnt; j0 += kPlainRows * kPairThreads) {
                const int j1 = min(j0 + kPlainRows * kPairThreads, cnt);
                double sum = 0.0;
                for (int j = j0; j < j1; j += kPairThreads) {
                    const Member u = mem[j];
                    const Member *grp = mem + u.first;
                    const RowRange r = row_range(u.code, j - (int)u.first);
                    const unsigned cls = (u.code >> 13) & 3u, cu = u.code & 0x1FFFu;
                    const double *t = cls == 2u ? mixed : table;
                    const int stride = cls == 2u ? n2 : n1;
                    double row = 0.0;
                    int at = r.at;
                    for (int k0 = 0; k0 < r.n; k0 += 8) {
                        double part = 0.0;
                        const int k1 = min(k0 + 8, r.n);
#pragma unroll 4
                        for (int k = k0; k < k1; ++k) {
                            const Member w = grp[at];
                            at = at + 1 == r.wrap ? 0 : at + 1;
                            if (((w.code >> 13) & 3u) == cls) part = __fma_rn(pair_entry(t, stride, cu, w.code & 0x1FFFu), w.v, part);
                        }
                        row = __dadd_rn(row, part);
                    }
                    sum = __fma_rn(u.v, row, sum);
                }
                csum_add(acc, sum);
            }
        }
    }
    acc = block_csum(acc, s_red);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = acc.s;
        partial[2 * blockIdx.x + 1] = acc.c;
    }
}

// One block: the blocks' sums (pairs twice: both orders), merged in a fixed order; over c^T c.
__global__ void __launch_bounds__(1024) k_energy_finish(const double *partial, int n, const RdmState *st, double *e) {
    __shared__ CSum s_red[32];
    CSum tot{0.0, 0.0};
    for (int b = threadIdx.x; b < n; b += blockDim.x) csum_merge(tot, CSum{2.0 * partial[2 * b], 2.0 * partial[2 * b + 1]});
    tot = block_csum(tot, s_red);
    if (threadIdx.x == 0) *e = __ddiv_rn(__dadd_rn(tot.s, tot.c), st->norm);
}

// The two-body density matrix over pair codes: v v' of every pair of members added at (smaller code, larger code) with
// one FP64 reduction in L2. Blocks as in k_pair_energy; in large groups a warp's reductions fall in one table row.
__global__ void __launch_bounds__(kPairThreads) k_pair_grad(const Member *members, const unsigned *base_p, const unsigned *count_p,
                                                        int parts, const Task *tasks, unsigned long long n_tasks, int large,
                                                        int n1, int n2, double *table) {
    double *mixed = table + (size_t)n1 * n1;
    auto add = [&](const Member &u, const Member &w) {
        const unsigned cls = (u.code >> 13) & 3u, cu = u.code & 0x1FFFu, cw = w.code & 0x1FFFu;
        if (((w.code >> 13) & 3u) == cls)
            atomicAdd((cls == 2u ? mixed : table) + (size_t)min(cu, cw) * (cls == 2u ? n2 : n1) + max(cu, cw), __dmul_rn(u.v, w.v));
    };
    if ((int)blockIdx.x < large) {
        constexpr unsigned kWarps = kPairThreads / 32;
        for_task_rows(members, tasks, n_tasks, blockIdx.x * kWarps + (threadIdx.x >> 5), (unsigned)large * kWarps,
                      [&](const Member &u, const Member *grp, unsigned k0, unsigned k1) {
#pragma unroll 4
            for (unsigned k = k0; k < k1; ++k) add(u, grp[k]);
        });
        return;
    }
    for (int p = (int)blockIdx.x - large; p < parts; p += (int)gridDim.x - large) {
        const Member *mem = members + base_p[p];
        const int cnt = (int)count_p[p];
        for (int j = threadIdx.x; j < cnt; j += kPairThreads) {
            const Member u = mem[j];
            const Member *grp = mem + u.first;
            const RowRange r = row_range(u.code, j - (int)u.first);
            int at = r.at;
#pragma unroll 4
            for (int k = 0; k < r.n; ++k) {
                const Member w = grp[at];
                at = at + 1 == r.wrap ? 0 : at + 1;
                add(u, w);
            }
        }
    }
}

// Maps the density matrix over pair codes (rows < columns) and the occupation-pair sums onto h and the packed ERIs. A
// one-electron element comes once per shared key: gh holds N - 1 times its value off the diagonal (k_scale_out divides).
__global__ void __launch_bounds__(kThreads) k_fold(const double *table, const double *occ_pair, int n_orb, int n1, int n2,
                                                   double *gh, double *ge) {
    auto one_body = [&](int a, int b, double v) {  // both h[a][b] and h[b][a]
        atomicAdd(&gh[a * n_orb + b], v);
        atomicAdd(&gh[b * n_orb + a], v);
    };
    const int row = blockIdx.y;
    if (row < n1) {
        int p, q;
        triangle_of(row, p, q);
        for (int col = row + 1 + blockIdx.x * blockDim.x + threadIdx.x; col < n1; col += gridDim.x * blockDim.x) {
            const double g = table[(size_t)row * n1 + col];
            if (g == 0.0) continue;
            int r, s;
            triangle_of(col, r, s);
            atomicAdd(&ge[fq::eidx(p, r, q, s)], 2.0 * g);
            atomicAdd(&ge[fq::eidx(p, s, q, r)], -2.0 * g);
            if (q == s) one_body(p, r, g);
            if (p == r) one_body(q, s, g);
            if (q == r) one_body(p, s, -g);
            if (p == s) one_body(q, r, -g);
        }
    } else if (row < n1 + n2) {
        const int row2 = row - n1, p = row2 / n_orb, q = row2 - p * n_orb;
        for (int col = row2 + 1 + blockIdx.x * blockDim.x + threadIdx.x; col < n2; col += gridDim.x * blockDim.x) {
            const double g = table[(size_t)n1 * n1 + (size_t)row2 * n2 + col];
            if (g == 0.0) continue;
            const int r = col / n_orb, s = col - r * n_orb;
            atomicAdd(&ge[fq::eidx(p, r, q, s)], 2.0 * g);
            if (q == s) one_body(p, r, g);
            if (p == r) one_body(q, s, g);
        }
    } else if (blockIdx.x == 0) {  // spin orbital q: O_pq for p <= q
        const int q = row - n1 - n2, Q = q >> 1;
        for (int p = threadIdx.x; p <= q; p += blockDim.x) {
            const double v = occ_pair[q * (q + 1) / 2 + p];
            if (v == 0.0) continue;
            const int P = p >> 1;
            if (p == q) {
                atomicAdd(&gh[P * n_orb + P], v);
            } else {
                atomicAdd(&ge[fq::eidx(P, P, Q, Q)], v);
                if ((p & 1) == (q & 1)) atomicAdd(&ge[fq::eidx(P, Q, Q, P)], -v);
            }
        }
    }
}

// Connected pairs for fciqmc_rdm_info: pairs of members with one spin orbital in common (each single excitation
// N - 1 times, once per shared key) and with none (the double excitations). Blocks as in the pair passes (as rows of the
// partition's block, one key of 8,128 determinants took 27 ms); dynamic shared memory: the spin orbitals of a code.
__global__ void __launch_bounds__(kPairThreads) k_pair_count(const Member *members, const unsigned *base_p, const unsigned *count_p,
                                                         int parts, const Task *tasks, unsigned long long n_tasks, int large,
                                                         int n_orb, int n1, int n2, RdmState *st) {
    extern __shared__ unsigned short s_orb[];  // x | y << 8: alpha alpha, beta beta, mixed
    for (int k = threadIdx.x; k < n1; k += kPairThreads) {
        int p, q;
        triangle_of(k, p, q);
        s_orb[k] = (unsigned short)(2 * p | (2 * q) << 8);
        s_orb[n1 + k] = (unsigned short)((2 * p + 1) | (2 * q + 1) << 8);
    }
    for (int k = threadIdx.x; k < n2; k += kPairThreads) s_orb[2 * n1 + k] = (unsigned short)(2 * (k / n_orb) | (2 * (k % n_orb) + 1) << 8);
    __syncthreads();
    unsigned long long shared_n = 0, apart = 0;
    auto orbitals = [&](unsigned code) { return (unsigned)s_orb[((code >> 13) & 3u) * (unsigned)n1 + (code & 0x1FFFu)]; };
    auto count = [&](unsigned u, unsigned w) {
        const unsigned ux = u & 0xFFu, uy = u >> 8, wx = w & 0xFFu, wy = w >> 8;
        const int same = (ux == wx) + (ux == wy) + (uy == wx) + (uy == wy);
        shared_n += same == 1 ? 1 : 0;
        apart += same == 0 ? 1 : 0;
    };
    if ((int)blockIdx.x < large) {
        constexpr unsigned kWarps = kPairThreads / 32;
        for_task_rows(members, tasks, n_tasks, blockIdx.x * kWarps + (threadIdx.x >> 5), (unsigned)large * kWarps,
                      [&](const Member &u, const Member *grp, unsigned k0, unsigned k1) {
            const unsigned o = orbitals(u.code);
            for (unsigned k = k0; k < k1; ++k) count(o, orbitals(grp[k].code));
        });
    } else {
        for (int p = (int)blockIdx.x - large; p < parts; p += (int)gridDim.x - large) {
            const Member *mem = members + base_p[p];
            const int cnt = (int)count_p[p];
            for (int j = threadIdx.x; j < cnt; j += kPairThreads) {
                const Member u = mem[j];
                const Member *grp = mem + u.first;
                const RowRange r = row_range(u.code, j - (int)u.first);
                const unsigned o = orbitals(u.code);
                int at = r.at;
                for (int k = 0; k < r.n; ++k) {
                    count(o, orbitals(grp[at].code));
                    at = at + 1 == r.wrap ? 0 : at + 1;
                }
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        shared_n += __shfl_down_sync(0xFFFFFFFFu, shared_n, o);
        apart += __shfl_down_sync(0xFFFFFFFFu, apart, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (shared_n) atomicAdd(&st->n_shared, shared_n);
        if (apart) atomicAdd(&st->n_apart, apart);
    }
}

__global__ void k_scale_out(const double *gh, const double *ge, int n_orb, long long n_e, double keys, const double *scale,
                            const RdmState *st, double *out_h, double *out_e) {
    const double f = __ddiv_rn(*scale, st->norm);
    const int n_h = n_orb * n_orb;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n_h + n_e; k += (long long)gridDim.x * blockDim.x) {
        if (k < n_h) out_h[k] = __dmul_rn((int)k / n_orb == (int)k % n_orb ? gh[k] : __ddiv_rn(gh[k], keys), f);
        else out_e[k - n_h] = __dmul_rn(ge[k - n_h], f);
    }
}

}  // namespace

struct fciqmc_rdm {
    Dims d;
    RdmLayout L;
    char *ws;
    cudaStream_t s;
    RdmState host;
    bool rdm_ready;  // unscaled density matrices computed
};

namespace {
template <typename T>
T *ptr(const fciqmc_rdm *r, size_t off) {
    return reinterpret_cast<T *>(r->ws + off);
}

// Warps of a k_occ_pairs block that add determinants: as many copies of the occupation triangle as fit in 208 KB, at most
// all of them.
int occ_warps(const Dims &d) {
    const size_t nent = (size_t)d.n_so * (d.n_so + 1) / 2;
    return (int)std::max<size_t>(1, std::min<size_t>(kOccThreads / 32, (208u << 10) / (sizeof(double) * nent)));
}

template <int W>
int construct(fciqmc_rdm *r) {
    const Dims &d = r->d;
    cudaStream_t s = r->s;
    RdmState *st = ptr<RdmState>(r, r->L.state);
    const unsigned long long *dets = ptr<unsigned long long>(r, r->L.dets);
    const double *c = ptr<double>(r, r->L.c);
    unsigned *total = ptr<unsigned>(r, r->L.total_p), *base = ptr<unsigned>(r, r->L.base_p);
    unsigned *cursor = ptr<unsigned>(r, r->L.cursor_p), *coarse = ptr<unsigned>(r, r->L.coarse_p);
    unsigned long long *records = ptr<unsigned long long>(r, r->L.records);
    const size_t sm_hist = sizeof(unsigned) * d.parts, sm_group = sizeof(GroupShared<W>);
    const size_t sm_scatter = sizeof(ScatterShared);
    const size_t nent = (size_t)d.n_so * (d.n_so + 1) / 2, sm_occ = sizeof(double) * nent * occ_warps(d);
    if (cudaFuncSetAttribute(k_key_hist<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(unsigned) * kPartMax)) != cudaSuccess ||
        cudaFuncSetAttribute(k_key_scatter<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_scatter) != cudaSuccess ||
        cudaFuncSetAttribute(k_group<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_group) != cudaSuccess ||
        cudaFuncSetAttribute(k_occ_pairs<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, 208 << 10) != cudaSuccess)
        return FCIQMC_ERR_CUDA;
    cudaMemsetAsync(st, 0, sizeof(RdmState), s);
    cudaMemsetAsync(total, 0, sizeof(unsigned) * d.parts, s);
    k_key_hist<W><<<d.hash_blocks, kHashThreads, sm_hist, s>>>(dets, d.n, d.n_elec, d.parts, d.pbits, total);
    const int fine = d.parts > kBins ? kFineBits : 0, cbits = d.pbits - fine;  // bits of the two scatter passes
    k_part_scan<<<1, 1024, 0, s>>>(total, d.parts, fine, base, cursor, coarse);
    const long long per = std::max(1, kTileKeys / d.npairs);
    const int gs = (int)std::min<long long>(2 * kSms, (d.n + per - 1) / per);
    // with two passes the first one's records lie where the members will be written last
    unsigned long long *first = fine ? reinterpret_cast<unsigned long long *>(ptr<Member>(r, r->L.members)) : records;
    k_key_scatter<W><<<gs, kHashThreads, sm_scatter, s>>>(dets, d.n, d.n_elec, cbits, d.tbits, coarse, first);
    if (fine) {
        const long long tiles = ((d.n_keys >> cbits) + 4095) / 4096;  // of an average coarse bin
        k_refine<<<dim3((unsigned)std::min<long long>(tiles + 1, 1024), 1u << cbits), kHashThreads, 0, s>>>(first, d.tbits, base, cursor, records);
    }
    k_group<W><<<d.parts, kGroupThreads, sm_group, s>>>(dets, c, d.n_elec, d.n_orb, d.tbits, records, base, ptr<Member>(r, r->L.members),
                                                        ptr<unsigned>(r, r->L.count_p), ptr<Head>(r, r->L.heads), st);
    double *norm_part = ptr<double>(r, r->L.partial) + 2 * (kPairGrid + kLargeGrid + kDiagBlocks);
    const int nw = occ_warps(d);
    const int go = (int)std::min<long long>(kSms, (d.n + nw - 1) / nw), gn = (int)std::min<long long>(kNormGrid, (d.n + kThreads - 1) / kThreads);
    k_norm<<<gn, kThreads, 0, s>>>(c, d.n, norm_part);
    k_occ_pairs<W><<<go, kOccThreads, sm_occ, s>>>(dets, c, d.n, d.n_elec, d.n_so, nw, ptr<CSum>(r, r->L.occ_part));
    const int n_merge = (int)((nent + kMergeThreads / 4 - 1) / (kMergeThreads / 4));
    k_occ_merge<<<n_merge + 1 + kSms, kMergeThreads, 0, s>>>(ptr<CSum>(r, r->L.occ_part), go, (int)nent, ptr<double>(r, r->L.occ_pair),
                                                             n_merge, norm_part, gn, ptr<Head>(r, r->L.heads),
                                                             ptr<Task>(r, r->L.records), st);
    if (cudaGetLastError() != cudaSuccess) return FCIQMC_ERR_CUDA;
    if (cudaMemcpyAsync(&r->host, st, sizeof(RdmState), cudaMemcpyDeviceToHost, s) != cudaSuccess) return FCIQMC_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return FCIQMC_ERR_CUDA;
    return r->host.status;
}

dim3 table_grid(const Dims &d, int extra_rows) {
    return dim3((unsigned)std::max(1, (std::max(d.n1, d.n2) + 4 * kThreads - 1) / (4 * kThreads)), (unsigned)(d.n1 + d.n2 + extra_rows));
}
int pair_grid(const Dims &d) { return std::min(kPairGrid, d.parts); }
int large_grid(const fciqmc_rdm *r) {
    constexpr unsigned long long kWarps = kPairThreads / 32;
    return (int)std::min<unsigned long long>(kLargeGrid, (r->host.n_tasks + kWarps - 1) / kWarps);
}

void launch_energy(fciqmc_rdm *r, const double *h, const double *eri, double *e) {
    const Dims &d = r->d;
    cudaStream_t s = r->s;
    const RdmState *st = ptr<RdmState>(r, r->L.state);
    double *partial = ptr<double>(r, r->L.partial), *table = ptr<double>(r, r->L.table), *share = ptr<double>(r, r->L.share);
    const int g = pair_grid(d), gl = large_grid(r);
    k_share<<<(d.n_orb * d.n_orb + kThreads - 1) / kThreads, kThreads, 0, s>>>(h, d.n_orb * d.n_orb, (double)(d.n_elec - 1), share);
    k_pair_table<<<table_grid(d, 0), kThreads, 0, s>>>(share, eri, d.n_orb, d.n1, d.n2, table);
    k_pair_energy<<<g + gl + kDiagBlocks, kPairThreads, 0, s>>>(ptr<Member>(r, r->L.members), ptr<unsigned>(r, r->L.base_p),
                                                            ptr<unsigned>(r, r->L.count_p), d.parts, ptr<Task>(r, r->L.records),
                                                            r->host.n_tasks, gl, d.n1, d.n2, table, ptr<double>(r, r->L.occ_pair),
                                                            h, eri, d.n_orb, partial);
    k_energy_finish<<<1, 1024, 0, s>>>(partial, g + gl + kDiagBlocks, st, e);
}

void launch_rdm(fciqmc_rdm *r) {
    const Dims &d = r->d;
    cudaStream_t s = r->s;
    double *gh = ptr<double>(r, r->L.gh), *ge = ptr<double>(r, r->L.ge), *table = ptr<double>(r, r->L.table);
    cudaMemsetAsync(gh, 0, sizeof(double) * d.n_orb * d.n_orb, s);
    cudaMemsetAsync(ge, 0, sizeof(double) * d.n_eri, s);
    cudaMemsetAsync(table, 0, sizeof(double) * ((size_t)d.n1 * d.n1 + (size_t)d.n2 * d.n2), s);
    const int gl = large_grid(r);
    k_pair_grad<<<pair_grid(d) + gl, kPairThreads, 0, s>>>(ptr<Member>(r, r->L.members), ptr<unsigned>(r, r->L.base_p),
                                                       ptr<unsigned>(r, r->L.count_p), d.parts, ptr<Task>(r, r->L.records),
                                                       r->host.n_tasks, gl, d.n1, d.n2, table);
    k_fold<<<table_grid(d, d.n_so), kThreads, 0, s>>>(table, ptr<double>(r, r->L.occ_pair), d.n_orb, d.n1, d.n2,
                                                      gh, ge);
}
}  // namespace

extern "C" {

size_t fciqmc_rdm_workspace_bytes(int n_elec, int n_orb, int64_t n_dets) {
    Dims d;
    if (!dims_of(n_elec, n_orb, n_dets, d)) return 0;
    return layout_of(d).total;
}

int fciqmc_rdm_create(int n_elec, int n_orb, const uint64_t *dets_dev, const double *c_dev, int64_t n_dets,
                      void *workspace, size_t workspace_bytes, void *cuda_stream, fciqmc_rdm **out) {
    if (!out) return FCIQMC_ERR_INVALID_ARG;
    *out = nullptr;
    Dims d;
    if (!dims_of(n_elec, n_orb, n_dets, d)) return FCIQMC_ERR_UNSUPPORTED;
    if (!dets_dev || !c_dev) return FCIQMC_ERR_INVALID_ARG;
    RdmLayout L = layout_of(d);
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) % 256) != 0 || workspace_bytes < L.total)
        return FCIQMC_ERR_WORKSPACE;
    fciqmc_rdm *r = new (std::nothrow) fciqmc_rdm();
    if (!r) return FCIQMC_ERR_INVALID_ARG;
    r->d = d;
    r->L = L;
    r->ws = static_cast<char *>(workspace);
    r->s = static_cast<cudaStream_t>(cuda_stream);
    if (cudaMemcpyAsync(ptr<unsigned long long>(r, L.dets), dets_dev, sizeof(uint64_t) * d.W * d.n, cudaMemcpyDeviceToDevice, r->s) != cudaSuccess ||
        cudaMemcpyAsync(ptr<double>(r, L.c), c_dev, sizeof(double) * d.n, cudaMemcpyDeviceToDevice, r->s) != cudaSuccess) {
        delete r;
        return FCIQMC_ERR_CUDA;
    }
    const int rc = d.W == 1 ? construct<1>(r) : construct<2>(r);
    if (rc != FCIQMC_OK) {
        delete r;
        return rc;
    }
    *out = r;
    return FCIQMC_OK;
}

int fciqmc_rdm_energy(fciqmc_rdm *r, const double *h_dev, const double *eri_dev, double *e_dev) {
    if (!r || !h_dev || !eri_dev || !e_dev) return FCIQMC_ERR_INVALID_ARG;
    launch_energy(r, h_dev, eri_dev, e_dev);
    return cudaGetLastError() == cudaSuccess ? FCIQMC_OK : FCIQMC_ERR_CUDA;
}

int fciqmc_rdm_gradient(fciqmc_rdm *r, const double *scale_dev, double *grad_h_dev, double *grad_eri_dev) {
    if (!r || !scale_dev || !grad_h_dev || !grad_eri_dev) return FCIQMC_ERR_INVALID_ARG;
    if (!r->rdm_ready) {
        launch_rdm(r);
        r->rdm_ready = true;
    }
    const long long nh = (long long)r->d.n_orb * r->d.n_orb;
    const int g = (int)std::min<long long>(kSms * 4, (nh + r->d.n_eri + kThreads - 1) / kThreads);
    k_scale_out<<<g, kThreads, 0, r->s>>>(ptr<double>(r, r->L.gh), ptr<double>(r, r->L.ge), r->d.n_orb, r->d.n_eri, (double)(r->d.n_elec - 1),
                                          scale_dev, ptr<RdmState>(r, r->L.state), grad_h_dev, grad_eri_dev);
    return cudaGetLastError() == cudaSuccess ? FCIQMC_OK : FCIQMC_ERR_CUDA;
}

int fciqmc_rdm_info(fciqmc_rdm *r, int64_t *counts) {
    if (!r || !counts) return FCIQMC_ERR_INVALID_ARG;
    RdmState *st = ptr<RdmState>(r, r->L.state);
    RdmState h;
    if (r->rdm_ready) {
        if (cudaMemsetAsync(&st->n_shared, 0, 2 * sizeof(unsigned long long), r->s) != cudaSuccess) return FCIQMC_ERR_CUDA;
        const Dims &d = r->d;
        const int gl = large_grid(r);
        k_pair_count<<<pair_grid(d) + gl, kPairThreads, sizeof(unsigned short) * (2 * d.n1 + d.n2), r->s>>>(
            ptr<Member>(r, r->L.members), ptr<unsigned>(r, r->L.base_p), ptr<unsigned>(r, r->L.count_p), d.parts, ptr<Task>(r, r->L.records),
            r->host.n_tasks, gl, d.n_orb, d.n1, d.n2, st);
    }
    if (cudaMemcpyAsync(&h, st, sizeof(RdmState), cudaMemcpyDeviceToHost, r->s) != cudaSuccess ||
        cudaStreamSynchronize(r->s) != cudaSuccess)
        return FCIQMC_ERR_CUDA;
    counts[0] = (int64_t)h.n_buckets;
    counts[1] = (int64_t)h.n_members;
    counts[2] = (int64_t)h.n_pairs;
    counts[3] = (int64_t)(h.n_shared / (unsigned long long)(r->d.n_elec - 1));
    counts[4] = (int64_t)h.n_apart;
    return h.status;
}

void fciqmc_rdm_destroy(fciqmc_rdm *r) {
    if (!r) return;
    cudaStreamSynchronize(r->s);
    delete r;
}

}  // extern "C"
