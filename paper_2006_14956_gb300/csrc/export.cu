// export.cu -- moving the walker list between the host and the bucket layout.
// Import: the compact input is checked, counted per bucket (to choose the
// bucket count) and placed on the device, each determinant into the next free
// slot of its bucket (order inside a bucket affects no result: every draw is
// keyed and every sum exact), and its slot listed for the H_ii kernel.
// Export, in (alpha, beta) order: the occupied slots of every bucket are
// compacted with a sort key, sorted by a least-significant-digit radix sort
// (8-bit digits, each pass stable), and the keys, C, H_ii - E_ref and the flags
// are gathered in that order.  Only the n live entries then cross to the host.
// The sort key of a determinant is the pair of its words' ranks among all
// words with as many electrons (the rank grows with the word): 68 bits instead
// of 100 at 50 orbitals and 10 + 10 electrons, so 9 passes over 20 bytes per
// determinant instead of 14 passes over 24; with at most 64 bits, 12 bytes.
#include <cuda_runtime.h>

#include "fq_device.cuh"

namespace fq {

constexpr int XS_THREADS = 256;  // one thread per digit value in the scatter
constexpr int XS_WARPS = XS_THREADS / 32;
constexpr int XS_ITEMS = 16;     // keys per thread: the block's barriers are per tile of 4096 keys
constexpr int XS_TILE = XS_THREADS * XS_ITEMS;
constexpr int XG_THREADS = 1024;

// ------------------------------------------------------------------ ranks
// binomial(p, i) for p, i < 64: the rank of a word is the sum over its set
// bits, lowest first, of binomial(position of bit i, i + 1)
struct Binomials {
    u64 c[64][64];
};
static constexpr Binomials binomials()
{
    Binomials B{};
    for (int p = 0; p < 64; p++) {
        B.c[p][0] = 1;
        for (int i = 1; i < 64; i++) B.c[p][i] = p ? B.c[p - 1][i - 1] + B.c[p - 1][i] : 0;
    }
    return B;
}
__device__ const Binomials d_binom = binomials();

// bits of the rank of a word with k of n bits set: the smallest r with binomial(n, k) <= 2^r
static int rank_bits(int n, int k)
{
    unsigned __int128 c = 1;
    for (int i = 1; i <= k; i++) c = c * (unsigned)(n - k + i) / (unsigned)i;
    int r = 0;
    while (((unsigned __int128)1 << r) < c) r++;
    return r;
}

__device__ __forceinline__ u64 word_rank(u64 w)
{
    u64 r = 0;
    for (int i = 1; w; i++) {
        const int p = __ffsll((long long)w) - 1;
        w &= w - 1;
        r += i < 64 ? __ldg(&d_binom.c[p][i]) : 0ULL;  // 64 electrons: one word only
    }
    return r;
}

// the low `bits` bits, 0 to 64 (a shift by 64 has no value in C++)
__host__ __device__ constexpr u64 low_mask(int bits) { return bits >= 64 ? ~0ULL : (1ULL << bits) - 1ULL; }
static_assert(low_mask(0) == 0 && low_mask(8) == 255 && low_mask(56) == ~0ULL >> 8 && low_mask(64) == ~0ULL, "low_mask");

// ------------------------------------------------------------------ compaction
// determinants of every group of XC_GROUP buckets, one thread each
__global__ void __launch_bounds__(XS_THREADS) k_export_count(const int *__restrict__ cnt, int nbk, int ng, long long *gsum)
{
    const int g = blockIdx.x * XS_THREADS + threadIdx.x;
    if (g >= ng) return;
    long long v = 0;
    for (int b = g * XC_GROUP; b < min((g + 1) * XC_GROUP, nbk); b++) v += cnt[b];
    gsum[g] = v;
}

// gsum[0 .. ng) to its exclusive prefix, the total in gsum[ng] (one block)
__global__ void __launch_bounds__(XG_THREADS) k_export_groups(long long *gsum, int ng)
{
    __shared__ long long s_w[XG_THREADS / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    long long carry = 0;
    for (int q0 = 0; q0 < ng; q0 += XG_THREADS) {
        const long long v = q0 + t < ng ? gsum[q0 + t] : 0;
        long long incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_w[warp] = incl;
        __syncthreads();
        long long before = carry, all = 0;
        for (int w = 0; w < XG_THREADS / 32; w++) {
            before += w < warp ? s_w[w] : 0;
            all += s_w[w];
        }
        if (q0 + t < ng) gsum[q0 + t] = before + incl - v;
        carry += all;
        __syncthreads();
    }
    if (t == 0) gsum[ng] = carry;
}

// the occupied slots of a group's buckets in bucket order, with their sort
// keys: a warp per bucket; rank(alpha) * 2^bits_b + rank(beta), the low
// lo_bits of it in `lo`, the rest in `hi`
__global__ void __launch_bounds__(XS_THREADS) k_export_compact(const ulonglong2 *__restrict__ key, const int *__restrict__ cnt,
                                                               const long long *__restrict__ gsum, int nbk, int bits_b,
                                                               int lo_bits, u64 *hi, u64 *lo, unsigned *idx)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b0 = blockIdx.x * XC_GROUP;
    static_assert(XC_GROUP <= 32, "a lane per bucket of the group");
    const int mine = lane < XC_GROUP && b0 + lane < nbk ? cnt[b0 + lane] : 0;
    int incl = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const long long o0 = gsum[blockIdx.x];
    for (int q = warp; q < XC_GROUP; q += XS_WARPS) {
        const int m = __shfl_sync(0xffffffffu, mine, q), before = __shfl_sync(0xffffffffu, incl - mine, q);
        for (int e = lane; e < m; e += 32) {
            const size_t s = (size_t)(b0 + q) * CAP_M + e;
            const ulonglong2 k = key[s];
            const u128 r = ((u128)word_rank(k.x) << bits_b) | word_rank(k.y);
            const long long o = o0 + before + e;
            hi[o] = (u64)(r >> lo_bits);
            if (lo) lo[o] = (u64)r & low_mask(lo_bits);
            idx[o] = (unsigned)s;
        }
    }
}

// ------------------------------------------------------------------ radix sort
// digit counts of every tile, stored digit-major: hist[d * ntiles + tile]
__global__ void __launch_bounds__(XS_THREADS) k_export_hist(const u64 *__restrict__ word, long long n, int shift, int *hist,
                                                            int ntiles)
{
    __shared__ int s_h[256];
    const int t = threadIdx.x;
    s_h[t] = 0;
    __syncthreads();
    const long long i0 = (long long)blockIdx.x * XS_TILE;
#pragma unroll 4
    for (int r = 0; r < XS_ITEMS; r++) {
        const long long i = i0 + (long long)r * XS_THREADS + t;
        if (i < n) atomicAdd(&s_h[(int)((word[i] >> shift) & 255u)], 1);
    }
    __syncthreads();
    hist[(size_t)t * ntiles + blockIdx.x] = s_h[t];
}

// exclusive scan of each digit's row of tile counts, hist[d * ntiles ..
// (d + 1) * ntiles), in place (block d), and the row total in dtot[d]
__global__ void __launch_bounds__(XS_THREADS) k_export_scan(int *hist, int ntiles, int *dtot)
{
    __shared__ int s_w[XS_WARPS];
    __shared__ int s_carry;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int *row = hist + (size_t)blockIdx.x * ntiles;
    if (t == 0) s_carry = 0;
    __syncthreads();
    for (int q0 = 0; q0 < ntiles; q0 += XS_THREADS) {
        const int q = q0 + t;
        const int v = q < ntiles ? row[q] : 0;
        int incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_w[warp] = incl;
        __syncthreads();
        int before = s_carry;
        for (int w = 0; w < warp; w++) before += s_w[w];
        if (q < ntiles) row[q] = before + incl - v;
        __syncthreads();
        if (t == XS_THREADS - 1) s_carry = before + incl;
        __syncthreads();
    }
    if (t == 0) dtot[blockIdx.x] = s_carry;
}

// the tile's elements of one array through shared memory: element r of a
// thread is at place pos[r] in digit order, so that neighbouring threads write
// neighbouring addresses
template <typename V>
__device__ __forceinline__ void scatter_array(const V *__restrict__ src, V *dst, long long i0, int cnt, V *stage,
                                              const unsigned char *s_dig, const int *s_gbase, const unsigned short (&pos)[XS_ITEMS])
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < XS_ITEMS; r++) {
        const int j = warp * (32 * XS_ITEMS) + r * 32 + lane;
        if (j < cnt) stage[pos[r]] = src[i0 + j];
    }
    __syncthreads();
    for (int j = t; j < cnt; j += XS_THREADS) dst[s_gbase[s_dig[j]] + j] = stage[j];
}

// stable scatter of one tile by the digit of `word` (hi or lo): warp w ranks
// elements [512 w, 512 (w + 1)) among the equal digits before them (a counter
// per digit and warp, no block barrier), one scan over the warps and digits
// places them, and the arrays follow one after the other.  hist = NULL: the
// only tile.
__global__ void __launch_bounds__(XS_THREADS) k_export_scatter(const u64 *__restrict__ word, int shift, long long n,
                                                               const int *__restrict__ hist, int ntiles,
                                                               const int *__restrict__ dtot, const u64 *__restrict__ hi,
                                                               const u64 *__restrict__ lo,
                                                               const unsigned *__restrict__ idx, u64 *hi2, u64 *lo2,
                                                               unsigned *idx2)
{
    __shared__ u64 s_stage[XS_TILE];
    __shared__ unsigned char s_dig[XS_TILE];
    __shared__ unsigned short s_cnt[XS_WARPS][256];
    __shared__ int s_gbase[256];  // global place of a digit's first element of this tile, minus its place in the tile
    __shared__ int s_sum[2][XS_WARPS];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned below = (1u << lane) - 1u;
    const long long i0 = (long long)blockIdx.x * XS_TILE;
    const int cnt = (int)min((long long)XS_TILE, n - i0);
    for (int q = lane; q < 256; q += 32) s_cnt[warp][q] = 0;
    __syncwarp();
    unsigned short pos[XS_ITEMS];
    unsigned char dig[XS_ITEMS];
#pragma unroll
    for (int r = 0; r < XS_ITEMS; r++) {
        const int j = warp * (32 * XS_ITEMS) + r * 32 + lane;
        dig[r] = j < cnt ? (unsigned char)((word[i0 + j] >> shift) & 255u) : 0;
    }
#pragma unroll
    for (int r = 0; r < XS_ITEMS; r++) {
        const bool valid = warp * (32 * XS_ITEMS) + r * 32 + lane < cnt;
        const unsigned peers = __match_any_sync(0xffffffffu, valid ? (int)dig[r] : 256);  // a value no key has
        const unsigned before = valid ? s_cnt[warp][dig[r]] : 0u;
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) s_cnt[warp][dig[r]] = (unsigned short)(before + __popc(peers));
        __syncwarp();
        pos[r] = (unsigned short)(before + __popc(peers & below));
    }
    __syncthreads();
    {
        // thread t, digit t: the warps' prefix, then exclusive scans over the
        // digits of this tile's counts and of all tiles' totals
        int c = 0;
        for (int w = 0; w < XS_WARPS; w++) {
            const int x = s_cnt[w][t];
            s_cnt[w][t] = (unsigned short)c;
            c += x;
        }
        const int v[2] = {c, hist ? dtot[t] : c};
        int in[2] = {v[0], v[1]};
        for (int o = 1; o < 32; o <<= 1)
            for (int k = 0; k < 2; k++) {
                const int y = __shfl_up_sync(0xffffffffu, in[k], o);
                if (lane >= o) in[k] += y;
            }
        if (lane == 31) { s_sum[0][warp] = in[0]; s_sum[1][warp] = in[1]; }
        __syncthreads();
        int l = in[0] - v[0], g = in[1] - v[1];
        for (int w = 0; w < warp; w++) { l += s_sum[0][w]; g += s_sum[1][w]; }
        s_gbase[t] = g + (hist ? hist[(size_t)t * ntiles + blockIdx.x] : 0) - l;
        for (int w = 0; w < XS_WARPS; w++) s_cnt[w][t] = (unsigned short)(s_cnt[w][t] + l);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < XS_ITEMS; r++)
        if (warp * (32 * XS_ITEMS) + r * 32 + lane < cnt) {
            pos[r] = (unsigned short)(pos[r] + s_cnt[warp][dig[r]]);
            s_dig[pos[r]] = dig[r];
        }
    scatter_array(hi, hi2, i0, cnt, s_stage, s_dig, s_gbase, pos);
    if (lo) scatter_array(lo, lo2, i0, cnt, s_stage, s_dig, s_gbase, pos);
    scatter_array(idx, idx2, i0, cnt, reinterpret_cast<unsigned *>(s_stage), s_dig, s_gbase, pos);
}

__global__ void k_export_gather(const unsigned *__restrict__ idx, long long n, const ulonglong2 *__restrict__ key,
                                const double *__restrict__ c, const double *__restrict__ hd,
                                const uint8_t *__restrict__ fl, u64 *oa, u64 *ob, double *oc, double *ohd, int32_t *ofl)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const unsigned s = idx[i];
        const ulonglong2 k = key[s];
        oa[i] = k.x;
        ob[i] = k.y;
        oc[i] = c[s];
        ohd[i] = hd[s];
        ofl[i] = fl[s];
    }
}

// import, step 1: flags bit 0 = an entry with a wrong electron count, an
// orbital beyond norb or a non-finite amplitude; bit 1 = the reference present
__global__ void k_import_check(const u64 *__restrict__ a, const u64 *__restrict__ b, const double *__restrict__ c,
                               long long n, int na, int nb, u64 normask, u64 ra, u64 rb, int *flags)
{
    int f = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const u64 x = a[i], y = b[i];
        const bool finite = (dbits(c[i]) & 0x7ff0000000000000ULL) != 0x7ff0000000000000ULL;
        if (__popcll(x) != na || __popcll(y) != nb || ((x | y) & ~normask) || !finite) f |= 1;
        if (x == ra && y == rb) f |= 2;
    }
    f = __reduce_or_sync(0xffffffffu, f);
    if ((threadIdx.x & 31) == 0 && f) atomicOr(flags, f);
}

// import, step 2: bucket counts at 2^bb buckets; *over = 1 once a bucket
// holds more than IMPORT_M
__global__ void k_import_count(const u64 *__restrict__ a, const u64 *__restrict__ b, long long n, int bb, int *cnt,
                               int *over)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int o = atomicAdd(&cnt[bucket_of(det_hash(a[i], b[i]), bb)], 1);
        if (o == IMPORT_M) atomicOr(over, 1);
    }
}

// import, step 3: each determinant into the next free slot of its bucket
// (fill = the zeroed counts of the list), flags (the reference's), and its
// slot into list[i]
__global__ void k_import_place(const u64 *__restrict__ a, const u64 *__restrict__ b, const double *__restrict__ c,
                               long long n, int bb, u64 ra, u64 rb, int *fill, ulonglong2 *key, double *oc,
                               uint8_t *ofl, unsigned *list)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const u64 x = a[i], y = b[i];
        const int bk = bucket_of(det_hash(x, y), bb);
        const size_t s = (size_t)bk * CAP_M + (size_t)atomicAdd(&fill[bk], 1);
        key[s] = make_ulonglong2(x, y);
        oc[s] = c[i];
        ofl[s] = (uint8_t)((x == ra && y == rb) ? DFLAG_REF : 0);
        list[i] = (unsigned)s;
    }
}

static unsigned grid_for(long long n)
{
    const long long g = (n + 255) / 256;
    return (unsigned)(g < 1 ? 1 : (g < 4096 ? g : 4096));
}

cudaError_t launch_import_check(const u64 *a, const u64 *b, const double *c, long long n, int na, int nb, u64 normask,
                                u64 ra, u64 rb, int *flags, cudaStream_t s)
{
    if (n > 0) k_import_check<<<grid_for(n), 256, 0, s>>>(a, b, c, n, na, nb, normask, ra, rb, flags);
    return cudaGetLastError();
}

cudaError_t launch_import_count(const u64 *a, const u64 *b, long long n, int bb, int *cnt, int *over, cudaStream_t s)
{
    k_import_count<<<grid_for(n), 256, 0, s>>>(a, b, n, bb, cnt, over);
    return cudaGetLastError();
}

cudaError_t launch_import_place(const u64 *a, const u64 *b, const double *c, long long n, int bb, u64 ra, u64 rb,
                                int *fill, ulonglong2 *key, double *oc, uint8_t *ofl, unsigned *list, cudaStream_t s)
{
    k_import_place<<<grid_for(n), 256, 0, s>>>(a, b, c, n, bb, ra, rb, fill, key, oc, ofl, list);
    return cudaGetLastError();
}

// group prefix of the bucket counts into gsum (a word per group and one
// more), the number of determinants in *total (device pointer into gsum)
cudaError_t export_count(const int *cnt, int nbk, long long *gsum, const long long **total, cudaStream_t s)
{
    const int ng = (nbk + XC_GROUP - 1) / XC_GROUP;
    k_export_count<<<(ng + XS_THREADS - 1) / XS_THREADS, XS_THREADS, 0, s>>>(cnt, nbk, ng, gsum);
    k_export_groups<<<1, XG_THREADS, 0, s>>>(gsum, ng);
    *total = gsum + ng;
    return cudaGetLastError();
}

// Two buffers of sort keys and slots, and the outputs: after the last pass the
// keys are dead, and the outputs take their place (40 bytes per determinant)
size_t export_scratch_bytes(long long n)
{
    const long long ntiles = (n + XS_TILE - 1) / XS_TILE;
    return (size_t)n * (4 * sizeof(u64) + 2 * sizeof(unsigned)) + (size_t)ntiles * 256 * sizeof(int) + 256 * sizeof(int) +
           8 * 256;
}

// the n occupied determinants of a list sorted by (alpha, beta) into device
// arrays carved from `scratch` (export_scratch_bytes(n) bytes)
cudaError_t export_sorted(const ulonglong2 *key, const double *c, const double *hd, const uint8_t *fl, const int *cnt,
                          const long long *gsum, int nbk, long long n, int norb, int na, int nb, void *scratch,
                          const u64 **oa, const u64 **ob, const double **oc, const double **ohd, const int32_t **ofl,
                          cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    if (n > 0x7fffffffLL) return cudaErrorInvalidValue;  // 32-bit positions in the scatter
    const long long ntiles = (n + XS_TILE - 1) / XS_TILE;
    auto place = [&](size_t bytes) {  // each array on a 16-byte boundary
        unsigned char *p = (unsigned char *)scratch;
        scratch = p + ((bytes + 15) & ~(size_t)15);
        return (void *)p;
    };
    u64 *hi[2], *lo[2];
    unsigned *ix[2];
    for (int k = 0; k < 2; k++) {
        hi[k] = (u64 *)place((size_t)n * sizeof(u64));
        lo[k] = (u64 *)place((size_t)n * sizeof(u64));
        ix[k] = (unsigned *)place((size_t)n * sizeof(unsigned));
    }
    int *dtot = (int *)place(256 * sizeof(int));
    int *hist = (int *)place((size_t)ntiles * 256 * sizeof(int));

    const int bits_b = rank_bits(norb, nb), bits = rank_bits(norb, na) + bits_b;
    const int lo_bits = bits > 64 ? (bits - 64 + 7) / 8 * 8 : 0;  // whole digits below the top 64 bits
    k_export_compact<<<(nbk + XC_GROUP - 1) / XC_GROUP, XS_THREADS, 0, s>>>(key, cnt, gsum, nbk, bits_b, lo_bits, hi[0],
                                                                            lo_bits ? lo[0] : nullptr, ix[0]);
    int cur = 0;
    for (int bit = 0; bit < bits; bit += 8) {
        const bool low = bit < lo_bits;
        const u64 *word = low ? lo[cur] : hi[cur];
        const int shift = low ? bit : bit - lo_bits;
        const bool one = ntiles == 1;
        if (!one) {
            k_export_hist<<<(unsigned)ntiles, XS_THREADS, 0, s>>>(word, n, shift, hist, (int)ntiles);
            k_export_scan<<<256, XS_THREADS, 0, s>>>(hist, (int)ntiles, dtot);
        }
        // the low word is not looked at any more after its last digit
        const bool keep_lo = lo_bits > 0 && bit + 8 < lo_bits;
        k_export_scatter<<<(unsigned)ntiles, XS_THREADS, 0, s>>>(word, shift, n, one ? nullptr : hist, (int)ntiles, dtot,
                                                                  hi[cur], keep_lo ? lo[cur] : nullptr, ix[cur],
                                                                  hi[cur ^ 1], lo[cur ^ 1], ix[cur ^ 1]);
        cur ^= 1;
    }
    const int gb = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
    int32_t *df = (int32_t *)ix[cur ^ 1];
    k_export_gather<<<gb, 256, 0, s>>>(ix[cur], n, key, c, hd, fl, hi[0], hi[1], (double *)lo[0], (double *)lo[1], df);
    *oa = hi[0];
    *ob = hi[1];
    *oc = (double *)lo[0];
    *ohd = (double *)lo[1];
    *ofl = df;
    return cudaGetLastError();
}

}  // namespace fq
