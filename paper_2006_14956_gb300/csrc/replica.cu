// replica.cu -- the cross estimators of a replica pair (Sec. V: two
// independent walker distributions of the same system; Sec. VI: the
// Epstein-Nesbet PT2 correction from spawns discarded on both replicas).
//
// Both replicas keep the same bucket layout, so the determinants of bucket b
// of one replica can only meet those of bucket b of the other.  The
// annihilation kernel leaves, per bucket and replica, one entry per
// determinant of the iteration (start amplitude C, H_jj - E_ref when it was
// occupied, accepted and rejected spawn sums); k_replica_cross joins the two
// lists of a bucket through a shared-memory hash table of the first
// replica's entries and reduces, per bucket,
//   sum_j C^1_j C^2_j,  sum_j (C^1_j (H_jj - E_ref)) C^2_j,
//   sum_j (C^1_j S^2_j + C^2_j S^1_j)   (S = accepted + rejected spawns),
//   sum_j R^1_j R^2_j / (E_0 - (H_jj - E_ref))   over j with both rejected sums R nonzero,
// E_0 = the mean of the two shifts at the start of the iteration.  H_jj of
// the last kind (never in either list) is computed here, one warp each.
#include <cuda_runtime.h>

#include "fq_device.cuh"

namespace fq {

constexpr int XC_THREADS = 256, XC_WARPS = XC_THREADS / 32;
constexpr int XC_TABBITS = 14;   // the block's hash table: up to 8192 first-replica entries
constexpr int XC_WBITS = XC_TABBITS - 3;  // a warp's slice of it: up to 1024
constexpr int XC_PT2CAP = 1024;  // matched rejected determinants queued for the warps
static_assert((XC_WARPS << XC_WBITS) == (1 << XC_TABBITS), "a slice per warp");

// One bucket, by one warp (WARP: ordinary buckets, no block barrier) or by the
// whole block; tab: its hash table of 2^bits slots; np, pairs[cap]: its queue
template <bool WARP>
__device__ __forceinline__ void cross_bucket(const DevInst &A, const DevInst &B, double e0, int bk, int n0, int n1,
                                             unsigned *tab, int bits, int *np_, int (*pairs)[2], int cap,
                                             double (*red)[4])
{
    const int t = WARP ? (int)(threadIdx.x & 31) : (int)threadIdx.x, NT = WARP ? 32 : XC_THREADS;
    const int lane = threadIdx.x & 31;
    auto sync = [&]() { if (WARP) __syncwarp(); else __syncthreads(); };
    const SideEnt *S0 = A.side + (size_t)bk * A.side_cap;
    const SideEnt *S1 = B.side + (size_t)bk * B.side_cap;
    while (bits > 5 && (1 << (bits - 1)) >= 2 * n0) bits--;  // no larger table than the bucket needs
    const unsigned mask = (1u << bits) - 1u;
    const bool use_tab = 2 * n0 <= (int)(mask + 1u);
    if (use_tab) {
        for (int q = t; q <= (int)mask; q += NT) tab[q] = 0u;
        sync();
        for (int i = t; i < n0; i += NT) {
            unsigned s = (unsigned)det_hash(S0[i].a, S0[i].b) & mask;
            while (atomicCAS(&tab[s], 0u, (unsigned)(i + 1)) != 0u) s = (s + 1u) & mask;
        }
    }
    if (t == 0) *np_ = 0;
    sync();
    double ov = 0.0, hdg = 0.0, cr = 0.0, pt2 = 0.0;
    for (int j = t; j < n1; j += NT) {
        const SideEnt q = S1[j];
        int i = -1;
        if (use_tab) {
            unsigned s = (unsigned)det_hash(q.a, q.b) & mask;
            for (unsigned probe = 0; probe <= mask; probe++) {
                const unsigned v = tab[s];
                if (v == 0u) break;
                if (S0[v - 1].a == q.a && S0[v - 1].b == q.b) { i = (int)v - 1; break; }
                s = (s + 1u) & mask;
            }
        } else {
            for (int y = 0; y < n0; y++)
                if (S0[y].a == q.a && S0[y].b == q.b) { i = y; break; }
        }
        if (i < 0) continue;
        const SideEnt p = S0[i];
        ov = ov + p.c0 * q.c0;
        if (!is_zero(p.c0) && !is_zero(q.c0)) hdg = hdg + (p.c0 * p.hd) * q.c0;
        cr = cr + (p.c0 * (q.sacc + q.srej) + q.c0 * (p.sacc + p.srej));
        if (!is_zero(p.srej) && !is_zero(q.srej)) {
            const int k = atomicAdd(np_, 1);
            if (k < cap) { pairs[k][0] = i; pairs[k][1] = j; }
            else {
                const double den = e0 - diag_exact_thread(A, p.a, p.b);
                if (den != 0.0) pt2 = pt2 + (p.srej * q.srej) / den;  // undefined term left out
            }
        }
    }
    sync();
    const int np = min(*np_, cap);
    for (int k = WARP ? 0 : (int)(threadIdx.x >> 5); k < np; k += WARP ? 1 : XC_WARPS) {
        const SideEnt p = S0[pairs[k][0]], q = S1[pairs[k][1]];
        const u64 ka[1] = {p.a}, kb[1] = {p.b};
        double hd[1];
        diag_exact_warp_multi<1>(A, ka, kb, hd);
        if (lane == 0 && e0 - hd[0] != 0.0) pt2 = pt2 + (p.srej * q.srej) / (e0 - hd[0]);
    }
    for (int m = 16; m >= 1; m >>= 1) {
        ov = ov + __shfl_xor_sync(0xffffffffu, ov, m);
        hdg = hdg + __shfl_xor_sync(0xffffffffu, hdg, m);
        cr = cr + __shfl_xor_sync(0xffffffffu, cr, m);
        pt2 = pt2 + __shfl_xor_sync(0xffffffffu, pt2, m);
    }
    double r[4] = {ov, hdg, cr, pt2};
    if (!WARP) {
        if (lane == 0)
            for (int c = 0; c < 4; c++) red[threadIdx.x >> 5][c] = r[c];
        __syncthreads();
        for (int c = 0; c < 4; c++) {
            r[c] = 0.0;
            for (int w = 0; w < XC_WARPS; w++) r[c] = r[c] + red[w][c];
        }
    }
    if (t == 0) {
        Partial &P = A.part[bk];
        P.x_ov = r[0]; P.x_hd = r[1]; P.x_cr = r[2]; P.x_pt2 = r[3];
    }
    sync();
}

__global__ void __launch_bounds__(XC_THREADS) k_replica_cross(const DevInst *__restrict__ insts, int n_inst)
{
    extern __shared__ unsigned xtab[];
    __shared__ int s_np[XC_WARPS];
    __shared__ int s_pair[XC_PT2CAP][2];
    __shared__ double s_red[XC_WARPS][4];
    const int t = threadIdx.x, warp = t >> 5;
    for (int ii = 0; ii < n_inst; ii++) {
        const DevInst &A = insts[ii];
        if (A.partner <= ii || !A.side) continue;  // the first replica of each pair does the join
        const DevInst &B = insts[A.partner];
        const int errs = *(volatile int *)&A.st->err | *(volatile int *)&B.st->err;
        if ((errs & ERRB_STAGE) || A.st->err_at_start || B.st->err_at_start) continue;  // not committed: repeated
        const double e0 = (A.st->S + B.st->S) * 0.5;
        const int nbk = 1 << A.bb;
        if (A.bb != B.bb) {  // the host keeps the layouts equal; never join unequal ones
            for (int bk = blockIdx.x * blockDim.x + t; bk < nbk; bk += gridDim.x * blockDim.x) {
                Partial &P = A.part[bk];
                P.x_ov = 0.0; P.x_hd = 0.0; P.x_cr = 0.0; P.x_pt2 = 0.0;
            }
            continue;
        }
        // buckets whose table fits a warp's slice, a warp each; then the larger ones by the block
        constexpr int WMAX = 1 << (XC_WBITS - 1);
        for (int bk = blockIdx.x * XC_WARPS + warp; bk < nbk; bk += gridDim.x * XC_WARPS) {
            const int n0 = A.side_cnt[bk], n1 = B.side_cnt[bk];
            if (n0 <= WMAX)
                cross_bucket<true>(A, B, e0, bk, n0, n1, xtab + ((size_t)warp << XC_WBITS), XC_WBITS, &s_np[warp],
                                   s_pair + warp * (XC_PT2CAP / XC_WARPS), XC_PT2CAP / XC_WARPS, s_red);
        }
        __syncthreads();
        for (int bk0 = blockIdx.x * XC_WARPS; bk0 < nbk; bk0 += gridDim.x * XC_WARPS)
            for (int bk = bk0; bk < min(bk0 + XC_WARPS, nbk); bk++) {
                const int n0 = A.side_cnt[bk], n1 = B.side_cnt[bk];
                if (n0 > WMAX) cross_bucket<false>(A, B, e0, bk, n0, n1, xtab, XC_TABBITS, &s_np[0], s_pair, XC_PT2CAP, s_red);
            }
        __syncthreads();
    }
}

// shared-memory opt-in of the join kernel (called before any stream capture)
cudaError_t replica_kernel_init()
{
    return cudaFuncSetAttribute(k_replica_cross, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(sizeof(unsigned) << XC_TABBITS));
}

cudaError_t launch_replica_cross(const DevInst *dinst, int n_inst, int max_buckets, cudaStream_t s)
{
    const size_t smem = sizeof(unsigned) << XC_TABBITS;
    int dev = 0, sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev);
    int blocks = sm * 3;
    const int need = (max_buckets + XC_WARPS - 1) / XC_WARPS;
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    k_replica_cross<<<blocks, XC_THREADS, smem, s>>>(dinst, n_inst);
    return cudaGetLastError();
}

}  // namespace fq
