// kernels.cu -- the projector iteration of initiator-FCIQMC on GB300.
//
// One iteration (Eq. (4) of Guther et al. 2020) is a handful of launches over
// the bucketed walker list of every run in the batch:
//   k_spawn        (a) ceil(|C_i|) attempts per determinant, one Philox block,
//                  one excitation and one Slater-Condon element per attempt;
//                  survivors of the rounding of Eq. (3) are appended to the
//                  spawn bucket of their target.  Every warp works alone on
//                  32 attempts at a time.
//   k_spawn_heavy  the same for determinants with many walkers, split into
//                  fixed-size slices so no warp waits on one heavily
//                  populated determinant.
//   k_annihilate   (b)+(c) one warp per bucket, the bucket's walkers and
//                  spawns in the warp's shared memory: equal determinants
//                  found through a small hash table, death and rounding, the
//                  spawns summed exactly, the initiator rule and rounding, the
//                  new bucket written, exact H_jj of the new determinants, and
//                  N_w, E_num (Eq. (9)) and the counts added to the run's
//                  exact totals by global reductions.
//   k_annihilate_big  the same for buckets with more records, a block each.
//   k_finalize     per run: read and clear the exact totals, update the
//                  shift, append the statistics row, flip the buffers.
// Options add work to these launches or one more: the semi-stochastic
// projection (semistoch.cu) before annihilation, the trial-estimator probe
// (trial.cu tables) and the adaptive shift's weight sums inside spawning and
// annihilation, and for a replica pair the cross join (replica.cu) before
// k_finalize.
// All of them read the iteration state from device memory, so one iteration
// is captured once as a CUDA graph and replayed.
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "fq_device.cuh"
#include "warp_table.cuh"

namespace fq {

__device__ __forceinline__ int find_inst(const int *unit_start, int n_inst, int u)
{
    int lo = 0, hi = n_inst;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (__ldg(unit_start + mid) <= u) lo = mid; else hi = mid;
    }
    return lo;
}

// D membership (open addressing on the determinant hash; empty slot = (0,0),
// which is never a valid determinant because every run has electrons)
__device__ __forceinline__ bool in_D(const DevInst &I, u64 a, u64 b)
{
    if (I.nd == 0) return false;
    u64 m = (1ULL << I.dhash_bits) - 1;
    u64 s = det_hash(a, b) & m;
    for (int probe = 0; probe < (1 << I.dhash_bits); probe++) {
        u64 ka = __ldg(I.dhash_keys + 2 * s), kb = __ldg(I.dhash_keys + 2 * s + 1);
        if (ka == a && kb == b) return true;
        if (ka == 0 && kb == 0) return false;
        s = (s + 1) & m;
    }
    return false;
}

// ------------------------------------------------------------------ spawning
// One spawning attempt k from parent (pa, pb) draws the Philox block
// (pa, pb, iteration, (k << 8) | spawn); the words an attempt consumes and
// every decision depend on that counter alone, so attempts may be evaluated
// in any order and by any thread.

// how a kernel finds the run of a bucket: one run whose descriptor is a
// kernel parameter (its fields are constant-bank operands), or a table of
// runs with the first unit (bucket) of each
struct OneRun {
    static constexpr bool SINGLE = true;
    const DevInst &I;
    __device__ __forceinline__ const DevInst &inst(int) const { return I; }
    __device__ __forceinline__ int find(int) const { return 0; }
    __device__ __forceinline__ IterState *claims() const { return I.st; }
};
struct RunTable {
    static constexpr bool SINGLE = false;
    const DevInst *__restrict__ t;
    const int *__restrict__ start;
    int n;
    __device__ __forceinline__ const DevInst &inst(int ii) const { return t[ii]; }
    __device__ __forceinline__ int find(int u) const { return find_inst(start, n, u); }
    __device__ __forceinline__ IterState *claims() const { return t[0].st; }  // the first run counts for the launch
};

// How a launch's n units (buckets, or parts of them) come to its nw warps:
// dealt out in turn, u = warp, warp + nw, ...  Over many rounds the warps drift
// apart (heavily populated determinants, uneven buckets, SMs at different
// distances from the data): with 27 rounds 14 % of the spawning's and 8 % of
// the annihilation's warp time was idle at the end.  So from CLAIM_ROUNDS
// rounds on (CLAIM kernels) the last quarter is claimed by whichever warp gets
// there first.  50 orbitals, spawning and annihilation: 484 + 500 -> 447 +
// 461 us at 7.7e6 determinants, 4.46 + 4.36 -> 4.17 + 4.18 ms at 7.6e7;
// claiming the last half: 4.18 + 4.21 ms.  Below that it costs more than it
// gives (3.4 rounds: 75 -> 78 us).
constexpr int CLAIM_ROUNDS = 8;
__host__ __device__ __forceinline__ int dealt_units(int n, int nw)
{
    const int rounds = n / nw;
    return (rounds - rounds / 4) * nw;
}

struct AdaptQueue;
// what the spawning code knows about the parent beyond its key: its
// main-list slot, the list parity and the shift at the start of the iteration
// (aq: the warp's queue of the adaptive shift)
struct SpawnCtx {
    unsigned pslot;
    int par;
    double S;
    AdaptQueue *aq;
};

// 128-bit add of q to the words p[0] (low), p[1] (high)
__device__ __forceinline__ void atomic_add128(u64 *p, u128 q)
{
    const u64 lo = (u64)q, hi = (u64)(q >> 64);
    const u64 old = atomicAdd((unsigned long long *)p, (unsigned long long)lo);
    atomicAdd((unsigned long long *)(p + 1), (unsigned long long)(hi + (old + lo < old ? 1ULL : 0ULL)));
}

// a spawn whose weight in the adaptive shift's sums is still to be found
struct AdaptRec {
    u64 a, b;       // target
    double H;
    unsigned slot;  // parent's main-list slot
    unsigned bt;    // target's bucket
};
struct AdaptQueue {
    AdaptRec r[64];  // fewer than 32 before 32 attempts are evaluated
    unsigned n;
};

// adaptive shift (Sec. V): the weight |H_ji| / |H_jj - E_ref - S| of a spawn
// from a non-initiator, truncated to 2^-64, into T of the parent, and into A
// as well when the target is occupied at the start of the iteration (the
// initiator rule accepts it); weights of 2^36 or more (|H_jj - E_ref - S| far
// below |H_ji|) and zero denominators are left out
__device__ __forceinline__ void adaptive_account(const DevInst &I, u64 ta, u64 tb, double H, int bt, const SpawnCtx &cx)
{
    const unsigned short *kx = I.kidx[cx.par] + (size_t)bt * KIDX;
    unsigned s = (unsigned)det_hash(ta, tb) & (unsigned)(KIDX - 1);
    double hdj = 0.0;
    bool occ = false, found = false;
    for (int probe = 0; probe < KIDX; probe++) {
        const unsigned v = __ldg(kx + s);
        if (!v) break;
        const size_t o = (size_t)bt * CAP_M + (v - 1);
        const ulonglong2 k = I.key[cx.par][o];
        if (k.x == ta && k.y == tb) {
            found = true;
            occ = !is_zero(I.c[cx.par][o]);
            hdj = I.hd[cx.par][o];
            break;
        }
        s = (s + 1) & (unsigned)(KIDX - 1);
    }
    if (!found) hdj = diag_exact_thread(I, ta, tb);
    const double den = bitsd(dbits(hdj - cx.S) & ~SIGN64);
    if (is_zero(den)) return;
    const double w = bitsd(dbits(H) & ~SIGN64) / den;
    u64 M;
    int E;
    split_abs(w, M, E);
    const int sh = E + 64;  // w 2^64 = M 2^sh
    if (sh + 53 > 100) return;  // w >= 2^36
    const u128 q = sh >= 0 ? ((u128)M << sh) : (sh > -64 ? (u128)(M >> (-sh)) : (u128)0);
    u64 *acc = I.facc[cx.par] + (size_t)cx.pslot * 4;
    atomic_add128(acc + 2, q);
    if (occ) atomic_add128(acc, q);
}

// append a surviving spawn (Eq. (3) rounding of the weight ws, D -> D filter)
// to its bucket: initiators' spawns from the front of the bucket's region,
// the others from its back
__device__ __forceinline__ void emit_weight(const DevInst &I, u64 ta, u64 tb, double ws, unsigned flags, u64 w3,
                                            double H, const SpawnCtx &cx)
{
    if (abs_lt(ws, I.cmin)) {
        ws = round_stoch(ws, I.cmin, I.cmin_log2, I.cmin_pow2, w3);
        if (is_zero(ws)) return;
    }
    if (!abs_lt(ws, 0x1p31)) { atomicOr(&I.st->err, ERRB_NUMERIC); return; }
    if ((flags & 2u) && in_D(I, ta, tb)) return;  // D -> D is applied exactly
    const int bt = bucket_of(det_hash(ta, tb), I.bb);
    if (cx.aq && I.adaptive && !(flags & 1u)) {  // weighed by full warps: H_jj of a new target is ~n^2/2 loads
        AdaptRec &r = cx.aq->r[atomicAdd(&cx.aq->n, 1u)];
        r.a = ta; r.b = tb; r.H = H; r.slot = cx.pslot; r.bt = (unsigned)bt;
    }
    const bool init = flags & 1u;
    const int s = atomicAdd((init ? I.scnt_i : I.scnt_n) + bt, 1);
    if (s < I.cap_s) {
        const size_t o = (size_t)bt * I.cap_s + (init ? s : I.cap_s - 1 - s);
        I.skey[o] = make_ulonglong2(ta, tb);
        I.sw[o] = ws;
    }
}

// weight -H tau / p_gen(c) C_i / n_att of a uniformly generated excitation of class c
__device__ __forceinline__ void emit_spawn(const DevInst &I, u64 ta, u64 tb, double H, int cls, double cper,
                                           unsigned flags, u64 w3, const SpawnCtx &cx)
{
    if (is_zero(H)) return;
    emit_weight(I, ta, tb, neg_if(true, H * (I.lam[cls] * cper)), flags, w3, H, cx);
}

// the orbitals strictly between p and q (p != q, both below 64)
__device__ __forceinline__ u64 between(int p, int q)
{
    const int lo = min(p, q), hi = max(p, q);
    return (1ULL << hi) - (2ULL << lo);
}

// lattice hop (Hubbard): electron e (drawn from w1), neighbour slot w2
__device__ __forceinline__ void spawn_hop_e(const DevInst &I, u64 pa, u64 pb, double cper, unsigned flags, int e, u64 w2,
                                            u64 w3, const SpawnCtx &cx)
{
    const int sp = e >= I.na;
    u64 x = sp ? pb : pa;
    const int p = nth_set(x, sp ? e - I.na : e);
    const int q = __ldg(I.nbr + 4 * p + (int)pick(w2, (unsigned)I.z));
    if (q < 0 || ((x >> q) & 1ULL)) return;
    const double H = neg_if(__popcll(x & between(p, q)) & 1, I.tmt);
    x ^= (1ULL << p) | (1ULL << q);
    emit_spawn(I, sp ? pa : x, sp ? x : pb, H, CLS_HOP, cper, flags, w3, cx);
}

// single excitation (App. A): electron e (drawn from w1), hole of its spin w2
__device__ __forceinline__ void spawn_single_e(const DevInst &I, u64 pa, u64 pb, double cper, unsigned flags, int e,
                                               u64 w2, u64 w3, const SpawnCtx &cx)
{
    const int sp = e >= I.na;
    u64 x = sp ? pb : pa;
    const int i = nth_set(x, sp ? e - I.na : e);
    const int m = sp ? I.mb : I.ma;
    const int a = nth_set(~x & I.normask, (int)pick(w2, (unsigned)m));
    const double v = single_exact(I, pa, pb, sp, i, a);
    const double H = neg_if(__popcll(x & between(i, a)) & 1, v);
    x ^= (1ULL << i) | (1ULL << a);
    emit_spawn(I, sp ? pa : x, sp ? x : pb, H, sp ? CLS_SINGLE_B : CLS_SINGLE_A, cper, flags, w3, cx);
}

// double excitation (App. A): ordered electron pair ep = e1 | e2 << 8 (drawn
// from w1), then the hole pair from w2.  Uniform generator: any pair of empty
// orbitals of the electrons' spins.  Pre-computed heat-bath sampling: the
// alias table of that pair of spin orbitals, bin k = floor(w2 K / 2^64), coin
// = the low 64 bits of w2 K (top 53 bits); an occupied hole or an empty table
// fails the attempt, and with p_gen = p_pair |H| / S the weight is
// -sign(H) lambda_ij C_i / n_att, lambda_ij = tau S / p_pair (per table).
// The sign: a_a+ a_b+ a_j a_i = (a_a+ a_i)(a_b+ a_j) for distinct orbitals,
// so it is the product of the two singles' signs, the second taken in the
// determinant the first leaves (which differs only for equal spins).
template <bool PCHB>
__device__ __forceinline__ void spawn_double(const DevInst &I, u64 pa, u64 pb, double cper, unsigned flags, unsigned ep,
                                             u64 w2, u64 w3, const SpawnCtx &cx)
{
    const int na = I.na;
    const int e1 = (int)(ep & 0xffu), e2 = (int)(ep >> 8);
    const int s1 = e1 >= na, s2 = e2 >= na;
    const int o1 = nth_set(s1 ? pb : pa, s1 ? e1 - na : e1);
    const int o2 = nth_set(s2 ? pb : pa, s2 ? e2 - na : e2);
    const bool opp = s1 != s2;
    // opposite spins: (oi, oa) alpha and (oj, ob) beta; equal spins: oi < oj, oa < ob
    const int oi = opp ? (s1 ? o2 : o1) : min(o1, o2), oj = opp ? (s1 ? o1 : o2) : max(o1, o2);
    const u64 xi = (!opp && s1) ? pb : pa, xj = (opp || s1) ? pb : pa;  // the words oi and oj are in
    int oa, ob;
    double lamS = 0.0;
    if (PCHB) {
        const int N = I.norb;
        int t, K;
        u64 off;
        if (opp) {
            t = oi * N + oj;
            K = N * N;
            off = (u64)t * (u64)K;
        } else {
            const int p = oj * (oj - 1) / 2 + oi;
            t = N * N + p;
            K = N * (N - 1) / 2;
            off = I.pchb_ss_base + (u64)p * (u64)K;
        }
        const double2 mt = __ldg(I.pchb_meta + t);
        if (!(dbits(mt.y) != 0)) return;  // S = 0: nothing to propose
        lamS = mt.x;
        const u64 low = w2 * (u64)K;
        const ulonglong2 e = __ldg(I.pchb_ent + off + pick(w2, (unsigned)K));
        const unsigned hp = ((low >> 11) < e.x) ? (unsigned)(e.y & 0xffffu) : (unsigned)((e.y >> 16) & 0xffffu);
        oa = (int)(hp & 0xffu);
        ob = (int)(hp >> 8);
        if (((xi >> oa) & 1ULL) || ((xj >> ob) & 1ULL)) return;
    } else {
        // two different holes of one spin are drawn as an ordered pair (h1, rank among the others)
        const unsigned d = opp ? (unsigned)I.mb : (unsigned)((s1 ? I.mb : I.ma) - 1);
        const unsigned tot = opp ? (unsigned)(I.ma * I.mb) : d * (d + 1u);
        const unsigned y = pick(w2, tot);
        const unsigned yh = div_by(y, opp ? I.mg_mb : (s1 ? I.mg_mb1 : I.mg_ma1));
        const unsigned rr = y - yh * d;
        const int q1 = nth_set(~xi & I.normask, (int)yh);
        const int q2 = nth_set(~xj & I.normask, (int)(rr + (!opp && rr >= yh ? 1u : 0u)));
        oa = opp ? q1 : min(q1, q2);
        ob = opp ? q2 : max(q1, q2);
    }
    const u64 fi = (1ULL << oi) | (1ULL << oa), fj = (1ULL << oj) | (1ULL << ob);
    const u64 yi = opp ? xi : xi ^ fj;  // oi -> oa follows oj -> ob
    const int par = (__popcll(xj & between(oj, ob)) ^ __popcll(yi & between(oi, oa))) & 1;
    const u64 ta = pa ^ (opp ? fi : (s1 ? 0ULL : fi ^ fj)), tb = pb ^ (opp ? fj : (s1 ? fi ^ fj : 0ULL));
    double v = eri4(I, oa, oi, ob, oj);
    if (!opp) v = v - eri4(I, oa, oj, ob, oi);
    const double H = neg_if(par, v);
    if (PCHB) {
        if (is_zero(H)) return;
        emit_weight(I, ta, tb, neg_if(!(dbits(H) & SIGN64), lamS * cper), flags, w3, H, cx);
    } else {
        emit_spawn(I, ta, tb, H, opp ? CLS_DOUBLE_AB : (s1 ? CLS_DOUBLE_BB : CLS_DOUBLE_AA), cper, flags, w3, cx);
    }
}

// How the attempts of a kernel are generated: the runs of a batch may differ
// (GEN_ANY looks at each run), a kernel of one run holds that run's code only
// (smaller code: the warps of the spawning kernel are at different places of
// it, and instruction fetch was its largest stall).
enum { GEN_UNIFORM = 0, GEN_PCHB = 1, GEN_HOP = 2, GEN_ANY = 3 };
template <int GEN>
__device__ __forceinline__ bool gen_is(const DevInst &I, int g)
{
    if (GEN != GEN_ANY) return GEN == g;
    return g == GEN_HOP ? I.kind == FCIQMC_HUBBARD : (I.kind != FCIQMC_HUBBARD && (I.pchb != 0) == (g == GEN_PCHB));
}

// class of one attempt from its first two words, or -1 for a failed attempt;
// *ep = the electron of a single or a hop, or for a double e1 | e2 << 8 (the
// ordered electron pair), all drawn from w1
enum { Q_DOUBLE = 0, Q_SINGLE = 1, Q_HOP = 2 };
template <int GEN>
__device__ __forceinline__ int classify(const DevInst &I, u64 w0, u64 w1, unsigned *ep)
{
    const int n = I.n;
    const bool hop = gen_is<GEN>(I, GEN_HOP), single = !hop && (w0 >> 11) < I.tsingle;
    const unsigned xe = pick(w1, (unsigned)(hop || single ? n : n * (n - 1)));
    if (hop) {
        *ep = xe;
        return Q_HOP;
    }
    if (single) {
        *ep = xe;
        return ((int)xe >= I.na ? I.mb : I.ma) == 0 ? -1 : Q_SINGLE;
    }
    if (n < 2) return -1;
    const unsigned q1 = div_by(xe, I.mg_n1);
    const int e1 = (int)q1, r = (int)(xe - q1 * (unsigned)(n - 1));
    const int e2 = r + (r >= e1 ? 1 : 0);
    *ep = (unsigned)e1 | ((unsigned)e2 << 8);
    const int s1 = e1 >= I.na, s2 = e2 >= I.na;
    if (s1 != s2) return (I.ma == 0 || I.mb == 0) ? -1 : Q_DOUBLE;
    return (s1 ? I.mb : I.ma) < 2 ? -1 : Q_DOUBLE;
}

// The spawning kernel.  Every warp works alone: it takes tiles of 32 list
// slots, appends the occupied ones to a ring of parents in shared memory with
// a running number of attempts, and evaluates 32 attempts at a time, one per
// lane, whatever tiles (and buckets) their parents came from.  Doubles and
// hops are evaluated where they are drawn; singles, whose exact sum is ten
// times as long, wait in a queue of the warp until there are 32 of them.
// Parents whose C / n_att needs a binary64 division (n_att not a power of two;
// the division costs a whole warp's turn whatever its active lanes) wait too.
// There is no block barrier and an attempt never leaves the chip: at 7.3e7
// determinants and 9.1e7 attempts (50 orbitals) a block-per-bucket draw with
// 48-byte attempt records in global memory and a second kernel for the
// evaluation took 8.6 ms; this takes 4.1 ms, issue slots 61 % used (the ten
// Philox rounds' 32 x 32 products alone keep the heavy FMA pipe at 42 %).
constexpr int SP_THREADS = 256, SP_WARPS = SP_THREADS / 32, RING = 64;
constexpr int CHUNK_S = 512;  // attempts per slice of a heavily populated determinant
static_assert(HEAVY_ATT == (unsigned)CHUNK_S, "heavy slices");

struct SpawnRec {    // a drawn single excitation
    u64 ka, kb;      // parent
    double cper;     // C_i / n_att
    u64 w2, w3;      // hole word, rounding word
    unsigned slot;   // parent's main-list slot (adaptive shift)
    unsigned info;   // electron | parent flags << 16
};
struct SpawnWarp {
    ulonglong2 key[RING];    // ring of parents: the pending ones hold fewer than 32
    double cper[RING];       // attempts before a tile of at most 32 more is appended
    unsigned off[RING];      // running number of the parent's first attempt
    unsigned slot[RING];
    SpawnRec q[RING];        // singles waiting (fewer than 32 before 32 attempts are drawn)
    unsigned divq[RING];     // slots waiting for their division
    unsigned char fl[RING];  // initiator | in-D bits
};

struct SpawnRun {  // the run a warp works on, at the start of the iteration
    long long it;
    double S;
    int par;
    AdaptQueue *aq;  // the warp's queue of the adaptive shift (NULL: no run of the launch uses it)
};

constexpr size_t SP_SMEM = SP_WARPS * sizeof(SpawnWarp), SP_SMEM_ADAPT = SP_SMEM + SP_WARPS * sizeof(AdaptQueue);
static_assert(4 * (SP_SMEM + 1024) <= 233472 && 3 * (SP_SMEM_ADAPT + 1024) <= 233472, "resident spawning blocks per SM");

// up to 32 of the spawns that wait to be weighed
__device__ __forceinline__ void eval_adaptive(const DevInst &I, const SpawnRun &R)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const unsigned q = R.aq->n, n = min(q, 32u);
    if (lane < n) {
        const AdaptRec r = R.aq->r[q - n + lane];
        adaptive_account(I, r.a, r.b, r.H, (int)r.bt, SpawnCtx{r.slot, R.par, R.S, nullptr});
    }
    __syncwarp();
    if (lane == 0) R.aq->n = q - n;
    __syncwarp();
}

// up to 32 queued singles, from the end of the queue
__device__ __forceinline__ void eval_singles(const DevInst &I, SpawnWarp &W, int &nq, const SpawnRun &R)
{
    const int lane = threadIdx.x & 31;
    const int n = min(nq, 32);
    __syncwarp();
    if (lane < n) {
        const SpawnRec r = W.q[nq - n + lane];
        const SpawnCtx cx{r.slot, R.par, R.S, R.aq};
        spawn_single_e(I, r.ka, r.kb, r.cper, r.info >> 16, (int)(r.info & 0xffffu), r.w2, r.w3, cx);
    }
    nq -= n;
    __syncwarp();
}

// ... until fewer than `keep` wait
__device__ __forceinline__ void drain_adaptive(const DevInst &I, const SpawnRun &R, unsigned keep)
{
    if (!R.aq) return;
    for (;;) {
        __syncwarp();
        if (R.aq->n < keep) return;
        __syncwarp();
        eval_adaptive(I, R);
    }
}

// one attempt per lane (lanes with `on`): draw, classify, evaluate or queue
template <int GEN>
__device__ __forceinline__ void attempts32(const DevInst &I, SpawnWarp &W, int &nq, const SpawnRun &R, bool on,
                                           ulonglong2 key, u64 k, double cper, unsigned fl, unsigned slot)
{
    const int lane = threadIdx.x & 31;
    u64 w[4];
    philox(key.x, key.y, (u64)R.it, (k << 8) | (u64)PURPOSE_SPAWN, I.seed, I.replica, w);
    unsigned ep = 0;
    int cls = classify<GEN>(I, w[0], w[1], &ep);
    if (!on) cls = -1;
    const SpawnCtx cx{slot, R.par, R.S, R.aq};
    if (!gen_is<GEN>(I, GEN_HOP)) {
        const unsigned ms = __ballot_sync(0xffffffffu, cls == Q_SINGLE);
        if (cls == Q_SINGLE) {
            SpawnRec &r = W.q[nq + __popc(ms & ((1u << lane) - 1u))];
            r.ka = key.x; r.kb = key.y; r.cper = cper; r.w2 = w[2]; r.w3 = w[3]; r.slot = slot; r.info = ep | (fl << 16);
        }
        nq += __popc(ms);
        if (cls == Q_DOUBLE) {
            if (gen_is<GEN>(I, GEN_PCHB)) spawn_double<true>(I, key.x, key.y, cper, fl, ep, w[2], w[3], cx);
            else spawn_double<false>(I, key.x, key.y, cper, fl, ep, w[2], w[3], cx);
        }
    } else if (cls == Q_HOP) {
        spawn_hop_e(I, key.x, key.y, cper, fl, (int)ep, w[2], w[3], cx);
    }
}

struct SpawnCursor {       // running numbers: ring entries [r0, r1) pending, attempts [done, tot)
    unsigned r0, r1, done, tot;
    int nq, nd;            // singles and divisions waiting
};

// 32 pending attempts (or the last ones): lane l takes attempt done + l, whose
// parent is found from the pending entries that start inside the window
template <int GEN>
__device__ __forceinline__ void spawn_window(const DevInst &I, SpawnWarp &W, SpawnCursor &C, const SpawnRun &R)
{
    const int lane = threadIdx.x & 31;
    unsigned bit = 0;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const unsigned j = (unsigned)(h * 32 + lane);
        if (j < C.r1 - C.r0) {
            const unsigned o = W.off[(C.r0 + j) & (RING - 1)] - C.done;
            if (o - 1u < 31u) bit |= 1u << o;  // o in 1 .. 31 (the entry at r0 starts at or before `done`)
        }
    }
    const unsigned m = __reduce_or_sync(0xffffffffu, bit);
    const unsigned r = (C.r0 + __popc(m & (0xffffffffu >> (31 - lane)))) & (RING - 1);
    const bool on = C.done + lane - C.tot >= 0x80000000u;
    attempts32<GEN>(I, W, C.nq, R, on, W.key[r], (u64)(C.done + lane - W.off[r]), W.cper[r], W.fl[r], W.slot[r]);
    C.done += 32;
    if (C.tot - C.done - 1u >= 0x7fffffffu) {  // done >= tot: nothing is pending
        C.done = C.tot;
        C.r0 = C.r1;
    } else {
        C.r0 += __popc(m);
        if (C.r0 + 1 != C.r1 && W.off[(C.r0 + 1) & (RING - 1)] == C.done) C.r0++;
    }
}

// the lanes' parents (valid lanes, nat >= 1 attempts each) into the ring
__device__ __forceinline__ void spawn_append(SpawnWarp &W, SpawnCursor &C, bool valid, ulonglong2 key, unsigned nat,
                                             double cper, unsigned fl, unsigned slot)
{
    const int lane = threadIdx.x & 31;
    const unsigned mv = __ballot_sync(0xffffffffu, valid), below = (1u << lane) - 1u;
    const unsigned many = __ballot_sync(0xffffffffu, valid && nat > 1);
    const unsigned pos = (unsigned)__popc(mv & below);
    unsigned ex = pos, total = (unsigned)__popc(mv);
    if (many) {
        unsigned v = valid ? nat : 0u;
        const unsigned mine = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        ex = v - mine;
        total = __shfl_sync(0xffffffffu, v, 31);
    }
    __syncwarp();
    if (valid) {
        const unsigned r = (C.r1 + pos) & (RING - 1);
        W.key[r] = key;
        W.cper[r] = cper;
        W.off[r] = C.tot + ex;
        W.slot[r] = slot;
        W.fl[r] = (unsigned char)fl;
    }
    __syncwarp();
    C.r1 += (unsigned)__popc(mv);
    C.tot += total;
}

// slices of a determinant with more attempts than one warp should draw
__device__ __noinline__ void queue_heavy(const DevInst &I, ulonglong2 kk, double c, unsigned nat, unsigned fl, unsigned slot)
{
    const double ch = c / (double)nat;
    const unsigned nch = (nat + HEAVY_ATT - 1) / HEAVY_ATT;
    const int q0 = atomicAdd(&I.st->heavy_n, (int)nch);
    if ((long long)q0 + nch > (long long)I.heavy_cap) {
        atomicOr(&I.st->err, ERRB_HEAVY_CAP);
        return;
    }
    for (unsigned q = 0; q < nch; q++) {
        HeavyChunk h;
        h.a = kk.x; h.b = kk.y; h.cper = ch; h.k0 = (u64)q * HEAVY_ATT;
        const unsigned left = nat - q * HEAVY_ATT;
        h.count = left < HEAVY_ATT ? left : HEAVY_ATT;
        h.flags = fl;
        h.slot = slot;
        h.pad = 0;
        I.heavy[q0 + q] = h;
    }
}

// parts: warps per bucket, so that a small list still reaches every SM; part
// p takes slots p, p + parts, ... (the oldest determinants, the most
// populated ones, come first in a bucket).  Determinants with more than
// heavy_min attempts go to the heavy queue.  The loop holds every piece of
// work once (code size): each turn evaluates a full window of attempts or of
// singles, or else appends parents; a run's last turns empty what is left.
template <int GEN, bool ADAPT, bool CLAIM, typename RUNS>
__device__ __forceinline__ void spawn_body(const RUNS &runs, int n_units, int parts, unsigned heavy_min)
{
    extern __shared__ __align__(16) unsigned char sp_raw[];
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    SpawnWarp &W = reinterpret_cast<SpawnWarp *>(sp_raw)[threadIdx.x >> 5];
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nw = (int)((gridDim.x * blockDim.x) >> 5);
    SpawnCursor C{0, 0, 0, 0, 0, 0};
    SpawnRun R{0, 0.0, 0, nullptr};
    if (ADAPT) {
        R.aq = reinterpret_cast<AdaptQueue *>(sp_raw + SP_WARPS * sizeof(SpawnWarp)) + (threadIdx.x >> 5);
        if (lane == 0) R.aq->n = 0;
        __syncwarp();
    }
    unsigned long long att = 0;
    int cur = -1, err = 0;
    int v = gw, u = 0, ii = -1, b = 0, t = 0, m = 0;  // unit and part; next tile of bucket b
    const int n_work = n_units * parts, dealt = CLAIM ? dealt_units(n_work, nw) : n_work;
    int claim = 0;                                    // lane 0: the warp's next unit after the dealt ones
    bool have = false, drain = false;                 // v is set up (t, m valid); the run's list is done
    while (true) {
        if (ADAPT) {
            __syncwarp();
            const unsigned na = R.aq->n;
            if (na >= 32 || (drain && na > 0 && C.nq == 0 && C.tot == C.done)) {
                eval_adaptive(runs.inst(cur), R);
                continue;
            }
        }
        if (C.nq >= 32 || (drain && C.nq > 0)) {
            eval_singles(runs.inst(cur), W, C.nq, R);
            continue;
        }
        if (C.tot - C.done >= 32u || (drain && C.tot != C.done)) {  // a full window, or a run's last one
            spawn_window<GEN>(runs.inst(cur), W, C, R);
            continue;
        }
        // the next tile of this warp, in this run or another
        while (!have || t >= m) {
            if (have) {
                v = !CLAIM || v + nw < dealt ? v + nw : dealt + __shfl_sync(0xffffffffu, claim, 0);
                have = false;
            }
            if (v >= n_work) { ii = -1; break; }
            u = v / parts;
            ii = runs.find(u);
            if (ii != cur) break;
            if (!err) {
                b = u - runs.inst(ii).unit0;
                m = runs.inst(ii).cnt[R.par][b];
                t = v - u * parts;
            } else {
                m = t = 0;
            }
            if (CLAIM && v + nw >= dealt && lane == 0) claim = atomicAdd(&runs.claims()->claim_spawn, 1);
            have = true;
        }
        const bool more = have && t < m;
        if (cur >= 0 && !err) {
            const DevInst &I = runs.inst(cur);
            const bool divide = C.nd >= 32 || (!more && C.nd > 0);
            if (more || divide) {
                // parents from the list (a tile) or from the division queue
                const int n = min(C.nd, 32);
                unsigned slot;
                bool in;
                __syncwarp();
                if (divide) {
                    in = lane < n;
                    slot = W.divq[in ? C.nd - n + lane : 0];
                    C.nd -= n;
                } else {
                    const int d = t + lane * parts;
                    in = d < m;
                    slot = (unsigned)((size_t)b * CAP_M + d);
                    t += 32 * parts;
                }
                ulonglong2 kk = make_ulonglong2(0, 0);
                double c = 0.0;
                uint8_t f = 0;
                if (in) {
                    kk = I.key[R.par][slot];
                    c = I.c[R.par][slot];
                    f = I.fl[R.par][slot];
                }
                unsigned nat = 0;
                bool valid = !is_zero(c), later = false;
                double cper = c;  // C / 1 is C
                const bool init = (dbits(c) & ~SIGN64) > dbits(I.n_a) || (f & (DFLAG_REF | DFLAG_D));
                const unsigned fl = (init ? 1u : 0u) | ((f & DFLAG_D) ? 2u : 0u);
                if (valid && !abs_lt(c, 0x1p31)) {
                    atomicOr(&I.st->err, ERRB_NUMERIC);
                    valid = false;
                }
                if (valid) nat = (unsigned)ceil_abs(c);
                if (divide) {
                    cper = c / (double)max(nat, 1u);
                } else {
                    att += nat;
                    if (nat > max(heavy_min, I.heavy_floor)) {
                        queue_heavy(I, kk, c, nat, fl, slot);
                        valid = false;
                    } else if (nat & (nat - 1)) {
                        later = true;
                        valid = false;
                    } else if (valid) {  // n_att = 2^s <= 2 |C|: the quotient is C with its exponent lowered by s
                        cper = bitsd(dbits(c) - ((u64)(31 - __clz(nat)) << 52));
                    }
                }
                const unsigned md = __ballot_sync(0xffffffffu, later);
                if (later) W.divq[C.nd + __popc(md & below)] = slot;
                C.nd += __popc(md);
                spawn_append(W, C, valid, kk, nat, cper, fl, slot);
                continue;
            }
            // the run is at its end for this warp: what is still pending
            if (C.tot != C.done || C.nq > 0 || (ADAPT && R.aq->n > 0)) {
                drain = true;
                continue;
            }
            for (int o = 16; o >= 1; o >>= 1) att += __shfl_xor_sync(0xffffffffu, att, o);
            if (lane == 0 && att) red_add(&I.acc[(gw % NSHARD) * ACC_STRIDE + ACC_ATT], (u64)att);
        }
        if (ii < 0) return;
        drain = false;
        // a new run: its state, read once per run a warp meets (a flag raised
        // by another warp during this kernel makes the host repeat the
        // iteration, whose output is then discarded)
        cur = ii;
        const DevInst &I = runs.inst(cur);
        C = SpawnCursor{0, 0, 0, 0, 0, 0};
        att = 0;
        err = __shfl_sync(0xffffffffu, *(volatile int *)&I.st->err, 0);
        R.par = I.st->parity;
        R.it = I.st->iter;
        R.S = I.st->S;
        if (lane == 0 && v == I.unit0 * parts) I.st->err_at_start = err;  // the state seen when this run's spawning began
    }
}

template <int GEN, bool ADAPT, bool CLAIM>
__global__ void __launch_bounds__(SP_THREADS, ADAPT ? 3 : 4) k_spawn(const __grid_constant__ DevInst I, int n_units,
                                                                     int parts, unsigned heavy_min)
{
    spawn_body<GEN, ADAPT, CLAIM>(OneRun{I}, n_units, parts, heavy_min);
}

template <bool ADAPT, bool CLAIM>
__global__ void __launch_bounds__(SP_THREADS, ADAPT ? 3 : 4) k_spawn_batch(const DevInst *__restrict__ insts,
                                                                        const int *__restrict__ unit_start, int n_inst,
                                                                        int n_units, int parts, unsigned heavy_min)
{
    spawn_body<GEN_ANY, ADAPT, CLAIM>(RunTable{insts, unit_start, n_inst}, n_units, parts, heavy_min);
}

// the slices of heavily populated determinants, one block each
template <typename RUNS>
__device__ __forceinline__ void heavy_body(const RUNS &runs, int n_inst)
{
    extern __shared__ __align__(16) unsigned char sp_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    SpawnWarp &W = reinterpret_cast<SpawnWarp *>(sp_raw)[warp];
    AdaptQueue *aq = reinterpret_cast<AdaptQueue *>(sp_raw + SP_WARPS * sizeof(SpawnWarp)) + warp;
    if (lane == 0) aq->n = 0;
    __syncwarp();
    // between the spawning that claimed units and the annihilation that will
    if (blockIdx.x == 0 && threadIdx.x == 0) runs.claims()->claim_spawn = runs.claims()->claim_anni = 0;
    // lane l looks at run i0 + l (a look costs an L2 round trip: 64 runs one
    // after the other took 100 us); only runs with work for this block follow.
    // The slices of all runs are dealt out in one sequence (`first` slices
    // before the run's own, modulo the grid).  Dealt out from block 0 for every
    // run they piled up on the first blocks: 64 lattice runs 1.61 ms per
    // iteration of all kernels, now 1.44 (the deferred buckets' share included)
    int first = 0;
    for (int i0 = 0; i0 < n_inst; i0 += 32) {
        int nh_l = 0, ex = 0;
        if (i0 + lane < n_inst) {
            const IterState *st = runs.inst(i0 + lane).st;
            const int err = *(volatile const int *)&st->err, n = *(volatile const int *)&st->heavy_n;
            nh_l = err ? 0 : n;
            ex = (int)((unsigned)n % gridDim.x);  // a run's flag may rise meanwhile: it does not move the others' slices
        }
        int q_l = (int)blockIdx.x;
        if (!RUNS::SINGLE) {
            const int mine = ex;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, ex, o);
                if (lane >= o) ex += y;
            }
            q_l = (int)((blockIdx.x + gridDim.x - (unsigned)(first + ex - mine) % gridDim.x) % gridDim.x);
            first = (int)((unsigned)(first + __shfl_sync(0xffffffffu, ex, 31)) % gridDim.x);
        }
        unsigned todo = __ballot_sync(0xffffffffu, q_l < nh_l);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            const int nh = __shfl_sync(0xffffffffu, nh_l, src), q0 = __shfl_sync(0xffffffffu, q_l, src);
            const DevInst &I = runs.inst(i0 + src);
            const SpawnRun R{I.st->iter, I.st->S, I.st->parity, I.adaptive ? aq : nullptr};
            int nq = 0;
            for (int q = q0; q < nh; q += gridDim.x) {
                const HeavyChunk h = I.heavy[q];
                for (unsigned a = 32u * warp; a < h.count; a += SP_THREADS) {
                    attempts32<GEN_ANY>(I, W, nq, R, a + lane < h.count, make_ulonglong2(h.a, h.b), h.k0 + a + lane, h.cper,
                                    h.flags, h.slot);
                    drain_adaptive(I, R, 32);  // each step below and above queues at most 32 more
                    if (nq >= 32) eval_singles(I, W, nq, R);
                    drain_adaptive(I, R, 32);
                }
            }
            if (nq > 0) eval_singles(I, W, nq, R);
            drain_adaptive(I, R, 1);
        }
    }
}

__global__ void __launch_bounds__(SP_THREADS, 3) k_spawn_heavy(const __grid_constant__ DevInst I)
{
    heavy_body(OneRun{I}, 1);
}

__global__ void __launch_bounds__(SP_THREADS, 3) k_spawn_heavy_batch(const DevInst *__restrict__ insts, int n_inst)
{
    heavy_body(RunTable{insts, nullptr, n_inst}, n_inst);
}

// slot of determinant (a, b) in the trial-estimator table, or -1
__device__ __forceinline__ int trial_find(const DevInst &I, u64 a, u64 b)
{
    const u64 mask = (1ULL << I.trial_bits) - 1;
    u64 s = det_hash(a, b) & mask;
    for (u64 probe = 0; probe <= mask; probe++) {
        if (__ldg(I.trial_state + s) == 0u) return -1;
        if (__ldg(&I.trial_tab[s].a) == a && __ldg(&I.trial_tab[s].b) == b) return (int)s;
        s = (s + 1) & mask;
    }
    return -1;
}

// ------------------------------------------------------------------ annihilation
// One warp per bucket: the bucket's walkers and spawns (up to AW_E records;
// larger buckets go to k_annihilate_big) meet in the warp's own shared
// memory, without a block barrier:
//   A  walkers: keys and C into shared memory and into a small hash table
//      (one byte per slot: the record);
//   B  spawns: each finds its target or becomes the record of a new
//      determinant; the initiator rule (Sec. I: a non-initiator's spawn
//      survives only onto a determinant occupied at the start of the
//      iteration); an accepted spawn is pushed on its target's list;
//   C  rounds of 32 records: walkers (death (b) and Eq. (3), then their
//      spawns added), new determinants (the sum of their spawns), and last
//      the records whose sum needs the rounding draw of the annihilation,
//      few enough that they are collected first.  Kept records go to the new
//      bucket in order.  Sums are exact and rounded once, so no order matters.
// New determinants wait in a queue of the warp for H_jj until there are 32.
// The table needs no atomics (warp_table.cuh).  A block of 256 threads per
// bucket of 1024 slots (three barriers per bucket, 128-bit shared
// accumulators, two blocks per SM) spent
// 5.6 of 14 stall cycles per instruction at those barriers: 7.13 ms at 7.3e7
// determinants and 3.5e7 spawns (50 orbitals), and 0.87 ms more for H_jj in a
// kernel of its own; this takes 4.2 ms for both.  It is bound by instruction
// issue (56 % of the slots; the warps of an SM are at different places of a
// long code) and latency, DRAM at 17 %.
constexpr int AN_THREADS = 256, AN_WARPS = AN_THREADS / 32;
constexpr int AW_E = 192;          // records per warp (bytes of the table index them: below 255)
constexpr int AW_TAB = 512;
constexpr unsigned AW_NONE = 0xffu;
constexpr int BIG_SCRATCH = 1 << 30;  // big_list: the bucket needs the global scratch (written when it is deferred: a
                                      // bucket's counts say nothing once another block has annihilated it)
constexpr int ND_MAX = 64;         // electrons the pair table covers
constexpr int ND_PAIRS = ND_MAX * (ND_MAX - 1) / 2;

struct AnniWarp {
    ulonglong2 key[AW_E];          // walkers [0, m), spawns [m, m + s)
    double val[AW_E];              // C (walkers), w (spawns); the sum of a record waiting for its draw
    int head[AW_E];                // the record last pushed on this record's list, -1: none
    unsigned short next[AW_E];     // the one pushed before it (0xffff: none); bit 15 of the index: rejected
    unsigned char tab[AW_TAB];
    unsigned char list[2 * AW_E];  // records of new determinants, then those waiting for the annihilation draw
    unsigned newq[32 + AW_E];      // slots of new determinants waiting for H_jj
    unsigned enq[32 + AW_E];       // slots of determinants connected to the reference waiting for their E_num term
    unsigned char orb[4][ND_MAX];
};
constexpr size_t AN_SMEM = AN_WARPS * sizeof(AnniWarp) + ND_PAIRS * sizeof(unsigned short);
static_assert(KIDX * sizeof(unsigned short) <= AW_E * sizeof(ulonglong2), "the new list's index is built over the keys");
static_assert(3 * (AN_SMEM + 1024) <= 233472, "resident annihilation blocks per SM");
static_assert(AW_E < (int)AW_NONE && CAP_M <= 0x7fff, "records in a byte, list links in 15 bits");

// A warp's share of a run's exact integer totals over the buckets it meets
// in one launch (integer sums: any order gives the same total)
struct AnniTotals {
    u128 nw = 0;            // N_w * 2^32
    i128 ann = 0;           // annihilated walkers * 2^32
    i128 enm = 0;           // E_num * 2^Fe (terms truncated to the grid)
    long long rej = 0;      // rejected non-initiator spawns
    long long ndet = 0;     // determinants kept (lane 0)
    long long spawns = 0;   // spawns received (lane 0)
};

// the totals of a warp into the run's accumulators (line w % NSHARD), then zero
__device__ __forceinline__ void anni_flush(const DevInst &I, AnniTotals &T, int w)
{
    const int lane = threadIdx.x & 31;
    for (int mm = 16; mm >= 1; mm >>= 1) {
        T.rej += __shfl_xor_sync(0xffffffffu, T.rej, mm);
        T.ann += shfl_xor_i128(T.ann, mm);
        T.nw += (u128)shfl_xor_i128((i128)T.nw, mm);
        T.enm += shfl_xor_i128(T.enm, mm);
    }
    if (lane == 0) {
        u64 *acc = I.acc + (w % NSHARD) * ACC_STRIDE;
        limb_add(acc + ACC_NW, (i128)T.nw);
        limb_add(acc + ACC_ANN, T.ann);
        limb_add(acc + ACC_ENUM, T.enm);
        if (T.rej) red_add(&acc[ACC_REJ], (u64)T.rej);
        if (T.ndet) red_add(&acc[ACC_NDET], (u64)T.ndet);
        if (T.spawns) red_add(&acc[ACC_SPAWNS], (u64)T.spawns);
    }
    T = AnniTotals{};
}

// the E_num term of a determinant connected to the reference, on the grid
// 2^-Fe (R12)
__device__ __noinline__ i128 enum_term(const DevInst &I, u64 a, u64 b, double c)
{
    if (I.kind == FCIQMC_HUBBARD) {  // only a hop along a bond couples: H = -+ t = h_ai
        const u64 d = a == I.ref_a ? b ^ I.ref_b : a ^ I.ref_a, x = a == I.ref_a ? b : a;
        if ((a != I.ref_a && b != I.ref_b) || __popcll(d) != 2) return 0;
        const int i = __ffsll((long long)d) - 1, j = 63 - __clzll((long long)d);
        const double H = neg_if(__popcll(x & between(i, j)) & 1, __ldg(I.h + i * I.norb + j));
        return is_zero(H) ? (i128)0 : to_fixed(H * c, I.Fe);
    }
    return to_fixed(hoff_generic(I, a, b, I.ref_a, I.ref_b) * c, I.Fe);
}

// death of a determinant in D (the exact projection's result) or, with the
// adaptive shift (Sec. V), of a non-initiator: S_i = f_i S
__device__ __noinline__ double death_special(const DevInst &I, u64 a, u64 b, double c, double hd, unsigned f, int par,
                                             size_t slot, double shift)
{
    if (f & DFLAG_D) return I.dc_new[d_index_of(I, a, b)];
    double Si = shift;
    if ((dbits(c) & ~SIGN64) <= dbits(I.n_a) && !(f & DFLAG_REF)) {
        const u64 *acc = I.facc[par] + slot * 4;
        const u128 A = ((u128)acc[1] << 64) | acc[0], T = ((u128)acc[3] << 64) | acc[2];
        if (T != 0) Si = (u128_to_double(A) / u128_to_double(T)) * shift;
    }
    return c * (1.0 - I.tau * (hd - Si));
}

// a kept determinant of D, and the reference
__device__ __noinline__ void keep_special(const DevInst &I, u64 a, u64 b, double c, unsigned f, int np)
{
    if (f & DFLAG_REF) I.st->e_den = c;
    if (f & DFLAG_D) I.dc_buf[np][d_index_of(I, a, b)] = c;
}

// H_jj - E_ref of a lattice: U times the doubly occupied sites
__device__ __noinline__ double lattice_diag(const DevInst &I, u64 a, u64 b)
{
    const i128 xr = (i128)(((u128)I.xref_hi << 64) | (u128)I.xref_lo);
    return fixed_to_double((i128)__popcll(a & b) * fx_load(I.Jfx, 0) - xr, I.F);
}

// (numerator, denominator) of the trial-wave-function estimator (Sec. IV)
__device__ __noinline__ double2 trial_terms(const DevInst &I, u64 a, u64 b, double c)
{
    const int ts = is_zero(c) ? -1 : trial_find(I, a, b);
    if (ts < 0) return make_double2(0.0, 0.0);
    return make_double2(__ldg(&I.trial_tab[ts].w) * c, __ldg(&I.trial_tab[ts].cT) * c);
}

// the lines of bucket b that its warp will read, into L2: one line per lane
// (the first 64 keys, C and H_ii, the flags, the spawns at both ends of their region)
__device__ __forceinline__ void prefetch_bucket(const DevInst &I, int b, int par)
{
    const int lane = threadIdx.x & 31;
    const size_t base = (size_t)b * CAP_M, s0 = (size_t)b * I.cap_s, s1 = s0 + I.cap_s;
    const char *p;
    if (lane < 8) p = (const char *)(I.key[par] + base) + 128 * lane;
    else if (lane < 12) p = (const char *)(I.c[par] + base) + 128 * (lane - 8);
    else if (lane < 16) p = (const char *)(I.hd[par] + base) + 128 * (lane - 12);
    else if (lane == 16) p = (const char *)(I.fl[par] + base);
    else if (lane < 19) p = (const char *)(I.skey + s0) + 128 * (lane - 17);
    else if (lane < 22) p = (const char *)(I.skey + s1) - 16 - 128 * (lane - 19);
    else if (lane == 22) p = (const char *)(I.sw + s0);
    else if (lane < 25) p = (const char *)(I.sw + s1) - 8 - 128 * (lane - 23);
    else return;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// exact sum of a list of three or more accepted spawns, rounded once
__device__ __noinline__ double list_sum(const AnniWarp &W, int h, int Fw)
{
    i128 x = 0;
    for (int e = h; e >= 0;) {
        const unsigned nx = W.next[e & 0x7fff];
        if (!(e & 0x8000)) x += to_fixed(W.val[e], Fw);
        e = nx == 0xffffu ? -1 : (int)nx;
    }
    return fixed_to_double(x, Fw);
}

// exact sum of the rejected spawns of a list, rounded once (replica pairs)
__device__ __noinline__ double list_sum_rejected(const AnniWarp &W, int h, int Fw)
{
    i128 x = 0;
    for (int e = h; e >= 0;) {
        const unsigned nx = W.next[e & 0x7fff];
        if (e & 0x8000) x += to_fixed(W.val[e & 0x7fff], Fw);
        e = nx == 0xffffu ? -1 : (int)nx;
    }
    return fixed_to_double(x, Fw);
}

// H_jj - E_ref of up to four determinants of list `np` (slots q[0 .. cnt)),
// eight lanes each: their terms h_pp (electron e1) and pairs e1 < e2 (listed
// in `pair`, e1 | e2 << 8), four loads in flight per lane, exact sum, rounded once
__device__ __forceinline__ void diag_four(const DevInst &I, const unsigned *q, int cnt, int np,
                                          const unsigned short *pair, unsigned char (*orb)[ND_MAX])
{
    const int lane = threadIdx.x & 31, g = lane >> 3, sl = lane & 7;
    const int n = I.n, na = I.na, N = I.norb, T = n + n * (n - 1) / 2;
    const unsigned d = q[g < cnt ? g : 0];
    const ulonglong2 key = I.key[np][d];
    for (int e = sl; e < n; e += 8)
        orb[g][e] = (unsigned char)(e < na ? nth_set(key.x, e) : nth_set(key.y, e - na));
    __syncwarp();
    i128 part = 0;
    for (int t0 = sl; t0 < T; t0 += 32) {
        ulonglong2 v[4];
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int t = t0 + 8 * r;
            v[r] = make_ulonglong2(0, 0);
            if (t < n) v[r] = __ldg(I.hfx + orb[g][t]);
            else if (t < T) {
                const unsigned tm = pair[t - n];
                const int e1 = (int)(tm & 0xffu), e2 = (int)(tm >> 8);
                v[r] = __ldg((((e1 < na) == (e2 < na)) ? I.JKfx : I.Jfx) + orb[g][e1] * N + orb[g][e2]);
            }
        }
#pragma unroll
        for (int r = 0; r < 4; r++) part += (i128)(((u128)v[r].y << 64) | (u128)v[r].x);
    }
    for (int m = 4; m >= 1; m >>= 1) part += shfl_xor_i128(part, m);
    const i128 xref = (i128)(((u128)I.xref_hi << 64) | (u128)I.xref_lo);
    if (sl == 0 && g < cnt) I.hd[np][d] = fixed_to_double(part - xref, I.F);
    __syncwarp();
}

// the same for more electrons than the pair table covers
__device__ __noinline__ void diag_generic(const DevInst &I, const unsigned *q, int cnt, int np)
{
    for (int k = 0; k < cnt; k++) {
        const ulonglong2 kk = I.key[np][q[k]];
        const double hdv = diag_exact_warp(I, kk.x, kk.y);
        if ((threadIdx.x & 31) == 0) I.hd[np][q[k]] = hdv;
    }
    __syncwarp();
}

// the pairs e1 < e2 of up to ND_MAX electrons, in the order of e2 (whole block)
__device__ __forceinline__ void fill_pairs(unsigned short *pair)
{
    for (int c = 1 + (int)(threadIdx.x >> 5); c < ND_MAX; c += (int)(blockDim.x >> 5))
        for (int r = (int)(threadIdx.x & 31); r < c; r += 32) pair[c * (c - 1) / 2 + r] = (unsigned short)(r | (c << 8));
    __syncthreads();
}

// H_jj of queued new determinants: 32 at a time, one per lane (half the
// instructions of eight lanes per determinant, and no reduction); a run's
// last few by eight lanes each (a quarter of the latency).  On short lists
// every warp ends with a few: 40 orbitals, 2e4 walkers 43.5 us per iteration,
// 61.5 with those by a lane each (24 orbitals 40.9 and 48.5, 50 orbitals at
// 1e5 54.8 and 71.7); with the line at 31 in place of 8 they are the same.
__device__ __forceinline__ void new_diag(const DevInst &I, AnniWarp &W, int &nq, int np, const unsigned short *pair, bool all)
{
    __syncwarp();
    while (nq >= 32 || (all && nq > 8)) {
        const int lane = threadIdx.x & 31, cnt = min(nq, 32);
        nq -= cnt;
        if (lane < cnt) {
            const unsigned d = W.newq[nq + lane];
            const ulonglong2 kk = I.key[np][d];
            I.hd[np][d] = diag_exact_thread(I, kk.x, kk.y);
        }
        __syncwarp();
    }
    while (all && nq > 0) {
        const int cnt = min(nq, 4);
        nq -= cnt;
        if (I.n <= ND_MAX) diag_four(I, W.newq + nq, cnt, np, pair, W.orb);
        else diag_generic(I, W.newq + nq, cnt, np);
    }
}

// the E_num terms of queued determinants, 32 at a time (one determinant in a
// hundred is connected to the reference, but its term costs a warp hundreds of
// instructions whatever its active lanes: taken where it was found it was 235
// of 756 us at 7.6e6 determinants, 50 orbitals)
__device__ __forceinline__ void enum_queue(const DevInst &I, AnniWarp &W, int &ne, int np, bool all, AnniTotals &T)
{
    __syncwarp();
    while (ne >= 32 || (all && ne > 0)) {
        const int lane = threadIdx.x & 31, cnt = min(ne, 32);
        ne -= cnt;
        if (lane < cnt) {
            const unsigned d = W.enq[ne + lane];
            const ulonglong2 kk = I.key[np][d];
            T.enm += enum_term(I, kk.x, kk.y, I.c[np][d]);
        }
        __syncwarp();
    }
}

// EXTRA: some run of the launch has replica side lists or the adaptive shift
template <bool EXTRA>
__device__ __forceinline__ void anni_bucket_warp(const DevInst &I, AnniWarp &W, int b, int par, long long it,
                                                 double shift, int m, int si, int sn, AnniTotals &T, int &nq, int &ne)
{
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u, full = 0xffffffffu;
    const int E = m + si + sn, np = par ^ 1;
    const size_t base = (size_t)b * CAP_M, sbase = (size_t)b * I.cap_s;
    constexpr unsigned tmask = AW_TAB - 1;
    const bool side = EXTRA && I.side != nullptr, adaptive = EXTRA && I.adaptive;

    // A
    __syncwarp();
    {
        uint4 *tz = reinterpret_cast<uint4 *>(W.tab);
        for (int q = lane; q < AW_TAB / 16; q += 32) tz[q] = make_uint4(full, full, full, full);
    }
    for (int e = lane; e < E; e += 32) W.head[e] = -1;
    __syncwarp();
    // A and B in rounds of 32 records: walkers and spawns share the rounds'
    // code; a round holds one kind
    const int ra = (m + 31) >> 5, rb = (si + sn + 31) >> 5;
    long long rejected = 0;
    for (int r = 0; r < ra + rb; r++) {
        const bool walk = r < ra;
        const int q = (walk ? r : r - ra) * 32 + lane;    // walker or spawn number
        const bool on = q < (walk ? m : si + sn);
        const int e = walk ? q : m + q;
        ulonglong2 k = make_ulonglong2(0, 0);
        double v = 0.0;
        if (on) {
            const size_t o = walk ? base + q : sbase + (q < si ? q : I.cap_s - 1 - (q - si));
            k = (walk ? I.key[par] : I.skey)[o];
            v = (walk ? I.c[par] : I.sw)[o];
            W.key[e] = k;
            W.val[e] = v;
        }
        __syncwarp();
        // (walkers are distinct: they are not compared)
        const int target = warp_claim(W.tab, tmask, (unsigned)det_hash(k.x, k.y) & tmask, (unsigned char)e,
                                      (unsigned char)AW_NONE, on, [&](unsigned char x) {
                                          if (walk) return false;
                                          const ulonglong2 kk = W.key[x];
                                          return kk.x == k.x && kk.y == k.y;
                                      });
        if (!walk && on) {
            const bool accepted = q < si || (target < m && !is_zero(W.val[target]));
            if (accepted || side) {
                const int old = atomicExch(&W.head[target], accepted ? e : (e | 0x8000));
                W.next[e] = (unsigned short)(old < 0 ? 0xffff : old);
            }
            if (!accepted) rejected++;
        }
    }
    __syncwarp();
    T.rej += rejected;

    // new determinants that hold spawns (side lists: every new one)
    int nown = 0;
    for (int q0 = 0; q0 < si + sn; q0 += 32) {
        const bool own = q0 + lane < si + sn && W.head[m + q0 + lane] >= 0;
        const unsigned mo = __ballot_sync(full, own);
        if (own) W.list[nown + __popc(mo & below)] = (unsigned char)(m + q0 + lane);
        nown += __popc(mo);
    }
    __syncwarp();

    // C: items [0, m) walkers, [m, m + nown) new determinants, then those
    // waiting for their draw (W.list past nown), which join as they appear
    int total = 0, items = m + nown;
    bool bad = false;
    double tnum = 0.0, tden = 0.0;
    for (int i0 = 0; i0 < items;) {
        const int i = i0 + lane;
        const bool on = i < items, walk = i < m, pend = i >= m + nown;
        i0 = min(i0 + 32, items);
        const int e = !on ? 0 : (walk ? i : (int)W.list[i - m]);
        const bool old = on && e < m;  // a determinant of the old list
        int h = -1;
        ulonglong2 k = make_ulonglong2(0, 0);
        double v = 0.0, hd = 0.0;
        unsigned f = 0;
        if (on) {
            k = W.key[e];
            if (!pend) h = W.head[e];
            if (walk || pend) v = W.val[e];
            if (old) {
                hd = I.hd[par][base + e];
                f = I.fl[par][base + e];
            }
        }
        const double c0 = v;
        bool draw = on && pend;
        if (on && walk) {
            if ((f & DFLAG_D) || adaptive) v = death_special(I, k.x, k.y, v, hd, f, par, base + e, shift);
            else v = v * (1.0 - I.tau * (hd - shift));  // C (1 - tau (H_ii - E_ref - S))
            draw = !(f & DFLAG_D) && !is_zero(v) && abs_lt(v, I.cmin);
        }
        if (__any_sync(full, draw)) {
            u64 w[4];
            philox<2>(k.x, k.y, (u64)it, (u64)(pend ? PURPOSE_ANNIH : PURPOSE_DEATH), I.seed, I.replica, w);
            if (draw) v = round_stoch(v, I.cmin, I.cmin_log2, I.cmin_pow2, w[0]);
        }
        bool later = false;
        double sacc = 0.0;
        if (h >= 0) {
            // the accepted spawns: one is exact, the exact sum of two rounded
            // once is the binary64 sum; more go through the fixed-point sum
            const double cp = v;
            int cnt = 0;
            for (int x = h; x >= 0;) {
                const unsigned nx = W.next[x & 0x7fff];
                if (!EXTRA || !(x & 0x8000)) {
                    const double wv = W.val[x];
                    sacc = cnt ? sacc + wv : wv;
                    cnt++;
                    T.ann += (i128)fx32(wv);
                }
                x = nx == 0xffffu ? -1 : (int)nx;
            }
            if (cnt > 2) sacc = list_sum(W, h, I.Fw);
            if (cnt) {
                v = walk ? cp + sacc : sacc;
                T.ann += (walk ? (i128)fx32(cp) : (i128)0) - (i128)fx32(v);
                later = !(f & DFLAG_D) && !is_zero(v) && abs_lt(v, I.cmin);
            }
        }
        if (side && on && !pend) {  // replica pair: the record's entry
            SideEnt &se = I.side[(size_t)b * I.side_cap + i];
            se.a = k.x; se.b = k.y;
            se.c0 = walk ? c0 : 0.0;
            se.hd = walk ? hd : 0.0;
            se.sacc = sacc;
            se.srej = h >= 0 ? list_sum_rejected(W, h, I.Fw) : 0.0;
        }
        const unsigned ml = __ballot_sync(full, later);
        if (later) {
            W.list[items - m + __popc(ml & below)] = (unsigned char)e;
            W.val[e] = v;
        }
        items += __popc(ml);
        const bool keep = on && !later && (!is_zero(v) || (f & (DFLAG_REF | DFLAG_D)));
        const unsigned mk = __ballot_sync(full, keep);
        const int pos = total + __popc(mk & below);
        total += __popc(mk);
        const bool write = keep && pos < CAP_M, lattice = I.kind == FCIQMC_HUBBARD;
        const unsigned mn = __ballot_sync(full, write && !old && !lattice);
        if (write) {
            const size_t dst = base + pos;
            I.key[np][dst] = k;
            I.c[np][dst] = v;
            I.fl[np][dst] = (uint8_t)(f & (DFLAG_REF | DFLAG_D));
            if (!old && lattice) hd = lattice_diag(I, k.x, k.y);
            if (old || lattice) I.hd[np][dst] = hd;
            else W.newq[nq + __popc(mn & below)] = (unsigned)dst;
            if (!abs_lt(v, 0x1p31)) bad = true;
            else T.nw += fx32(v);
            if (f & (DFLAG_REF | DFLAG_D)) keep_special(I, k.x, k.y, v, f, np);
            if (I.trial_bits) {
                const double2 x = trial_terms(I, k.x, k.y, v);
                tnum = tnum + x.x;
                tden = tden + x.y;
            }
            if (adaptive) {
                u64 *acc = I.facc[np] + dst * 4;
                acc[0] = 0; acc[1] = 0; acc[2] = 0; acc[3] = 0;
            }
        }
        nq += __popc(mn);
        const bool conn = write && !(f & DFLAG_REF) && !is_zero(v) &&
                          __popcll(k.x ^ I.ref_a) + __popcll(k.y ^ I.ref_b) <= 4;
        const unsigned me = __ballot_sync(full, conn);
        if (conn) W.enq[ne + __popc(me & below)] = (unsigned)(base + pos);
        ne += __popc(me);
        __syncwarp();
    }
    if (bad) atomicOr(&I.st->err, ERRB_NUMERIC);
    if (adaptive && total <= CAP_M) {
        // the new list's index (hash -> position + 1) for the next iteration's
        // spawns, built where the keys were
        unsigned short *kx = reinterpret_cast<unsigned short *>(W.key);
        for (int q = lane; q < KIDX; q += 32) kx[q] = 0;
        __syncwarp();
        for (int p0 = 0; p0 < total; p0 += 32) {
            const int p = p0 + lane;
            unsigned s = 0;
            if (p < total) {
                const ulonglong2 k = I.key[np][base + p];
                s = (unsigned)det_hash(k.x, k.y) & (unsigned)(KIDX - 1);
            }
            warp_claim(kx, (unsigned)(KIDX - 1), s, (unsigned short)(p + 1), (unsigned short)0, p < total,
                       [](unsigned short) { return false; });
        }
        __syncwarp();
        for (int q = lane; q < KIDX; q += 32) I.kidx[np][(size_t)b * KIDX + q] = kx[q];
    }
    if (I.trial_bits)  // binary64 sums, only when the estimator is on
        for (int mm = 16; mm >= 1; mm >>= 1) {
            tnum = tnum + __shfl_xor_sync(full, tnum, mm);
            tden = tden + __shfl_xor_sync(full, tden, mm);
        }
    if (lane == 0) {
        if (total > CAP_M) { atomicOr(&I.st->err, ERRB_MAIN_CAP); atomicMax(&I.st->need_main, total); }
        else I.cnt[np][b] = total;
        T.ndet += total;
        T.spawns += si + sn;
        if (I.trial_bits) { I.part[b].t_num = tnum; I.part[b].t_den = tden; }
        if (side) I.side_cnt[b] = m + nown;
        I.scnt_i[b] = 0;
        I.scnt_n[b] = 0;
    }
}

template <bool EXTRA, bool CLAIM, typename RUNS>
__device__ __forceinline__ void anni_body(const RUNS &runs, int n_units)
{
    extern __shared__ __align__(16) unsigned char an_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    AnniWarp &W = reinterpret_cast<AnniWarp *>(an_raw)[warp];
    unsigned short *pair = reinterpret_cast<unsigned short *>(an_raw + AN_WARPS * sizeof(AnniWarp));
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nw = (int)((gridDim.x * blockDim.x) >> 5);
    fill_pairs(pair);
    AnniTotals T;
    int cur = -1, err = 0, par = 0, nq = 0, ne = 0;
    long long it = 0;
    double shift = 0.0;
    const int dealt = CLAIM ? dealt_units(n_units, nw) : n_units;
    int claim = 0;  // lane 0: the bucket after the next one, which is known already to be prefetched
    auto after = [&](int x) { return x + nw < dealt ? x + nw : dealt + __shfl_sync(0xffffffffu, claim, 0); };
    for (int u = gw, nx = gw + nw;; u = CLAIM ? nx : u + nw, nx = CLAIM ? after(nx) : nx) {
        const int ii = u < n_units ? runs.find(u) : -1;
        if (ii < 0 && cur < 0) return;  // a warp without buckets
        if (cur >= 0 && (nq >= 32 || (ii != cur && nq > 0))) new_diag(runs.inst(cur), W, nq, par ^ 1, pair, ii != cur);
        if (cur >= 0 && (ne >= 32 || (ii != cur && ne > 0))) enum_queue(runs.inst(cur), W, ne, par ^ 1, ii != cur, T);
        if (ii != cur) {
            // the run's state at the start of the iteration, read once per run a warp meets
            if (cur >= 0) anni_flush(runs.inst(cur), T, gw);
            if (ii < 0) return;
            const DevInst &I = runs.inst(ii);
            cur = ii;
            err = __shfl_sync(0xffffffffu, *(volatile int *)&I.st->err, 0);
            par = I.st->parity;
            it = I.st->iter;
            shift = I.st->S;
        }
        if (CLAIM && nx + nw >= dealt && lane == 0) claim = atomicAdd(&runs.claims()->claim_anni, 1);
        if (err) continue;
        const DevInst &I = runs.inst(cur);
        const int b = u - I.unit0;
        const int m = I.cnt[par][b], si = I.scnt_i[b], sn = I.scnt_n[b];
        const int next = CLAIM ? nx : u + nw;
        if (RUNS::SINGLE && next < n_units) prefetch_bucket(I, next, par);
        if (si + sn > I.cap_s) {
            if (lane == 0) {
                atomicOr(&I.st->err, ERRB_SPAWN_CAP);
                atomicMax(&I.st->need_spawn, si + sn);
                atomicAdd(&I.st->n_spawn_over, 1);
            }
        } else if (m + si + sn > AW_E) {  // deferred to k_annihilate_big
            if (lane == 0) I.big_list[atomicAdd(&I.st->big_n, 1)] = b | (m + si + sn > EMAX ? BIG_SCRATCH : 0);
        } else {
            anni_bucket_warp<EXTRA>(I, W, b, par, it, shift, m, si, sn, T, nq, ne);
        }
    }
}

template <bool EXTRA, bool CLAIM>
__global__ void __launch_bounds__(AN_THREADS, 3) k_annihilate(const __grid_constant__ DevInst I, int n_units)
{
    anni_body<EXTRA, CLAIM>(OneRun{I}, n_units);
}

template <bool EXTRA, bool CLAIM>
__global__ void __launch_bounds__(AN_THREADS, 3) k_annihilate_batch(const DevInst *__restrict__ insts,
                                                                            const int *__restrict__ unit_start,
                                                                            int n_inst, int n_units)
{
    anni_body<EXTRA, CLAIM>(RunTable{insts, unit_start, n_inst}, n_units);
}

// ------------------------------------------------------------------ large buckets
// A bucket with more records than a warp holds: one block, the records staged
// (shared memory for up to EMAX, a global scratch slice beyond) and every
// distinct determinant given one owner record through an open-addressing
// table: walkers are inserted first, then every spawn finds its target or
// inserts itself as the owner of a new determinant.  Accepted weights are
// added to the owner's exact 128-bit accumulator with two 64-bit atomics (the
// low word's carry goes to the high word), so the sum does not depend on the
// order of arrival.
template <typename IDX>
struct Stage {
    ulonglong2 *key;
    double *val;      // C (walkers) or w (spawns); after death C', after annihilation the result
    u64 *acc_lo;
    u64 *acc_hi;
    int *nacc;        // accepted spawns per owner
    int *eflag;       // EF_* bits
    IDX *tab;         // hash table: element index + 1, 0 = empty
    IDX *opos;        // output position of kept owners
};
enum { EF_OWNER = 1, EF_OCC = 2, EF_KEEP = 4, EF_REF = 16, EF_D = 32, EF_REJ = 64, EF_RREC = 128 };
// EF_REJ: a rejected spawn arrived (owners); EF_RREC: this spawn was rejected

struct K3Shared {
    int wsum[K3_THREADS / 32];
    double red_t[K3_THREADS / 32][2];
    u64 red_u[K3_THREADS / 32][8];
    int n_new, side_n;
    int hdr_err, hdr_par;
    long long hdr_it;
    double hdr_S;
};

struct K3Smem {
    K3Shared sh;
    ulonglong2 key[EMAX];
    double val[EMAX];
    u64 acc_lo[EMAX];
    u64 acc_hi[EMAX];
    int nacc[EMAX];
    int eflag[EMAX];
    unsigned short tab[1 << TABBITS];
    unsigned short opos[EMAX];
};
static_assert(3 * (sizeof(K3Smem) + 1024) <= 233472, "three large-bucket blocks per SM");

__device__ __forceinline__ int block_excl_scan(int v, int *wsum, int *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int s = lane < K3_THREADS / 32 ? wsum[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < K3_THREADS / 32) wsum[lane] = s;
    }
    __syncthreads();
    int r = x - v + (warp ? wsum[warp - 1] : 0);
    *total = wsum[K3_THREADS / 32 - 1];
    return r;  // wsum is written again only after the caller's next barrier
}

// Death, annihilation and the reductions of one bucket b (steps (b) and (c)
// of Eq. (4)).  All threads of the block call this together.
template <typename IDX>
__device__ void anni_bucket(const DevInst &I, K3Shared &S, Stage<IDX> W, int tabbits, int b, int par, long long it,
                            double shift, int m, int si, int sn)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int E = m + si + sn, cap_s = I.cap_s, TAB = 1 << tabbits;
    const u64 tmask = (u64)(TAB - 1);
    const size_t base = (size_t)b * CAP_M, sbase = (size_t)b * cap_s;
    const ulonglong2 *okey = I.key[par];
    const double *oc = I.c[par], *ohd = I.hd[par];
    const uint8_t *ofl = I.fl[par];

    // 1. stage: walkers [0, m), initiator spawns [m, m+si), other spawns [m+si, E);
    //    four records per thread per round, all loads issued before the stores
    for (int q = t; q < TAB; q += K3_THREADS) W.tab[q] = 0;
    if (t == 0) S.n_new = 0;
    for (int e0 = 0; e0 < E; e0 += 4 * K3_THREADS) {
        ulonglong2 k[4];
        double v[4];
        int f[4];
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int e = e0 + r * K3_THREADS + t;
            k[r] = make_ulonglong2(0, 0);
            v[r] = 0.0;
            f[r] = 0;
            if (e < m) {
                k[r] = okey[base + e];
                v[r] = oc[base + e];
                const uint8_t fl = ofl[base + e];
                f[r] = EF_OWNER | ((fl & DFLAG_REF) ? EF_REF : 0) | ((fl & DFLAG_D) ? EF_D : 0);
            } else if (e < m + si) {
                k[r] = I.skey[sbase + (e - m)];
                v[r] = I.sw[sbase + (e - m)];
            } else if (e < E) {
                const int slot = cap_s - 1 - (e - m - si);
                k[r] = I.skey[sbase + slot];
                v[r] = I.sw[sbase + slot];
            }
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int e = e0 + r * K3_THREADS + t;
            if (e < E) {
                W.key[e] = k[r];
                W.val[e] = v[r];
                W.acc_lo[e] = 0;
                W.acc_hi[e] = 0;
                W.nacc[e] = 0;
                W.eflag[e] = f[r] | ((e < m && !is_zero(v[r])) ? EF_OCC : 0);
            }
        }
    }
    __syncthreads();
    // 2. walkers (thread t holds walkers t + r K3_THREADS, r < 4): insert into
    //    the table (keys are distinct); death (b) and Eq. (3), the rounding
    //    draws two at a time
    static_assert(CAP_M <= 4 * K3_THREADS, "walkers per thread");
    double hdr[4];
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const int e = t + r * K3_THREADS;
        hdr[r] = e < m ? ohd[base + e] : 0.0;
    }
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const int e = t + r * K3_THREADS;
        if (e < m) {
            const ulonglong2 k = W.key[e];
            u64 s = det_hash(k.x, k.y) & tmask;
            while (atomicCAS(&W.tab[s], (IDX)0, (IDX)(e + 1)) != (IDX)0) s = (s + 1) & tmask;
        }
    }
#pragma unroll
    for (int r0 = 0; r0 < 4; r0 += 2) {
        double cp[2];
        bool draw[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int e = t + (r0 + h) * K3_THREADS;
            draw[h] = false;
            cp[h] = 0.0;
            if (e < m) {
                if (W.eflag[e] & EF_D) {
                    const ulonglong2 k = W.key[e];
                    cp[h] = I.dc_new[d_index_of(I, k.x, k.y)];
                } else {
                    // C (1 - tau (H_ii - E_ref - S_i)), then rounding with the death draw;
                    // S_i = f_i S for a non-initiator with the adaptive shift (Sec. V)
                    double Si = shift;
                    const bool init = (dbits(W.val[e]) & ~SIGN64) > dbits(I.n_a) || (W.eflag[e] & EF_REF);
                    if (I.adaptive && !init) {
                        const u64 *acc = I.facc[par] + (base + e) * 4;
                        const u128 A = ((u128)acc[1] << 64) | acc[0], T = ((u128)acc[3] << 64) | acc[2];
                        if (T != 0) Si = (u128_to_double(A) / u128_to_double(T)) * shift;
                    }
                    const double fct = 1.0 - I.tau * (hdr[r0 + h] - Si);
                    cp[h] = W.val[e] * fct;
                    draw[h] = !is_zero(cp[h]) && abs_lt(cp[h], I.cmin);
                }
            }
        }
        if (I.side)  // replica pair: walkers' entries (start amplitude, H_ii - E_ref)
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int e = t + (r0 + h) * K3_THREADS;
                if (e < m) {
                    SideEnt &se = I.side[(size_t)b * I.side_cap + e];
                    const ulonglong2 k = W.key[e];
                    se.a = k.x; se.b = k.y; se.c0 = W.val[e]; se.hd = hdr[r0 + h]; se.sacc = 0.0; se.srej = 0.0;
                }
            }
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int e = t + (r0 + h) * K3_THREADS;
            if (draw[h]) {
                const ulonglong2 k = W.key[e];
                u64 w[4];
                philox(k.x, k.y, (u64)it, (u64)PURPOSE_DEATH, I.seed, I.replica, w);
                cp[h] = round_stoch(cp[h], I.cmin, I.cmin_log2, I.cmin_pow2, w[0]);
            }
            if (e < m) W.val[e] = cp[h];
        }
    }
    __syncthreads();
    // 3. spawns: find the target or become the owner of a new determinant;
    //    initiator rule (Sec. I): a non-initiator spawn survives only onto a
    //    determinant occupied at the start of the iteration
    long long rejected = 0;
    i128 ann = 0;
    for (int e = m + t; e < E; e += K3_THREADS) {
        const ulonglong2 k = W.key[e];
        u64 s = det_hash(k.x, k.y) & tmask;
        int target = -1;
        while (true) {
            IDX v = ((volatile IDX *)W.tab)[s];
            if (v == 0) {
                IDX old = atomicCAS(&W.tab[s], (IDX)0, (IDX)(e + 1));
                if (old == 0) { target = e; break; }
                v = old;
            }
            const int tt = (int)v - 1;
            const ulonglong2 kk = W.key[tt];
            if (kk.x == k.x && kk.y == k.y) { target = tt; break; }
            s = (s + 1) & tmask;
        }
        if (target == e) atomicOr(&W.eflag[e], EF_OWNER);
        const bool init = e < m + si;
        const bool accepted = init || (target < m && (W.eflag[target] & EF_OCC));
        if (!accepted) {
            rejected++;
            if (I.side) {
                W.opos[e] = (IDX)target;
                atomicOr(&W.eflag[e], EF_RREC);
                atomicOr(&W.eflag[target], EF_REJ);
            }
            continue;
        }
        const double w = W.val[e];
        const i128 x = to_fixed(w, I.Fw);
        const u64 lo = (u64)x, hi = (u64)((u128)x >> 64);
        const u64 old = atomicAdd((unsigned long long *)&W.acc_lo[target], (unsigned long long)lo);
        atomicAdd((unsigned long long *)&W.acc_hi[target], (unsigned long long)(hi + (old + lo < old ? 1ULL : 0ULL)));
        atomicAdd(&W.nacc[target], 1);
        ann += (i128)fx32(w);
    }
    __syncthreads();
    // replica pair: every owner's entry receives the accepted and the rejected
    // spawn sums (exact, rounded once each); the rejected weights are summed
    // in the accumulators once the accepted sums have been read
    const bool side = I.side != nullptr;
    if (side) {
        if (t == 0) S.side_n = 0;
        __syncthreads();
        for (int e = t; e < E; e += K3_THREADS) {
            const int f = W.eflag[e];
            if (!(f & EF_OWNER)) continue;
            const bool had = W.nacc[e] > 0;
            const double sacc = had ? fixed_to_double((i128)(((u128)W.acc_hi[e] << 64) | (u128)W.acc_lo[e]), I.Fw)
                                    : 0.0;
            const int slot = e < m ? e : m + atomicAdd(&S.side_n, 1);
            SideEnt &se = I.side[(size_t)b * I.side_cap + slot];
            if (e >= m) {
                const ulonglong2 k = W.key[e];
                se.a = k.x; se.b = k.y; se.c0 = 0.0; se.hd = 0.0; se.srej = 0.0;
            }
            se.sacc = sacc;
            W.nacc[e] = (slot << 1) | (had ? 1 : 0);
            W.acc_lo[e] = 0;
            W.acc_hi[e] = 0;
        }
        __syncthreads();
        for (int e = m + t; e < E; e += K3_THREADS) {
            if (!(W.eflag[e] & EF_RREC)) continue;
            const int target = (int)W.opos[e];
            const i128 x = to_fixed(W.val[e], I.Fw);
            const u64 lo = (u64)x, hi = (u64)((u128)x >> 64);
            const u64 old = atomicAdd((unsigned long long *)&W.acc_lo[target], (unsigned long long)lo);
            atomicAdd((unsigned long long *)&W.acc_hi[target], (unsigned long long)(hi + (old + lo < old ? 1ULL : 0ULL)));
        }
        __syncthreads();
        for (int e = t; e < E; e += K3_THREADS) {
            const int f = W.eflag[e];
            if (!(f & EF_OWNER) || !(f & EF_REJ)) continue;
            const i128 X = (i128)(((u128)W.acc_hi[e] << 64) | (u128)W.acc_lo[e]);
            I.side[(size_t)b * I.side_cap + (W.nacc[e] >> 1)].srej = fixed_to_double(X, I.Fw);
        }
        if (t == 0) I.side_cnt[b] = m + S.side_n;
    }
    // 4. owners: sum = C' + exact spawn sum, then Eq. (3) with the annihilation draw
    for (int e = t; e < E; e += K3_THREADS) {
        const int f = W.eflag[e];
        if (!(f & EF_OWNER)) continue;
        const bool present = e < m;
        const double cp = present ? W.val[e] : 0.0;
        double accv = cp;
        if (side ? (W.nacc[e] & 1) : W.nacc[e] > 0) {
            const double sw = side ? I.side[(size_t)b * I.side_cap + (W.nacc[e] >> 1)].sacc
                                   : fixed_to_double((i128)(((u128)W.acc_hi[e] << 64) | (u128)W.acc_lo[e]), I.Fw);
            accv = present ? cp + sw : sw;
            ann += (present ? (i128)fx32(cp) : (i128)0) - (i128)fx32(accv);
            if (!(f & EF_D) && !is_zero(accv) && abs_lt(accv, I.cmin)) {
                const ulonglong2 k = W.key[e];
                u64 w[4];
                philox(k.x, k.y, (u64)it, (u64)PURPOSE_ANNIH, I.seed, I.replica, w);
                accv = round_stoch(accv, I.cmin, I.cmin_log2, I.cmin_pow2, w[0]);
            }
        }
        W.val[e] = accv;
        if (!is_zero(accv) || (f & (EF_REF | EF_D))) W.eflag[e] = f | EF_KEEP;
    }
    // 5. output positions in element order
    int total;
    const int per = (E + K3_THREADS - 1) / K3_THREADS;
    const int e0 = t * per, e1 = min(E, e0 + per);
    int cnt = 0;
    __syncthreads();
    for (int e = e0; e < e1; e++) cnt += (W.eflag[e] & EF_KEEP) ? 1 : 0;
    int o = block_excl_scan(cnt, S.wsum, &total);
    const bool overflow = total > CAP_M;
    if (overflow && t == 0) { atomicOr(&I.st->err, ERRB_MAIN_CAP); atomicMax(&I.st->need_main, total); }
    for (int e = e0; e < e1; e++)
        if (W.eflag[e] & EF_KEEP) W.opos[e] = (IDX)(o++);
    __syncthreads();

    // 6. write the new bucket; reductions
    const int np = par ^ 1;
    ulonglong2 *nkey = I.key[np];
    double *nc = I.c[np], *nhd = I.hd[np];
    uint8_t *nfl = I.fl[np];
    u128 nw = 0;
    i128 enm = 0;  // E_num: each term truncated to the grid 2^-Fe (R12), summed exactly
    double tnum = 0.0, tden = 0.0;
    bool bad = false;
    if (!overflow) {
        for (int r = 0; t + r * K3_THREADS < E; r++) {
            const int e = t + r * K3_THREADS;
            const int f = W.eflag[e];
            if (!(f & EF_KEEP)) continue;
            const ulonglong2 k = W.key[e];
            const double c = W.val[e];
            const size_t dst = base + W.opos[e];
            nkey[dst] = k;
            nc[dst] = c;
            nfl[dst] = (uint8_t)(((f & EF_REF) ? DFLAG_REF : 0) | ((f & EF_D) ? DFLAG_D : 0));
            if (e < m) nhd[dst] = ohd[base + e];  // read again: an L2 hit, fewer live registers
            else {
                const int qn = atomicAdd(&S.n_new, 1);
                W.nacc[qn] = e;  // accumulators are free now: reuse as the list of new determinants
            }
            if (!abs_lt(c, 0x1p31)) bad = true;
            else nw += fx32(c);
            if (f & EF_REF) I.st->e_den = c;
            else {
                const int lev = __popcll(k.x ^ I.ref_a) + __popcll(k.y ^ I.ref_b);
                if (lev <= 4 && !is_zero(c)) enm += to_fixed(hoff_generic(I, k.x, k.y, I.ref_a, I.ref_b) * c, I.Fe);
            }
            if (f & EF_D) I.dc_buf[par ^ 1][d_index_of(I, k.x, k.y)] = c;
            if (I.trial_bits && !is_zero(c)) {  // trial-wave-function estimator (Sec. IV)
                const int ts = trial_find(I, k.x, k.y);
                if (ts >= 0) {
                    tnum = tnum + __ldg(&I.trial_tab[ts].w) * c;
                    tden = tden + __ldg(&I.trial_tab[ts].cT) * c;
                }
            }
        }
    }
    if (bad) atomicOr(&I.st->err, ERRB_NUMERIC);
    __syncthreads();
    // adaptive shift: the new list's index (hash -> position + 1) and zeroed
    // weight sums for the next iteration's spawns
    if (I.adaptive && !overflow) {
        for (int q = t; q < KIDX; q += K3_THREADS) W.tab[q] = 0;
        __syncthreads();
        for (int r = 0; t + r * K3_THREADS < E; r++) {
            const int e = t + r * K3_THREADS;
            if (!(W.eflag[e] & EF_KEEP)) continue;
            const ulonglong2 k = W.key[e];
            unsigned sl = (unsigned)det_hash(k.x, k.y) & (unsigned)(KIDX - 1);
            while (atomicCAS(&W.tab[sl], (IDX)0, (IDX)(W.opos[e] + 1)) != (IDX)0) sl = (sl + 1) & (unsigned)(KIDX - 1);
            u64 *acc = I.facc[np] + (base + W.opos[e]) * 4;
            acc[0] = 0; acc[1] = 0; acc[2] = 0; acc[3] = 0;
        }
        __syncthreads();
        for (int q = t; q < KIDX; q += K3_THREADS) I.kidx[np][(size_t)b * KIDX + q] = (unsigned short)W.tab[q];
    }
    // 7. H_jj - E_ref of the new determinants, a warp each
    if (!overflow) {
        const int nnew = S.n_new;
        for (int q = warp; q < nnew; q += K3_THREADS / 32) {
            const int e = W.nacc[q];
            const ulonglong2 k = W.key[e];
            const double hdv = diag_exact_warp(I, k.x, k.y);
            if (lane == 0) nhd[base + W.opos[e]] = hdv;
        }
    }
    // 8. bucket reductions (fixed order: lanes by xor tree, warps in index order)
    if (I.trial_bits)  // binary64 adds are slow on this part: only when the estimator is on
        for (int mm = 16; mm >= 1; mm >>= 1) {
            tnum = tnum + __shfl_xor_sync(0xffffffffu, tnum, mm);
            tden = tden + __shfl_xor_sync(0xffffffffu, tden, mm);
        }
    for (int mm = 16; mm >= 1; mm >>= 1) {
        enm += shfl_xor_i128(enm, mm);
        rejected += __shfl_xor_sync(0xffffffffu, rejected, mm);
        ann += shfl_xor_i128(ann, mm);
        nw += (u128)shfl_xor_i128((i128)nw, mm);
    }
    if (lane == 0) {
        S.red_t[warp][0] = tnum;
        S.red_t[warp][1] = tden;
        S.red_u[warp][0] = (u64)nw;
        S.red_u[warp][1] = (u64)(nw >> 64);
        S.red_u[warp][2] = (u64)ann;
        S.red_u[warp][3] = (u64)((u128)ann >> 64);
        S.red_u[warp][4] = (u64)rejected;
        S.red_u[warp][5] = (u64)enm;
        S.red_u[warp][6] = (u64)((u128)enm >> 64);
    }
    __syncthreads();
    if (t == 0) {
        double tn = 0.0, td = 0.0;
        u128 nws = 0;
        i128 anns = 0, ens = 0;
        long long rej = 0;
        for (int k = 0; k < K3_THREADS / 32; k++) {
            if (I.trial_bits) {
                tn = tn + S.red_t[k][0];
                td = td + S.red_t[k][1];
            }
            nws += ((u128)S.red_u[k][1] << 64) | S.red_u[k][0];
            anns += (i128)(((u128)S.red_u[k][3] << 64) | S.red_u[k][2]);
            rej += (long long)S.red_u[k][4];
            ens += (i128)(((u128)S.red_u[k][6] << 64) | S.red_u[k][5]);
        }
        // the bucket's share of the run's exact totals (its line b % NSHARD)
        u64 *acc = I.acc + (b % NSHARD) * ACC_STRIDE;
        limb_add(acc + ACC_NW, (i128)nws);
        limb_add(acc + ACC_ANN, anns);
        limb_add(acc + ACC_ENUM, ens);
        red_add(&acc[ACC_NDET], (u64)total);
        if (rej) red_add(&acc[ACC_REJ], (u64)rej);
        red_add(&acc[ACC_SPAWNS], (u64)(si + sn));
        if (I.trial_bits) {
            Partial &P = I.part[b];
            P.t_num = tn;
            P.t_den = td;
        }
        if (!overflow) I.cnt[np][b] = total;
        I.scnt_i[b] = 0;
        I.scnt_n[b] = 0;
    }
    // no closing barrier: what thread 0 still reads (the warp sums) is written
    // again only after the next bucket's barriers
}

// one run's deferred buckets (whole block; every block of the launch calls it;
// q0: the first one of this block)
__device__ void annihilate_deferred(const DevInst &I, K3Smem &Sm, int q0)
{
    K3Shared &S = Sm.sh;
    const int t = threadIdx.x;
    __syncthreads();
    if (t == 0) {
        S.hdr_err = *(volatile int *)&I.st->err;
        S.hdr_par = I.st->parity;
        S.hdr_it = I.st->iter;
        S.hdr_S = I.st->S;
        S.n_new = I.st->big_n;
    }
    __syncthreads();
    const int err = S.hdr_err, par = S.hdr_par, nbig = S.n_new;
    const long long it = S.hdr_it;
    const double shift = S.hdr_S;
    __syncthreads();
    if (err || nbig == 0) return;
    const Stage<unsigned short> Ws{Sm.key, Sm.val, Sm.acc_lo, Sm.acc_hi, Sm.nacc, Sm.eflag, Sm.tab, Sm.opos};
    for (int q = q0; q < nbig; q += gridDim.x) {
        const int b = I.big_list[q];
        if (b & BIG_SCRATCH) continue;
        anni_bucket<unsigned short>(I, S, Ws, TABBITS, b, par, it, shift, I.cnt[par][b], I.scnt_i[b], I.scnt_n[b]);
        __syncthreads();
    }
    if (blockIdx.x >= BIG_BLOCKS) return;
    // beyond shared memory: this block's slice of the global scratch
    const int Ecap = CAP_M + I.cap_s, tabbits = I.big_tabbits;
    unsigned char *p = I.big_scratch + (size_t)blockIdx.x * I.big_stride;
    Stage<unsigned> W;
    W.key = (ulonglong2 *)p; p += (size_t)Ecap * sizeof(ulonglong2);
    W.val = (double *)p; p += (size_t)Ecap * sizeof(double);
    W.acc_lo = (u64 *)p; p += (size_t)Ecap * 8;
    W.acc_hi = (u64 *)p; p += (size_t)Ecap * 8;
    W.nacc = (int *)p; p += (size_t)Ecap * 4;
    W.eflag = (int *)p; p += (size_t)Ecap * 4;
    W.opos = (unsigned *)p; p += (size_t)Ecap * 4;
    W.tab = (unsigned *)p;
    for (int q = blockIdx.x; q < nbig; q += BIG_BLOCKS) {
        int b = I.big_list[q];
        if (!(b & BIG_SCRATCH)) continue;
        b &= ~BIG_SCRATCH;
        if (!I.big_scratch) {  // no scratch yet: report, the host allocates it and repeats the iteration
            if (t == 0) atomicOr(&I.st->err, ERRB_SPAWN_CAP);
            break;
        }
        anni_bucket<unsigned>(I, S, W, tabbits, b, par, it, shift, I.cnt[par][b], I.scnt_i[b], I.scnt_n[b]);
        __syncthreads();
    }
}

__global__ void __launch_bounds__(K3_THREADS) k_annihilate_big(const DevInst *__restrict__ insts, int n_inst)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    K3Smem &Sm = *reinterpret_cast<K3Smem *>(smem_raw);
    K3Shared &S = Sm.sh;
    const int t = threadIdx.x;
    int first = 0;
    for (int i0 = 0; i0 < n_inst; i0 += K3_THREADS) {
        // thread t looks at run i0 + t; only runs with deferred buckets follow,
        // whose buckets are dealt out to the blocks in one sequence (every
        // block sees the same counts; flags that rise meanwhile move nothing)
        const int n = i0 + t < n_inst ? insts[i0 + t].st->big_n : 0;
        int nwork, sum;
        __syncthreads();
        const int pos = block_excl_scan(n > 0, S.wsum, &nwork);
        __syncthreads();
        const int ex = block_excl_scan((int)((unsigned)n % gridDim.x), S.wsum, &sum);
        if (n > 0) {
            Sm.eflag[pos] = i0 + t;
            Sm.nacc[pos] = (int)((blockIdx.x + gridDim.x - (unsigned)(first + ex) % gridDim.x) % gridDim.x);
        }
        first = (int)((unsigned)(first + sum) % gridDim.x);
        __syncthreads();
        // the arrays are reused below: thread w keeps entry w
        const int mine = t < nwork ? Sm.eflag[t] : 0, mine_q = t < nwork ? Sm.nacc[t] : 0;
        for (int w = 0; w < nwork; w++) {
            __syncthreads();
            if (t == w) { S.n_new = mine; S.side_n = mine_q; }
            __syncthreads();
            annihilate_deferred(insts[S.n_new], Sm, S.side_n);
        }
    }
}

// ------------------------------------------------------------------ finalize
// one run's iteration committed by one block; insts, self: the table the run
// lies in (its replica partner is looked up there), NULL for a run alone
__device__ __forceinline__ void finalize_run(const DevInst &I, const DevInst *insts, int self)
{
    IterState *st = I.st;
    __shared__ int s_err;
    __shared__ double s_r[6][K5_THREADS / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int nbk = 1 << I.bb;
    const bool pair = insts && I.partner > self;  // the first replica reports the cross estimators
    const bool trial = I.trial_bits != 0;
    const bool tree = trial || pair;  // binary64 estimator sums need the whole block; otherwise warp 0 alone
    if (!tree && warp != 0) return;
    int e = 0;
    if (t == 0) {
        e = *(volatile int *)&st->err;
        // a replica commits its iteration only together with its partner: not
        // if the partner skipped it (a flag was up when its spawning began) or
        // failed in it
        const IterState *pst = insts && I.partner >= 0 ? insts[I.partner].st : nullptr;
        if (!e && pst && (*(volatile const int *)&pst->err_at_start ||
                          (*(volatile const int *)&pst->err & ERRB_STAGE))) {
            st->err = ERRB_PARTNER;
            e = ERRB_PARTNER;
        }
    }
    if (tree) {
        if (t == 0) s_err = e;
        __syncthreads();
        e = s_err;
    } else {
        e = __shfl_sync(0xffffffffu, e, 0);
    }
    if (e) return;
    // Binary64 sums of the estimators that have them (trial numerator and
    // denominator; replica-pair terms): every thread adds its buckets in order,
    // then a halving tree over the threads
    constexpr int NF = 6;  // words 0 .. 5 of a partial
    double dsum[NF];
#pragma unroll
    for (int f = 0; f < NF; f++) dsum[f] = 0.0;
    if (tree) {
        for (int u = t; u < nbk; u += K5_THREADS) {
            const double *p = reinterpret_cast<const double *>(I.part + u);
#pragma unroll
            for (int f = 0; f < NF; f++)
                if (f < 2 ? trial : pair) dsum[f] = dsum[f] + p[f];
        }
#pragma unroll
        for (int f = 0; f < NF; f++) {
            if (f < 2 ? !trial : !pair) continue;
            double v = dsum[f];
            for (int mm = 16; mm >= 1; mm >>= 1) v = v + __shfl_xor_sync(0xffffffffu, v, mm);
            if (lane == 0) s_r[f][warp] = v;
        }
        __syncthreads();
        if (warp == 0)
#pragma unroll
            for (int f = 0; f < NF; f++) {
                if (f < 2 ? !trial : !pair) continue;
                double v = lane < K5_THREADS / 32 ? s_r[f][lane] : 0.0;
                for (int mm = 16; mm >= 1; mm >>= 1) v = v + __shfl_xor_sync(0xffffffffu, v, mm);
                dsum[f] = v;
            }
    }
    if (warp != 0) return;
    // the shift state, loaded now so that its latency overlaps the totals'
    const long long it = st->iter, cnt0 = st->cnt, shift_start0 = st->shift_start, stop_iter = st->stop_iter;
    const long long semi_built = st->semi_built, trial_built = st->trial_built;
    const int vary0 = st->vary, par0 = st->parity;
    const double S0 = st->S, e_den = st->e_den;
    const u64 nwl_lo0 = st->nwl_lo, nwl_hi0 = st->nwl_hi;
    // the exact totals the buckets added up: lane k sums word k of the NSHARD
    // lines (each limb's total stays below 2^64) and clears it
    u64 v = 0;
    if (lane < NACC) {
        u64 x[NSHARD];
#pragma unroll
        for (int j = 0; j < NSHARD; j++) x[j] = I.acc[j * ACC_STRIDE + lane];
#pragma unroll
        for (int j = 0; j < NSHARD; j++) {
            I.acc[j * ACC_STRIDE + lane] = 0;
            v += x[j];
        }
    }
    u64 w[NACC];
#pragma unroll
    for (int k = 0; k < NACC; k++) w[k] = __shfl_sync(0xffffffffu, v, k);
    if (lane != 0) return;
    const u128 W = (u128)limb_total(w + ACC_NW);
    const i128 A = limb_total(w + ACC_ANN), EN = limb_total(w + ACC_ENUM);
    const long long nd = (long long)w[ACC_NDET], rj = (long long)w[ACC_REJ], sps = (long long)w[ACC_SPAWNS],
                    at = (long long)w[ACC_ATT];
    const double e_num = fixed_to_double(EN, I.Fe);
    const double t_num = trial ? dsum[0] : 0.0, t_den = trial ? dsum[1] : 0.0;
    const double x_ov = pair ? dsum[2] : 0.0, x_hd = pair ? dsum[3] : 0.0, x_cr = pair ? dsum[4] : 0.0;
    const double x_pt = pair ? dsum[5] : 0.0;
    const double nwd = u128_to_double(W) * 0x1p-32;
    // shift update (Booth, Thom, Alavi 2009)
    int vary = vary0;
    long long cnt = cnt0, shift_start = shift_start0;
    double S = S0;
    u64 nwl_lo = nwl_lo0, nwl_hi = nwl_hi0;
    if (!vary) {
        if (nwd >= I.target) {
            vary = 1;
            shift_start = it;
            nwl_lo = (u64)W; nwl_hi = (u64)(W >> 64);
            cnt = 0;
        }
    } else if (++cnt == I.A) {
        const u128 L = ((u128)nwl_hi << 64) | nwl_lo;
        const double ratio = nwd / (u128_to_double(L) * 0x1p-32);
        S = S - I.cz * fq_ln(ratio);
        nwl_lo = (u64)W; nwl_hi = (u64)(W >> 64);
        cnt = 0;
    }
    int flags = 0;
    if (!(S == S) || !(nwd == nwd)) flags |= ERRB_NUMERIC;
    fciqmc_iter_stats &R = I.ring[it & (long long)(I.ring_cap - 1)];  // ring_cap is a power of two
    R.iteration = it; R.nw = nwd; R.shift = S; R.e_num = e_num; R.e_den = e_den;
    R.ndet = nd; R.attempts = at; R.spawns = sps; R.rejected = rj;
    R.annihilated = i128_to_double(A) * 0x1p-32; R.vary = vary; R.pad0 = 0;
    R.trial_num = t_num; R.trial_den = t_den;
    R.x_overlap = x_ov;
    R.x_var_num = pair ? x_hd - x_cr / (2.0 * I.tau) : 0.0;
    R.x_pt2 = pair ? x_pt / (I.tau * I.tau) : 0.0;
    st->vary = vary; st->shift_start = shift_start; st->cnt = cnt; st->S = S;
    st->nwl_lo = nwl_lo; st->nwl_hi = nwl_hi;
    st->iter = it + 1;
    st->parity = par0 ^ 1;
    st->heavy_n = 0;
    st->big_n = 0;
    if (I.semi_size > 0 && !semi_built && vary && it + 1 == shift_start + I.semi_start) flags |= ERRB_PAUSE_SEMI;
    if (I.trial_size > 0 && !trial_built && vary && it + 1 == shift_start + I.trial_start) flags |= ERRB_PAUSE_TRIAL;
    if (it + 1 >= stop_iter) flags |= ERRB_STOP;
    if (flags) st->err |= flags;
}

__global__ void __launch_bounds__(K5_THREADS) k_finalize(const DevInst *__restrict__ insts, int n_inst)
{
    finalize_run(insts[blockIdx.x], insts, (int)blockIdx.x);
}

// the end of one run's iteration in one launch: its deferred buckets, if any,
// then the block that is done last commits it (a launch of their own for
// buckets that are hardly ever there cost 2 to 6 us of 37 to 83 us)
static_assert(K3_THREADS == K5_THREADS, "one block does both");
__global__ void __launch_bounds__(K3_THREADS) k_finish(const __grid_constant__ DevInst I)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int s_last;
    const int nbig = I.st->big_n;  // changed by the committing block alone
    if (nbig == 0) {
        if (blockIdx.x) return;
    } else {
        annihilate_deferred(I, *reinterpret_cast<K3Smem *>(smem_raw), (int)blockIdx.x);
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            s_last = atomicAdd(&I.st->done, 1) == (int)gridDim.x - 1;
        }
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        if (threadIdx.x == 0) I.st->done = 0;
    }
    finalize_run(I, nullptr, 0);
}

// ------------------------------------------------------------------ growth and import
// per-bucket list index of list `par` (adaptive shift), and zeroed weight sums
__global__ void k_build_kidx(const DevInst *__restrict__ Ip, int par, int nb)
{
    __shared__ unsigned short tab[KIDX];
    const DevInst &I = *Ip;
    for (int b = blockIdx.x; b < nb; b += gridDim.x) {
        for (int q = threadIdx.x; q < KIDX; q += blockDim.x) tab[q] = 0;
        __syncthreads();
        const int m = min(I.cnt[par][b], CAP_M);
        for (int e = threadIdx.x; e < m; e += blockDim.x) {
            const ulonglong2 k = I.key[par][(size_t)b * CAP_M + e];
            unsigned sl = (unsigned)det_hash(k.x, k.y) & (unsigned)(KIDX - 1);
            while (atomicCAS(&tab[sl], (unsigned short)0, (unsigned short)(e + 1)) != 0) sl = (sl + 1) & (unsigned)(KIDX - 1);
            u64 *acc = I.facc[par] + ((size_t)b * CAP_M + e) * 4;
            acc[0] = 0; acc[1] = 0; acc[2] = 0; acc[3] = 0;
        }
        __syncthreads();
        for (int q = threadIdx.x; q < KIDX; q += blockDim.x) I.kidx[par][(size_t)b * KIDX + q] = tab[q];
        __syncthreads();
    }
}

// split every bucket of src (bb bits) into two buckets of dst (bb+1 bits)
__global__ void k_rebucket(const DevInst *__restrict__ src, const DevInst *__restrict__ dst, int nb_src, int par)
{
    for (int b = blockIdx.x; b < nb_src; b += gridDim.x) {
        const int m = src->cnt[par][b];
        for (int e = threadIdx.x; e < m; e += blockDim.x) {
            size_t o = (size_t)b * CAP_M + e;
            ulonglong2 k = src->key[par][o];
            int nbk = bucket_of(det_hash(k.x, k.y), dst->bb);
            int slot = atomicAdd(dst->cnt[par] + nbk, 1);
            if (slot >= CAP_M) { atomicOr(&dst->st->err, ERRB_MAIN_CAP); continue; }
            size_t d = (size_t)nbk * CAP_M + slot;
            dst->key[par][d] = k;
            dst->c[par][d] = src->c[par][o];
            dst->hd[par][d] = src->hd[par][o];
            dst->fl[par][d] = src->fl[par][o];
        }
    }
}

// H_ii - E_ref and reference flags for every determinant of buffer par
__global__ void k_diag(const DevInst *__restrict__ I, int par, int nb)
{
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int b = gw; b < nb; b += nw) {
        const int m = I->cnt[par][b];
        for (int e = 0; e < m; e++) {
            size_t o = (size_t)b * CAP_M + e;
            ulonglong2 k = I->key[par][o];
            double hdv = diag_exact_warp(*I, k.x, k.y);
            if (lane == 0) {
                I->hd[par][o] = hdv;
                uint8_t f = I->fl[par][o] & DFLAG_D;
                if (k.x == I->ref_a && k.y == I->ref_b) f |= DFLAG_REF;
                I->fl[par][o] = f;
            }
        }
    }
}

// ------------------------------------------------------------------ time-step bound
// sum_j |<D_j|H|D_ref>| over every single and double excitation of the
// reference; fixed grid, fixed per-thread order and fixed reduction tree, so
// the result is deterministic.
constexpr int REFSUM_BLOCKS = 64;
__global__ void __launch_bounds__(256) k_ref_abs_sum(const DevInst *__restrict__ Ip, double *partial)
{
    const DevInst &I = *Ip;
    const u64 ra = I.ref_a, rb = I.ref_b, va = ~ra & I.normask, vb = ~rb & I.normask;
    const long long na = I.na, nb = I.nb, ma = I.ma, mb = I.mb;
    const long long s1 = na * ma, s2 = nb * mb, s3 = na * nb * ma * mb, s4 = na * na * ma * ma, s5 = nb * nb * mb * mb;
    const long long total = s1 + s2 + s3 + s4 + s5;
    double acc = 0.0;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        long long q = idx;
        u64 ta = ra, tb = rb;
        if (q < s1) {
            ta ^= (1ULL << nth_set(ra, (int)(q / ma))) | (1ULL << nth_set(va, (int)(q % ma)));
        } else if ((q -= s1) < s2) {
            tb ^= (1ULL << nth_set(rb, (int)(q / mb))) | (1ULL << nth_set(vb, (int)(q % mb)));
        } else if ((q -= s2) < s3) {
            const int b = (int)(q % mb); q /= mb;
            const int a = (int)(q % ma); q /= ma;
            const int j = (int)(q % nb), i = (int)(q / nb);
            ta ^= (1ULL << nth_set(ra, i)) | (1ULL << nth_set(va, a));
            tb ^= (1ULL << nth_set(rb, j)) | (1ULL << nth_set(vb, b));
        } else if ((q -= s3) < s4) {
            const int b = (int)(q % ma); q /= ma;
            const int a = (int)(q % ma); q /= ma;
            const int j = (int)(q % na), i = (int)(q / na);
            if (!(i < j && a < b)) continue;
            ta ^= (1ULL << nth_set(ra, i)) | (1ULL << nth_set(ra, j)) | (1ULL << nth_set(va, a)) | (1ULL << nth_set(va, b));
        } else {
            q -= s4;
            const int b = (int)(q % mb); q /= mb;
            const int a = (int)(q % mb); q /= mb;
            const int j = (int)(q % nb), i = (int)(q / nb);
            if (!(i < j && a < b)) continue;
            tb ^= (1ULL << nth_set(rb, i)) | (1ULL << nth_set(rb, j)) | (1ULL << nth_set(vb, a)) | (1ULL << nth_set(vb, b));
        }
        acc = acc + fabs(hoff_generic(I, ra, rb, ta, tb));
    }
    __shared__ double sm[8];
    for (int m = 16; m >= 1; m >>= 1) acc = acc + __shfl_xor_sync(0xffffffffu, acc, m);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < 8; k++) s = s + sm[k];
        partial[blockIdx.x] = s;
    }
}

cudaError_t ref_abs_sum(const DevInst *dinst, double *dpartial, double *out, cudaStream_t s)
{
    k_ref_abs_sum<<<REFSUM_BLOCKS, 256, 0, s>>>(dinst, dpartial);
    double hp[REFSUM_BLOCKS];
    cudaError_t e = cudaMemcpyAsync(hp, dpartial, sizeof(hp), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    double acc = 0.0;
    for (int k = 0; k < REFSUM_BLOCKS; k++) acc = acc + hp[k];
    *out = acc;
    return cudaSuccess;
}

// ------------------------------------------------------------------ launchers
static int g_num_sms = 0;
static int num_sms()
{
    if (!g_num_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_num_sms <= 0) g_num_sms = 1;
    }
    return g_num_sms;
}

void launch_build_kidx(const DevInst *dinst, int parity, int nb, cudaStream_t s)
{
    int grid = nb < num_sms() * 8 ? nb : num_sms() * 8;
    k_build_kidx<<<grid, 256, 0, s>>>(dinst, parity, nb);
}

// launch geometry, chosen by fciqmc_autotune (grid blocks per SM; beyond the
// resident count, 4 per SM for the spawning kernel and 3 for the annihilation,
// the hardware hands the next block to whichever slot frees first, which evens
// out buckets of unequal size)
// g_spawn_bps = 0 and 1 and g_anni_bps = 0 select one resident wave of blocks
static int g_spawn_bps = 1, g_heavy_bps = 2, g_anni_bps = 0;
static int g_geometry_gen = 0;  // changes with every set_launch_geometry
int launch_geometry_generation() { return g_geometry_gen; }
void set_launch_geometry(int spawn_bps, int heavy_bps, int anni_bps)
{
    g_geometry_gen++;
    g_spawn_bps = spawn_bps;
    g_heavy_bps = heavy_bps;
    g_anni_bps = anni_bps;
}
void get_launch_geometry(int *spawn_bps, int *heavy_bps, int *anni_bps)
{
    *spawn_bps = g_spawn_bps;
    *heavy_bps = g_heavy_bps;
    *anni_bps = g_anni_bps;
}

// How a list's buckets are dealt to warps: as many warps per bucket as it
// takes to reach every resident warp of the GPU, and the number of attempts
// above which a determinant goes to the heavy queue (a warp draws its
// attempts 32 at a time, one after the other).  On a short list, where one
// determinant's windows are the launch's longest chain, that is 64: a 4x4
// lattice at 1e5 walkers takes 2.38 ms per 40 iterations, 2.64 with 512 (the
// 8-site ring at 1e4, 20 iterations: 0.907 and 0.888).  On a long list it is
// half a slice: a batch of eight served requests takes 362 ms, 374 with 512;
// 64 lattice runs and 50 orbitals at 1e7 walkers are the same with 64, 256 and
// 512 within 1 %.
struct SpawnSplit {
    int parts, grid;
    unsigned heavy_min;
};
static SpawnSplit spawn_split(int n_units, int bps)
{
    SpawnSplit p;
    const int warps = num_sms() * 4 * SP_WARPS;
    p.parts = 1;
    while (p.parts < CAP_M / 32 && (long long)n_units * p.parts < 2 * warps) p.parts *= 2;
    p.heavy_min = p.parts > 1 ? 64 : HEAVY_ATT / 2;
    const long long need = ((long long)n_units * p.parts + SP_WARPS - 1) / SP_WARPS;
    p.grid = (int)(need < (long long)num_sms() * bps ? need : (long long)num_sms() * bps);
    return p;
}

static int spawn_blocks(int spawn_bps, bool adaptive) { return spawn_bps > 1 ? spawn_bps : (adaptive ? 3 : 4); }
static int anni_grid(int n_units, int anni_bps)
{
    const int need = (n_units + AN_WARPS - 1) / AN_WARPS, full = num_sms() * (anni_bps > 0 ? anni_bps : 3);
    return need < full ? need : full;
}

// the grids a launch configuration gives a batch of n_units buckets (for
// fciqmc_autotune: configurations of the same grid are the same launch)
void batch_grids(int n_units, bool adaptive, int spawn_bps, int anni_bps, int *spawn, int *anni)
{
    *spawn = spawn_split(n_units, spawn_blocks(spawn_bps, adaptive)).grid;
    *anni = anni_grid(n_units, anni_bps);
}

// whether the last units of a launch are claimed (with the adaptive shift and
// with replica lists, whose kernels have no registers to spare, never)
static bool claims(int n, int nw) { return n / nw >= CLAIM_ROUNDS; }

// spawning of one run (`one`, the host image of its descriptor) or of a table
// of runs (one = NULL); adaptive: some run uses the adaptive shift
template <int GEN>
static void launch_spawn_one(const DevInst *one, int grid, int n_units, int parts, unsigned heavy_min, cudaStream_t s)
{
    const bool claim = claims(n_units * parts, grid * SP_WARPS);
    if (one->adaptive) k_spawn<GEN, true, false><<<grid, SP_THREADS, SP_SMEM_ADAPT, s>>>(*one, n_units, parts, heavy_min);
    else if (claim) k_spawn<GEN, false, true><<<grid, SP_THREADS, SP_SMEM, s>>>(*one, n_units, parts, heavy_min);
    else k_spawn<GEN, false, false><<<grid, SP_THREADS, SP_SMEM, s>>>(*one, n_units, parts, heavy_min);
}
void launch_spawn(const DevInst *one, const DevInst *dinst, const int *unit_start, int n_inst, int n_units, bool adaptive,
                  cudaStream_t s)
{
    const SpawnSplit p = spawn_split(n_units, spawn_blocks(g_spawn_bps, adaptive));
    const int grid = p.grid, parts = p.parts;
    const unsigned heavy_min = p.heavy_min;
    if (one && one->kind == FCIQMC_HUBBARD) launch_spawn_one<GEN_HOP>(one, grid, n_units, parts, heavy_min, s);
    else if (one && one->pchb) launch_spawn_one<GEN_PCHB>(one, grid, n_units, parts, heavy_min, s);
    else if (one) launch_spawn_one<GEN_UNIFORM>(one, grid, n_units, parts, heavy_min, s);
    else if (adaptive) k_spawn_batch<true, false><<<grid, SP_THREADS, SP_SMEM_ADAPT, s>>>(dinst, unit_start, n_inst, n_units, parts, heavy_min);
    else if (claims(n_units * parts, grid * SP_WARPS)) k_spawn_batch<false, true><<<grid, SP_THREADS, SP_SMEM, s>>>(dinst, unit_start, n_inst, n_units, parts, heavy_min);
    else k_spawn_batch<false, false><<<grid, SP_THREADS, SP_SMEM, s>>>(dinst, unit_start, n_inst, n_units, parts, heavy_min);
}

void launch_spawn_heavy(const DevInst *one, const DevInst *dinst, int n_inst, cudaStream_t s)
{
    const int grid = num_sms() * g_heavy_bps;
    if (one) k_spawn_heavy<<<grid, SP_THREADS, SP_SMEM_ADAPT, s>>>(*one);
    else k_spawn_heavy_batch<<<grid, SP_THREADS, SP_SMEM_ADAPT, s>>>(dinst, n_inst);
}

__global__ void k_diag_list_long(const __grid_constant__ DevInst I, int par, const unsigned *list, int nn);
cudaError_t init_kernels()
{
    cudaError_t e = cudaFuncSetAttribute(k_annihilate_big, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(K3Smem));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(K3Smem));
    if (e == cudaSuccess)  // 64 orbitals at most
        e = cudaFuncSetAttribute(k_diag_list_long, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)((2 * 64 * 64 + 64) * sizeof(ulonglong2)));
    auto warp_smem = [&](auto *f, size_t bytes, int blocks) {  // the resident blocks need their shared memory at once
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)((blocks * (bytes + 1024) * 100 + 233471) / 233472));
    };
    warp_smem(k_spawn<GEN_UNIFORM, false, false>, SP_SMEM, 4);
    warp_smem(k_spawn<GEN_UNIFORM, false, true>, SP_SMEM, 4);
    warp_smem(k_spawn<GEN_PCHB, false, false>, SP_SMEM, 4);
    warp_smem(k_spawn<GEN_PCHB, false, true>, SP_SMEM, 4);
    warp_smem(k_spawn<GEN_HOP, false, false>, SP_SMEM, 4);
    warp_smem(k_spawn<GEN_HOP, false, true>, SP_SMEM, 4);
    warp_smem(k_spawn_batch<false, false>, SP_SMEM, 4);
    warp_smem(k_spawn_batch<false, true>, SP_SMEM, 4);
    warp_smem(k_spawn<GEN_UNIFORM, true, false>, SP_SMEM_ADAPT, 3);
    warp_smem(k_spawn<GEN_PCHB, true, false>, SP_SMEM_ADAPT, 3);
    warp_smem(k_spawn<GEN_HOP, true, false>, SP_SMEM_ADAPT, 3);
    warp_smem(k_spawn_batch<true, false>, SP_SMEM_ADAPT, 3);
    warp_smem(k_spawn_heavy, SP_SMEM_ADAPT, 3);
    warp_smem(k_spawn_heavy_batch, SP_SMEM_ADAPT, 3);
    warp_smem(k_annihilate<false, false>, AN_SMEM, 3);
    warp_smem(k_annihilate<false, true>, AN_SMEM, 3);
    warp_smem(k_annihilate_batch<false, false>, AN_SMEM, 3);
    warp_smem(k_annihilate_batch<false, true>, AN_SMEM, 3);
    warp_smem(k_annihilate<true, false>, AN_SMEM, 3);
    warp_smem(k_annihilate_batch<true, false>, AN_SMEM, 3);
    return e;
}

// annihilation of one run (`one`) or of a table of runs; extra: some run has
// replica side lists or the adaptive shift.  g_anni_bps = 0: one resident
// wave of blocks, else that many blocks per SM
cudaError_t launch_annihilate(const DevInst *one, const DevInst *dinst, const int *unit_start, int n_inst, int n_units,
                              bool extra, cudaStream_t s)
{
    const int grid = anni_grid(n_units, g_anni_bps);
    const bool claim = claims(n_units, grid * AN_WARPS);
    if (one && extra) k_annihilate<true, false><<<grid, AN_THREADS, AN_SMEM, s>>>(*one, n_units);
    else if (one && claim) k_annihilate<false, true><<<grid, AN_THREADS, AN_SMEM, s>>>(*one, n_units);
    else if (one) k_annihilate<false, false><<<grid, AN_THREADS, AN_SMEM, s>>>(*one, n_units);
    else if (extra) k_annihilate_batch<true, false><<<grid, AN_THREADS, AN_SMEM, s>>>(dinst, unit_start, n_inst, n_units);
    else if (claim) k_annihilate_batch<false, true><<<grid, AN_THREADS, AN_SMEM, s>>>(dinst, unit_start, n_inst, n_units);
    else k_annihilate_batch<false, false><<<grid, AN_THREADS, AN_SMEM, s>>>(dinst, unit_start, n_inst, n_units);
    return cudaGetLastError();
}

// the buckets beyond a warp's records; every block takes those that fit
// shared memory, the first BIG_BLOCKS the others
void launch_annihilate_big(const DevInst *dinst, int n_inst, cudaStream_t s)
{
    k_annihilate_big<<<num_sms() * 3 > BIG_BLOCKS ? num_sms() * 3 : BIG_BLOCKS, K3_THREADS, sizeof(K3Smem), s>>>(dinst, n_inst);
}

// the deferred buckets of one run and its commit
void launch_finish(const DevInst *one, cudaStream_t s)
{
    k_finish<<<num_sms() * 3 > BIG_BLOCKS ? num_sms() * 3 : BIG_BLOCKS, K3_THREADS, sizeof(K3Smem), s>>>(*one);
}

void launch_finalize(const DevInst *dinst, int n_inst, cudaStream_t s)
{
    k_finalize<<<n_inst, K5_THREADS, 0, s>>>(dinst, n_inst);
}

// H_ii - E_ref of every determinant of list `par`, given by its slots (import)
__global__ void __launch_bounds__(256) k_diag_list(const __grid_constant__ DevInst I, int par, const unsigned *list, int nn)
{
    __shared__ unsigned short s_pair[ND_PAIRS];
    __shared__ unsigned char s_orb[8][4][ND_MAX];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nwarp = (int)((gridDim.x * blockDim.x) >> 5);
    if (I.n > ND_MAX) {  // beyond the table: the generic warp sum
        for (int q = 2 * gw; q < nn; q += 2 * nwarp) {
            const unsigned d0 = list[q], d1 = q + 1 < nn ? list[q + 1] : d0;
            const ulonglong2 k0 = I.key[par][d0], k1 = I.key[par][d1];
            const u64 ka[2] = {k0.x, k1.x}, kb[2] = {k0.y, k1.y};
            double hdv[2];
            diag_exact_warp_multi<2>(I, ka, kb, hdv);
            if (lane == 0) {
                I.hd[par][d0] = hdv[0];
                if (q + 1 < nn) I.hd[par][d1] = hdv[1];
            }
        }
        return;
    }
    fill_pairs(s_pair);
    for (int q = 4 * gw; q < nn; q += 4 * nwarp) diag_four(I, list + q, min(4, nn - q), par, s_pair, s_orb[wl]);
}

// the same for a long list: one determinant per lane, the tables in shared
// memory.  A sum is n (n + 1) / 2 16-byte loads at scattered places; from
// global memory every lane's load is an L1 line of its own (1.47 ms for 3e6
// determinants of 20 electrons, 1.16 ms with one determinant per lane)
constexpr int DL_THREADS = 1024;
__global__ void __launch_bounds__(DL_THREADS, 1) k_diag_list_long(const __grid_constant__ DevInst I, int par,
                                                                  const unsigned *list, int nn)
{
    extern __shared__ ulonglong2 dl_tab[];
    const int N = I.norb, N2 = N * N;
    ulonglong2 *JK = dl_tab, *J = dl_tab + N2, *hp = dl_tab + 2 * N2;
    for (int q = threadIdx.x; q < N2; q += DL_THREADS) {
        JK[q] = __ldg(I.JKfx + q);
        J[q] = __ldg(I.Jfx + q);
        if (q < N) hp[q] = __ldg(I.hfx + q);
    }
    __syncthreads();
    const i128 xref = (i128)(((u128)I.xref_hi << 64) | (u128)I.xref_lo);
    auto at = [](const ulonglong2 &v) { return (i128)(((u128)v.y << 64) | (u128)v.x); };
    for (long long i = (long long)blockIdx.x * DL_THREADS + threadIdx.x; i < nn; i += (long long)gridDim.x * DL_THREADS) {
        const unsigned d = list[i];
        const ulonglong2 kk = I.key[par][d];
        i128 x = -xref;
        for (int s = 0; s < 2; s++) {
            u64 w = s ? kk.y : kk.x;
            while (w) {
                const int p = __ffsll((long long)w) - 1;
                w &= w - 1;
                x += at(hp[p]);
                for (u64 o = w; o; o &= o - 1) x += at(JK[p * N + __ffsll((long long)o) - 1]);
                if (!s)
                    for (u64 o = kk.y; o; o &= o - 1) x += at(J[p * N + __ffsll((long long)o) - 1]);
            }
        }
        I.hd[par][d] = fixed_to_double(x, I.F);
    }
}

// ------------------------------------------------------------------ integral tables
// The fixed-point tables of a run (h_pp, (pp|qq), (pp|qq) - (pq|qp), and per
// (a, i, k) the pair (ai|kk), (ai|kk) - (ak|ki)) from its integrals, one entry
// per thread; every integral lies on the grid 2^-F (the host checked).  On the
// host the 2 N^3 + 2 N^2 conversions of 50 orbitals took 7 of the 13 ms that
// creating a run takes.
__global__ void __launch_bounds__(256) k_tables(int N, int F, const double *__restrict__ h, const double *__restrict__ eri,
                                                ulonglong2 *hfx, ulonglong2 *J, ulonglong2 *JK, ulonglong2 *S)
{
    auto fixed = [&](const double *p) { return to_fixed(__ldg(p), F); };
    auto put = [](ulonglong2 *d, i128 v) { *d = make_ulonglong2((u64)(u128)v, (u64)((u128)v >> 64)); };
    const long long n3 = (long long)N * N * N;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n3; q += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(q % N), i = (int)(q / N % N), a = (int)(q / N / N);
        const i128 c = fixed(eri + pidx(pidx(a, i), pidx(k, k))), x = fixed(eri + pidx(pidx(a, k), pidx(k, i)));
        put(S + 2 * q, c);
        put(S + 2 * q + 1, c - x);
        if (a == i) {
            put(J + a * N + k, c);        // (aa|kk)
            put(JK + a * N + k, c - x);   // (aa|kk) - (ak|ka)
            if (k == 0) put(hfx + a, fixed(h + a * N + a));
        }
    }
}

cudaError_t launch_tables(int N, int F, const double *h, const double *eri, ulonglong2 *hfx, ulonglong2 *J, ulonglong2 *JK,
                          ulonglong2 *S, cudaStream_t s)
{
    const int blocks = (N * N * N + 255) / 256;
    k_tables<<<blocks < num_sms() * 8 ? blocks : num_sms() * 8, 256, 0, s>>>(N, F, h, eri, hfx, J, JK, S);
    return cudaGetLastError();
}

void launch_diag_list(const DevInst *one, int par, const unsigned *list, int nn, cudaStream_t s)
{
    // the line: a determinant for every thread of the long list's kernel (one
    // block per SM, which first copies the tables)
    const size_t smem = (size_t)(2 * one->norb * one->norb + one->norb) * sizeof(ulonglong2);
    if (nn >= num_sms() * DL_THREADS) k_diag_list_long<<<num_sms(), DL_THREADS, smem, s>>>(*one, par, list, nn);
    else if (nn > 0) k_diag_list<<<num_sms() * 4, 256, 0, s>>>(*one, par, list, nn);
}

void launch_rebucket(const DevInst *src, const DevInst *dst, int nb_src, int parity, cudaStream_t s)
{
    int grid = nb_src < num_sms() * 8 ? nb_src : num_sms() * 8;
    k_rebucket<<<grid, 256, 0, s>>>(src, dst, nb_src, parity);
}

void launch_diag(const DevInst *dinst, int parity, int nb, cudaStream_t s)
{
    int warps = nb;
    int blocks = (warps * 32 + 255) / 256;
    if (blocks > num_sms() * 16) blocks = num_sms() * 16;
    if (blocks < 1) blocks = 1;
    k_diag<<<blocks, 256, 0, s>>>(dinst, parity, nb);
}

u64 det_hash_host(u64 a, u64 b) { return det_hash(a, b); }

}  // namespace fq
