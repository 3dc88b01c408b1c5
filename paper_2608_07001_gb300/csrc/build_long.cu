// build_long.cu -- the prototype trees of units whose slot is longer than the
// 128 tokens the unit kernel (build.cu) keeps in shared memory: supplied
// partitions may hold slots of thousands of tokens (App. A.2 atomic units are
// whatever slots the partition gives; the trees still recurse to single-token
// leaves, App. A.3 "Recursive refinement rule").
//
// The arithmetic is the unit kernel's, node by node: for a node I = [a, b) the
// binary cuts X_v (top-K positions by curvature in [a, b-2], cut xi = t + 1,
// plus the midpoint a + floor(n/2); App. B.4 Eq. app_tree_split_candidates),
// the salient-token extraction at p* = argmax R_tok (or the singleton-floor
// position of largest score, forced), candidate intervals that are prefixes
// [a, xi) and suffixes [xi, b) of I, RoPE-consistent prototypes (Eqs.
// app_rope_prototype, app_value_prototype, app_effective_multiplicity), the
// probe statistics Z_u, M_u of every candidate from one forward and one
// backward scan over the node (Eq. app_original_attention_stats), D_u and the
// mass-weighted D (Eqs. app_probe_distortion, app_node_and_drop_distortion),
// the refinement decision (Eqs. app_binary_split .. app_split_choice), gains,
// costs, utilities clamped at 0 and bottleneck keys (Eqs.
// app_operation_gains .. app_unit_utility), with the same node records, op
// list and pending-node key bounds, so the allocation, the pruning passes and
// the gather treat both kinds of unit alike.
//
// What differs is the work split.  The tree of a long unit is built one level
// per launch sequence, across CTAs:
//   long_collect  (CTA per listed unit) the nodes to evaluate -- a fresh root,
//                 or the pending nodes whose key bound reaches tau -- as one
//                 contiguous, ordered block of work items per unit;
//   long_eval     (CTA per work item, taken from a counter) one node: cut
//                 candidates, per-segment sums between the candidate boundaries
//                 (at most 20 segments; each candidate's prototype sums are the
//                 sum of its segments), the probe scans reading V and the probe
//                 weights through a staging ring, the decision.  Only the cut of
//                 largest curvature reward is evaluated at first; a cut whose
//                 exact bound is below it is never evaluated (build.cu);
//   long_commit   (warp per unit) children numbered in work-item order after
//                 the unit's existing nodes (deterministic), records, Split ops,
//                 pending bounds.
// The probe scans fold their fp32 running sums every 32 tokens (and at every
// candidate end) into a second fp32 sum, so that sums over thousands of
// tokens keep the rounding of short ones.
#include "gkv_internal.cuh"

#include <algorithm>
#include <cfloat>

#include <type_traits>

namespace gkv {
namespace {

constexpr int kLT = 256;          // threads per CTA
constexpr int kLPP = 32;          // probe pairs: thread handles probes p and p + 32 (W <= 64)
constexpr int kLCL = 8;           // threads per probe pair (4-element groups, interleaved)
constexpr int kLPPW = 32 / kLCL;  // probe pairs per warp
constexpr int kLNW = kLT / 32;    // warps
constexpr int kLNCD = 20;         // candidate rows per direction (17 cuts + p* side + whole node)
constexpr int kLMaxK = 16;        // largest K
constexpr int kLMaxCut = 18;      // K + midpoint (+1 spare)
constexpr int kLMaxSeg = 24;      // segments between the boundaries a, b, the cuts, p*, p* + 1
constexpr int kLFold = 32;        // tokens per fp32 partial sum of a scan
constexpr int kLChunk = 32;       // tokens per staged chunk of a scan
constexpr int kLU = 4;            // tokens loaded at a time by the segment sums (divides kLFold)

struct LongRes {
    int nch;               // -1: pending (root only), 0: leaf (non-finite inputs), 2 or 3
    int ca[3], cb[3];      // children, absolute positions
    float cD[3], rch[3];   // their distortion and value
    float bnd[3];          // key bound of a child left pending (n >= 2)
    float U, kap;          // the node's split utility and bottleneck key
    float bound;           // pending root: the bound of its split key
};

struct LongArgs {
    const void *K, *V, *Q;
    const int32_t *slots;
    const float2 *rope;
    const double *kappa;
    const float *rtok, *row_m, *row_Z, *omega;
    const float2 *Eg;              // nullable: [L G][N_c][32] probe weights (u, u + 32) of every token
    const uint8_t *fl_acc;         // nullable: [L G][N_c] accepted singleton-floor positions
    const float *fl_f;             //           and their floor scores
    int L, G, Hq, T, d, W, gq, cs, Nc, J, k_cand;
    float inv_sqrt_d, lamZ, lamM, eps, lam_kappa, base_frac;
    int fresh;                     // 1: the roots of the listed slots; 0: pending nodes of listed units
    int root_only;                 // fresh: only the root's own distortion (its split stays pending)
    int prune;                     // lambda_Z, lambda_M >= 0, so every D >= 0: cuts and nodes may be ruled out by bounds
    float tau;                     // resume: evaluate pending nodes whose key bound >= tau
    const int32_t *list;           // fresh: slot indices; resume: unit ids
    int n_list, lg0, nlg;          // fresh units: slot list x (l, g) in [lg0, lg0 + nlg)
    // work items of the level
    int64_t *it_gv, *it_uid;
    float *it_kin;                 // bottleneck key of the op that created the node
    uint8_t *it_ufl;               // the node's unit holds a singleton-floor position
    LongRes *res;
    int32_t *u_start, *u_cnt;      // per listed unit: its block of work items
    unsigned int *n_items;         // [4]: work items, small subtrees of each class
    unsigned int *it_next;         // the next work item to take (zero at the level's start)
    int32_t *sub;                  // [kUnitClasses][cap_items] small subtrees' roots (global node indices)
    int64_t cap_items;
    // node records and unit arrays (build.cu's layout)
    int32_t *nd_a, *nd_b, *nd_child0, *nd_parent, *nd_unit;
    int8_t *nd_nchild, *nd_cost;
    float *nd_D, *nd_R, *nd_U, *nd_kappa;
    uint8_t *nd_sel;
    uint2 *ops;
    unsigned int *n_ops;
    int32_t *u_nnodes;
    float *u_Uadd, *u_Ddrop, *u_pend;
    uint8_t *u_sel;
    int *status;
    unsigned long long *work;
};

// Upper bound of a split's utility (see build.cu: U <= omega R D where both factors are >= 0, rounded up).
__device__ __forceinline__ float lkey_bound(float x) { return x + fabsf(x) * 1e-5f; }

__device__ __forceinline__ unsigned long long lokey(double x) {
    unsigned long long u = (unsigned long long)__double_as_longlong(x);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double lokey_inv(unsigned long long k) {
    unsigned long long u = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)u);
}

__device__ __forceinline__ int lround_half_even_mid(int a, int b) {
    int s = a + b - 1;
    if ((s & 1) == 0) return s >> 1;
    int lo = (s - 1) >> 1;
    return (lo & 1) == 0 ? lo : lo + 1;
}

__device__ __forceinline__ float4 lld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 lld4(const __nv_bfloat16 *p) {
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
// N consecutive elements of a row, held raw until they are used (one load for N = 2).
template <typename T, int N> struct LRaw;
template <int N> struct LRaw<float, N> {
    float v[N];
    __device__ __forceinline__ void load(const float *p) {
        if constexpr (N == 2) {
            const float2 x = *reinterpret_cast<const float2 *>(p);
            v[0] = x.x; v[1] = x.y;
        } else {
            v[0] = p[0];
        }
    }
    __device__ __forceinline__ float get(int j) const { return v[j]; }
};
template <int N> struct LRaw<__nv_bfloat16, N> {
    uint32_t u;
    __device__ __forceinline__ void load(const __nv_bfloat16 *p) {
        if constexpr (N == 2) u = *reinterpret_cast<const uint32_t *>(p);
        else u = *reinterpret_cast<const uint16_t *>(p);
    }
    __device__ __forceinline__ float get(int j) const {   // bf16 -> fp32 is exact: the bits move to the high half
        return __uint_as_float(j ? u & 0xFFFF0000u : u << 16);
    }
};

// Block-wide sum of a float (fixed order: lanes, then warps ascending).
__device__ __forceinline__ float block_sum(float v, float *sf) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_sum(v);
    if (lane == 0) sf[warp] = v;
    __syncthreads();
    float s = 0.f;
    for (int w = 0; w < kLNW; w++) s += sf[w];
    __syncthreads();
    return s;
}

// ---------------------------------------------------------------------------
// long_collect: the level's work items of one listed unit (CTA per unit)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void unit_of(const LongArgs &A, int i, int64_t &uid, int &lg, int &j) {
    if (A.fresh) {
        j = A.list[i / A.nlg];
        lg = A.lg0 + i % A.nlg;
        uid = (int64_t)lg * A.J + j;
    } else {
        uid = A.list[i];
        lg = (int)(uid / A.J);
        j = (int)(uid - (int64_t)lg * A.J);
    }
}

__global__ void __launch_bounds__(kLT) long_collect_kernel(LongArgs A) {
    __shared__ float sf[kLNW];
    __shared__ int wcnt[kLNW];
    __shared__ int base_s;
    const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t uid;
    int lg, j;
    unit_of(A, i, uid, lg, j);
    const int sa = A.slots[j], sb = A.slots[j + 1], n = sb - sa;
    const int64_t nbase = node_base(lg, sa, A.cs, A.Nc);
    const size_t rbase = (size_t)lg * A.Nc + (sa - A.cs);
    // does the slot hold an accepted singleton-floor position (its Add is then a floor op)
    int ufl = 0;
    if (A.fl_acc) {
        int any = 0;
        for (int t = tid; t < n; t += kLT) any |= A.fl_acc[rbase + t];
        ufl = __syncthreads_or(any);
    }
    if (A.fresh) {
        float r = 0.f;
        for (int t = tid; t < n; t += kLT) r += A.rtok[rbase + t];
        const float rootR = block_sum(r, sf);
        for (int k = tid; k < 2 * n; k += kLT) A.nd_cost[nbase + k] = 0;   // unused slots carry no op
        if (tid == 0) {
            const unsigned int pos = atomicAdd(&A.n_items[0], 1u);
            if ((int64_t)pos < A.cap_items) {
                A.it_gv[pos] = nbase;
                A.it_uid[pos] = uid;
                A.it_kin[pos] = 0.f;   // a fresh root's creator is its Add, formed by long_eval
                A.it_ufl[pos] = (uint8_t)ufl;
                A.u_start[i] = (int32_t)pos;
                A.u_cnt[i] = 1;
            } else {
                atomicOr(A.status, 64);
                A.u_start[i] = 0;
                A.u_cnt[i] = 0;
            }
            A.nd_a[nbase] = sa; A.nd_b[nbase] = sb; A.nd_R[nbase] = rootR; A.nd_D[nbase] = 0.f;
            A.nd_parent[nbase] = (int32_t)(-2 - uid); A.nd_unit[nbase] = (int32_t)uid;
            A.nd_child0[nbase] = -1; A.nd_nchild[nbase] = 0; A.nd_U[nbase] = 0.f;
            A.nd_kappa[nbase] = 0.f; A.nd_sel[nbase] = 0;
            A.u_nnodes[uid] = 1; A.u_pend[uid] = -1.f; A.u_sel[uid] = 0;
            A.u_Uadd[uid] = 0.f; A.u_Ddrop[uid] = 0.f;
        }
        return;
    }
    // resume: pending nodes (child count -1) whose key bound reaches tau, in
    // node order; the others keep the unit's largest pending bound
    const int nn = A.u_nnodes[uid];
    int cnt = 0;
    float pend = -1.f;
    for (int k = tid; k < nn; k += kLT) {
        const int64_t v = nbase + k;
        if (A.nd_nchild[v] != -1) continue;
        const float bnd = A.nd_U[v];
        if (bnd < A.tau) { pend = fmaxf(pend, bnd); continue; }
        const int len = A.nd_b[v] - A.nd_a[v];
        if (len > kMaxUnit) { cnt++; continue; }
        // a small node: its subtree goes to the unit kernel (subtree mode), into
        // the slots reserved for it.  A node the unit kernel left pending inside
        // a subtree has none, but its bound is below a threshold that only
        // rises, so it never reaches this point; it is skipped all the same.
        if (A.nd_child0[v] < 0) continue;
        const int cls = unit_class(len);
        const unsigned int pos = atomicAdd(&A.n_items[1 + cls], 1u);
        if ((int64_t)pos < A.cap_items) A.sub[(size_t)cls * A.cap_items + pos] = (int32_t)v;
        else atomicOr(A.status, 64);
    }
    pend = warp_max(pend);
    if (lane == 0) sf[warp] = pend;
    cnt = (int)block_sum((float)cnt, reinterpret_cast<float *>(wcnt));   // counts are far below 2^24
    if (tid == 0) {
        float pm = -1.f;
        for (int w = 0; w < kLNW; w++) pm = fmaxf(pm, sf[w]);
        A.u_pend[uid] = pm;
        int b0 = 0;
        if (cnt > 0) {
            const unsigned int pos = atomicAdd(&A.n_items[0], (unsigned)cnt);
            if ((int64_t)pos + cnt <= A.cap_items) {
                b0 = (int)pos;
            } else {
                atomicOr(A.status, 64);
                cnt = 0;
            }
        }
        A.u_start[i] = b0;
        A.u_cnt[i] = cnt;
        base_s = cnt > 0 ? b0 : -1;
    }
    __syncthreads();
    if (base_s < 0) return;
    // ordered compaction, 256 nodes at a time
    int out = base_s;
    for (int k0 = 0; k0 < nn; k0 += kLT) {
        const int k = k0 + tid;
        bool q = false;
        if (k < nn && A.nd_nchild[nbase + k] == -1)
            q = A.nd_U[nbase + k] >= A.tau && A.nd_b[nbase + k] - A.nd_a[nbase + k] > kMaxUnit;
        const unsigned bal = __ballot_sync(0xffffffffu, q);
        if (lane == 0) wcnt[warp] = __popc(bal);
        __syncthreads();
        int before = 0, tot = 0;
        for (int w = 0; w < kLNW; w++) {
            before += w < warp ? wcnt[w] : 0;
            tot += wcnt[w];
        }
        if (q) {
            const int pos = out + before + __popc(bal & ((1u << lane) - 1u));
            const int64_t v = nbase + k;
            const int32_t pg = A.nd_parent[v];
            A.it_gv[pos] = v;
            A.it_uid[pos] = uid;
            A.it_kin[pos] = pg < 0 ? (ufl ? FLT_MAX : A.u_Uadd[uid]) : A.nd_kappa[pg];
            A.it_ufl[pos] = (uint8_t)ufl;
        }
        out += tot;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// long_eval: one node per CTA (grid-stride over the level's work items)
// ---------------------------------------------------------------------------
template <int DH, typename Tin>
struct LongSmem {
    static constexpr int RB = DH * (int)sizeof(Tin);                // bytes of a K or V row
    static constexpr int AB = RB > kLPP * 8 ? RB : kLPP * 8;        // of a key row or a row of probe weights
    float sk[kLMaxSeg][DH];          // per segment: sum of k_circ
    float srv[kLMaxSeg][DH];         //              sum of R v
    float ssv[kLMaxSeg][DH];         //              sum of v
    float ktil[2 * kLNCD][DH], vtil[2 * kLNCD][DH];
    union {
        // the probe scans' staging ring: per buffer kLChunk value rows, then as
        // many probe-weight rows (32 float2) or key rows
        __align__(16) unsigned char ring[2][kLChunk * (RB + AB)];
        float red[kLNW][3 * DH + 2];     // per-warp partials of one segment (before the scans)
        struct {                         // the warps' largest curvatures (before the segments)
            unsigned long long key[kLNW * kLMaxK];
            int pos[kLNW * kLMaxK];
        } top;
    };
    float redD[2 * kLNCD][kLNW], redP[2 * kLNCD][kLNW];
    float sR[kLMaxSeg], sKn[kLMaxSeg];
    int sF[kLMaxSeg];                // accepted floor positions in the segment
    float candD[2 * kLNCD], candP[2 * kLNCD], meff[2 * kLNCD];
    int ca[2 * kLNCD], cb[2 * kLNCD];   // prefixes at [0, npre) by ascending end, suffixes at
                                        // [kLNCD, kLNCD + nsuf) by descending start (absolute)
    uint8_t need[2 * kLNCD];            // rows that the next scans evaluate
    int segb[kLMaxSeg + 1];
    int nseg;
    int sel[kLMaxCut], cut[kLMaxCut], pidx[kLMaxCut], sidx[kLMaxCut];
    float kh[kLMaxCut];              // normalised curvature of the cuts
    int ncut, npre, nsuf, eL, eR, whole, pstar, forced, k1;
    unsigned long long kmaxk;        // largest curvature key
    unsigned long long bk[kLNW];     // per warp: smallest curvature key
    unsigned rk[kLNW], fk[kLNW];     //           largest token value, floor score (keys)
    int rp[kLNW], fp[kLNW];          //           and their positions
    int bad;
    unsigned pmask, alive;           // cuts whose prefix, whose both sides are evaluated
    unsigned rest;                   // cuts under evaluation
    int extP, extn, extr;            // the extraction's left side is evaluated; both are; under evaluation
    int more;                        // rows are left to evaluate
};

// Order-preserving 32-bit key of a float (larger value -> larger key).
__device__ __forceinline__ unsigned fokey(float x) {
    const uint32_t u = __float_as_uint(x);
    return (u >> 31) ? ~u : u | 0x80000000u;
}

// Bound by the fp32 FMAs of the probe scan (2 W d per token) and by latency, so
// two CTAs share an SM: the staging ring's bytes hold the segment partials and
// the curvature candidates before the scans, and the queries are read back for
// each evaluated row.  Skew 64K at 32x, all 16 launches: 161 -> 60 ms with the
// bound (half of the scanned tokens, 3 rows of about 36 for most nodes), the
// second CTA, tokens loaded four at a time by the segment sums, scans in
// stretches between fold points without a test per token, and the top-K drawn
// per warp in place of 16 block-wide passes over the curvature.
// EG: the probe weights of every token were written by the score pass; only
// then the queries need no registers during the scans.
template <int DH, typename Tin, bool EG>
__global__ void __launch_bounds__(kLT, EG ? 2 : 1) long_eval_kernel(LongArgs A) {
    using S = LongSmem<DH, Tin>;
    constexpr int HALF = DH / 2, NG = DH / (4 * kLCL), CH = 4 * NG, PPL = HALF / 32;
    static_assert(kLPP * kLCL == kLT && DH % (4 * kLCL) == 0 && HALF % 32 == 0, "layout");
    extern __shared__ __align__(16) unsigned char lsm_raw[];
    S &sm = *reinterpret_cast<S *>(lsm_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = lane / kLPPW, pp = warp * kLPPW + (lane & (kLPPW - 1));
    const int64_t n_items = min((int64_t)*A.n_items, A.cap_items);
    const float inv_sqrt_d = A.inv_sqrt_d, lamZ = A.lamZ, lamM = A.lamM, epsf = A.eps;
    // work items are taken from a counter, so that CTAs finishing short nodes
    // take the next ones (the nodes of a level range from 129 to 16384 tokens)
    __shared__ long long s_it;
    for (;;) {
        __syncthreads();   // the previous item's reads of s_it are done
        if (tid == 0) s_it = (long long)atomicAdd(A.it_next, 1u);
        __syncthreads();
        const int64_t it = s_it;
        if (it >= n_items) break;
        const int64_t gv = A.it_gv[it], uid = A.it_uid[it];
        const int lg = (int)(uid / A.J), l = lg / A.G, g = lg - l * A.G;
        const int a = A.nd_a[gv], b = A.nd_b[gv], n = b - a;
        const bool root = A.fresh != 0, ronly = root && A.root_only != 0;
        const bool cands = n >= 3 && !ronly;
        const float om = A.omega ? A.omega[lg] : 1.0f;
        const float *Rg = A.rtok + (size_t)lg * A.Nc - A.cs;   // Rg[t]: token value at absolute t
        const Tin *Kl = static_cast<const Tin *>(A.K) + (size_t)lg * A.T * DH;
        const Tin *Vl = static_cast<const Tin *>(A.V) + (size_t)lg * A.T * DH;
        const unsigned FULL = 0xffffffffu;
        if (tid == 0) sm.bad = 0;
        __syncthreads();
        // ---- phase A: cut candidates, curvature range, p*, forced floor position
        // top-K positions of [a, b-2] by (kappa descending, position ascending):
        // every warp draws its own K, a lane looking for its next position only
        // when its last one was taken; the K best of them are ranked by counting.
        {
            unsigned long long kmin = ~0ull, bkey = 0ull;
            int bpos = INT_MAX;
#pragma unroll 4
            for (int t = a + tid; t <= b - 2; t += kLT) {
                const unsigned long long k = lokey(A.kappa[t]);
                kmin = min(kmin, k);
                if (bpos == INT_MAX || k > bkey) { bkey = k; bpos = t; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) kmin = min(kmin, __shfl_xor_sync(FULL, kmin, o));
            // salient token p* = argmax R_tok over [a, b) (ties: lower t)
            unsigned rkey = 0u;
            int rpos = INT_MAX;
            bool nonf = false;
#pragma unroll 4
            for (int t = a + tid; t < b; t += kLT) {
                const float r = Rg[t];
                nonf |= !isfinite(r);
                const unsigned k = fokey(r);
                if (rpos == INT_MAX || k > rkey) { rkey = k; rpos = t; }
            }
            if (nonf) sm.bad = 1;
            // a node holding an accepted floor position is extracted at the one of
            // largest floor score (ties: lower t)
            unsigned fkey = 0u;
            int fpos = INT_MAX;
            if (A.fl_acc)
                for (int t = a + tid; t < b; t += kLT) {
                    const size_t q = (size_t)lg * A.Nc + (t - A.cs);
                    if (!A.fl_acc[q]) continue;
                    const unsigned k = fokey(A.fl_f[q]);
                    if (fpos == INT_MAX || k > fkey) { fkey = k; fpos = t; }
                }
            const unsigned rmx = __reduce_max_sync(FULL, rpos != INT_MAX ? rkey : 0u);
            const int rmp = __reduce_min_sync(FULL, rpos != INT_MAX && rkey == rmx ? rpos : INT_MAX);
            const unsigned fmx = __reduce_max_sync(FULL, fpos != INT_MAX ? fkey : 0u);
            const int fmp = __reduce_min_sync(FULL, fpos != INT_MAX && fkey == fmx ? fpos : INT_MAX);
            if (lane == 0) {
                sm.bk[warp] = kmin;
                sm.rk[warp] = rmx; sm.rp[warp] = rmp;
                sm.fk[warp] = fmx; sm.fp[warp] = fmp;
            }
            // one at least, for the curvature range (n > kMaxUnit > K)
            const int K = cands ? max(A.k_cand, 1) : 0;
            for (int r = 0; r < K; r++) {
                const unsigned hi = (unsigned)(bkey >> 32), lo = (unsigned)bkey;
                const bool v0 = bpos != INT_MAX;
                const unsigned mh = __reduce_max_sync(FULL, v0 ? hi : 0u);
                const bool v1 = v0 && hi == mh;
                const unsigned ml = __reduce_max_sync(FULL, v1 ? lo : 0u);
                const int mp = __reduce_min_sync(FULL, v1 && lo == ml ? bpos : INT_MAX);
                if (lane == 0) {
                    sm.top.key[warp * kLMaxK + r] = ((unsigned long long)mh << 32) | ml;
                    sm.top.pos[warp * kLMaxK + r] = mp;   // INT_MAX: the warp's positions are used up
                }
                if (bpos == mp && v0) {   // this lane's position was taken: its next one
                    const unsigned long long pk = bkey;
                    const int ppos = bpos;
                    bkey = 0ull;
                    bpos = INT_MAX;
#pragma unroll 4
                    for (int t = a + tid; t <= b - 2; t += kLT) {
                        const unsigned long long k = lokey(A.kappa[t]);
                        if ((k < pk || (k == pk && t > ppos)) && (bpos == INT_MAX || k > bkey)) { bkey = k; bpos = t; }
                    }
                }
            }
            __syncthreads();
            if (K > 0 && tid < kLNW * K) {
                const int i = (tid / K) * kLMaxK + tid % K;
                const unsigned long long k = sm.top.key[i];
                const int pos = sm.top.pos[i];
                int rank = 0;
                for (int w = 0; w < kLNW; w++)
                    for (int r = 0; r < K; r++) {
                        const unsigned long long k2 = sm.top.key[w * kLMaxK + r];
                        const int p2 = sm.top.pos[w * kLMaxK + r];
                        rank += p2 != INT_MAX && (k2 > k || (k2 == k && p2 < pos));
                    }
                if (pos != INT_MAX && rank < K) {
                    sm.sel[rank] = pos;
                    if (rank == 0) sm.kmaxk = k;
                }
            }
            __syncthreads();
        }
        // candidate rows, segment boundaries and the rows evaluated first (warp 0)
        if (warp == 0) {
            const int wl = lane < kLNW ? lane : 0;
            const unsigned rmx = __reduce_max_sync(FULL, sm.rp[wl] != INT_MAX ? sm.rk[wl] : 0u);
            int ps = __reduce_min_sync(FULL, sm.rp[wl] != INT_MAX && sm.rk[wl] == rmx ? sm.rp[wl] : INT_MAX);
            const unsigned fmx = __reduce_max_sync(FULL, sm.fp[wl] != INT_MAX ? sm.fk[wl] : 0u);
            const int fps = __reduce_min_sync(FULL, sm.fp[wl] != INT_MAX && sm.fk[wl] == fmx ? sm.fp[wl] : INT_MAX);
            if (!(ps >= a && ps < b)) ps = a;
            const bool forced = fps != INT_MAX;
            if (forced) ps = fps;
            const int er = ps + 1;
            const int K = cands ? A.k_cand : 0;   // n > kMaxUnit > K: K positions were found
            // cuts in ascending order: the positions' successors and the midpoint
            const int mid = a + n / 2;
            int xi = lane < K ? sm.sel[lane] + 1 : INT_MAX;
            const bool have = __any_sync(FULL, xi == mid);
            int ncut = K;
            if (cands && !have) {
                if (lane == K) xi = mid;
                ncut++;
            }
            int at = 0;
            for (int q = 0; q < ncut; q++) at += __shfl_sync(FULL, xi, q) < xi;
            __syncwarp();
            if (lane < ncut) sm.cut[at] = xi;
            __syncwarp();
            xi = lane < ncut ? sm.cut[lane] : INT_MAX;
            float kh = 0.f;
            if (lane < ncut) {
                unsigned long long mn = ~0ull;
                for (int w = 0; w < kLNW; w++) mn = min(mn, sm.bk[w]);
                const double kmn = lokey_inv(mn), kmx = lokey_inv(sm.kmaxk);
                const float krange = kmx > kmn ? 1.0f / (float)(kmx - kmn) : 0.f;
                kh = (float)(A.kappa[xi - 1] - kmn) * krange;
                sm.kh[lane] = kh;
            }
            const unsigned rew = lane < ncut ? fokey(A.lam_kappa * kh + 0.f) : 0u;
            const unsigned rew_mx = __reduce_max_sync(FULL, rew);
            const int k1 = __ffs(__ballot_sync(FULL, rew == rew_mx)) - 1;
            // rows: prefixes [a, xi) and [a, p*) by ascending end, the node itself
            // last; suffixes [xi, b) and [p* + 1, b) by descending start
            const unsigned lt = (1u << lane) - 1u, gt = ~((2u << lane) - 1u);
            const bool pv = lane < ncut && xi - a >= 2, sv = lane < ncut && b - xi >= 2;
            const bool elv = cands && ps - a >= 2, erv = cands && b - er >= 2;
            const unsigned pm = __ballot_sync(FULL, pv), sm_ = __ballot_sync(FULL, sv);
            const unsigned pdup = __ballot_sync(FULL, pv && xi == ps), sdup = __ballot_sync(FULL, sv && xi == er);
            const bool elr = elv && !pdup, err = erv && !sdup;   // rows of their own
            const int prow = __popc(pm & lt) + (elr && ps < xi ? 1 : 0);
            const int srow = kLNCD + __popc(sm_ & gt) + (err && er > xi ? 1 : 0);
            const int el_at = __popc(__ballot_sync(FULL, pv && xi < ps));
            const int er_at = kLNCD + __popc(__ballot_sync(FULL, sv && xi > er));
            const int npre0 = __popc(pm) + elr, npre = npre0 + root, nsuf = __popc(sm_) + err;
            if (pv) { sm.ca[prow] = a; sm.cb[prow] = xi; }
            if (sv) { sm.ca[srow] = xi; sm.cb[srow] = b; }
            if (lane < ncut) { sm.pidx[lane] = pv ? prow : -1; sm.sidx[lane] = sv ? srow : -1; }
            for (int q = lane; q < 2 * kLNCD; q += 32) sm.need[q] = 0;
            __syncwarp();
            const int eL = elv ? el_at : -1, eR = erv ? er_at : -1;
            if (lane == 0) {
                if (elr) { sm.ca[eL] = a; sm.cb[eL] = ps; }
                if (err) { sm.ca[eR] = er; sm.cb[eR] = b; }
                if (root) { sm.ca[npre0] = a; sm.cb[npre0] = b; sm.need[npre0] = 1; }
                sm.npre = npre; sm.nsuf = nsuf; sm.eL = eL; sm.eR = eR; sm.whole = root ? npre0 : -1;
                sm.ncut = ncut; sm.pstar = ps; sm.forced = forced; sm.k1 = k1;
                sm.alive = 0u;
                sm.extn = 0;
            }
            // Stage 0 evaluates prefixes: of the cut of largest reward, of the cuts
            // that D alone would not rule out against that reward (all of a root's,
            // whose D is not known yet: a row costs far less than a second scan),
            // and the forced extraction's; a fresh root's own row comes with them.
            const float DI0 = root || !A.prune ? INFINITY : A.nd_D[gv];
            const float rew1 = __shfl_sync(FULL, A.lam_kappa * kh, k1);
            const bool first = cands && !forced && lane < ncut &&
                               (lane == k1 || !(fmaf(A.lam_kappa, kh, DI0) < rew1));
            const unsigned fm = __ballot_sync(FULL, first);
            const bool fext = cands && (forced || !(rew1 >= DI0));
            if (first && pv) sm.need[prow] = 1;
            if (lane == 0) {
                if (fext && eL >= 0) sm.need[eL] = 1;
                sm.rest = fm;
                sm.extr = fext;
            }
            // segment boundaries: a, b, the cuts, p*, p* + 1
            const bool ps_in = ps > a && !__any_sync(FULL, xi == ps), er_in = er < b && !__any_sync(FULL, xi == er);
            int bd = xi;
            if (lane == 30) bd = ps_in ? ps : INT_MAX;
            if (lane == 31) bd = er_in ? er : INT_MAX;
            int slot = 1;
            for (int q = 0; q < 32; q++) slot += __shfl_sync(FULL, bd, q) < bd;
            if (bd != INT_MAX) sm.segb[slot] = bd;
            const int nin = __popc(__ballot_sync(FULL, bd != INT_MAX));
            if (lane == 0) { sm.segb[0] = a; sm.segb[nin + 1] = b; sm.nseg = nin + 1; }
        }
        __syncthreads();
        // ---- phase B: per-segment sums of k_circ, R v, v, R, ||k|| and floor positions
        // Warp w takes the tokens x + w, x + w + 8, ...; lane owns the rotation
        // pairs (i, i + d/2), i = PPL lane + j.  Each warp's running sums are
        // folded every kLFold of its tokens.
        // Tokens are loaded kLU at a time before any is added (a token at a time
        // was bound by the loads' latency).
        const int nseg = sm.nseg;
        const int i0 = lane * PPL;
        struct Acc {
            float k0[PPL], k1[PPL], r0[PPL], r1[PPL], v0[PPL], v1[PPL], rs, ks;
            __device__ __forceinline__ void clear() {
#pragma unroll
                for (int j = 0; j < PPL; j++) k0[j] = k1[j] = r0[j] = r1[j] = v0[j] = v1[j] = 0.f;
                rs = ks = 0.f;
            }
            __device__ __forceinline__ void add(const Acc &o) {
#pragma unroll
                for (int j = 0; j < PPL; j++) {
                    k0[j] += o.k0[j]; k1[j] += o.k1[j]; r0[j] += o.r0[j]; r1[j] += o.r1[j];
                    v0[j] += o.v0[j]; v1[j] += o.v1[j];
                }
                rs += o.rs;
                ks += o.ks;
            }
        };
        struct Tok {
            LRaw<Tin, PPL> k0, k1, v0, v1;
            float2 cs[PPL];
            float r;
        };
        auto load_tok = [&](Tok &x, int t) {
            const size_t e = (size_t)t * DH + i0;
            x.k0.load(Kl + e); x.k1.load(Kl + e + HALF);
            x.v0.load(Vl + e); x.v1.load(Vl + e + HALF);
            const float2 *rp = A.rope + (size_t)t * HALF + i0;
            if constexpr (PPL == 2) {
                const float4 c4 = *reinterpret_cast<const float4 *>(rp);
                x.cs[0] = make_float2(c4.x, c4.y);
                x.cs[1] = make_float2(c4.z, c4.w);
            } else {
                x.cs[0] = rp[0];
            }
            x.r = Rg[t];
        };
        auto norm_tok = [&](const Tok &x) {   // ||k_t||^2, the same in every lane
            float nn = 0.f;
#pragma unroll
            for (int j = 0; j < PPL; j++) {
                const float k0 = x.k0.get(j), k1 = x.k1.get(j);
                nn = fmaf(k0, k0, fmaf(k1, k1, nn));
            }
            return warp_sum(nn);
        };
        auto add_tok = [&](Acc &c, const Tok &x, float nn) {
#pragma unroll
            for (int j = 0; j < PPL; j++) {
                const float k0 = x.k0.get(j), k1 = x.k1.get(j), v0 = x.v0.get(j), v1 = x.v1.get(j);
                // k_circ = RoPE^-1(k, t): rotation by -t
                c.k0[j] += fmaf(k0, x.cs[j].x, k1 * x.cs[j].y);
                c.k1[j] += fmaf(k1, x.cs[j].x, -(k0 * x.cs[j].y));
                c.r0[j] = fmaf(x.r, v0, c.r0[j]);
                c.r1[j] = fmaf(x.r, v1, c.r1[j]);
                c.v0[j] += v0;
                c.v1[j] += v1;
            }
            c.rs += x.r;
            c.ks += sqrtf(nn);
        };
        // segments of at most kLNW tokens: one token per partial sum, a segment
        // per warp and no barrier (clustered curvature peaks make many of them)
        for (int s = 0, k = 0; s < nseg; s++) {
            const int x = sm.segb[s], y = sm.segb[s + 1];
            if (y - x > kLNW || k++ % kLNW != warp) continue;
            Acc v;
            v.clear();
            for (int t0 = x; t0 < y; t0 += kLU) {
                Tok tk[kLU];
                float nn[kLU];
#pragma unroll
                for (int u = 0; u < kLU; u++) load_tok(tk[u], min(t0 + u, y - 1));
#pragma unroll
                for (int u = 0; u < kLU; u++) nn[u] = norm_tok(tk[u]);
#pragma unroll
                for (int u = 0; u < kLU; u++)
                    if (t0 + u < y) {
                        Acc c;
                        c.clear();
                        add_tok(c, tk[u], nn[u]);
                        v.add(c);
                    }
            }
#pragma unroll
            for (int j = 0; j < PPL; j++) {
                sm.sk[s][i0 + j] = v.k0[j];  sm.sk[s][i0 + j + HALF] = v.k1[j];
                sm.srv[s][i0 + j] = v.r0[j]; sm.srv[s][i0 + j + HALF] = v.r1[j];
                sm.ssv[s][i0 + j] = v.v0[j]; sm.ssv[s][i0 + j + HALF] = v.v1[j];
            }
            bool f = false;
            if (A.fl_acc && lane < y - x) f = A.fl_acc[(size_t)lg * A.Nc + (x + lane - A.cs)] != 0;
            f = __any_sync(FULL, f);
            if (lane == 0) { sm.sR[s] = v.rs; sm.sKn[s] = v.ks; sm.sF[s] = f; }
        }
        for (int s = 0; s < nseg; s++) {
            const int x = sm.segb[s], y = sm.segb[s + 1];
            if (y - x <= kLNW) continue;
            Acc tot, c;
            tot.clear();
            c.clear();
            int fold = 0;
            for (int t0 = x + warp; t0 < y; t0 += kLU * kLNW) {
                Tok tk[kLU];
                float nn[kLU];
#pragma unroll
                for (int u = 0; u < kLU; u++) load_tok(tk[u], min(t0 + u * kLNW, y - 1));
#pragma unroll
                for (int u = 0; u < kLU; u++) nn[u] = norm_tok(tk[u]);
#pragma unroll
                for (int u = 0; u < kLU; u++)
                    if (t0 + u * kLNW < y) add_tok(c, tk[u], nn[u]);
                fold += kLU;
                if (fold == kLFold) {   // the last, partial sum may be folded here too: it adds the same
                    tot.add(c);
                    c.clear();
                    fold = 0;
                }
            }
            tot.add(c);
            float *rw = sm.red[warp];
#pragma unroll
            for (int j = 0; j < PPL; j++) {
                rw[i0 + j] = tot.k0[j];
                rw[i0 + j + HALF] = tot.k1[j];
                rw[DH + i0 + j] = tot.r0[j];
                rw[DH + i0 + j + HALF] = tot.r1[j];
                rw[2 * DH + i0 + j] = tot.v0[j];
                rw[2 * DH + i0 + j + HALF] = tot.v1[j];
            }
            if (lane == 0) { rw[3 * DH] = tot.rs; rw[3 * DH + 1] = tot.ks; }
            int fc = 0;
            if (A.fl_acc)
                for (int t = x + tid; t < y; t += kLT) fc += A.fl_acc[(size_t)lg * A.Nc + (t - A.cs)] ? 1 : 0;
            fc = __syncthreads_count(fc != 0);   // also orders the partials above
            for (int e = tid; e < 3 * DH + 2; e += kLT) {
                float v = 0.f;
#pragma unroll
                for (int w = 0; w < kLNW; w++) v += sm.red[w][e];
                if (e < DH) sm.sk[s][e] = v;
                else if (e < 2 * DH) sm.srv[s][e - DH] = v;
                else if (e < 3 * DH) sm.ssv[s][e - 2 * DH] = v;
                else if (e == 3 * DH) sm.sR[s] = v;
                else sm.sKn[s] = v;
            }
            if (tid == 0) sm.sF[s] = fc;
            __syncthreads();
        }
        __syncthreads();
        const int npre = sm.npre, nsuf = sm.nsuf;
        unsigned long long w_scan = 0, w_eval = 0, w_len = 0;   // work counters (thread 0)
        // Stages, one scan each: 0 the prefixes chosen above, 1 the suffixes of those
        // that may still be the best cut; then, rarely, 2 the prefixes and 3 the
        // suffixes of cuts that the best one found does not rule out.
        for (int stage = 0;; stage++) {
        // ---- phase C: candidate prototypes from their segments (warp per candidate)
        auto seg_of = [&](int pos) {   // index of the boundary at pos (every candidate end is one)
            int s = 0;
            while (s < nseg && sm.segb[s] != pos) s++;
            return s;
        };
        for (int q = warp; q < npre + nsuf; q += kLNW) {
            const int k = q < npre ? q : kLNCD + (q - npre);
            if (!sm.need[k]) continue;
            const int x = sm.ca[k], y = sm.cb[k], nJ = y - x;
            const int s0 = seg_of(x), s1 = seg_of(y);
            const int p = lround_half_even_mid(x, y);
            float2 rot[PPL];
#pragma unroll
            for (int j = 0; j < PPL; j++) rot[j] = A.rope[(size_t)p * HALF + i0 + j];
            float m0[PPL], m1[PPL], r0[PPL], r1[PPL], v0[PPL], v1[PPL];
            float rs = 0.f, ks = 0.f;
#pragma unroll
            for (int j = 0; j < PPL; j++) m0[j] = m1[j] = r0[j] = r1[j] = v0[j] = v1[j] = 0.f;
            for (int s = s0; s < s1; s++) {
#pragma unroll
                for (int j = 0; j < PPL; j++) {
                    m0[j] += sm.sk[s][i0 + j];  m1[j] += sm.sk[s][i0 + j + HALF];
                    r0[j] += sm.srv[s][i0 + j]; r1[j] += sm.srv[s][i0 + j + HALF];
                    v0[j] += sm.ssv[s][i0 + j]; v1[j] += sm.ssv[s][i0 + j + HALF];
                }
                rs += sm.sR[s];
                ks += sm.sKn[s];
            }
            const float ninv = 1.0f / (float)nJ;
            const float beta = A.base_frac * (rs * ninv);
            const float winv = 1.0f / ((rs + (float)nJ * beta) + epsf);
            float mu2 = 0.f;
#pragma unroll
            for (int j = 0; j < PPL; j++) {
                const float a0 = m0[j] * ninv, a1 = m1[j] * ninv;
                mu2 = fmaf(a0, a0, fmaf(a1, a1, mu2));
                sm.ktil[k][i0 + j] = a0 * rot[j].x - a1 * rot[j].y;
                sm.ktil[k][i0 + j + HALF] = a0 * rot[j].y + a1 * rot[j].x;
                sm.vtil[k][i0 + j] = fmaf(beta, v0[j], r0[j]) * winv;
                sm.vtil[k][i0 + j + HALF] = fmaf(beta, v1[j], r1[j]) * winv;
            }
            mu2 = warp_sum(mu2);
            if (lane == 0) {
                const float coh = sqrtf(mu2) / (ks * ninv + epsf);
                const float me = (float)nJ * coh * coh;
                sm.meff[k] = me < 1.0f ? 1.0f : (me > (float)nJ ? (float)nJ : me);
            }
        }
        __syncthreads();
        // ---- phase D: probe scans --------------------------------------------
        // thread (pp, c): probes pp and pp + 32, elements 4 c + 32 gi + j
        auto qrow = [&](int u) -> size_t { return ((size_t)l * A.Hq + g * A.gq + (u % A.gq)) * A.W + u; };
        auto load_q = [&](float2 *qd, int u) {
            if (u < A.W) {
                const Tin *qp = static_cast<const Tin *>(A.Q) + qrow(u) * DH + 4 * c;
#pragma unroll
                for (int gi = 0; gi < NG; gi++) {
                    const float4 x = lld4(qp + 32 * gi);
                    qd[2 * gi] = make_float2(x.x, x.y);
                    qd[2 * gi + 1] = make_float2(x.z, x.w);
                }
            } else {
#pragma unroll
                for (int q = 0; q < CH / 2; q++) qd[q] = make_float2(0.f, 0.f);
            }
        };
        const bool has0 = pp < A.W, has1 = pp + kLPP < A.W;
        const float mu0 = has0 ? A.row_m[qrow(pp)] : 0.f, mu1 = has1 ? A.row_m[qrow(pp + kLPP)] : 0.f;
        const float invZ0 = has0 ? 1.0f / A.row_Z[qrow(pp)] : 0.f, invZ1 = has1 ? 1.0f / A.row_Z[qrow(pp + kLPP)] : 0.f;
        // the queries: kept where every token needs them, else read back for each
        // evaluated row (a few per node)
        float2 qk0[EG ? 1 : CH / 2], qk1[EG ? 1 : CH / 2];
        if constexpr (!EG) {
            load_q(qk0, pp);
            load_q(qk1, pp + kLPP);
        }
        // D_u of candidate row k from the running statistics, weighted by the
        // probe's attention mass; per-warp partial sums (as in build.cu)
        auto evaluate = [&](int k, float Z0, float Z1, const float2 *M0, const float2 *M1) {
            float x0, x1;
            {
                float2 xa = make_float2(0.f, 0.f), xb = make_float2(0.f, 0.f);
                float2 ql0[EG ? CH / 2 : 1], ql1[EG ? CH / 2 : 1];
                if constexpr (EG) {
                    load_q(ql0, pp);
                    load_q(ql1, pp + kLPP);
                }
#pragma unroll
                for (int gi = 0; gi < NG; gi++) {
                    const float4 x = *reinterpret_cast<const float4 *>(&sm.ktil[k][4 * c + 32 * gi]);
                    const float2 kt[2] = {make_float2(x.x, x.y), make_float2(x.z, x.w)};
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int q = 2 * gi + h;
                        if constexpr (EG) {
                            xa = ffma2(ql0[q], kt[h], xa);
                            xb = ffma2(ql1[q], kt[h], xb);
                        } else {
                            xa = ffma2(qk0[q], kt[h], xa);
                            xb = ffma2(qk1[q], kt[h], xb);
                        }
                    }
                }
                x0 = xa.x + xa.y;
                x1 = xb.x + xb.y;
            }
#pragma unroll
            for (int o = kLPPW; o < 32; o <<= 1) {
                x0 += __shfl_xor_sync(0xffffffffu, x0, o);
                x1 += __shfl_xor_sync(0xffffffffu, x1, o);
            }
            const float me = sm.meff[k];
            const float zt0 = me * expf(x0 * inv_sqrt_d - mu0), zt1 = me * expf(x1 * inv_sqrt_d - mu1);
            const float2 nz0 = make_float2(-zt0, -zt0), nz1 = make_float2(-zt1, -zt1);
            float2 r0 = make_float2(0.f, 0.f), r1 = r0, m0 = r0, m1 = r0;
#pragma unroll
            for (int gi = 0; gi < NG; gi++) {
                const float4 x = *reinterpret_cast<const float4 *>(&sm.vtil[k][4 * c + 32 * gi]);
                const float2 va = make_float2(x.x, x.y), vb = make_float2(x.z, x.w);
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int q = 2 * gi + h;
                    const float2 vt = h ? vb : va;
                    const float2 d0 = ffma2(nz0, vt, M0[q]), d1 = ffma2(nz1, vt, M1[q]);
                    r0 = ffma2(d0, d0, r0);
                    r1 = ffma2(d1, d1, r1);
                    m0 = ffma2(M0[q], M0[q], m0);
                    m1 = ffma2(M1[q], M1[q], m1);
                }
            }
            float res0 = r0.x + r0.y, res1 = r1.x + r1.y, mm0 = m0.x + m0.y, mm1 = m1.x + m1.y;
#pragma unroll
            for (int o = kLPPW; o < 32; o <<= 1) {
                res0 += __shfl_xor_sync(0xffffffffu, res0, o);
                res1 += __shfl_xor_sync(0xffffffffu, res1, o);
                mm0 += __shfl_xor_sync(0xffffffffu, mm0, o);
                mm1 += __shfl_xor_sync(0xffffffffu, mm1, o);
            }
            const float dz0 = Z0 - zt0, dz1 = Z1 - zt1;
            const float D0 = lamZ * __fdividef(dz0 * dz0, fmaf(Z0, Z0, epsf)) + lamM * __fdividef(res0, mm0 + epsf);
            const float D1 = lamZ * __fdividef(dz1 * dz1, fmaf(Z1, Z1, epsf)) + lamM * __fdividef(res1, mm1 + epsf);
            const float p0 = Z0 * invZ0, p1 = Z1 * invZ1;
            float pd = fmaf(p0, D0, p1 * D1), pw = p0 + p1;
#pragma unroll
            for (int o = 1; o < kLPPW; o <<= 1) {
                pd += __shfl_xor_sync(0xffffffffu, pd, o);
                pw += __shfl_xor_sync(0xffffffffu, pw, o);
            }
            if (lane == 0) { sm.redD[k][warp] = pd; sm.redP[k][warp] = pw; }
        };
        // one direction: the running sums over the node's tokens, folded every
        // kLFold tokens and at every candidate end, evaluated at each end.  The
        // tokens are staged kLChunk at a time in a two-buffer cp.async ring:
        // their value rows and their probe weights (pass B) or key rows.
        auto scan = [&](bool suffix) {
            // the direction's rows; the scan ends at the last one needed
            const int r0 = suffix ? kLNCD : 0;
            int nk = suffix ? nsuf : npre;
            while (nk > 0 && !sm.need[r0 + nk - 1]) nk--;
            if (nk == 0) return;
            // tokens of the scan: forward a, a + 1, ..; backward b - 1, b - 2, ..
            auto end_of = [&](int k) { return suffix ? b - sm.ca[r0 + k] : sm.cb[r0 + k] - a; };
            const int ntok = end_of(nk - 1);
            float2 Mt0[CH / 2], Mt1[CH / 2], Mc0[CH / 2], Mc1[CH / 2];
            float Zt0 = 0.f, Zt1 = 0.f, Zc0 = 0.f, Zc1 = 0.f;
#pragma unroll
            for (int q = 0; q < CH / 2; q++) Mt0[q] = Mt1[q] = Mc0[q] = Mc1[q] = make_float2(0.f, 0.f);
            auto fold_in = [&]() {
#pragma unroll
                for (int q = 0; q < CH / 2; q++) {
                    Mt0[q].x += Mc0[q].x; Mt0[q].y += Mc0[q].y; Mt1[q].x += Mc1[q].x; Mt1[q].y += Mc1[q].y;
                    Mc0[q] = Mc1[q] = make_float2(0.f, 0.f);
                }
                Zt0 += Zc0; Zt1 += Zc1; Zc0 = Zc1 = 0.f;
            };
            // chunk c holds the scan's tokens [c kLChunk, (c + 1) kLChunk): rows
            // tlo .. tlo + m - 1 of the input, tlo the smallest position
            auto chunk_rows = [&](int c0, int &tlo, int &m) {
                m = min(kLChunk, ntok - c0);
                tlo = suffix ? b - c0 - m : a + c0;
            };
            auto issue = [&](int c0, int buf) {
                if (c0 < ntok) {
                    int tlo, m;
                    chunk_rows(c0, tlo, m);
                    unsigned char *dst = sm.ring[buf];
                    constexpr int RB = S::RB;
                    const char *vsrc = reinterpret_cast<const char *>(Vl + (size_t)tlo * DH);
                    for (int q = tid; q < m * RB / 16; q += kLT) cp_async16(dst + 16 * q, vsrc + 16 * q, true);
                    unsigned char *dst2 = dst + kLChunk * RB;
                    if constexpr (EG) {
                        const char *esrc = reinterpret_cast<const char *>(A.Eg + ((size_t)lg * A.Nc + (tlo - A.cs)) * kLPP);
                        for (int q = tid; q < m * kLPP * 8 / 16; q += kLT) cp_async16(dst2 + 16 * q, esrc + 16 * q, true);
                    } else {
                        const char *ksrc = reinterpret_cast<const char *>(Kl + (size_t)tlo * DH);
                        for (int q = tid; q < m * RB / 16; q += kLT) cp_async16(dst2 + 16 * q, ksrc + 16 * q, true);
                    }
                }
                cp_async_commit();
            };
            // The sums are folded every kLFold tokens and at every row's end, also of
            // rows not needed now, so that a row's bits do not depend on which
            // others are evaluated.
            int kk = 0, kend = end_of(0), next_fold = kLFold;
            unsigned ebits = 0u;   // largest probe-weight bits: weights are >= 0, non-finite ones on top
            issue(0, 0);
            for (int c0 = 0, buf = 0; c0 < ntok; c0 += kLChunk, buf ^= 1) {
                issue(c0 + kLChunk, buf ^ 1);
                cp_async_wait<1>();   // this chunk's copies have landed (each thread its own)
                __syncthreads();
                int tlo, m;
                chunk_rows(c0, tlo, m);
                const Tin *vrow0 = reinterpret_cast<const Tin *>(sm.ring[buf]) + 4 * c;
                const unsigned char *aux = sm.ring[buf] + kLChunk * S::RB;
                for (int i = 0; i < m;) {
                    const int lim = max(i + 1, min(m, min(next_fold, kend) - c0));
#pragma unroll 2
                    for (; i < lim; i++) {
                        const int r = suffix ? m - 1 - i : i;   // row of the scan's token c0 + i
                        float e0, e1;
                        if constexpr (EG) {   // zero for probes past W
                            const float2 e = reinterpret_cast<const float2 *>(aux)[r * kLPP + pp];
                            e0 = e.x;
                            e1 = e.y;
                        } else {
                            const Tin *krow = reinterpret_cast<const Tin *>(aux) + (size_t)r * DH;
                            float2 ya = make_float2(0.f, 0.f), yb = ya;
#pragma unroll
                            for (int gi = 0; gi < NG; gi++) {
                                const float4 kv = lld4(krow + 4 * c + 32 * gi);
                                const float2 ka = make_float2(kv.x, kv.y), kb = make_float2(kv.z, kv.w);
                                ya = ffma2(qk0[2 * gi], ka, ya); ya = ffma2(qk0[2 * gi + 1], kb, ya);
                                yb = ffma2(qk1[2 * gi], ka, yb); yb = ffma2(qk1[2 * gi + 1], kb, yb);
                            }
                            float y0 = ya.x + ya.y, y1 = yb.x + yb.y;
#pragma unroll
                            for (int o = kLPPW; o < 32; o <<= 1) {
                                y0 += __shfl_xor_sync(0xffffffffu, y0, o);
                                y1 += __shfl_xor_sync(0xffffffffu, y1, o);
                            }
                            e0 = has0 ? expf(y0 * inv_sqrt_d - mu0) : 0.f;
                            e1 = has1 ? expf(y1 * inv_sqrt_d - mu1) : 0.f;
                        }
                        ebits = max(ebits, max(__float_as_uint(e0), __float_as_uint(e1)));
                        const float2 ee0 = make_float2(e0, e0), ee1 = make_float2(e1, e1);
                        Zc0 += e0;
                        Zc1 += e1;
                        const Tin *vrow = vrow0 + r * DH;
#pragma unroll
                        for (int gi = 0; gi < NG; gi++) {
                            const float4 x = lld4(vrow + 32 * gi);
                            const float2 va = make_float2(x.x, x.y), vb = make_float2(x.z, x.w);
                            Mc0[2 * gi] = ffma2(ee0, va, Mc0[2 * gi]);
                            Mc0[2 * gi + 1] = ffma2(ee0, vb, Mc0[2 * gi + 1]);
                            Mc1[2 * gi] = ffma2(ee1, va, Mc1[2 * gi]);
                            Mc1[2 * gi + 1] = ffma2(ee1, vb, Mc1[2 * gi + 1]);
                        }
                    }
                    const int done = c0 + i;
                    if (done == next_fold || done == kend) {
                        fold_in();
                        next_fold = done + kLFold;
                    }
                    while (done == kend) {
                        if (sm.need[r0 + kk]) evaluate(r0 + kk, Zt0, Zt1, Mt0, Mt1);
                        kend = ++kk < nk ? end_of(kk) : INT_MAX;
                    }
                }
                __syncthreads();   // the buffer is refilled by the next issue
            }
            cp_async_wait<0>();
            if (ebits >= 0x7f800000u) sm.bad = 1;
        };
        scan(false);
        scan(true);
        __syncthreads();
        // ---- phase E: candidate D, the decision, gains and keys -----------------
        const float invW = 1.0f / (float)A.W;
        for (int q = tid; q < npre + nsuf; q += kLT) {
            const int k = q < npre ? q : kLNCD + (q - npre);
            if (!sm.need[k]) continue;
            float d = 0.f, pw = 0.f;
#pragma unroll
            for (int w = 0; w < kLNW; w++) { d += sm.redD[k][w]; pw += sm.redP[k][w]; }
            sm.candD[k] = d * invW;
            sm.candP[k] = pw * invW;
        }
        __syncthreads();
        // G_bin of a cut is ((D - D_L) - D_R) + lambda_kappa kh with D_L, D_R >= 0,
        // so D + lambda_kappa kh, and (D - D_L) + lambda_kappa kh once D_L is known,
        // bound it, also as rounded (every operation is monotone).  A cut whose
        // bound is below the best G_bin evaluated cannot be the best one; the
        // extraction's sides cannot matter when that G_bin reaches D.
        if (warp == 0) {
            if (tid == 0) {
                int pe = a, ssn = b;
                for (int q = 0; q < npre; q++)
                    if (sm.need[q]) { pe = max(pe, sm.cb[q]); w_len += sm.cb[q] - a; w_eval++; }
                for (int q = kLNCD; q < kLNCD + nsuf; q++)
                    if (sm.need[q]) { ssn = min(ssn, sm.ca[q]); w_len += b - sm.ca[q]; w_eval++; }
                w_scan += (pe - a) + (b - ssn);
            }
            const int k1 = sm.k1, ncut = sm.ncut;
            const bool decide = cands && !sm.bad && stage < 3;
            const float DI = root ? sm.candD[sm.whole] : A.nd_D[gv];
            const int i = lane < ncut ? lane : 0;
            const unsigned rest = sm.rest;
            const bool extr = sm.extr != 0, mine = (rest >> lane) & 1u;
            unsigned pmask = stage == 0 ? rest : stage == 2 ? sm.pmask | rest : sm.pmask;
            unsigned alive = sm.alive, next = 0u;
            bool extP = stage == 0 ? extr : stage == 2 ? sm.extP || extr : sm.extP != 0;
            bool extn = sm.extn != 0, next_ext = false;
            __syncwarp();
            for (int q = lane; q < 2 * kLNCD; q += 32) sm.need[q] = 0;
            if (stage == 1 || stage == 3) {
                alive |= rest;
                extn |= extr;
            }
            const bool known = (pmask >> lane) & 1u;
            const float DL = known && sm.pidx[i] >= 0 ? sm.candD[sm.pidx[i]] : 0.f;
            const float ub = fmaf(A.lam_kappa, sm.kh[i], DI - DL);
            // the best G_bin of the cuts evaluated
            float lb = -INFINITY;
            if ((alive >> lane) & 1u) {
                const float DR = sm.sidx[i] >= 0 ? sm.candD[sm.sidx[i]] : 0.f;
                lb = fmaf(A.lam_kappa, sm.kh[i], (DI - DL) - DR);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) lb = fmaxf(lb, __shfl_xor_sync(FULL, lb, o));
            if (decide && sm.forced) {
                next_ext = stage == 0;
            } else if (decide) {
                bool q;
                if (stage == 0) {
                    // the suffixes that are likely needed, in one scan: bounds within D of
                    // the first cut's (what its own suffix may take off); the check
                    // after stage 1 is the exact one
                    const float ub1 = __shfl_sync(FULL, ub, k1);
                    q = mine && (lane == k1 || !A.prune || !(ub < ub1 - DI));
                    next_ext = extr && !(A.prune && A.lam_kappa * sm.kh[k1] >= DI);
                } else if (stage == 2) {
                    q = mine && (!A.prune || !(ub < lb));
                    next_ext = extr;
                } else {
                    q = lane < ncut && !((alive >> lane) & 1u) && (!A.prune || !(ub < lb));
                    next_ext = !extn && !(A.prune && lb >= DI);
                }
                next = __ballot_sync(FULL, q);
            }
            __syncwarp();
            {
                const bool pre = stage == 1;   // the next stage's scan
                const bool todo = ((next >> lane) & 1u) && !(pre && known);
                const int row = todo ? (pre ? sm.pidx[i] : sm.sidx[i]) : -1;
                const int erow = next_ext && !(pre && extP) ? (pre ? sm.eL : sm.eR) : -1;
                if (row >= 0) sm.need[row] = 1;
                if (lane == 0) {
                    if (erow >= 0) sm.need[erow] = 1;
                    sm.pmask = pmask;
                    sm.alive = alive;
                    sm.rest = next;
                    sm.extP = extP;
                    sm.extn = extn;
                    sm.extr = next_ext;
                    sm.more = next != 0u || next_ext;
                }
            }
        }
        __syncthreads();
        if (!sm.more) break;
        }   // stages
        if (warp == 0) {
            LongRes rs;
            rs.nch = 0;
            rs.U = rs.kap = rs.bound = 0.f;
            for (int q = 0; q < 3; q++) { rs.ca[q] = rs.cb[q] = 0; rs.cD[q] = rs.rch[q] = rs.bnd[q] = 0.f; }
            const int forced = sm.forced, ps = sm.pstar, ncut = sm.ncut;
            const bool ufl = A.it_ufl[it] != 0;
            float kin = A.it_kin[it];
            float DI;
            const bool bounded = A.prune && om >= 0.f;   // build.cu
            auto split_bound = [&](float k, float R, float D) { return bounded ? fminf(k, lkey_bound(om * R * D)) : k; };
            const float nodeR = A.nd_R[gv];
            if (root) {   // D, D_drop and the Add gain of the slot (Eq. app_operation_gains)
                const float Pd = sm.candP[sm.whole];
                DI = sm.candD[sm.whole];
                float gain = om * nodeR * (Pd - DI);
                if (gain < 0.f) gain = 0.f;
                kin = ufl ? FLT_MAX : gain;   // a floor slot's Add is a floor op
                if (lane == 0) {
                    A.u_Uadd[uid] = sm.bad ? 0.f : gain;
                    A.u_Ddrop[uid] = sm.bad ? 0.f : Pd;
                    A.nd_D[gv] = sm.bad ? 0.f : DI;
                }
            } else {
                DI = A.nd_D[gv];
            }
            // value of [x, y) from the segment sums; does it hold a floor position
            auto seg_sum = [&](int x, int y, float &r, bool &fl) {   // x, y are boundaries
                int s = 0;
                while (s < nseg && sm.segb[s] != x) s++;
                r = 0.f;
                fl = false;
                for (; s < nseg && sm.segb[s] != y; s++) { r += sm.sR[s]; fl |= sm.sF[s] != 0; }
            };
            if (sm.bad) {
                if (lane == 0) atomicOr(A.status, 8);   // non-finite: a leaf with zero gain
                rs.nch = 0;
            } else if (ronly) {   // the root's split is decided later: bound its key
                rs.nch = -1;
                rs.bound = forced ? FLT_MAX : split_bound(kin, nodeR, DI);
            } else {
                int nch;
                if (n == 2) {
                    nch = 2;
                    rs.ca[0] = a; rs.cb[0] = a + 1; rs.cD[0] = 0.f;
                    rs.ca[1] = a + 1; rs.cb[1] = b; rs.cD[1] = 0.f;
                } else {
                    // binary cut: lane q evaluates cut q; max G_bin, ties -> smallest xi
                    float best = -INFINITY;
                    int bq = 0x7fffffff;
                    if ((sm.alive >> lane) & 1u) {   // the cuts that no bound ruled out
                        const float DL = sm.pidx[lane] >= 0 ? sm.candD[sm.pidx[lane]] : 0.f;
                        const float DR = sm.sidx[lane] >= 0 ? sm.candD[sm.sidx[lane]] : 0.f;
                        best = fmaf(A.lam_kappa, sm.kh[lane], (DI - DL) - DR);
                        bq = lane;
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const float ov = __shfl_xor_sync(0xffffffffu, best, o);
                        const int oq = __shfl_xor_sync(0xffffffffu, bq, o);
                        if (ov > best || (ov == best && oq < bq)) { best = ov; bq = oq; }
                    }
                    int bxi = -1;
                    float bL = 0.f, bR = 0.f;
                    if (bq < ncut && best > -INFINITY) {
                        bxi = sm.cut[bq];
                        bL = sm.pidx[bq] >= 0 ? sm.candD[sm.pidx[bq]] : 0.f;
                        bR = sm.sidx[bq] >= 0 ? sm.candD[sm.sidx[bq]] : 0.f;
                    }
                    // extraction at p* (its D are read only where they were evaluated)
                    const bool ext = sm.extn != 0;
                    int ea[3], eb[3], ne = 0;
                    float eD[3];
                    if (ps > a) { ea[ne] = a; eb[ne] = ps; eD[ne] = ext && ps - a >= 2 ? sm.candD[sm.eL] : 0.f; ne++; }
                    ea[ne] = ps; eb[ne] = ps + 1; eD[ne] = 0.f; ne++;
                    if (ps + 1 < b) { ea[ne] = ps + 1; eb[ne] = b; eD[ne] = ext && b - ps - 1 >= 2 ? sm.candD[sm.eR] : 0.f; ne++; }
                    float gext = DI;
                    for (int q = 0; q < ne; q++) gext -= eD[q];
                    if (bxi < 0) {   // only reachable with non-finite gains
                        bxi = sm.cut[0];
                        bL = sm.pidx[0] >= 0 ? sm.candD[sm.pidx[0]] : 0.f;
                        bR = sm.sidx[0] >= 0 ? sm.candD[sm.sidx[0]] : 0.f;
                    }
                    const float rho_ext = ne == 3 ? 0.5f * gext : gext;   // G_ext / (|children| - 1)
                    if (forced || (ext && rho_ext > best)) {
                        nch = ne;
                        for (int q = 0; q < ne; q++) { rs.ca[q] = ea[q]; rs.cb[q] = eb[q]; rs.cD[q] = eD[q]; }
                    } else {
                        nch = 2;
                        rs.ca[0] = a; rs.cb[0] = bxi; rs.cD[0] = bL;
                        rs.ca[1] = bxi; rs.cb[1] = b; rs.cD[1] = bR;
                    }
                }
                bool chf[3] = {false, false, false};
                for (int q = 0; q < nch; q++) seg_sum(rs.ca[q], rs.cb[q], rs.rch[q], chf[q]);
                const float rnode = (rs.rch[0] + rs.rch[1]) + rs.rch[2];   // R of the node = sum over its children
                const float dsum = (rs.cD[0] + rs.cD[1]) + (nch == 3 ? rs.cD[2] : 0.f);
                const int cost = nch - 1;
                float gain = om * rnode * (DI - dsum);
                if (gain < 0.f) gain = 0.f;
                rs.U = cost == 2 ? 0.5f * gain : gain;
                rs.kap = forced ? FLT_MAX : fminf(rs.U, kin);
                for (int q = 0; q < nch; q++)
                    rs.bnd[q] = rs.cb[q] - rs.ca[q] >= 2
                                    ? (chf[q] ? FLT_MAX : split_bound(rs.kap, rs.rch[q], rs.cD[q]))
                                    : 0.f;
                rs.nch = nch;
            }
            if (lane == 0) {
                A.res[it] = rs;
                atomicAdd(&A.work[0], w_scan);
                atomicAdd(&A.work[1], w_eval);
                atomicAdd(&A.work[2], w_len);
                atomicAdd(&A.work[3], 1ull);
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// long_commit: children numbered after the unit's nodes, in work-item order
// (warp per listed unit)
// ---------------------------------------------------------------------------
__global__ void long_commit_kernel(LongArgs A) {
    const int i = blockIdx.x, lane = threadIdx.x;
    const int start = A.u_start[i], cnt = A.u_cnt[i];
    if (cnt <= 0) return;
    const int64_t uid = A.it_uid[start];
    const int lg = (int)(uid / A.J), j = (int)(uid - (int64_t)lg * A.J);
    const int64_t nbase = node_base(lg, A.slots[j], A.cs, A.Nc);
    int base = A.u_nnodes[uid];
    float pend = A.u_pend[uid];
    for (int k0 = 0; k0 < cnt; k0 += 32) {
        const int k = k0 + lane;
        const bool in = k < cnt;
        LongRes rs;
        int64_t gv = 0;
        int nch = 0, used = 0;
        if (in) {
            rs = A.res[start + k];
            gv = A.it_gv[start + k];
            nch = rs.nch > 0 ? rs.nch : 0;
            // the children's slots, then for each child of 2 .. kMaxUnit tokens the
            // 2 len - 2 slots its subtree can need (the unit kernel fills them)
            used = nch;
            for (int q = 0; q < nch; q++) {
                const int len = rs.cb[q] - rs.ca[q];
                if (len >= 2 && len <= kMaxUnit) used += 2 * len - 2;
            }
        }
        int incl = used;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const int tot = __shfl_sync(0xffffffffu, incl, 31);
        if (in) {
            if (rs.nch < 0) {   // pending root: its split key is bounded
                A.nd_child0[gv] = -1; A.nd_nchild[gv] = -1; A.nd_cost[gv] = 0;
                A.nd_U[gv] = rs.bound; A.nd_kappa[gv] = 0.f; A.nd_sel[gv] = 0;
                pend = fmaxf(pend, rs.bound);
            } else if (rs.nch == 0) {
                A.nd_child0[gv] = -1; A.nd_nchild[gv] = 0; A.nd_cost[gv] = 0;
                A.nd_U[gv] = 0.f; A.nd_kappa[gv] = 0.f; A.nd_sel[gv] = 0;
            } else {
                const int child0 = base + incl - used;   // unit-relative index
                const int cost = nch - 1;
                A.nd_child0[gv] = child0; A.nd_nchild[gv] = (int8_t)nch; A.nd_cost[gv] = (int8_t)cost;
                A.nd_U[gv] = rs.U; A.nd_kappa[gv] = rs.kap; A.nd_sel[gv] = 0;
                A.ops[atomicAdd(A.n_ops, 1u)] =
                    make_uint2(__float_as_uint(rs.kap), ((uint32_t)gv << 1) | (uint32_t)(cost - 1));
                int res = child0 + nch;
                for (int q = 0; q < nch; q++) {
                    const int64_t gc = nbase + child0 + q;
                    const int len = rs.cb[q] - rs.ca[q];
                    const bool pending = len >= 2;
                    A.nd_a[gc] = rs.ca[q]; A.nd_b[gc] = rs.cb[q];
                    A.nd_parent[gc] = (int32_t)gv; A.nd_unit[gc] = (int32_t)uid;
                    A.nd_D[gc] = rs.cD[q]; A.nd_R[gc] = rs.rch[q];
                    // a pending child of at most kMaxUnit tokens keeps its reservation in
                    // child0; the reserved slots are marked unused (child count -2) until
                    // the unit kernel fills them
                    A.nd_child0[gc] = (pending && len <= kMaxUnit) ? res : -1;
                    if (pending && len <= kMaxUnit) {
                        for (int r = res; r < res + 2 * len - 2; r++) {
                            A.nd_nchild[nbase + r] = -2; A.nd_cost[nbase + r] = 0; A.nd_sel[nbase + r] = 0;
                        }
                        res += 2 * len - 2;
                    }
                    A.nd_nchild[gc] = pending ? -1 : 0; A.nd_cost[gc] = 0;
                    A.nd_U[gc] = pending ? rs.bnd[q] : 0.f;   // a pending node's key bound
                    A.nd_kappa[gc] = 0.f; A.nd_sel[gc] = 0;
                    if (pending) pend = fmaxf(pend, rs.bnd[q]);
                }
            }
        }
        base += tot;
    }
    pend = warp_max(pend);
    if (lane == 0) {
        A.u_nnodes[uid] = base;
        A.u_pend[uid] = pend;
    }
}

// One resident wave: items are taken dynamically.
template <int DH, typename Tin, bool EG>
cudaError_t launch_eval(Ctx &c, const LongArgs &A, unsigned items, cudaStream_t s) {
    using S = LongSmem<DH, Tin>;
    static_assert(sizeof(S) <= 227 * 1024, "long-unit kernel shared memory above the per-CTA limit");
    static_assert(!EG || 2 * (sizeof(S) + 1024) <= 228 * 1024, "two CTAs per SM");
    const size_t sm = sizeof(S);
    cudaError_t e = cudaFuncSetAttribute(long_eval_kernel<DH, Tin, EG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sm);
    int occ = 1;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, long_eval_kernel<DH, Tin, EG>, kLT, sm);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::min<int64_t>((int64_t)c.num_sms * std::max(occ, 1), (int64_t)items);
    long_eval_kernel<DH, Tin, EG><<<grid, kLT, sm, s>>>(A);
    c.launches += 1;
    return cudaGetLastError();
}

template <int DH>
cudaError_t launch_eval_d(Ctx &c, const LongArgs &A, unsigned items, cudaStream_t s) {
    if (c.p.dtype != GKV_BF16) return launch_eval<DH, float, false>(c, A, items, s);
    return A.Eg ? launch_eval<DH, __nv_bfloat16, true>(c, A, items, s)
                : launch_eval<DH, __nv_bfloat16, false>(c, A, items, s);
}

__global__ void long_units_kernel(const int32_t *long_slots, int n_long, int lg0, int nlg, int J, int32_t *out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_long * nlg) return;
    const int q = k / nlg, i = k - q * nlg;
    out[k] = (lg0 + i) * J + long_slots[q];
}

}  // namespace

size_t long_res_bytes() { return sizeof(LongRes); }

cudaError_t launch_long_units(Ctx &c, const int32_t *long_slots, int n_long, int lg0, int nlg, int J,
                              int32_t *out, cudaStream_t s) {
    const int n = n_long * nlg;
    if (n <= 0) return cudaSuccess;
    long_units_kernel<<<(n + 255) / 256, 256, 0, s>>>(long_slots, n_long, lg0, nlg, J, out);
    c.launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_long_level(Ctx &c, const void *K, const void *V, const void *Q, const float *omega,
                              const int32_t *slots, int J, int fresh, int root_only, float tau,
                              const int32_t *list, int n_list, int lg0, int nlg, cudaStream_t s,
                              unsigned int *n_items_host, float tau_prune) {
    const gkv_params &p = c.p;
    Workspace &w = c.w;
    if (nlg < 0) nlg = p.L * p.G - lg0;
    const int64_t n_units = fresh ? (int64_t)n_list * nlg : (int64_t)n_list;
    if (n_items_host) *n_items_host = 0;
    if (n_units <= 0) return cudaSuccess;
    if (n_units > w.long_units_cap) return cudaErrorInvalidValue;
    LongArgs A;
    A.K = K; A.V = V; A.Q = Q;
    A.slots = slots; A.rope = w.rope; A.kappa = w.kappa;
    A.rtok = w.rtok; A.row_m = w.row_m; A.row_Z = w.row_Z; A.omega = omega;
    A.Eg = use_tc(c) ? reinterpret_cast<const float2 *>(w.Eg) : nullptr;
    A.fl_acc = p.alpha_floor > 0.0 ? w.fl_acc : nullptr;
    A.fl_f = w.fl_f;
    A.L = p.L; A.G = p.G; A.Hq = p.Hq; A.T = p.T; A.d = p.d; A.W = p.W; A.gq = p.Hq / p.G;
    A.cs = p.ctx_start; A.Nc = c.Nc; A.J = J; A.k_cand = p.k_cand;
    A.inv_sqrt_d = (float)(1.0 / sqrt((double)p.d));
    A.lamZ = (float)p.lambda_Z; A.lamM = (float)p.lambda_M; A.eps = (float)p.eps;
    A.lam_kappa = (float)p.lambda_kappa; A.base_frac = (float)p.base_frac;
    A.prune = p.lambda_Z >= 0.0 && p.lambda_M >= 0.0;
    A.fresh = fresh; A.root_only = root_only; A.tau = tau;
    A.list = list; A.n_list = n_list; A.lg0 = lg0; A.nlg = nlg;
    A.it_gv = w.long_gv; A.it_uid = w.long_uid; A.it_kin = w.long_kin; A.it_ufl = w.long_ufl;
    A.res = static_cast<LongRes *>(w.long_res);
    A.u_start = w.long_start; A.u_cnt = w.long_cnt; A.n_items = w.long_n; A.cap_items = w.long_cap;
    A.nd_a = w.nd_a; A.nd_b = w.nd_b; A.nd_child0 = w.nd_child0; A.nd_parent = w.nd_parent;
    A.nd_unit = w.nd_unit; A.nd_nchild = w.nd_nchild; A.nd_cost = w.nd_cost;
    A.nd_D = w.nd_D; A.nd_R = w.nd_R; A.nd_U = w.nd_U; A.nd_kappa = w.nd_kappa; A.nd_sel = w.nd_sel;
    A.ops = w.ops; A.n_ops = w.n_ops;
    A.u_nnodes = w.u_nnodes; A.u_Uadd = w.u_Uadd; A.u_Ddrop = w.u_Ddrop; A.u_pend = w.u_pend;
    A.u_sel = w.u_sel;
    A.status = w.dev_int + 1;
    A.work = w.work;
    A.sub = w.long_sub;
    A.it_next = w.long_n + 1 + kUnitClasses;
    cudaError_t e = cudaMemsetAsync(w.long_n, 0, (2 + kUnitClasses) * sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    long_collect_kernel<<<(unsigned)n_units, kLT, 0, s>>>(A);
    c.launches += 1;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the level's counts: long work items, small subtrees of each class
    unsigned int cnt[1 + kUnitClasses] = {0, 0, 0, 0};
    e = cudaMemcpyAsync(cnt, w.long_n, sizeof cnt, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    for (int q = 0; q <= kUnitClasses; q++) cnt[q] = (unsigned)std::min<int64_t>((int64_t)cnt[q], w.long_cap);
    if (n_items_host) *n_items_host = cnt[0] + cnt[1] + cnt[2] + cnt[3];
    if (cnt[0] > 0) {
        e = p.d == 128 ? launch_eval_d<128>(c, A, cnt[0], s) : launch_eval_d<64>(c, A, cnt[0], s);
        if (e != cudaSuccess) return e;
        long_commit_kernel<<<(unsigned)n_units, 32, 0, s>>>(A);
        c.launches += 1;
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    // nodes of at most kMaxUnit tokens: their subtrees on the unit kernel
    return launch_unit_subtrees(c, K, V, Q, omega, slots, J,
                                {w.long_sub, w.long_cap, {(int)cnt[1], (int)cnt[2], (int)cnt[3]}}, tau_prune, s);
}

}  // namespace gkv
